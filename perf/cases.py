"""The work that users of this package have it do, as cases that can be timed and compared.

Every case goes through the package's public entry points (the plan of `sfmm.Plan`,
`autograd.deflection`, `sfmm.sort_keys_static`) on inputs drawn on the GPU from a seed.
The kinds of case:

deflect   potential and deflection of N masses at M targets, device arrays in and out
host      the same from pinned host arrays, results read back to the host
grad      one training step of the gradient workload: forward, loss, dL/dq and dL/dy
shells    independent lensing shells of very different sizes, solved as one batch
sort      order-29 keys and stable sort without any device allocation

Settings (p, leaf size, MAC constants) are those of the benchmark's paths; skies are the
random, uniform and clustered ones of the tests and the benchmark.
"""
import math

import numpy as np
import torch

from paper_2210_07021_gb300 import autograd, sfmm, workloads

DEV = "cuda"
ARCMIN = math.pi / (180.0 * 60.0)

# the number formats with the order, leaf size and MAC constants they are run with:
# `default` is Plan() as it comes (FP64, order from the tolerance), the others the settings
# of the benchmark (the 1e-6, 1e-10, FP64 and all-FP32 paths) and of its gradient workload
PATHS = {
    "default": dict(precision=sfmm.SFMM_FP64, p=0, tol=1e-10, leaf_size=32, c_s=2.0, c_t=0.5),
    "fp64": dict(precision=sfmm.SFMM_FP64, p=32, leaf_size=32, c_s=1.5, c_t=0.45),
    "mixed": dict(precision=sfmm.SFMM_MIXED, p=20, leaf_size=96, c_s=1.5, c_t=0.5),
    "mixed_df": dict(precision=sfmm.SFMM_MIXED_DF, p=28, leaf_size=64, c_s=1.6, c_t=0.45),
    "fp32": dict(precision=sfmm.SFMM_FP32, p=20, leaf_size=64, c_s=1.3, c_t=0.5),
    "grad": dict(precision=sfmm.SFMM_MIXED_DF, p=28, leaf_size=64, c_s=2.0, c_t=0.45),
}


def listed():
    return [
        # a plugin that may not allocate sorts its particles: the largest size the entry point takes
        dict(name="sort_262144", kind="sort", n=262_144),
        # the smallest solve: the tests' random sky at its own points, the plan as it comes
        dict(name="random_4096_default", kind="deflect", path="default", sky="random", n=4096, m=0, psi=True,
             q32=False),
        # the smallest lensing shell (deflection only), on a coarse pixel grid
        dict(name="shell_10000_grid64", kind="deflect", path="mixed", sky="clustered", n=10_000, nside=64, psi=False,
             q32=False),
        # a uniform sky of unequal masses at its own points, odd size, 1e-10
        dict(name="uniform_100003_df", kind="deflect", path="mixed_df", sky="random", n=100_003, m=0, psi=True,
             q32=False),
        # the clustered sky of one million masses on the N_side 512 pixel grid, 1e-6
        dict(name="clustered_1e6_grid512", kind="deflect", path="mixed", sky="clustered", n=1_000_000, nside=512,
             psi=True, q32=False),
        # the benchmark's sky: N = M = 1.6e7, float32 masses, the 1e-6 path
        dict(name="pair_16e6_mixed", kind="deflect", path="mixed", sky="pair", n=16_000_000, m=16_000_000, psi=True,
             q32=True),
        # the same sky at 1e-10
        dict(name="pair_16e6_df", kind="deflect", path="mixed_df", sky="pair", n=16_000_000, m=16_000_000, psi=True,
             q32=True),
        # a quarter of it on the all-FP32 path (M2L on the tensor cores)
        dict(name="pair_4e6_fp32", kind="deflect", path="fp32", sky="pair", n=4_000_000, m=4_000_000, psi=True,
             q32=True),
        # float64 throughout at a million points
        dict(name="pair_1e6_fp64", kind="deflect", path="fp64", sky="pair", n=1_000_000, m=1_000_000, psi=True,
             q32=True),
        # one training step of the gradient workload (1e-10 forward, adjoint backward)
        dict(name="grad_1e6_grid256", kind="grad", path="grad", n=1_000_000, nside=256),
        # sixteen lensing shells of 1e4 to 2e6 masses, deflection at the N_side 128 pixel centres
        dict(name="shells_16", kind="shells", path="mixed", shells=16, n_min=10_000, n_max=2_000_000, nside=128),
        # the headline call end to end: host arrays in, host arrays out
        dict(name="host_4e6_mixed", kind="host", path="mixed", n=4_000_000, m=4_000_000),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sort", "random", "grid", "grid", "pair", "pair", "pair", "grad", "shells", "host"])
    if kind == "sort":
        return dict(kind="sort", n=_logint(rng, 1000, 262_144))
    if kind == "random":
        path = rng.choice(["default", "mixed", "mixed_df"])
        return dict(kind="deflect", path=path, sky="random", n=_logint(rng, 2000, 150_000), m=0,
                    psi=rng.random() < 0.7, q32=rng.random() < 0.3)
    if kind == "grid":
        path = rng.choice(["mixed", "mixed", "mixed_df", "fp64"])
        top = 1_000_000 if path != "fp64" else 300_000
        return dict(kind="deflect", path=path, sky="clustered", n=_logint(rng, 10_000, top),
                    nside=rng.randrange(24, 400 if path != "fp64" else 160), psi=rng.random() < 0.5,
                    q32=rng.random() < 0.5)
    if kind == "pair":
        path = rng.choice(["mixed", "mixed_df", "fp32", "fp64"])
        top = {"mixed": 12_000_000, "mixed_df": 8_000_000, "fp32": 4_000_000, "fp64": 800_000}[path]
        return dict(kind="deflect", path=path, sky="pair", n=_logint(rng, 50_000, top), m=_logint(rng, 50_000, top),
                    psi=rng.random() < 0.7, q32=rng.random() < 0.6)
    if kind == "grad":
        return dict(kind="grad", path="grad", n=_logint(rng, 10_000, 1_000_000), nside=rng.randrange(24, 256))
    if kind == "shells":
        return dict(kind="shells", path="mixed", shells=rng.randrange(4, 17), n_min=_logint(rng, 5_000, 20_000),
                    n_max=_logint(rng, 100_000, 2_000_000), nside=rng.randrange(32, 128))
    return dict(kind="host", path="mixed", n=_logint(rng, 50_000, 4_000_000), m=_logint(rng, 50_000, 4_000_000))


# --------------------------------------------------------------------- inputs
def _gen(seed, stream=0):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1009 + stream) & 0x7FFFFFFFFFFF)


def _unit(v):
    return v / torch.linalg.norm(v, dim=1, keepdim=True)


def _uniform(g, n):
    return _unit(torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64))


def _nfw_table():
    """x and enclosed-mass CDF of the projected NFW profile truncated at 20 scale radii."""
    x = np.geomspace(1e-6, 20.0, 8001)
    f = np.where(x < 1, np.arccosh(np.maximum(1 / x, 1)), np.arccos(np.minimum(1 / x, 1))) / np.sqrt(np.abs(1 - x * x))
    c = np.maximum.accumulate(np.maximum(np.log(x / 2) + f, 0.0))
    return x, c / c[-1]


def _interp(u, xp, fp):
    k = torch.searchsorted(xp, u).clamp(1, xp.numel() - 1)
    x0, x1, f0, f1 = xp[k - 1], xp[k], fp[k - 1], fp[k]
    return f0 + (f1 - f0) * ((u - x0) / (x1 - x0).clamp_min(1e-300)).clamp(0, 1)


def _clumps(g, n):
    rs = torch.exp(torch.empty(n, device=DEV, dtype=torch.float64).uniform_(math.log(0.1), math.log(2.0), generator=g))
    return _uniform(g, n), rs * ARCMIN


def _clustered(g, n, clumps):
    """70 % of the points in NFW clumps, the rest uniform, in random order."""
    centres, rs = clumps
    n_cl = int(round(0.7 * n))
    which = torch.randint(0, centres.shape[0], (n_cl,), generator=g, device=DEV)
    xs, cdf = (torch.as_tensor(t, device=DEV) for t in _nfw_table())
    th = _interp(torch.rand(n_cl, generator=g, device=DEV, dtype=torch.float64), cdf, xs) * rs[which]
    ph = 2 * math.pi * torch.rand(n_cl, generator=g, device=DEV, dtype=torch.float64)
    c = centres[which]
    a = torch.zeros_like(c)
    a[:, 2] = (c[:, 2].abs() < 0.9).double()
    a[:, 0] = 1.0 - a[:, 2]
    e1 = _unit(torch.linalg.cross(c, a))
    e2 = torch.linalg.cross(c, e1)
    y = torch.cos(th)[:, None] * c + torch.sin(th)[:, None] * (torch.cos(ph)[:, None] * e1 + torch.sin(ph)[:, None] * e2)
    pts = torch.cat([_unit(y), _uniform(g, n - n_cl)])
    return pts[torch.randperm(n, generator=g, device=DEV)].contiguous()


def _grid(nside):
    return torch.as_tensor(workloads.healpix_ring_centres(nside), device=DEV)


def _inputs(case, seed):
    """(src, q, tgt) of a deflect, host or grad case."""
    n, sky = case["n"], case.get("sky", "pair" if "m" in case else "clustered")
    q32 = case.get("q32", case["kind"] == "host")
    g = _gen(seed)
    if sky == "random":              # lognormal masses at their own points
        src = _uniform(g, n)
        q = torch.exp(0.5 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
        tgt = src
    else:                            # equal masses on a clustered sky
        clumps = _clumps(_gen(seed, 1), max(1, n // 800 if sky == "pair" else n // 500))
        src = _clustered(g, n, clumps)
        q = torch.full((n,), 4 * math.pi / n, device=DEV, dtype=torch.float64)
        tgt = _clustered(_gen(seed, 2), case["m"], clumps) if sky == "pair" else _grid(case["nside"])
    return src, q.float() if q32 else q, tgt


def _shell_sizes(case):
    return [int(v) for v in np.geomspace(case["n_min"], case["n_max"], case["shells"])]


def _shells(case, seed):
    tgt = _grid(case["nside"])
    out = []
    for k, n in enumerate(_shell_sizes(case)):
        src = _clustered(_gen(seed, 10 + 2 * k), n, _clumps(_gen(seed, 11 + 2 * k), max(1, n // 500)))
        out.append((src, torch.full((n,), 4 * math.pi / n, device=DEV, dtype=torch.float64), tgt))
    return out


def _pinned(t):
    return t.cpu().pin_memory().numpy()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sort":
        return dict(kind=kind, xyz=_uniform(_gen(seed), case["n"]))
    path = PATHS[case["path"]]
    if kind == "shells":
        return dict(kind=kind, shells=_shells(case, seed), plan=sfmm.Plan(**path))
    src, q, tgt = _inputs(case, seed)
    n, m = src.shape[0], tgt.shape[0]
    plan = sfmm.Plan(q_f32=q.dtype == torch.float32, n_max=max(n, m) if kind == "grad" else n,
                     m_max=max(n, m) if kind == "grad" else m, **path)
    if kind == "host":
        hs, hq, ht = _pinned(src), _pinned(q), _pinned(tgt)
        psi = torch.empty(m, dtype=torch.float64, pin_memory=True).numpy()
        alpha = torch.empty((m, 2), dtype=torch.float64, pin_memory=True).numpy()
        return dict(kind=kind, plan=plan, src=hs, q=hq, tgt=ht, psi=psi, alpha=alpha)
    st = dict(kind=kind, plan=plan, src=src, q=q, tgt=tgt, with_psi=case.get("psi", True))
    if kind == "grad":               # weights and reference deflections of the loss
        g = _gen(seed, 3)
        st["w"] = 0.5 + torch.rand((m, 1), generator=g, device=DEV, dtype=torch.float64)
        st["ref"] = 0.3 * torch.randn((m, 2), generator=g, device=DEV, dtype=torch.float64)
        src.requires_grad_()
        q.requires_grad_()
    return st


def run(state):
    kind = state["kind"]
    if kind == "sort":
        return sfmm.sort_keys_static(state["xyz"])
    plan = state["plan"]
    if kind == "shells":
        return [alpha for _, alpha in plan.deflection_batch(state["shells"], with_psi=False, lanes=4)]
    src, q, tgt = state["src"], state["q"], state["tgt"]
    if kind == "host":
        return plan.deflection_host(src, q, tgt, psi=state["psi"], alpha=state["alpha"])
    if kind == "grad":
        psi, alpha = autograd.deflection(src, q, tgt, plan)
        loss = (state["w"] * (alpha - state["ref"]) ** 2).sum()
        g_src, g_q = torch.autograd.grad(loss, (src, q))
        return psi.detach(), alpha.detach(), g_src, g_q
    return plan.deflection(src, q, tgt, with_psi=state["with_psi"])


# ------------------------------------------------------------ what a pass needs
def work(case):
    """Bytes: every input read once, every output written once.  Operations: the
    expansions formed and evaluated once per point (8 p each) and 14 operations
    per near pair, a target meeting about 9 leaves of half the leaf size."""
    kind = case["kind"]
    if kind == "sort":
        return dict(bytes=case["n"] * (24 + 8 + 4), flops=0)
    path = PATHS[case["path"]]
    per_point = 8 * (path["p"] or 32)
    near = 14 * 9 * path["leaf_size"] // 2

    def solve(n, m, q_bytes, out):
        return n * (24 + q_bytes) + m * (24 + out), n * per_point + m * (per_point + near)

    if kind == "shells":
        m = 12 * case["nside"] ** 2
        parts = [solve(n, m, 8, 16) for n in _shell_sizes(case)]
        return dict(bytes=sum(b for b, _ in parts), flops=sum(f for _, f in parts))
    n = case["n"]
    m = 12 * case["nside"] ** 2 if "nside" in case else case["m"] or n
    psi = case.get("psi", True)
    b, f = solve(n, m, 4 if case.get("q32", kind == "host") else 8, 24 if psi else 16)
    if kind == "grad":
        b2, f2 = solve(m, n, 16, 32)
        b, f = b + b2, f + f2
    return dict(bytes=b, flops=f)


# ------------------------------------------------------- the same in 64 bits
def _basis(x):
    rho = torch.sqrt(x[:, 0] ** 2 + x[:, 1] ** 2)
    safe = rho.clamp_min(1e-300)
    cp = torch.where(rho > 0, x[:, 0] / safe, torch.ones_like(rho))
    sp = torch.where(rho > 0, x[:, 1] / safe, torch.zeros_like(rho))
    et = torch.stack([x[:, 2] * cp, x[:, 2] * sp, -rho], 1)
    return et, torch.stack([-sp, cp, torch.zeros_like(rho)], 1)


def _direct(src, q, tgt, dip=None):
    """sum_j q_j G(x_i, y_j) (+ the dipoles' g_j . grad_y G) and its covariant gradient in x, as 3-vectors."""
    m, n = tgt.shape[0], src.shape[0]
    psi = torch.empty(m, dtype=torch.float64, device=DEV)
    grad = torch.empty((m, 3), dtype=torch.float64, device=DEV)
    step = max(1, 200_000_000 // n)
    for a in range(0, m, step):
        x = tgt[a:a + step]
        d = [x[:, k:k + 1] - src[None, :, k] for k in range(3)]
        d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        far = d2 > 0
        d2 = torch.where(far, d2, torch.ones_like(d2))
        w = torch.where(far, q[None, :] / d2, torch.zeros_like(d2))
        qs = torch.where(far, q[None, :].expand_as(d2), torch.zeros_like(d2))
        p = (qs * (torch.log(d2) - math.log(4.0))).sum(1) / (4 * math.pi)
        s = torch.stack([(w * d[k]).sum(1) for k in range(3)], 1) - 0.5 * x * qs.sum(1, keepdim=True)
        if dip is not None:
            gd = -(dip[None, :, 0] * d[0] + dip[None, :, 1] * d[1] + dip[None, :, 2] * d[2]) / d2
            gd = torch.where(far, gd, torch.zeros_like(gd))
            p += gd.sum(1) / (2 * math.pi)
            inv = torch.where(far, 1.0 / d2, torch.zeros_like(d2))
            s += torch.stack([(-2.0 * gd * inv * d[k]).sum(1) - inv @ dip[:, k] for k in range(3)], 1)
        s -= (s * x).sum(1, keepdim=True) * x      # tangent to the sphere at x
        psi[a:a + step] = p
        grad[a:a + step] = s / (2 * math.pi)
    return psi, grad


def _alpha(tgt, grad):
    et, ep = _basis(tgt)
    return torch.stack([(grad * et).sum(1), (grad * ep).sum(1)], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sort", "shells"):      # whole numbers; too many shells to sum directly
        return None
    n = case["n"]
    m = 12 * case["nside"] ** 2 if "nside" in case else case["m"] or n
    if n * m > 1.2e10 or (kind == "grad" and n * m > 4e9):
        return None
    src, q, tgt = _inputs(case, seed)
    q = q.double()
    psi, grad = _direct(src, q, tgt)
    alpha = _alpha(tgt, grad)
    if kind == "grad":
        g = _gen(seed, 3)
        w = 0.5 + torch.rand((m, 1), generator=g, device=DEV, dtype=torch.float64)
        ref = 0.3 * torch.randn((m, 2), generator=g, device=DEV, dtype=torch.float64)
        ga = 2.0 * w * (alpha - ref)
        et, ep = _basis(tgt)
        dip = ga[:, :1] * et + ga[:, 1:] * ep
        g_q, g_y = _direct(tgt, torch.zeros(m, dtype=torch.float64, device=DEV), src, dip)
        return psi, alpha, q[:, None] * g_y, g_q
    return (psi if case.get("psi", True) else None), alpha
