"""The FP64 near field's reciprocal and product logarithm: runs of equal masses and
masses that all differ, separations from coincident through 1e-150 (d^2 below the fast
path's range, still normal) to antipodal, and a non-finite mass.  With 12 boxes and a MAC that takes none of their pairs
every result is a plain sum, so the tolerance is rounding: 2^-45 of the sum of the
terms' magnitudes (the terms' own errors are a few 2^-53 each, 64 terms)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_07021_gb300 import sfmm
from conftest import unit

TOL = 2.0 ** -45


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def points():
    rng = np.random.default_rng(8)
    north = np.array([0.0, 0.0, 1.0])
    near = [np.array([d, 0.0, 1.0]) for d in (1e-150, 1e-130, 1e-20, 1e-9, 1e-4)]
    src = np.vstack([unit(rng.normal(size=(50, 3))), [north], near, [-north]])
    return src, np.vstack([src, [[3e-150, 2e-150, 1.0]], unit(rng.normal(size=(20, 3)))])


def direct(src, q, tgt):
    """psi, alpha and the sums of the terms' magnitudes, in 80-bit floats."""
    s, x, q = (a.astype(np.longdouble) for a in (src, tgt, q))
    d = x[:, None, :] - s[None]
    d2 = (d * d).sum(2)
    ok = d2 > 0
    d2 = np.where(ok, d2, 1)
    w = np.where(ok, q[None] / d2, 0)
    lg = np.where(ok, q[None] * (np.log(d2) - np.log(np.longdouble(4))), 0)
    a3 = (w[:, :, None] * d).sum(1) - x * np.where(ok, q[None], 0).sum(1)[:, None] / 2
    rho = np.hypot(x[:, 0], x[:, 1])
    cp = np.where(rho > 0, x[:, 0] / np.where(rho > 0, rho, 1), 1)
    sp = np.where(rho > 0, x[:, 1] / np.where(rho > 0, rho, 1), 0)
    al = np.stack([a3[:, 0] * x[:, 2] * cp + a3[:, 1] * x[:, 2] * sp - a3[:, 2] * rho, a3[:, 1] * cp - a3[:, 0] * sp], 1)
    mag = (np.abs(w)[:, :, None] * np.abs(d)).sum((1, 2)) + np.abs(q).sum()
    return lg.sum(1) / (4 * np.pi), al / (2 * np.pi), np.abs(lg).sum(1) + np.abs(q).sum(), mag


@pytest.mark.parametrize("masses", ["equal", "runs", "distinct"])
def test_pairs(masses):
    src, tgt = points()
    n = src.shape[0]
    q = {"equal": np.full(n, 0.7), "runs": np.repeat([1.0, 3.0, 0.25], 20)[:n],
         "distinct": np.random.default_rng(1).lognormal(0, 1, n)}[masses]
    plan = sfmm.Plan(p=8, leaf_size=64, c_s=4.0)
    psi, alpha = plan.deflection(dev(src), dev(q), dev(tgt))
    only = plan.deflection(dev(src), dev(q), dev(tgt), with_psi=False)[1]
    assert plan.stats()["n_nodes"] == 12 and plan.stats()["n_m2l"] == 0
    rp, ra, mp, ma = direct(src, q, tgt)
    assert np.all(np.abs(psi.cpu().numpy() - rp) <= TOL * mp)
    for a in (alpha, only):
        assert np.all(np.abs(a.cpu().numpy() - ra) <= TOL * ma[:, None])


def test_a_mass_that_is_not_finite_is_left_out_where_it_coincides():
    src, _ = points()
    q = np.ones(src.shape[0])
    q[3] = np.inf
    psi, alpha = sfmm.Plan(p=8, leaf_size=64, c_s=4.0).deflection(dev(src), dev(q), dev(src[3:4]))
    keep = np.arange(src.shape[0]) != 3
    rp, ra, mp, ma = direct(src[keep], q[keep], src[3:4])
    assert np.all(np.abs(psi.cpu().numpy() - rp) <= TOL * mp)
    assert np.all(np.abs(alpha.cpu().numpy() - ra) <= TOL * ma[:, None])


@pytest.mark.parametrize("what", ["deflection", "shear", "npm"])
def test_few_and_many_targets_give_the_same(what):
    """A few targets' items are each shared by a CTA's warps, many targets' are not: the
    same sums in another order (rounding, 2^-45 of the largest; mu, a reciprocal of a
    difference of these, is not a sum)."""
    rng = np.random.default_rng(3)
    src, tgt = unit(rng.normal(size=(600, 3))), unit(rng.normal(size=(160_000, 3)))
    q = dev(rng.lognormal(0, 0.5, 600))
    plan = sfmm.Plan(p=12, leaf_size=8, sigma=0.05 if what == "npm" else 0.0)
    call = (lambda t: plan.shear(dev(src), q, t, True, True)[:3]) if what == "shear" else \
        (lambda t: plan.deflection(dev(src), q, t))
    for a, b in zip(call(dev(tgt[:300])), call(dev(tgt))):
        a, b = a.cpu().numpy(), b.cpu().numpy()[:300]
        assert np.abs(a - b).max() <= TOL * np.abs(b).max()
