"""FP64: a target on a mass that outweighs all others near it.  The mass does not act on
the target, so neither may its rounding: the tolerance, 2^-45, is of the other masses'
terms alone.  12 boxes and a MAC that takes none of their pairs, so every result is a
plain sum (test_gpu_fp64_near.py); few targets take the kernel that shares an item between
warps, many the other one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_07021_gb300 import sfmm
from conftest import unit

TOL = 2.0 ** -45


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def sky(heavy):
    """Sources of masses about 1, `heavy` ones at every eighth of their places (a list:
    all at one place)."""
    rng = np.random.default_rng(5)
    base = unit(rng.normal(size=(64, 3)))
    q = rng.lognormal(0, 0.5, 64)
    at = base[::8].repeat(len(heavy), 0)
    return np.vstack([base, at]), np.concatenate([q, np.tile(heavy, 8)]), base[::8]


def psi_of_the_others(src, q, x):
    d2 = ((x[:, None] - src[None]).astype(np.longdouble) ** 2).sum(2)
    ok = d2 > 0
    t = np.where(ok, q[None] * (np.log(np.where(ok, d2, 1)) - np.log(np.longdouble(4))), 0) / (4 * np.pi)
    return t.sum(1), np.abs(t).sum(1) + np.abs(np.where(ok, q[None], 0)).sum(1)


@pytest.mark.parametrize("n_tgt", [8, 160_000])
@pytest.mark.parametrize("heavy", [[1e5], [1e8], [1e16], [1e12, -1e12], [1.0, 0.25]])
def test_a_heavy_mass_at_the_target(heavy, n_tgt):
    src, q, x = sky(heavy)
    x = np.tile(x, (n_tgt // 8, 1))
    plan = sfmm.Plan(p=8, leaf_size=256, c_s=4.0)
    for i in range(8):                     # one heavy place at a time
        m = q.copy()
        m[64:] = np.where(np.arange(len(q) - 64) // len(heavy) == i, m[64:], 0.0)
        psi = plan.deflection(dev(src), dev(m), dev(x))[0]
        assert plan.stats()["n_m2l"] == 0
        ref, mag = psi_of_the_others(src, m, x[i:i + 1])
        got = psi.cpu().numpy()[i::8]
        assert np.all(np.abs(got - ref) <= TOL * mag), np.abs(got - ref).max() / mag


def test_a_lone_mass_does_not_act_on_itself():
    x = dev(np.array([[0.6, 0.0, 0.8]]))
    psi, alpha = sfmm.Plan(p=8).deflection(x, dev(np.array([0.7])), x)
    assert psi.item() == 0.0 and torch.equal(alpha, torch.zeros_like(alpha))


@pytest.mark.parametrize("heavy", [[1e8], [1e16], [1e12, -1e12]])
def test_the_adjoint_of_a_heavy_charge(heavy):
    tgt, h, x = sky(heavy)                 # forward targets, whose charges act on the sources x
    plan = sfmm.Plan(p=8, leaf_size=256, c_s=4.0)
    for i in range(8):
        c = h.copy()
        c[64:] = np.where(np.arange(len(h) - 64) // len(heavy) == i, c[64:], 0.0)
        g_q = plan.adjoint(dev(x), dev(np.ones(8)), dev(tgt), g_psi=dev(c))[0]
        ref, mag = psi_of_the_others(tgt, c, x[i:i + 1])
        assert abs(g_q.cpu().numpy()[i] - ref) <= TOL * mag
