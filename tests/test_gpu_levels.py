"""The up- and down-pass on both sides of the lines between their kernels: narrow
levels (a warp per translation), wide ones (a thread per translation); the FP64 P2M
of small and of large trees; the FP64 M2L of lists within one warp's 32 pairs, over
two and over several, and of antipodal boxes.  The double-float and the FP64 paths
share no translation kernel, so each is the other's reference: the double-float
expansions carry 48 bits, and 1e-11 of the largest scaled coefficient is the
tolerance their equality is held to elsewhere."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_07021_gb300 import sfmm, workloads
from conftest import unit


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def scaled(plan, which, p):
    e = plan.debug(which, np.float64, 2 * p + 2)
    r = plan.debug(sfmm.ARR_NODE_GEOM, np.float64, 11)[:, 10]
    s = r[:, None] ** (np.arange(1, p + 1) * (1 if which == sfmm.ARR_LOCAL else -1.0))
    return e[:, :2], (e[:, 2::2] + 1j * e[:, 3::2]) * s


@pytest.mark.parametrize("n, m, p", [(300, 4, 1), (3000, 16, 2), (3000, 16, 20), (60_000, 4, 7), (60_000, 4, 20),
                                     (60_000, 4, 28), (30_000, 4, 32)])
def test_double_float_and_fp64_expansions_agree(n, m, p):
    rng = np.random.default_rng(n + p)
    src = np.vstack([unit(rng.normal(size=(n - n // 4, 3))), workloads.clustered(rng, n // 4, 5)])
    q, tgt = rng.lognormal(0, 0.5, n), unit(rng.normal(size=(n // 3, 3)))
    pd = sfmm.Plan(p=p, leaf_size=m)
    pm = sfmm.Plan(p=p, leaf_size=m, precision=sfmm.SFMM_MIXED_DF)
    pd.potential(dev(src), dev(q), dev(tgt))
    pm.potential(dev(src), dev(q), dev(tgt))
    lvl, lists = pd.debug(sfmm.ARR_NODE_LEVEL, np.int32), pd.debug(sfmm.ARR_M2L, np.int32, 2)[:, 1]
    if n == 60_000:
        assert np.bincount(lvl).max() > 4096 > np.bincount(lvl)[3]
    if n >= 3000:           # over several warps' pairs (a warp takes 16 of up to 19,456 pairs, else 32)
        assert np.bincount(lists).max() > (32 if lists.size <= 19456 else 64)
    for which in (sfmm.ARR_MULTIPOLE, sfmm.ARR_LOCAL):
        for a, b in zip(scaled(pd, which, p), scaled(pm, which, p)):
            assert np.abs(a - b).max() < 1e-11 * np.abs(a).max()
    local = pd.debug(sfmm.ARR_LOCAL, np.float64)
    pd.potential(dev(src), dev(q), dev(tgt))
    assert np.array_equal(local, pd.debug(sfmm.ARR_LOCAL, np.float64))      # sums in the list's order
