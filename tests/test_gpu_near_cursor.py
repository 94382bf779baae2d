"""The FP64 near field's walk through the near leaves as one list: leaves of none, one and
a few sources, fewer than the lanes of a target, for target groups of every size and for
few items (four warps share one) and many.  Twelve boxes and a MAC that takes none of
their pairs: every result is a plain sum, so the tolerance is rounding, 2^-45 of the sum
of the terms' magnitudes (the terms' own errors are a few 2^-53 each, 40 terms at most)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_07021_gb300 import sfmm
from conftest import unit
from test_gpu_fp64_near import TOL, dev, direct


@pytest.mark.parametrize("copies", [1, 9000])
@pytest.mark.parametrize("n,m", [(1, 1), (2, 3), (13, 47), (40, 75)])
def test_leaves_of_few_sources(n, m, copies):
    rng = np.random.default_rng(100 * n + m)
    src, tgt = unit(rng.normal(size=(n, 3))), unit(rng.normal(size=(m, 3)))
    tgt[:1] = src[:1]                                   # a coincident pair
    q = rng.lognormal(0, 1, n)
    plan = sfmm.Plan(p=8, leaf_size=64, c_s=4.0)
    psi, alpha = plan.deflection(dev(src), dev(q), dev(np.tile(tgt, (copies, 1))))
    assert plan.stats()["n_nodes"] == 12 and plan.stats()["n_m2l"] == 0
    rp, ra, mp, ma = direct(src, q, tgt)
    psi, alpha = psi.cpu().numpy().reshape(copies, m), alpha.cpu().numpy().reshape(copies, m, 2)
    assert np.all(np.abs(psi - rp) <= TOL * mp)
    assert np.all(np.abs(alpha - ra) <= TOL * ma[:, None])
