"""The tree and the lists where their construction changes hands: runs of narrow
levels by one CTA, wide levels by the whole GPU and narrow ones again, a depth limit
inside each, and the bounded waits of the leaf collection and of the walk (with a
limit of one poll tiles form the sums before them themselves: same lists)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle.healpix as hp
from oracle.tree import build_tree
from paper_2210_07021_gb300 import sfmm, workloads


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def sky(n, seed):
    rng = np.random.default_rng(seed)
    clumps = workloads.clump_set(rng, 12)
    return workloads.clustered(rng, n, 12, clumps=clumps), workloads.clustered(rng, n // 3, 12, clumps=clumps)


@pytest.mark.parametrize("n, m, depth", [(30, 64, 29), (5000, 1, 29), (40_000, 2, 29), (40_000, 2, 6), (40_000, 2, 3),
                                         (40_000, 2, 0)])
def test_tree(n, m, depth):
    src, tgt = sky(n, 3)
    keys = np.sort(hp.key29(src).astype(np.uint64))
    t = build_tree(keys, m, depth)
    if (n, depth) == (40_000, 29):
        assert np.bincount(t["level"]).max() > 4096 > np.bincount(t["level"])[-1]       # both kinds of level
    plan = sfmm.Plan(max_depth=depth, p=4, leaf_size=m)
    for _ in range(2):                       # with node arrays that have to grow, and grown ones
        plan.potential(dev(src), dev(np.ones(n)), dev(tgt))
        assert np.array_equal(plan.debug(sfmm.ARR_NODE_PREFIX, np.uint64), t["prefix"])
        assert np.array_equal(plan.debug(sfmm.ARR_NODE_LEVEL, np.int32), t["level"])
        rng = plan.debug(sfmm.ARR_NODE_RANGE, np.int32, 2)
        assert np.array_equal(rng[:, 0], t["first"]) and np.array_equal(rng[:, 1], t["count"])
        assert np.array_equal(plan.debug(sfmm.ARR_NODE_CHILD0, np.int32), t["child0"])
        assert np.array_equal(plan.debug(sfmm.ARR_NODE_PARENT, np.int32), t["parent"])
        st = plan.stats()
        assert st["n_nodes"] == len(t["level"]) and st["n_leaves"] == np.sum((t["child0"] < 0) & (t["count"] > 0))


def test_lists_and_results_with_waits_that_run_out():
    src, tgt = sky(30_000, 5)
    q = dev(np.ones(30_000))
    got = []
    for limit in (0, 1):
        plan = sfmm.Plan(p=16, leaf_size=8, wait_limit=limit)
        psi, alpha = plan.deflection(dev(src), q, dev(tgt))
        got.append([plan.debug(sfmm.ARR_M2L, np.int32), plan.debug(sfmm.ARR_P2P, np.int32), psi.cpu().numpy(),
                    alpha.cpu().numpy(), plan.stats()["n_leaves"]])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
