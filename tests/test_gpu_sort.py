"""The radix sort at the edges of its tiles (1024, 2048 and 4096 keys by size) and of
the sizes at which its method changes, and the look-back's bounded wait: with a limit of one poll tiles give up waiting and count the keys
before them instead, which must not change the result.  Keys and permutation are
compared with the oracle's keys and a stable argsort, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.healpix import key29
from paper_2210_07021_gb300 import sfmm, workloads


@pytest.mark.parametrize("n, wait_limit", [(n, w) for w in (0, 1) for n in (2, 1023, 1024, 1025, 4097, 150_000, 150_001,
                                                                           500_001)] + [(1_999_999, 0), (2_000_001, 0)])
def test_sorted_sources(n, wait_limit):
    rng = np.random.default_rng(n)
    src = workloads.clustered(rng, n, max(8, n // 500))
    src[n // 2:] = src[:n - n // 2]              # every key twice: equal keys keep their input order
    k = key29(src).astype(np.uint64)
    order = np.argsort(k, kind="stable")
    plan = sfmm.Plan(p=4, leaf_size=64, wait_limit=wait_limit)
    x = torch.as_tensor(src, device="cuda")
    plan.potential(x, torch.ones(n, dtype=torch.float64, device="cuda"), x[:10].clone())
    assert np.array_equal(plan.debug(sfmm.ARR_SRC_KEYS, np.uint64), k[order])
    assert np.array_equal(plan.debug(sfmm.ARR_SRC_PERM, np.uint32), order.astype(np.uint32))
