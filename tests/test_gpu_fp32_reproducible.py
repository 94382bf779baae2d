"""The all-FP32 path gives the same bits every time: the translations of a box's list are
added up in an order that does not depend on which tile of the tensor-core M2L ends first,
nor on the order in which pairs near antipodes were listed (c_s = 4: several of a box)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2210_07021_gb300 import sfmm, workloads


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n,leaf,c_s,p", [(400_000, 16, 1.3, 20), (60_001, 8, 4.0, 12), (60_001, 8, 4.0, 32)])
def test_same_bits_every_time(n, leaf, c_s, p):
    rng = np.random.default_rng(n + p)
    src = workloads.clustered(rng, n, 60)
    args = dev(src), dev(rng.lognormal(0, 0.5, n)), dev(workloads.clustered(rng, n, 60))
    plan = sfmm.Plan(p=p, leaf_size=leaf, c_s=c_s, precision=sfmm.SFMM_FP32)
    first = [t.clone() for t in plan.deflection(*args)]
    for _ in range(7):
        for a, b in zip(first, plan.deflection(*args)):
            assert torch.equal(a, b)
