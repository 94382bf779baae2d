"""The evaluation's work items: leaves with any number of targets are served in
chunks of 64, or of 32 where a problem has few targets.  Every number format
against the oracle at the chunks' edges, with most targets in one leaf; the
tolerances are the formats' stated errors."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.direct import adjoint as oracle_adjoint, direct_sum
from paper_2210_07021_gb300 import sfmm
from conftest import rand_cap, unit

MODES = [(sfmm.SFMM_FP64, 1e-10), (sfmm.SFMM_MIXED, 1e-6), (sfmm.SFMM_MIXED_DF, 1e-10), (sfmm.SFMM_FP32, 3e-5)]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def sky(m, seed):
    """40 sources around the sphere and m targets of a narrow cap (one leaf), three elsewhere."""
    rng = np.random.default_rng(seed)
    src = unit(rng.normal(size=(40, 3)))
    tgt = np.vstack([rand_cap(rng, unit([0.3, 0.5, 0.2]), 1e-3, m), unit(rng.normal(size=(3, 3)))])
    return src, rng.lognormal(0, 0.5, 40), tgt


@pytest.mark.parametrize("m, leaf", [(m, 8) for m in (1, 31, 32, 33, 50, 63, 64, 65, 95, 97, 129)]
                         + [(448 + m, 64) for m in (1, 31, 32, 33, 63, 64)])
def test_chunk_edges(m, leaf):
    """Chunks of 64 (few targets per node) and of 32 (12 nodes, 32 targets or more each)."""
    src, q, tgt = sky(m, m)
    ref = direct_sum(src, q, tgt)
    for prec, tol in MODES:
        plan = sfmm.Plan(p=32, leaf_size=leaf, precision=prec)
        psi, alpha = plan.deflection(dev(src), dev(q), dev(tgt))
        e = rel(psi.cpu().numpy(), ref["psi"]), rel(alpha.cpu().numpy(), ref["alpha"])
        assert max(e) < tol, (prec, e)
        plan.close()


def test_whole_chunks_of_a_large_leaf():
    """Enough targets for chunks of 64 (the other rule), almost all of them in one leaf."""
    src, q, tgt = sky(152 * 28 * 64 + 37, 5)
    ref = direct_sum(src, q, tgt)
    for prec, tol in MODES:
        plan = sfmm.Plan(p=32, leaf_size=8, precision=prec)
        psi, alpha = plan.deflection(dev(src), dev(q), dev(tgt))
        e = rel(psi.cpu().numpy(), ref["psi"]), rel(alpha.cpu().numpy(), ref["alpha"])
        assert max(e) < tol, (prec, e)
        plan.close()


@pytest.mark.parametrize("n", [33, 97, 130])
def test_adjoint_with_many_sources_in_one_leaf(n):
    """The adjoint evaluates at the forward sources: here n of them in one leaf."""
    tgt, _, src = sky(n, 70 + n)
    rng = np.random.default_rng(n)
    q, g = rng.lognormal(0, 0.5, src.shape[0]), rng.normal(size=(tgt.shape[0], 2))
    rq, rs = oracle_adjoint(src, q, tgt, g, None)
    for prec in (sfmm.SFMM_FP64, sfmm.SFMM_MIXED_DF):
        plan = sfmm.Plan(p=32, leaf_size=8, precision=prec)
        gq, gs = plan.adjoint(dev(src), dev(q), dev(tgt), g_alpha=dev(g))
        e = rel(gq.cpu().numpy(), rq), rel(gs.cpu().numpy(), rs)
        assert max(e) < 1e-10, (prec, e)
        plan.close()
