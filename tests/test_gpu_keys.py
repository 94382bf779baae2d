"""Keys of points whose floors the double-float path cannot decide: the centres of pixel
grids (of N_side a power of two every centre is a corner of order-29 pixels), the same
with a few ulp added to a coordinate, and coordinates at the ends of the exponent range.  The
divisions and roots made of integers must give the keys of the IEEE ones, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.healpix import key29, pix2vec_nest
from paper_2210_07021_gb300 import sfmm, workloads


def same_keys(x):
    x = np.ascontiguousarray(x)
    got = sfmm.keys(torch.as_tensor(x, device="cuda")).cpu().numpy().view(np.uint64)
    want = key29(x)
    bad = np.nonzero(got != want)[0]
    assert bad.size == 0, (bad.size, x[bad[:3]], got[bad[:3]], want[bad[:3]])


@pytest.mark.parametrize("nside", [1, 2, 3, 64, 100, 512])
def test_grid_centres(nside):
    same_keys(workloads.healpix_ring_centres(nside))


@pytest.mark.parametrize("order", [1, 8, 15, 22, 28])
def test_nested_centres_nudged(order):
    rng = np.random.default_rng(order)
    pix = rng.integers(0, 12 * 4 ** order, 200_000, dtype=np.int64).astype(np.uint64)
    x = pix2vec_nest(order, pix)
    same_keys(x)
    # an ulp or a few either way, one coordinate at a time
    for c in range(3):
        y = x.copy()
        y[:, c] *= 1.0 + rng.integers(-3, 4, len(y)) * 2.0 ** -52
        same_keys(y)


@pytest.mark.parametrize("tiny", [1e-320, 1e-305, 2.0 ** -301, 2.0 ** -299, 1e-60, 1e-17])
def test_exponents_at_the_range_of_the_integer_forms(tiny):
    """Coordinates on both sides of the exponents at which the FP64 routine takes over."""
    rng = np.random.default_rng(3)
    x = pix2vec_nest(6, np.arange(12 * 4 ** 6, dtype=np.uint64))
    for c in range(3):
        y = x.copy()
        y[:, c] = tiny * rng.choice([-1.0, 0.0, 1.0, 3.0], len(y))
        same_keys(y / np.linalg.norm(y, axis=1, keepdims=True))
