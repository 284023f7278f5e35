"""fp32 inner products: pairs of floats within a thread, fp64 across threads.  For vectors that one block of
threads holds (one 16-byte word each, n <= 1024) the thread's sum of four exact products is rounded twice
in fp64, and the block's tree of 8 + 5 additions and the sum over one block add at most 13 more roundings
of which those with zeros are exact: for n = 128 five remain.  So |dot - exact| <= 7 x 2^-53 sum |x y|.
Sums of products below the largest double stay finite although they exceed the largest float."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import Context, build_library
    build_library()
    return Context(0)


def _dot(ctx, x, y):
    return float(ctx.dot(torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda"))[0])


@pytest.mark.parametrize("seed", range(8))
def test_sum_over_a_warp_in_fp64(ctx, seed):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1, 1, 128).astype(np.float32)
    y = rng.uniform(-1, 1, 128).astype(np.float32)
    for a, b in ((x, x), (x, y)):
        p = a.astype(np.float64) * b.astype(np.float64)   # exact
        assert abs(_dot(ctx, a, b) - math.fsum(p)) <= 7 * 2.0 ** -53 * np.abs(p).sum()


@pytest.mark.parametrize("n", [4096, 70001, 1600000])
@pytest.mark.parametrize("value", [5e18, 1.5e19])
def test_sums_beyond_the_fp32_range(ctx, n, value):
    # one or two elements per accumulator at the smaller sizes, up to three at the largest: a thread's own sums
    # stay below 3.4e38, the sum over a warp does not
    x = np.full(n, value, np.float32)
    if n > 600000:
        x /= 2
    exact = n * float(x[0]) ** 2
    assert abs(_dot(ctx, x, x) - exact) <= 1e-13 * exact
