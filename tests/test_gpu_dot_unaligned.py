"""Inner products of vectors that do not start on 16-byte boundaries, and of batches with an odd stride: sizes
around the eight (fp32) or four (fp64) elements that a thread has in flight and the 155,648 threads of the
grid.  fp32 carries pairs of floats (48 bits) over at most 30 additions per thread: 2^-42 of sum |x y|; fp64
rounds each of at most 32 additions per thread and 30 across them: 2^-46."""
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


@pytest.mark.parametrize("n", [1, 2, 3, 5, 257, 4097, 155647, 155649, 1245185, 1400001])
@pytest.mark.parametrize("dtype,bound", [(np.float32, 2.0 ** -42), (np.float64, 2.0 ** -46)])
def test_unaligned_and_odd_strides(ctx, n, dtype, bound):
    rng = np.random.default_rng(n)
    x, y = (rng.uniform(-1, 1, 2 * n + 1).astype(dtype) for _ in range(2))
    X, Y = (torch.tensor(a, device="cuda") for a in (x, y))
    one = float(ctx.dot(X[1:n + 1], Y[1:n + 1])[0])
    two = ctx.dot(X[:2 * n], Y[:2 * n], nvec=2).cpu().numpy()
    for got, a, b in ((one, 1, n + 1), (two[0], 0, n), (two[1], n, 2 * n)):
        p = x[a:b].astype(np.longdouble) * y[a:b].astype(np.longdouble)
        exact = float(p.sum())
        assert abs(got - exact) <= bound * float(np.abs(p).sum()) + 1e-300, (got, exact)
