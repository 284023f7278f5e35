"""Work memory of batched fp32 applies on octrees: made when the operator is tuned, not by an apply, and given
back with the operator; solves of one right-hand side do not prepare for batches."""
import gc

import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _world():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import Context, DofMap, Mesh, build_library
    build_library()
    ctx = Context(0)
    dist = lambda X, Y, Z: syn.deformed_sphere_distance(X, Y, Z, 3)
    return ctx, DofMap(Mesh.octree(ctx, 10, 2, syn.refine_band_leaves(10, 2, dist, 2.0 / 40)), 2, 0)


def _reinit(ctx, m):
    from paper_2501_18781_gb300 import Operator
    op = Operator(ctx, "reinit", [m], eps=16.0, dtau=16.0 ** -3, coef_mode=1)
    op.set_field("phi", torch.tensor(np.tanh(4.0 * (m.coords()[:, 2] - 0.3)), device="cuda"))
    return op


def _free():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()   # the tensors' own cache is not the library's
    return torch.cuda.mem_get_info()[0]


def _batch(op, nrhs=8):
    u = torch.tensor(syn.uniform_pm1(11, op.n * nrhs), device="cuda").float()
    return u, torch.empty_like(u)


def test_memory_is_made_by_autotune_and_given_back():
    ctx, m = _world()
    area = 64 * m.n_dofs            # two interleaved vectors of eight right-hand sides
    assert area >= 8 << 20
    op = _reinit(ctx, m)            # loads every kernel once
    u, v = _batch(op)
    op.autotune()
    first = op.apply(u, nrhs=8)
    del op, ctx, m
    ctx, m = _world()
    before = _free()
    op = _reinit(ctx, m)
    op.autotune()
    tuned = _free()
    op.apply(u, v, nrhs=8)
    assert "interleaved8" in op.variant
    assert abs(_free() - tuned) < area // 4
    assert float((v - first).abs().max()) <= 1e-5 * float(first.abs().max())
    del op
    assert before - _free() < area // 4


def test_single_solves_prepare_nothing_for_batches():
    ctx, m = _world()
    tables = 448 * m.n_cells        # node numbers, levels and normals per leaf
    b = torch.tensor(syn.uniform_pm1(7, m.n_dofs), device="cuda")
    kw = dict(solver="defect_correction", precond="jacobi", tol=1e-8)
    used = []
    for _ in range(2):              # the first one fills the context's block pool
        op = _reinit(ctx, m)
        op.apply(b.float())
        start = _free()
        _, info = op.solve(b, **kw)
        assert info["status"] == 0
        used.append(start - _free())
        del op
    assert used[1] < tables // 2, used
