"""fp32 applies under a caller's stream capture where their own tables are not built yet (an fp64 apply has built the
Gauss-point tables): nothing can be allocated, so the general kernels serve, and the replayed graph gives the
fp32 result (2e-5, Oseen 5e-5 of each block's largest entry, as the kernels it stands in for)."""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cuda(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def _operator(ctx, name):
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    if name == "reinit_octree":
        dist = lambda X, Y, Z: syn.deformed_sphere_distance(X, Y, Z, 3)
        m = DofMap(Mesh.octree(ctx, 4, 2, syn.refine_band_leaves(4, 2, dist, 1.0 / 64)), 2, 0)
        op = Operator(ctx, "reinit", [m], eps=16.0, dtau=16.0 ** -3, coef_mode=1)
        op.set_field("phi", _cuda(np.tanh(4.0 * (m.coords()[:, 2] - 0.3))))
        return op, [(0, op.n)], 3
    mesh = Mesh.uniform(ctx, [10, 7, 5], (0.0,) * 3, (10 / 8, 7 / 8, 5 / 8))
    if name.startswith("oseen"):
        mu, mp = DofMap(mesh, 2, 0b011111), DofMap(mesh, 1, 0)
        op = Operator(ctx, "oseen", [mu, mp], sigma=16.0, rho_l=40.0, rho_g=0.4, mu_l=3.0, mu_g=0.03, rho_s=40.0,
                      mu_s=3.0, t_solidus=1900.0, t_liquidus=2200.0, darcy_c=1e3, darcy_b=1.0,
                      oseen_flags=7 if name == "oseen_meltpool" else 0)
        op.set_field("phi", _cuda(np.tanh(4.0 * (mu.coords()[:, 2] - 0.3))))
        op.set_field("beta", _cuda(syn.uniform_pm1(5, 3 * mu.n_dofs)))
        op.set_field("t_prev", _cuda(2000.0 + 400.0 * syn.uniform_pm1(7, mu.n_dofs)))
        return op, [(0, 3 * mu.n_dofs), (3 * mu.n_dofs, op.n)], 1
    m = DofMap(mesh, 2, 0b010000)
    op = Operator(ctx, "heat", [m], rhocp=1024.0, dt=1.0, k0=8.0, t_boil=1.0, coef_mode=1)
    op.set_field("t_prev", _cuda(1.0 + 0.5 * syn.uniform_pm1(3, m.n_dofs)))
    if name == "heat_convection":
        op.set_field("beta", _cuda(syn.uniform_pm1(5, 3 * m.n_dofs) / 8))
    return op, [(0, op.n)], 3


@pytest.mark.parametrize("name", ["heat", "heat_convection", "oseen", "oseen_meltpool", "reinit_octree"])
def test_captured_before_the_tables(name):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import Context, build_library
    build_library()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = Context(0, stream)
        op, blocks, nrhs = _operator(ctx, name)
        u = _cuda(syn.uniform_pm1(11, op.n * nrhs))
        ref = op.apply(u, nrhs=nrhs)
        u32, v = u.float(), torch.zeros(op.n * nrhs, device="cuda")
        # a first launch of every kernel outside the capture, on another operator
        warm, _, _ = _operator(ctx, name)
        warm.apply(u32, nrhs=nrhs)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        op.apply(u32, v, nrhs=nrhs)
    assert not any(k in op.variant for k in ("/march", "interleaved", "warp-per-component")), op.variant
    graph.replay()
    torch.cuda.synchronize()
    first = v.clone()
    with torch.cuda.stream(stream):
        own = op.apply(u32, nrhs=nrhs)     # now with tables of its own
    stream.synchronize()
    assert any(k in op.variant for k in ("/march", "interleaved", "warp-per-component")), op.variant
    for a, b in blocks:
        r = ref.view(nrhs, -1)[:, a:b]
        for x in (first, own):
            worst = float((x.double().view(nrhs, -1)[:, a:b] - r).abs().max())
            assert worst <= (2e-5 if name.startswith("heat") else 5e-5) * float(r.abs().max()), (name, (a, b), worst)
