"""The kernels that applies and solves take, by the operator's variant name and the launch count: where a
dispatch rule or a table build fell back to a general kernel, results alone would not show it."""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import Context, build_library
    build_library()
    return Context(0)


def _cuda(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def _heat(ctx, box, faces=0b010000):
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    m = DofMap(Mesh.uniform(ctx, list(box), (0.0,) * 3, tuple(n / 8 for n in box)), 2, faces)
    op = Operator(ctx, "heat", [m], rhocp=1024.0, dt=1.0, k0=8.0, t_boil=1.0, coef_mode=1)
    op.set_field("t_prev", _cuda(1.0 + 0.5 * syn.uniform_pm1(3, m.n_dofs)))
    return op, m


def test_fp32_uniform(ctx):
    op, m = _heat(ctx, (15, 12, 7))
    for nrhs in (1, 3):
        u = _cuda(syn.uniform_pm1(11, nrhs * m.n_dofs)).float()
        op.apply(u, nrhs=nrhs)
        assert op.variant.endswith("/uniform/f32/tabulated/march"), op.variant
    op.set_field("beta", _cuda(syn.uniform_pm1(5, 3 * m.n_dofs) / 8))
    for transpose, end in ((False, "/conv"), (True, "/conv-T")):
        op.apply(u, nrhs=3, transpose=transpose)
        assert op.variant.endswith("/uniform/f32/tabulated/march" + end), op.variant


@pytest.mark.parametrize("nrhs,lanes", [(1, 0), (2, 2), (3, 4), (4, 4), (5, 8), (8, 8), (9, 8), (17, 8)])
def test_fp32_octree_batches(ctx, nrhs, lanes):
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    dist = lambda X, Y, Z: syn.deformed_sphere_distance(X, Y, Z, 3)
    m = DofMap(Mesh.octree(ctx, 4, 2, syn.refine_band_leaves(4, 2, dist, 1.0 / 64)), 2, 0)
    op = Operator(ctx, "reinit", [m], eps=16.0, dtau=16.0 ** -3, coef_mode=1)
    op.set_field("phi", _cuda(np.tanh(4.0 * (m.coords()[:, 2] - 0.3))))
    op.apply(_cuda(syn.uniform_pm1(11, nrhs * m.n_dofs)).float(), nrhs=nrhs)
    assert op.variant.endswith("/interleaved%d" % lanes) if lanes else "interleaved" not in op.variant, op.variant


@pytest.mark.parametrize("flags", [0, 7])
def test_fp32_oseen(ctx, flags):
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    mesh = Mesh.uniform(ctx, [9, 5, 3], (0.0,) * 3, (9 / 8, 5 / 8, 3 / 8))
    mu, mp = DofMap(mesh, 2, 0b011111), DofMap(mesh, 1, 0)
    op = Operator(ctx, "oseen", [mu, mp], sigma=16.0, rho_l=40.0, rho_g=0.4, mu_l=3.0, mu_g=0.03, rho_s=40.0, mu_s=3.0,
                  t_solidus=1900.0, t_liquidus=2200.0, darcy_c=1e3, darcy_b=1.0, oseen_flags=flags)
    op.set_field("phi", _cuda(np.tanh(4.0 * (mu.coords()[:, 2] - 0.2))))
    op.set_field("beta", _cuda(syn.uniform_pm1(5, 3 * mu.n_dofs)))
    op.set_field("t_prev", _cuda(2000.0 + 400.0 * syn.uniform_pm1(7, mu.n_dofs)))
    op.apply(_cuda(syn.uniform_pm1(11, op.n)).float())
    assert op.variant == "oseen_q2q1/f32/tabulated/warp-per-component" + ("/meltpool" if flags else ""), op.variant


@pytest.mark.parametrize("box", [(1, 1, 1), (9, 5, 3), (19, 16, 15)])
@pytest.mark.parametrize("use_graph", [False, True])
def test_one_launch_cg_is_one_launch(ctx, box, use_graph):
    """The launches of a solve do not grow with its steps; step by step they do."""
    op, m = _heat(ctx, box, 0)
    op.set_variant("q2_line", 1)
    b = _cuda(syn.uniform_pm1(7, m.n_dofs))
    kw = dict(solver="cg", precond="jacobi", maxit=2000, use_graph=use_graph)
    counts, steps = [], []
    for tol in (1e-2, 1e-11):
        op.solve(b, tol=tol, **kw)
        before = ctx.launch_count()
        _, info = op.solve(b, tol=tol, **kw)
        assert info["status"] == 0
        counts.append(ctx.launch_count() - before)
        steps.append(info["iterations"])
    assert steps[1] > steps[0]
    # one more round at most: a restart from the true residual is a second launch and three vector kernels
    assert counts[1] - counts[0] <= 12, (counts, steps)
