"""Double-float applies at the ends of the fp64 range and on inputs that are not finite, against the fp64
apply of the same operator.  The operators are linear, so inputs scaled by 1e-280, 1e-300 or 1e300 keep
their bar: 1e-12 of the result's largest entry, plus what is flushed where a part of a result lies below
the smallest normal double, 2^-1022 (at most 64 parts per entry: eight cells, two floats each, folded
in a few steps).  An input that is not finite makes exactly the rows of the cells around it not finite."""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FLUSHED = 64 * 2.0 ** -1022


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import Context, build_library
    build_library()
    return Context(0)


def _cuda(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def _box(ctx, n=(9, 5, 6), h=0.125):
    from paper_2501_18781_gb300 import Mesh
    return Mesh.uniform(ctx, list(n), (0.0, 0.0, 0.0), tuple(h * m for m in n))


def _phi(m):
    return _cuda(np.tanh(4.0 * (m.coords()[:, 2] - 0.3) + 0.2 * syn.uniform_pm1(3, m.n_dofs)))


def _operator(ctx, name):
    """An operator with value and stiffness terms of one size, and its output blocks."""
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    rho, k = 2.0 * 8 ** 3, 8.0
    if name.startswith("oseen"):
        mesh = _box(ctx)
        mu, mp = DofMap(mesh, 2, 0b011111), DofMap(mesh, 1, 0)
        op = Operator(ctx, "oseen", [mu, mp], sigma=16.0, rho_l=40.0, rho_g=0.4, mu_l=3.0, mu_g=0.03, rho_s=40.0,
                      mu_s=3.0, t_solidus=1900.0, t_liquidus=2200.0, darcy_c=1e3, darcy_b=1.0,
                      oseen_flags=7 if name == "oseen_meltpool" else 0)
        op.set_field("phi", _phi(mu))
        op.set_field("beta", _cuda(syn.uniform_pm1(5, 3 * mu.n_dofs)))
        op.set_field("t_prev", _cuda(2000.0 + 400.0 * syn.uniform_pm1(7, mu.n_dofs)))
        return op, [(0, 3 * mu.n_dofs), (3 * mu.n_dofs, op.n)]
    if name == "reinit_octree":
        dist = lambda X, Y, Z: syn.deformed_sphere_distance(X, Y, Z, 3)
        m = DofMap(Mesh.octree(ctx, 4, 2, syn.refine_band_leaves(4, 2, dist, 1.0 / 64)), 2, 0)
        op = Operator(ctx, "reinit", [m], eps=16.0, dtau=16.0 ** -3, coef_mode=1)
        op.set_field("phi", _phi(m))
        return op, [(0, op.n)]
    m = DofMap(_box(ctx), 2, 0b010000)
    if name == "helmholtz":
        op = Operator(ctx, "helmholtz", [m], mass_coef=rho, a_liquid=10 * k, a_gas=k, coef_mode=1)
        op.set_field("phi", _phi(m))
    else:
        op = Operator(ctx, "heat", [m], rhocp=rho, dt=1.0, k0=k, t_boil=1.0, coef_mode=1)
        op.set_field("t_prev", _cuda(1.0 + 0.5 * syn.uniform_pm1(3, m.n_dofs)))
        op.set_field("beta", _cuda(syn.uniform_pm1(5, 3 * m.n_dofs) / 8))
    return op, [(0, op.n)]


OPERATORS = ["helmholtz", "heat_convection", "reinit_octree", "oseen", "oseen_meltpool"]


def _compare(op, blocks, u):
    ref = op.apply(u).cpu().numpy()
    v = op.apply(u, arith="df64").cpu().numpy()
    assert "/df64/" in op.variant, op.variant
    ok = np.isfinite(ref)
    assert np.array_equal(ok, np.isfinite(v)), (op.variant, int((~ok).sum()), int((~np.isfinite(v)).sum()))
    for a, b in blocks:
        r, w = ref[a:b][ok[a:b]], v[a:b][ok[a:b]]
        if r.size:
            worst = np.max(np.abs(w - r))
            assert worst <= 1e-12 * np.max(np.abs(r)) + FLUSHED, (op.variant, (a, b), worst, np.max(np.abs(r)))
    return ref


@pytest.mark.parametrize("name", OPERATORS)
@pytest.mark.parametrize("scale", [1e-280, 1e-300, 1e300])
def test_ends_of_the_range(ctx, name, scale):
    op, blocks = _operator(ctx, name)
    u = syn.uniform_pm1(11, op.n)
    _compare(op, blocks, _cuda(scale * u))
    # entries spread over 120 powers of two below the scale
    spread = 2.0 ** -np.floor(60.0 * (1.0 + syn.uniform_pm1(13, op.n)))
    _compare(op, blocks, _cuda(scale * u * spread))


@pytest.mark.parametrize("name", OPERATORS)
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_inputs_that_are_not_finite(ctx, name, bad):
    op, blocks = _operator(ctx, name)
    for at in (op.n // 3, op.n - 1 if name.startswith("oseen") else op.n // 2):
        u = syn.uniform_pm1(11, op.n)
        u[at] = bad
        ref = _compare(op, blocks, _cuda(u))
        assert 0 < (~np.isfinite(ref)).sum() < op.n


def test_results_beyond_the_range(ctx):
    from paper_2501_18781_gb300 import DofMap, Operator
    m = DofMap(_box(ctx), 2, 0)
    op = Operator(ctx, "helmholtz", [m], mass_coef=1e12, a_liquid=1.0, a_gas=1.0, coef_mode=1)
    op.set_field("phi", _phi(m))
    ref = _compare(op, [(0, op.n)], _cuda(np.full(op.n, 1.5e308)))
    assert not np.isfinite(ref).any()
