"""Applies on boxes whose extents are not multiples of the kernels' 8 x 4 x 4 bricks, against the fp64
apply of the same operator (itself pinned to the oracle on cubes): tile edges, lanes without a cell,
several right-hand sides, Dirichlet faces.  Bounds: double-float keeps 47 bits per operation, a few
1e-14 of |A||u| over a cell's few hundred operations, and is held to the fp64 bar 1e-12; fp32 has unit
roundoff 6e-8 and is held to its bar 2e-5 (5e-5 for Oseen).  Both are taken relative to the largest
entry of the result's block, which a row of |A||u| for uniform random u does not exceed by more than
the row's 125 to 425 entries."""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BOXES = [(1, 1, 1), (8, 4, 4), (9, 5, 3), (7, 13, 2), (17, 3, 9)]


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import Context, build_library
    build_library()
    return Context(0)


def _cuda(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def _mesh(ctx, n, h=0.125):
    from paper_2501_18781_gb300 import Mesh
    return Mesh.uniform(ctx, list(n), (0.0, 0.0, 0.0), tuple(h * m for m in n))


def _check(op, blocks, transpose=False, nrhs=1, rtol32=2e-5):
    """df64 and fp32 applies against the fp64 apply, each block (start, stop) by its largest entry."""
    n = op.n
    u = syn.uniform_pm1(11, n * nrhs)
    ref = op.apply(_cuda(u), nrhs=nrhs, transpose=transpose).cpu().numpy().reshape(nrhs, n)
    out = {"df64": (op.apply(_cuda(u), nrhs=nrhs, transpose=transpose, arith="df64"), 1e-12),
           "f32": (op.apply(_cuda(u.astype(np.float32)), nrhs=nrhs, transpose=transpose), rtol32)}
    for name, (v, rtol) in out.items():
        v = v.double().cpu().numpy().reshape(nrhs, n)
        for a, b in blocks:
            big = np.max(np.abs(ref[:, a:b]))
            worst = np.max(np.abs(v[:, a:b] - ref[:, a:b])) / big
            assert worst <= rtol, (name, op.variant, (a, b), worst)


@pytest.mark.parametrize("box", BOXES)
@pytest.mark.parametrize("faces", [0, 0b011010])
def test_scalar_operators(ctx, box, faces):
    from paper_2501_18781_gb300 import DofMap, Operator
    m = DofMap(_mesh(ctx, box), 2, faces)
    x = m.coords()
    rng = syn.uniform_pm1(3, m.n_dofs)
    # value and stiffness terms of one size (h = 1/8), Dirichlet rows of the same size as the others
    rho = 2.0 * 8 ** 3
    k = 8.0
    phi = _cuda(np.tanh(4.0 * (x[:, 2] - 0.3) + 0.2 * rng))
    helm = Operator(ctx, "helmholtz", [m], mass_coef=rho, a_liquid=10 * k, a_gas=k, coef_mode=1)
    helm.set_field("phi", phi)
    _check(helm, [(0, m.n_dofs)], nrhs=3)
    heat = Operator(ctx, "heat", [m], rhocp=rho, dt=1.0, k0=k, t_boil=1.0, coef_mode=1)
    heat.set_field("t_prev", _cuda(1.0 + 0.5 * rng))
    _check(heat, [(0, m.n_dofs)])
    beta = _cuda(8.0 ** -1 * syn.uniform_pm1(5, 3 * m.n_dofs))
    heat.set_field("beta", beta)
    for transpose in (False, True):
        _check(heat, [(0, m.n_dofs)], transpose=transpose, nrhs=2)
    heat.set_field("rhocp_qpoint", _cuda(rho * (1.5 + 0.5 * syn.uniform_pm1(6, 27 * m.n_cells))))
    for transpose in (False, True):
        _check(heat, [(0, m.n_dofs)], transpose=transpose)
    reinit = Operator(ctx, "reinit", [m], eps=k, dtau=1.0 / rho, coef_mode=1)
    reinit.set_field("phi", phi)
    _check(reinit, [(0, m.n_dofs)], nrhs=2)


@pytest.mark.parametrize("box", BOXES)
@pytest.mark.parametrize("flags", [0, 7])
def test_oseen(ctx, box, flags):
    from paper_2501_18781_gb300 import DofMap, Operator
    mesh = _mesh(ctx, box)
    mu, mp = DofMap(mesh, 2, 0b011111), DofMap(mesh, 1, 0)
    x = mu.coords()
    op = Operator(ctx, "oseen", [mu, mp], sigma=16.0, rho_l=40.0, rho_g=0.4, mu_l=3.0, mu_g=0.03, rho_s=40.0, mu_s=3.0,
                  t_solidus=1900.0, t_liquidus=2200.0, darcy_c=1e3, darcy_b=1.0, oseen_flags=flags)
    fields = [_cuda(np.tanh(4.0 * (x[:, 2] - 0.3) + 0.2 * syn.uniform_pm1(3, mu.n_dofs))),
              _cuda(syn.uniform_pm1(5, 3 * mu.n_dofs)), _cuda(2000.0 + 400.0 * syn.uniform_pm1(7, mu.n_dofs))]
    for name, f in zip(("phi", "beta", "t_prev"), fields):
        op.set_field(name, f)
    nu = mu.n_dofs
    _check(op, [(0, 3 * nu), (3 * nu, op.n)], nrhs=2, rtol32=5e-5)


@pytest.mark.parametrize("nrhs", [1, 2, 3, 8, 9, 17])
def test_octree_right_hand_sides(ctx, nrhs):
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    dist = lambda X, Y, Z: syn.deformed_sphere_distance(X, Y, Z, 3)
    leaves = syn.refine_band_leaves(4, 2, dist, 1.0 / 64)
    for faces in (0, 0b000101):
        m = DofMap(Mesh.octree(ctx, 4, 2, leaves), 2, faces)
        rng = syn.uniform_pm1(3, m.n_dofs)
        op = Operator(ctx, "reinit", [m], eps=16.0, dtau=16.0 ** -3, coef_mode=1)
        op.set_field("phi", _cuda(np.tanh(4.0 * (m.coords()[:, 2] - 0.3) + 0.2 * rng)))
        _check(op, [(0, m.n_dofs)], nrhs=nrhs, rtol32=5e-5)
