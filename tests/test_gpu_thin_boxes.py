"""fp32 applies on boxes that fill few lanes of the marching kernel's 8 x 4 columns: the general kernel serves
them, except several right-hand sides or Dirichlet rows on small meshes; on both sides of that line every form agrees with the
fp64 apply of the operator to the fp32 bar 2e-5 of the largest entry (unit roundoff 6e-8, a few hundred
operations per row)."""
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


# lanes with a cell: 3/8 (many tiles), 1/32, 9/16 twice, 19/24, all, 1/4 (many tiles); march: which of one right-hand side
# with Dirichlet rows, one without and three take the marching kernel
@pytest.mark.parametrize("box,march", [((3, 200, 40), ""), ((1, 1, 9), "rows,three"), ((9, 4, 5), "rows,three"),
                                       ((6, 3, 4), "rows,three"), ((19, 8, 5), "rows,one,three"),
                                       ((8, 4, 3), "rows,one,three"), ((2, 64, 64), "")])
@pytest.mark.parametrize("faces", [0, 0b010010])
def test_thin_boxes(ctx, box, march, faces):
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    m = DofMap(Mesh.uniform(ctx, list(box), (0.0,) * 3, tuple(n / 8 for n in box)), 2, faces)
    one, three = ("rows" if faces else "one") in march.split(","), "three" in march
    for kind in ("helmholtz", "heat", "convection", "convection+rhocp"):
        if kind == "helmholtz":
            op = Operator(ctx, "helmholtz", [m], mass_coef=1024.0, a_liquid=80.0, a_gas=8.0, coef_mode=1)
            op.set_field("phi", _cuda(np.tanh(4.0 * (m.coords()[:, 2] - 0.3))))
        else:
            op = Operator(ctx, "heat", [m], rhocp=1024.0, dt=1.0, k0=8.0, t_boil=1.0, coef_mode=1)
            op.set_field("t_prev", _cuda(1.0 + 0.5 * syn.uniform_pm1(3, m.n_dofs)))
        if kind.startswith("convection"):
            op.set_field("beta", _cuda(syn.uniform_pm1(5, 3 * m.n_dofs) / 8))
        if kind.endswith("rhocp"):
            op.set_field("rhocp_qpoint", _cuda(1024.0 * (1.5 + 0.5 * syn.uniform_pm1(6, 27 * m.n_cells))))
        for nrhs, taken in ((1, one), (3, three)):
            u = _cuda(syn.uniform_pm1(11, m.n_dofs * nrhs))
            for transpose in (False, True) if kind.startswith("convection") else (False,):
                ref = op.apply(u, nrhs=nrhs, transpose=transpose)
                v = op.apply(u.float(), nrhs=nrhs, transpose=transpose).double()
                assert ("/march" in op.variant) == taken, (kind, nrhs, op.variant)
                assert float((v - ref).abs().max()) <= 2e-5 * float(ref.abs().max()), (kind, nrhs, transpose)
