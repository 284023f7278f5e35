"""When the tables of the fp32 kernels are built: by mf_autotune also where it reads its choice from a record, so
that an apply under stream capture finds them; and once per set of fields where the memory is not there."""
import json

import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def build():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import build_library
    build_library()


def _heat(ctx, n, beta=False):
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    m = DofMap(Mesh.uniform(ctx, n, (0.0,) * 3, (1.0,) * 3), 2, 1 << 4)
    op = Operator(ctx, "heat", [m], rhocp=2.0 * n ** 3, dt=1.0, k0=float(n), t_boil=1.0, coef_mode=1)
    op.set_field("t_prev", torch.tensor(1.0 + 0.5 * syn.uniform_pm1(3, m.n_dofs), device="cuda"))
    if beta:
        op.set_field("beta", torch.tensor(syn.uniform_pm1(5, 3 * m.n_dofs) / n, device="cuda"))
    return op


def test_autotune_from_a_record_builds_the_tables(build, tmp_path):
    from paper_2501_18781_gb300 import Context
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = Context(0, stream)
        path = str(tmp_path / "tune.jsonl")
        _heat(ctx, 12).autotune(path)
        rec = json.loads(open(path).read().splitlines()[-1])
        with open(path, "a") as f:   # the tabulated form with one thread per cell
            f.write(json.dumps(dict(rec, mode32=1, q2_line32=0)) + "\n")
        op = _heat(ctx, 12)
        op.autotune(path)
        u = torch.tensor(syn.uniform_pm1(11, op.n), device="cuda").float()
        v = torch.zeros_like(u)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        op.apply(u, v)
    assert "/f32/tabulated/march" in op.variant, op.variant
    graph.replay()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        ref = op.apply(u.double())
    stream.synchronize()
    assert float((v.double() - ref).abs().max()) <= 2e-5 * float(ref.abs().max())


def test_a_failed_build_is_not_repeated_by_every_apply(build):
    from paper_2501_18781_gb300 import Context
    ctx = Context(0)
    op = _heat(ctx, 96, beta=True)
    table = 4 * 81 * 96 ** 3                    # the larger of its two tables
    u = torch.tensor(syn.uniform_pm1(11, op.n), device="cuda").float()
    v, w = torch.empty_like(u), torch.empty_like(u)
    ref = op.apply(u.double())                  # builds the fp64 and the general kernel's tables
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    left = 200 << 20
    assert left < table
    hold = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    op.apply(u, v)
    first = op.variant
    del hold
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    op.apply(u, w)                              # the memory is there again, but nothing asked for a new build
    assert "march" not in first and op.variant == first
    for x in (v, w):
        assert float((x.double() - ref).abs().max()) <= 2e-5 * float(ref.abs().max())
    op.set_field("t_prev", op._fields["t_prev"])
    op.apply(u, v)
    assert "march" in op.variant
    assert float((v.double() - ref).abs().max()) <= 2e-5 * float(ref.abs().max())
