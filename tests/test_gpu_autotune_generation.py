"""Records that a library with other kernels wrote to mf_autotune's cache file are not applied: their key does not
name the present generation of kernels, so the variants are timed and a record of their own is appended."""
import json
import re

import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_records_of_other_kernels_are_not_applied(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import Context, DofMap, Mesh, Operator, build_library
    build_library()
    ctx = Context(0)
    m = DofMap(Mesh.uniform(ctx, 6), 2, 0)
    fields = torch.tensor(syn.uniform_pm1(3, m.n_dofs), device="cuda")

    def tuned(path):
        op = Operator(ctx, "helmholtz", [m], mass_coef=1024.0, a_liquid=80.0, a_gas=8.0)
        op.set_field("phi", fields)
        op.autotune(path)
        return open(path).read().splitlines()

    path = str(tmp_path / "tune.jsonl")
    rec = json.loads(tuned(path)[-1])
    assert re.search(r" kernels=\d+$", rec["key"]), rec["key"]
    for key in (re.sub(r" kernels=\d+$", "", rec["key"]), re.sub(r"(?<= kernels=)\d+$", "1", rec["key"])):
        with open(path, "w") as f:   # as an earlier library wrote it
            f.write(json.dumps(dict(rec, key=key)) + "\n")
        lines = tuned(path)
        assert len(lines) == 2 and json.loads(lines[1])["key"] == rec["key"]
