"""Launch shapes of the general kernel on octrees: one right-hand side and batches each have their own, so what was timed
on one of them does not decide for the other."""
import json

import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_single_and_batched_applies_take_their_own_shape(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2501_18781_gb300 import Context, DofMap, Mesh, Operator, build_library
    build_library()
    ctx = Context(0)
    dist = lambda X, Y, Z: syn.deformed_sphere_distance(X, Y, Z, 3)
    m = DofMap(Mesh.octree(ctx, 4, 2, syn.refine_band_leaves(4, 2, dist, 1.0 / 64)), 2, 0)
    phi = torch.tensor(np.tanh(4.0 * (m.coords()[:, 2] - 0.3)), device="cuda")

    def tuned(path):
        op = Operator(ctx, "reinit", [m], eps=16.0, dtau=16.0 ** -3)
        op.set_field("phi", phi)
        op.autotune(path)
        return op

    path = str(tmp_path / "tune.jsonl")
    tuned(path)
    rec = json.loads(open(path).read().splitlines()[-1])
    u = torch.tensor(syn.uniform_pm1(11, 3 * m.n_dofs), device="cuda")
    ref = None
    for shapes in ((64, 8, 128, 0), (128, 0, 64, 8), (128, 2, 128, 4)):
        names = ("block", "persistent_blocks", "batch_block", "batch_persistent")
        with open(path, "a") as f:
            f.write(json.dumps(dict(rec, **dict(zip(names, shapes)))) + "\n")
        op = tuned(path)
        for nrhs, (block, persistent) in ((1, shapes[:2]), (3, shapes[2:])):
            v = op.apply(u[:nrhs * m.n_dofs], nrhs=nrhs)
            end = "/block%d" % block + ("/persistent%d" % persistent if persistent else "")
            assert op.variant.endswith(end), (op.variant, nrhs, shapes)
            if ref is None and nrhs == 3:
                ref = v.clone()
        assert float((v - ref).abs().max()) <= 1e-13 * float(ref.abs().max())
