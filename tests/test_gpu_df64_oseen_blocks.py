"""Double-float Oseen applies where only one of velocity and pressure is there, and small: each is scaled by
its own power of two, so neither may be lost against the zeros of the other.  Against the fp64 apply, at the
fp64 bar 1e-12 of each block's largest entry."""
import numpy as np
import pytest

import synthetic as syn
from test_gpu_df64_range import _cuda, _operator, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", ["oseen", "oseen_meltpool"])
@pytest.mark.parametrize("only", ["velocity", "pressure"])
@pytest.mark.parametrize("scale", [1e-30, 1e-60, 1e-200])
def test_one_field_alone(ctx, flags, only, scale):  # noqa: F811
    op, blocks = _operator(ctx, flags)
    nu3 = blocks[0][1]
    u = scale * syn.uniform_pm1(11, op.n)
    if only == "velocity":
        u[nu3:] = 0.0
    else:
        u[:nu3] = 0.0
    ref, v = (op.apply(_cuda(u), **kw).cpu().numpy() for kw in ({}, {"arith": "df64"}))
    assert "/df64/" in op.variant, op.variant
    for a, b in blocks if only == "velocity" else blocks[:1]:
        big = np.max(np.abs(ref[a:b]))
        assert big > 0 and np.max(np.abs(v[a:b] - ref[a:b])) <= 1e-12 * big, (a, b, big)
    if only == "pressure":
        assert not v[nu3:].any()
