"""Pipe contexts with an odd number of radial points: the bulk copies of the radial factors need
chunks of whole 16 bytes, which rows of 21 doubles give by themselves only for even counts.
Tolerance: that of test_gpu_pipe.py (2e-11 of the largest value, FP64)."""
import numpy as np
import pytest

from gpu_util import host, rel
from test_gpu_pipe import make, seeded, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr", [17, 33])
def test_pipe_odd_radial_grid(nr):
    ctx, orc = make(dict(nr=nr, mt=2, kz=3, nt=12, nz=12), max_batch=9)
    u, c, _, _ = seeded(ctx, orc)
    G = ctx.zeros()
    ctx.sp_step(to_dev(ctx, u, c), G)
    assert rel(host(ctx.pipe_split(G)[0]), orc.step((u, c))[0]) < 2e-11
    ctx.sp_set_base(to_dev(ctx, u, c))
    base = orc.base((u, c))
    d = ctx.zeros(9)
    for i in range(9):
        d[i] = to_dev(ctx, (i + 1.0) * u, 0.25 * i)
    out = ctx.zeros(9)
    ctx.sp_jvp(d, out)
    for i in (0, 8):
        ref, phase = orc.jvp(base, ((i + 1.0) * u, 0.25 * i))
        gu, gc = ctx.pipe_split(out[i])
        assert rel(host(gu), ref) < 2e-11
        assert abs(gc - phase) < 2e-11 * max(1.0, abs(phase))
