"""Pipe tangents in the batches that fill the radial solve's blocks of 16 directions (12, 17 with a block
of one, 64), at an even and an odd radial count and at the count with unrolled solves (64), with the phase
condition of every direction. FP64: against the oracle, with the tolerances of test_gpu_pipe.py (2e-11 of
the largest value, 1e-10 for the phase). Mixed: against one-direction calls; the float stages treat every
direction alike, so only the FP64 solve may round differently, and its tolerance holds."""
import numpy as np
import pytest

from gpu_util import host, rel
from test_gpu_pipe import make, seeded, to_dev

pytestmark = pytest.mark.gpu


def directions(ctx, orc, shape, n_dir):
    rng = np.random.default_rng(7)
    dirs = []
    d = ctx.zeros(n_dir)
    for i in range(n_dir):
        du = orc.sym(rng.standard_normal(shape) + 1j * rng.standard_normal(shape))
        du[:, :, :, 0] = 0.0
        dirs.append((du, 0.1 * i - 0.3))
        d[i] = to_dev(ctx, *dirs[i])
    return dirs, d


@pytest.mark.parametrize("nr", [24, 33, 64])
@pytest.mark.parametrize("n_dir", [12, 17, 64])
def test_fp64_batches(nr, n_dir):
    ctx, orc = make(dict(nr=nr, mt=2, kz=3, nt=12, nz=12), max_batch=n_dir)
    u, c, _, _ = seeded(ctx, orc)
    ctx.sp_set_base(to_dev(ctx, u, c))
    base = orc.base((u, c))
    dirs, d = directions(ctx, orc, u.shape, n_dir)
    out = ctx.zeros(n_dir)
    ctx.sp_jvp(d, out)
    for i in sorted({0, 7, 11, n_dir // 2, n_dir - 1}):
        ref, phase = orc.jvp(base, dirs[i])
        gu, gc = ctx.pipe_split(out[i])
        assert rel(host(gu), ref) < 2e-11
        assert abs(gc - phase) < 1e-10 * max(1.0, abs(phase))


@pytest.mark.parametrize("nr", [24, 33, 64])
@pytest.mark.parametrize("n_dir", [5, 12, 17])
def test_mixed_batches_match_single_calls(nr, n_dir):
    ctx, orc = make(dict(nr=nr, mt=2, kz=3, nt=12, nz=12), prec=1, max_batch=n_dir)
    u, c, _, _ = seeded(ctx, orc)
    ctx.sp_set_base(to_dev(ctx, u, c))
    _, d = directions(ctx, orc, u.shape, n_dir)
    out, one = ctx.zeros(n_dir), ctx.zeros()
    ctx.sp_jvp(d, out)
    for i in range(n_dir):
        ctx.sp_jvp(d[i].contiguous(), one)
        assert rel(host(out[i]), host(one)) < 2e-11
