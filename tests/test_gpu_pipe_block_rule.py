"""The radial solve's blocks of 16 directions, which need eight blocks per SM: 33 directions of 613 modes (a
last block of one) and 81 of 213 modes at an odd radial count, and a block of 8 for two and three directions,
beside one-direction calls. Tolerance: the FP64 one of test_gpu_pipe.py (the same chains, whose rounding may
differ with the unrolling)."""
import pytest

from gpu_util import host, rel
from test_gpu_pipe import make, seeded, to_dev
from test_gpu_pipe_batches import directions

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,n_dir", [(dict(nr=64, mt=12, kz=24, nt=48, nz=96), 33), (dict(nr=33, mt=8, kz=12, nt=32, nz=48), 81),
                                        (dict(nr=33, mt=2, kz=3, nt=12, nz=12), 2), (dict(nr=64, mt=2, kz=3, nt=12, nz=12), 3)])
def test_blocks(grid, n_dir):
    ctx, orc = make(grid, max_batch=n_dir)
    u, c, _, _ = seeded(ctx, orc)
    ctx.sp_set_base(to_dev(ctx, u, c))
    _, d = directions(ctx, orc, u.shape, n_dir)
    out, one = ctx.zeros(n_dir), ctx.zeros()
    ctx.sp_jvp(d, out)
    for i in sorted({0, 1, 15, 16, 32, n_dir - 2, n_dir - 1}):
        if i < n_dir:
            ctx.sp_jvp(d[i].contiguous(), one)
            assert rel(host(out[i]), host(one)) < 2e-11
