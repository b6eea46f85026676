"""sp_jvp_static beside the context's own calls on another stream: both give the bits that the same calls
give in turn. 48 x 65 x 48 and 64 x 9 x 64 are planes that a single sp_jvp passes through a buffer of the
context; 96 x 9 x 96 planes do not fit on chip and go through the static array."""
import numpy as np
import pytest
import torch

from gpu_util import dev, host, make, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,prec", [((48, 65, 48), 0), ((48, 65, 48), 1), ((64, 9, 64), 0), ((96, 9, 96), 0),
                                       ((16, 17, 24), 0)])
def test_static_beside_the_context(grid, prec):
    ctx, orc = make(*grid, prec=prec)
    u = dev(seeded(orc, 960, 0.1))
    d = dev(seeded(orc, 961, 1.0))
    ctx.sp_set_base(u)
    G, J, K = ctx.zeros(), ctx.zeros(), ctx.zeros()
    ctx.sp_step(d, G)
    ctx.sp_jvp(u, K)
    ctx.sp_jvp_static(d, J)
    ref = host(G), host(J), host(K)
    reps = 40
    outs = [(ctx.zeros(), ctx.zeros(), ctx.zeros()) for _ in range(reps)]
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for g, j, k in outs:
        ctx.sp_step(d, g, stream=a)
        ctx.sp_jvp_static(d, j, stream=b)
        ctx.sp_jvp(u, k, stream=a)
    for out in outs:
        for t, r in zip(out, ref):
            assert np.array_equal(host(t), r)
