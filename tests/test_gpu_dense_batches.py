"""The dense per-mode solve in batches: two directions per block (from nine blocks per SM), four (short
columns, from 36), with last blocks that are not full, beside one direction per call, whose bits a batch
must give; and against the oracle with the parity tests' tolerances (FP64 1e-12, mixed 1e-5)."""
import numpy as np
import pytest

from gpu_util import dev, host, make, rel, seeded

pytestmark = pytest.mark.gpu


# 113, 221, 481 and 113 solved modes; 152 SMs
@pytest.mark.parametrize("grid,n_dir", [((24, 25, 24), 13), ((32, 33, 32), 27), ((48, 65, 48), 3), ((24, 129, 24), 15)])
@pytest.mark.parametrize("prec", [0, 1])
def test_batch(grid, n_dir, prec):
    ctx, orc = make(*grid, max_batch=n_dir, prec=prec)
    u = seeded(orc, 1010, 0.1)
    ctx.sp_set_base(dev(u))
    base = orc.base(u)
    ds = np.stack([seeded(orc, 1011 + i, 1.0) for i in range(n_dir)])
    J, one = ctx.zeros(n_dir), ctx.zeros()
    ctx.sp_jvp(dev(ds), J)
    out = host(J)
    for i in range(n_dir):
        ctx.sp_jvp(dev(ds[i]), one)
        assert np.array_equal(out[i], host(one))
    for i in (0, n_dir - 1):
        assert rel(out[i], orc.jvp(base, ds[i])) < (1e-12 if prec == 0 else 1e-5)
