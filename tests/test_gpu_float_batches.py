"""The float forward transform of batched mixed tangents where its layout can go wrong: degrees around the
classes of rows (0 and 2 mod 4, odd) and their pairs, with and without the second split level, batches
that do not fill the directions of a block."""
import numpy as np
import pytest

from gpu_util import dev, host, make, rel, seeded

pytestmark = pytest.mark.gpu


# tolerance: that of the mixed tangent's parity tests at these degrees (about 170 float roundings)
@pytest.mark.parametrize("ny", [5, 7, 9, 11, 13, 15, 17, 35, 37, 63, 65])
@pytest.mark.parametrize("n_dir", [1, 6, 33])
def test_mixed_batches(ny, n_dir):
    ctx, orc = make(6, ny, 4, max_batch=33, prec=1)
    u = seeded(orc, 950, 0.1)
    ctx.sp_set_base(dev(u))
    base = orc.base(u)
    ds = np.stack([seeded(orc, 951 + i, 1.0) for i in range(n_dir)])
    J = ctx.zeros(n_dir)
    ctx.sp_jvp(dev(ds), J)
    for i in {0, n_dir // 2, n_dir - 1}:
        assert rel(host(J)[i], orc.jvp(base, ds[i])) < 1e-5
