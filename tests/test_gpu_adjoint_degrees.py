"""The transposed per-mode solve over Chebyshev degrees: the smallest, the edges of warps and of a
block's threads, even and odd half lengths, operators in shared memory and (N > 104) in place."""
import numpy as np
import pytest

import seeded_inputs as si
from gpu_util import dev, host, make, rel, seeded

pytestmark = pytest.mark.gpu


# the tolerance of the adjoint's FP64 parity tests
@pytest.mark.parametrize("ny", [5, 7, 17, 31, 33, 35, 65, 103, 105, 107, 129])
def test_vjp_degrees(ny):
    grid = (6, ny, 4)
    ctx, orc = make(*grid, max_batch=3)
    u = seeded(orc, 940, 0.1)
    ctx.sp_set_base(dev(u))
    base = orc.base(u)
    rs = np.stack([orc.seed_state(*si.couette_random_coeffs(941 + i, *grid, mmax=2), 1.0) for i in range(3)])
    out = ctx.zeros(3)
    ctx.sp_vjp(dev(rs), out)
    for i in range(3):
        assert rel(host(out)[i], orc.vjp(base, rs[i])) < 1e-12
