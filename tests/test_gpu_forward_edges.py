"""The forward Chebyshev transform where both points of a pair lie just below a power of two, which sets
the column's fixed-point scale. About the laminar state the x component of the tangent's product is
-v of the direction: one Chebyshev degree of v, whose interior extremes are such pairs (equal for even
degrees, opposite for odd ones). Tolerance 1e-12 of the largest value, as for every FP64 parity test."""
import numpy as np
import pytest

from gpu_util import dev, host, make, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,degree", [(9, 4), (7, 3), (13, 6), (33, 8), (19, 9)])
@pytest.mark.parametrize("n_dir", [1, 17])
def test_pairs_below_a_power_of_two(ny, degree, n_dir):
    ctx, orc = make(6, ny, 4, max_batch=1 if n_dir == 1 else 32)
    ctx.sp_set_base(ctx.zeros())
    base = orc.base(host(ctx.zeros()))
    ds = np.zeros((n_dir,) + tuple(ctx.zeros().shape), dtype=np.complex128)
    edges = [1.0 - 1e-11, 1.0 - 2.0 ** -40, -(1.0 - 1e-10)]
    for i in range(n_dir):
        ds[i][1, 1, 1, degree] = edges[i % 3] * (1.0 if i % 2 == 0 else 1.0j)
    J = ctx.zeros(n_dir)
    ctx.sp_jvp(dev(ds if n_dir > 1 else ds[0]), J)
    out = host(J).reshape(ds.shape)
    for i in range(min(n_dir, 3)):
        assert rel(out[i], orc.jvp(base, ds[i])) < 1e-12
