"""The fixed-point Chebyshev transforms and the dense and chained solves at the largest degree, N = 256,
one direction and a batch. Tolerance 1e-9 of the largest value: two exact inverses of the tau systems
agree to about that there (test_gpu_edges.py)."""
import numpy as np
import pytest

from gpu_util import dev, host, make, rel, seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_dir", [1, 33])
def test_tangents(n_dir):
    ctx, orc = make(4, 257, 4, max_batch=n_dir)
    u = seeded(orc, 990, 0.1)
    ctx.sp_set_base(dev(u))
    base = orc.base(u)
    ds = np.stack([seeded(orc, 991 + i, 1.0) for i in range(n_dir)])
    J = ctx.zeros(n_dir)
    ctx.sp_jvp(dev(ds), J)
    for i in (0, n_dir - 1):
        assert rel(host(J)[i], orc.jvp(base, ds[i])) < 1e-9
