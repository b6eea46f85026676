"""FP64 plane stage with fields of unlike size: a streak u at (kx, kz) = (0, 1) of order 1 beside a roll
(v, w) at (0, 2) of order eps. Of the x component of the products, which is of order eps, mode (0, 3) is
a response of its own: no input has that mode, and at kx = 0 the solve does not mix u with v and w. So its
largest value is known to the accuracy of FP64 transforms of each field by itself; tolerance 1e-12 of it, as
for every FP64 parity test."""
import numpy as np
import pytest

from gpu_util import dev, host, make, rel

pytestmark = pytest.mark.gpu


def states(orc, eps):
    rng = np.random.default_rng(970)
    streak, roll = np.zeros((2, 3, orc.MX, orc.MZ, orc.NY), complex)
    n = np.arange(orc.NY)
    decay = 0.5 ** n
    streak[0, 0, 1] = (rng.standard_normal(orc.NY) + 1j * rng.standard_normal(orc.NY)) * decay
    for c in (1, 2):
        roll[c, 0, 2] = eps * (rng.standard_normal(orc.NY) + 1j * rng.standard_normal(orc.NY)) * decay
    return streak, roll


def weak(a):
    return a[0, 0, 3]


@pytest.mark.parametrize("grid", [(16, 17, 24), (48, 9, 48), (12, 9, 96)])
@pytest.mark.parametrize("eps", [1e-4, 1e-8, 1e-12])
@pytest.mark.parametrize("n_dir", [1, 40])
def test_roll_beside_a_streak(grid, eps, n_dir):
    ctx, orc = make(*grid, max_batch=n_dir)
    streak, roll = states(orc, eps)
    G, J = ctx.zeros(), ctx.zeros(n_dir)
    ctx.sp_step(dev(streak + roll), G)
    assert rel(weak(host(G)), weak(orc.step(streak + roll))) < 1e-12
    # the weak field in the base, then in the direction
    for u, d in ((streak + roll, streak), (streak, streak + roll)):
        base = orc.base(u)
        ctx.sp_set_base(dev(u))
        ctx.sp_jvp(dev(np.stack([d] * n_dir)), J)
        ref = weak(orc.jvp(base, d))
        for i in (0, n_dir - 1):
            assert rel(weak(host(J)[i]), ref) < 1e-12
    base = orc.base(streak + roll)
    ctx.sp_set_base(dev(streak + roll))
    ctx.sp_vjp(dev(np.stack([streak] * n_dir)), J)
    ref = weak(orc.vjp(base, streak))
    for i in (0, n_dir - 1):
        assert rel(weak(host(J)[i]), ref) < 1e-12
