"""The fixed-point FP64 plane stage (xz_fx.cuh) where it can go wrong: every radix in both directions
and both orders of the factors, ragged chunks of row pairs, planes with one block and with several,
scales far from 1, zero and non-finite inputs. Tolerance 1e-12 of the largest value, as for every
FP64 parity test; linearity under powers of two 1e-13 (the scales follow the input exactly)."""
import numpy as np
import pytest
import torch

from gpu_util import dev, host, make, rel, seeded

pytestmark = pytest.mark.gpu

# sizes N1 x N2 of the two directions: 2x2 .. 12x12; 72 x 72 and 48 x 54 run in several blocks per plane
GRIDS = [(4, 9, 6), (6, 9, 4), (8, 13, 12), (12, 17, 8), (16, 17, 32), (32, 17, 18), (18, 9, 64), (36, 9, 24),
         (24, 9, 72), (54, 9, 16), (64, 9, 36), (72, 9, 72), (48, 11, 54), (16, 9, 108), (144, 9, 8)]


@pytest.mark.parametrize("grid", GRIDS)
def test_step_tangent_adjoint(grid):
    ctx, orc = make(*grid, max_batch=3)
    u = seeded(orc, 900, 0.1)
    base = orc.base(u)
    G, J = ctx.zeros(), ctx.zeros(3)
    ctx.sp_step(dev(u), G)
    assert rel(host(G), orc.step(u)) < 1e-12
    ctx.sp_set_base(dev(u))
    ds = np.stack([seeded(orc, 901 + i, 1.0) for i in range(3)])
    ctx.sp_jvp(dev(ds), J)
    for i in (0, 2):
        assert rel(host(J)[i], orc.jvp(base, ds[i])) < 1e-12
    ctx.sp_vjp(dev(ds), J)
    assert rel(host(J)[1], orc.vjp(base, ds[1])) < 1e-12


@pytest.mark.parametrize("grid", [(16, 17, 24), (48, 9, 48)])
def test_scales(grid):
    ctx, orc = make(*grid, max_batch=2)
    ctx.sp_set_base(dev(seeded(orc, 910, 0.1)))
    d = seeded(orc, 911, 1.0)
    J, Js = ctx.zeros(), ctx.zeros()
    ctx.sp_jvp(dev(d), J)
    for s in (2.0 ** -400, 2.0 ** -30, 2.0 ** 300):
        ctx.sp_jvp(dev(d * s), Js)
        assert rel(host(Js) / s, host(J)) < 1e-13
    ctx.sp_jvp(ctx.zeros(), J)
    assert float(J.abs().max()) == 0.0


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_input(value):
    ctx, orc = make(16, 17, 24)
    u = dev(seeded(orc, 920, 0.1))
    d = u.clone()
    u[1, 2, 3, 4] = value
    G = ctx.zeros()
    ctx.sp_step(u, G)
    assert not bool(torch.isfinite(torch.view_as_real(G)).all())
    ctx.sp_set_base(u)
    ctx.sp_jvp(d, G)
    assert not bool(torch.isfinite(torch.view_as_real(G)).all())


# Chebyshev degrees: the smallest, warps' edges, odd halves of N, the largest; one direction and
# passes of the batched solve's layouts (5: modes fastest, 17: directions fastest)
@pytest.mark.parametrize("ny", [5, 7, 31, 33, 35, 63, 65, 95, 127, 129])
@pytest.mark.parametrize("n_dir", [1, 5, 17])
def test_chebyshev_degrees(ny, n_dir):
    ctx, orc = make(6, ny, 4, max_batch=1 if n_dir == 1 else 32)
    u = seeded(orc, 930, 0.1)
    ctx.sp_set_base(dev(u))
    base = orc.base(u)
    ds = np.stack([seeded(orc, 931 + i, 1.0) for i in range(n_dir)])
    J = ctx.zeros(n_dir)
    ctx.sp_jvp(dev(ds), J)
    for i in (0, n_dir - 1):
        assert rel(host(J)[i], orc.jvp(base, ds[i])) < 1e-12
