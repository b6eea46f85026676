"""Pipe tangents and steps on square plane grids, with all modes of the 2/3 rule (the float register-FFT
plane kernel) and with fewer, whose arrays have other strides. Tolerances: those of test_gpu_pipe.py (FP64
2e-11 of the largest value, mixed 1e-5 per component at Nr = 64)."""
import numpy as np
import pytest

import seeded_inputs as si
from gpu_util import host, rel
from oracle.pipe import seed_state
from test_gpu_pipe import make, seeded, to_dev

pytestmark = pytest.mark.gpu

GRIDS = [(16, 5, 5), (16, 4, 5), (16, 5, 4), (24, 6, 7), (24, 7, 6), (32, 10, 10), (32, 8, 9), (48, 8, 9), (64, 6, 5)]


@pytest.mark.parametrize("n,mt,kz", GRIDS)
@pytest.mark.parametrize("prec", [0, 1])
def test_square_planes(n, mt, kz, prec):
    ctx, orc = make(dict(nr=64, mt=mt, kz=kz, nt=n, nz=n), prec=prec, max_batch=2)
    u, c, _, _ = seeded(ctx, orc)
    G, J = ctx.zeros(), ctx.zeros(2)
    ctx.sp_step(to_dev(ctx, u, c), G)
    assert rel(host(ctx.pipe_split(G)[0]), orc.step((u, c))[0]) < 2e-11
    ctx.sp_set_base(to_dev(ctx, u, c))
    streak, pol = si.pipe_random_coeffs(4100, orc.kzmax, orc.mt)
    du, _ = seed_state(orc, streak, pol, amp_streak=1.0, frac=1.0)
    d = ctx.zeros(2)
    d[0] = to_dev(ctx, -2.0 * du, 0.1)
    d[1] = to_dev(ctx, du, 0.2)
    ctx.sp_jvp(d, J)
    ref, _ = orc.jvp(orc.base((u, c)), (du, 0.2))
    got = host(ctx.pipe_split(J[1])[0])
    if prec == 0:
        assert rel(got, ref) < 2e-11
    else:
        for q in range(3):
            assert rel(got[q], ref[q]) < 1e-5
