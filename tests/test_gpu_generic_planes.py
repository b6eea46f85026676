"""The generic FP64 plane stage (kernels.cu, k_xz), which serves the sides that the fixed-point stage does
not factor (128, 162) or whose kept kz it does not hold, alone and in groups; and group members whose planes
do not fit on chip (96 x 96), which run launches of their own, with some members inactive. Tolerances: those
of every parity test, 1e-12 of the largest value in FP64, 1e-5 for the mixed tangent."""
import numpy as np
import pytest

from gpu_util import dev, host, make, rel, seeded
from oracle.gint import jvp_n
from test_gpu_gint import close
from test_gpu_group import make_group, seed_group

pytestmark = pytest.mark.gpu

GRIDS = [(128, 9, 4), (4, 9, 128), (162, 9, 6), (6, 9, 162)]


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("prec", [0, 1])
def test_single_context(grid, prec):
    ctx, orc = make(*grid, max_batch=2, prec=prec)
    u = seeded(orc, 980, 0.1)
    base = orc.base(u)
    G, J = ctx.zeros(), ctx.zeros(3)
    ctx.sp_step(dev(u), G)
    assert rel(host(G), orc.step(u)) < 1e-12
    ctx.sp_set_base(dev(u))
    ds = np.stack([seeded(orc, 981 + i, 1.0) for i in range(3)])
    tol = 1e-12 if prec == 0 else 1e-5
    ctx.sp_jvp(dev(ds), J)
    for i in range(3):
        assert rel(host(J)[i], orc.jvp(base, ds[i])) < tol
    ctx.sp_vjp(dev(ds), J)
    for i in range(3):
        assert rel(host(J)[i], orc.vjp(base, ds[i])) < tol
    ctx.sp_set_base_n(dev(u), 2)  # trajectory slots of the base fields
    ctx.sp_jvp_n(dev(ds), J)
    assert close(host(J)[2], jvp_n(orc, u, 2, ds[2]), ds[2], tol)


MEMBERS = [dict(nx=128, ny=9, nz=4, re=300.0), dict(nx=96, ny=9, nz=96, re=300.0), dict(nx=16, ny=17, nz=16, re=250.0),
           dict(nx=18, ny=9, nz=24, re=400.0), dict(nx=6, ny=9, nz=162, re=300.0)]


@pytest.mark.parametrize("prec", [0, 1])
def test_group(prec):
    g, orcs = make_group(prec, MEMBERS)
    U, states = seed_group(g, orcs, 9900, 0.1)
    D, dirs = seed_group(g, orcs, 9950, 1.0)
    G, J = g.zeros(), g.zeros()
    g.sp_group_step(U, G)
    g.sp_group_set_base(U)
    g.sp_group_jvp(D, J)
    for i, (m, orc) in enumerate(zip(g.members, orcs)):
        step, tan = host(g.member_view(G, i)), host(g.member_view(J, i))
        assert rel(step, orc.step(states[i])) < 1e-12
        assert rel(tan, orc.jvp(orc.base(states[i]), dirs[i])) < (1e-12 if prec == 0 else 1e-5)
        own = m.zeros()
        m.sp_step(g.member_view(U, i).contiguous(), own)
        assert np.array_equal(step, host(own))
        m.sp_set_base(g.member_view(U, i).contiguous())
        m.sp_jvp(g.member_view(D, i).contiguous(), own)
        assert np.array_equal(tan, host(own))


@pytest.mark.parametrize("prec", [0, 1])
def test_group_with_inactive_members(prec):
    """Members that start at the root, laminar flow, are inactive from the first iteration and stay there; the
    others' residuals fall, and are those of the oracle at the returned states (1e-10 of states of order 1)."""
    g, orcs = make_group(prec, MEMBERS)
    U, states = seed_group(g, orcs, 9970, 0.01)
    for i in (1, 3):
        g.member_view(U, i).zero_()
    _, reps = g.sp_group_newton_gmres(U, max_newton=3, max_krylov=100, tol=1e-10)
    for i, (r, orc) in enumerate(zip(reps, orcs)):
        u = host(g.member_view(U, i))
        if i in (1, 3):
            assert r["norm_F"] == 0.0 and np.all(u == 0.0)
            continue
        norm = orc.norm(orc.step(u))
        assert abs(norm - r["norm_F"]) < 1e-10
        assert norm < orc.norm(orc.step(states[i]))
