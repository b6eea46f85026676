"""The calls whose speed this library answers for: what a Newton-GMRES, continuation or
spectrum computation spends its time on, each through the public binding.

A case is a dict of plain values. ``kind`` says which call it is:

  step     sp_step: one BEFE step G(U) (the Newton residual, a hookstep trial)
  jvp      sp_jvp on ``n_dir`` directions; ``rebase``: with a new linearisation point each time
  grad     StokesStep forward and backward (the step, then the adjoint on an incoming gradient)
  group    sp_group_set_base + sp_group_jvp over uneven members (a parameter continuation)
  pstep    pipe: sp_step at a travelling-wave guess
  pjvp     pipe: sp_jvp on ``n_dir`` directions, speed component included
  newton   sp_newton_gmres: one Newton step with ``krylov`` Arnoldi columns

``exact`` restates the maps in plain torch, 64 bits: Fourier transforms by torch.fft, the
Chebyshev-tau (pipe: finite-difference) systems of every Fourier mode by dense LU.
"""
import math

import numpy as np
import torch

import paper_1804_05087_gb300 as sp

LX, LZ = 2 * math.pi / 1.14, 2 * math.pi / 2.5
GROUP_GRIDS = ((24, 33, 24), (32, 49, 32), (48, 65, 48), (64, 65, 64))


# ------------------------------------------------------------------ the cases
def _couette(name, kind, nx, ny, nz, prec, **kw):
    c = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, prec=prec, re=400.0, dt=100.0, box=1.0, lam_adv=0,
             n_dir=1, rebase=False)
    c.update(kw)
    return c


def _pipe(name, kind, prec, **kw):
    c = dict(name=name, kind=kind, prec=prec, nr=64, mt=12, kz=24, ntheta=48, nz=96, alpha=1.25, re=2500.0, dt=50.0,
             n_dir=1)
    c.update(kw)
    return c


def listed():
    return [
        # the inner loop of Newton-GMRES on the small grid: one Jacobian action of a Krylov vector
        _couette("krylov_fp64_16", "jvp", 16, 33, 16, "fp64"),
        # the same at the production grid, mixed precision as inexact Newton runs it
        _couette("krylov_mixed_48", "jvp", 48, 65, 48, "mixed"),
        # a Newton residual or hookstep trial at the production grid (always FP64)
        _couette("step_48", "step", 48, 65, 48, "fp64"),
        # many tangents at one linearisation point (the headline workload), both precisions
        _couette("tangents_fp64_48", "jvp", 48, 65, 48, "fp64", n_dir=256, rebase=True),
        _couette("tangents_mixed_48", "jvp", 48, 65, 48, "mixed", n_dir=256, rebase=True),
        # a block of tangents on an uneven, non-square grid (dense spectra, block Krylov methods)
        _couette("tangents_fp64_ragged", "jvp", 36, 45, 24, "fp64", n_dir=37, re=250.0, dt=10.0),
        # laminar advection in the implicit operator, the equilibrium searches' setting
        _couette("lamadv_mixed_48x35", "jvp", 48, 35, 48, "mixed", n_dir=16, lam_adv=1, re=380.0),
        # gradient of an objective of G(U) through torch.autograd on the large box
        _couette("grad_mixed_96", "grad", 96, 97, 96, "mixed", re=1000.0, box=2.0),
        # lock-step continuation: 64 problems on uneven grids, one Arnoldi action each
        dict(name="continuation_64", kind="group", prec="mixed", members=64, largest=3, re_lo=200.0, re_hi=1000.0,
             dt=100.0),
        # pipe flow: the residual of the travelling-wave search, and a block of mixed tangents
        _pipe("pipe_step", "pstep", "fp64"),
        _pipe("pipe_tangents_mixed", "pjvp", "mixed", n_dir=64),
        # one whole Newton step of the small problem: 100 Arnoldi columns, hookstep, update
        _couette("newton_16", "newton", 16, 33, 16, "fp64", krylov=100),
    ]


def draw(rng):
    kind = rng.choice(["jvp", "jvp", "jvp", "jvp", "step", "step", "grad", "group", "pstep", "pjvp", "newton"])
    prec = rng.choice(["fp64", "mixed"])

    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "group":
        return dict(kind=kind, prec=prec, members=rng.randint(8, 64), largest=rng.randint(1, 3),
                    re_lo=rng.choice([100.0, 200.0, 300.0]), re_hi=rng.choice([500.0, 800.0, 1000.0]),
                    dt=rng.choice([10.0, 50.0, 100.0]))
    if kind in ("pstep", "pjvp"):
        mt, kz = rng.randint(4, 12), rng.randint(6, 24)
        good = [n for n in (16, 18, 24, 32, 36, 48, 54, 64, 72, 96)]
        c = _pipe("", kind, "fp64" if kind == "pstep" else prec, nr=2 * rng.randint(16, 32), mt=mt, kz=kz,
                  ntheta=min(n for n in good if n >= 3 * mt + 1), nz=min(n for n in good if n >= 3 * kz + 1),
                  alpha=rng.choice([0.8, 1.25, 1.7]), re=round(rng.uniform(500, 3000), 1),
                  dt=rng.choice([10.0, 50.0, 100.0]), n_dir=1 if kind == "pstep" else spread(1, 64))
    else:
        lam = 1 if kind == "jvp" and rng.random() < 0.2 else 0
        sizes = [16, 18, 24, 32, 36, 48, 64]
        if kind in ("step", "grad"):
            sizes += [72, 96]
        if kind == "newton":
            sizes = [16, 18, 24]
        nx = rng.choice(sizes)
        nz = nx if rng.random() < 0.5 else rng.choice(sizes)
        ny = 2 * rng.randint(8, 20 if kind == "newton" else 40) + 1
        most = 256 * 48 * 65 * 48 // (nx * ny * nz * (4 if lam else 1))
        c = _couette("", kind, nx, ny, nz, "fp64" if kind == "step" else prec, re=round(rng.uniform(100, 1000), 1),
                     dt=rng.choice([1.0, 10.0, 100.0]), box=rng.choice([1.0, 1.0, 2.0]), lam_adv=lam)
        if kind == "jvp":
            c.update(n_dir=spread(1, min(256, most)), rebase=rng.random() < 0.5)
        if kind == "newton":
            c.update(krylov=rng.randint(20, 100))
    del c["name"]
    return c


# ------------------------------------------------------------------ grids
def _prec(case):
    return sp.SP_MIXED if case["prec"] == "mixed" else sp.SP_FP64


def _members(case):
    rng = np.random.default_rng(3000)
    out = []
    for _ in range(case["members"]):
        re = float(rng.uniform(case["re_lo"], case["re_hi"]))
        g = GROUP_GRIDS[int(rng.integers(0, 4)) % (case["largest"] + 1)]
        out.append(dict(nx=g[0], ny=g[1], nz=g[2], re=re, dt=case["dt"], box=1.0, lam_adv=0))
    return out


def _dims(c):
    kx, kz = (c["nx"] - 1) // 3, (c["nz"] - 1) // 3
    return kx, kz, 2 * kx + 1, kz + 1, c["ny"]


def _modes(kx):
    return torch.cat([torch.arange(0, kx + 1), torch.arange(-kx, 0)]).double().cuda()


def _waves(c):
    kx, kz, *_ = _dims(c)
    return _modes(kx) * (2 * math.pi / (LX * c["box"])), torch.arange(kz + 1).double().cuda() * (
        2 * math.pi / (LZ * c["box"]))


def _mirror(m):
    return [(-p) % m for p in range(m)]


def _sym(a):
    """Hermitian-consistent part: the half = 0 plane of [..., full, half, n]."""
    a = a.clone()
    p = a[..., :, 0, :]
    a[..., :, 0, :] = 0.5 * (p + p[..., _mirror(a.shape[-3]), :].conj())
    return a


def _weights(m):
    w = torch.full((m, 1), 2.0, dtype=torch.float64, device="cuda")
    w[0] = 1.0
    return w


def _norm(a):
    """Weighted coefficient norm of every state of [n, 3, full, half, n]."""
    return (_weights(a.shape[-2]) * a.abs() ** 2).sum(dim=(1, 2, 3, 4), keepdim=True).sqrt()


# ------------------------------------------------------------------ states
def _cheb(ny):
    n = ny - 1
    j = torch.arange(ny, dtype=torch.float64, device="cuda")
    k = torch.outer(j, j) % (2 * n)
    t = torch.cos(math.pi * k / n)                      # T_n(y_j)
    cb = torch.ones(ny, dtype=torch.float64, device="cuda")
    cb[0] = cb[n] = 2.0
    fwd = (2.0 / (n * cb))[:, None] * t.T / cb[None, :]  # values -> coefficients
    d = torch.zeros((ny, ny), dtype=torch.float64, device="cuda")
    for q in range(ny):
        d[q, q + 1::2] = 2.0 * j[q + 1::2]
    d[0] *= 0.5
    return t, fwd, d


def _cplx(shape, gen):
    return torch.complex(torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda"),
                         torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda"))


def _flow(c, n, amp, gen):
    """n divergence-free no-slip states of norm amp whose spectra decay as the workloads' do:
    10**(-n/8) in the Chebyshev degree, geometrically in the wavenumbers."""
    kx, kz, mx, mz, ny = _dims(c)
    t, fwd, d = _cheb(ny)
    k1, k3 = _waves(c)
    k1, k3 = k1[:, None, None], k3[None, :, None]
    fall = 10.0 ** (-torch.arange(ny, device="cuda") / 8.0) * torch.exp(
        -0.25 * (_modes(kx).abs()[:, None, None] + torch.arange(mz, device="cuda")[None, :, None]))
    y = torch.cos(math.pi * torch.arange(ny, dtype=torch.float64, device="cuda") / (ny - 1))
    a, b, m = (_cplx((n, mx, mz, ny), gen) * fall for _ in range(3))
    a[..., ny - 4:] = 0
    b[..., ny - 2:] = 0
    m[..., ny - 2:] = 0
    put = lambda coef, bump: ((coef @ t.T.to(coef.dtype)) * bump) @ fwd.T.to(coef.dtype)  # noqa: E731
    v, eta, mean = put(a, (1 - y * y) ** 2), put(b, 1 - y * y), put(m, 1 - y * y)
    k2 = k1 * k1 + k3 * k3
    k2[0, 0] = 1.0
    dv = v @ d.T.to(v.dtype)
    u = torch.stack([1j * (k1 * dv - k3 * eta) / k2, v, 1j * (k3 * dv + k1 * eta) / k2], dim=1)
    u[:, :, 0, 0] = 0
    u[:, 0, 0, 0] = eta[:, 0, 0].real.to(u.dtype)
    u[:, 2, 0, 0] = mean[:, 0, 0].real.to(u.dtype)
    u = _sym(u)
    return (u * (amp / _norm(u))).contiguous()


def _pipe_flow(c, n, amp, speed, gen):
    """n pipe states: axial streaks (1 - r^2) r^m and a divergence-free part from poloidal
    potentials (1 - r^2)^3 r^m p(r^2) in every mode, then the speed component."""
    mk, mt, nr = 2 * c["kz"] + 1, c["mt"] + 1, c["nr"]
    r = torch.cos(math.pi * torch.arange(nr, dtype=torch.float64, device="cuda") / (2 * nr - 1))
    m = 2.0 * torch.arange(mt, dtype=torch.float64, device="cuda")[None, :, None]
    k = (c["alpha"] * _modes(c["kz"]))[:, None, None]
    fall = torch.exp(-0.35 * (_modes(c["kz"]).abs()[:, None] + torch.arange(mt, device="cuda")[None, :]))
    u = torch.zeros((n, 3, mk, mt, nr), dtype=torch.complex128, device="cuda")
    for q in range(4):
        pol = (_cplx((n, mk, mt), gen) * fall * 2.0 ** -q)[..., None]
        for s, b in enumerate((1.0, -3.0, 3.0, -1.0)):
            e = m + 2 * q + 2 * s                                  # power of r of this term
            up = b * r ** (e - 1).clamp(min=0)
            low = b * (e * e - m * m) * r ** (e - 2).clamp(min=0)
            u[:, 0] += pol * (1j * k) * e * up
            u[:, 1] += pol * (-k * m) * up
            u[:, 2] -= pol * low
    u[:, :, 0] = 0
    u = _sym(u)
    u *= 0.1 / _norm(u)
    st = torch.zeros_like(u)
    st[:, 2, 0, 1:4] = torch.randn((n, 3, 1), generator=gen, dtype=torch.float64, device="cuda") * (1 - r * r) * r ** m[
        0, 1:4]
    u = (u + st / _norm(st)) * amp
    c0 = torch.full((n, 1), speed, dtype=torch.complex128, device="cuda")
    return torch.cat([u.reshape(n, -1), c0], dim=1).contiguous()


def _inputs(case, seed):
    """The tensors of one call: base state U and, where the call has them, directions."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    if kind == "group":
        mem = _members(case)
        return [_flow(c, 1, 0.1, gen)[0] for c in mem], [_flow(c, 1, 1.0, gen)[0] for c in mem]
    if kind in ("pstep", "pjvp"):
        u = _pipe_flow(case, 1, 0.05, 0.5, gen)[0]
        return u, _pipe_flow(case, case["n_dir"], 1.0, 0.1, gen) if kind == "pjvp" else None
    u = _flow(case, 1, 0.1, gen)[0]
    if kind == "jvp":
        return u, _flow(case, case["n_dir"], 1.0, gen)
    if kind == "grad":
        return u, _flow(case, 1, 1.0, gen)[0]
    return u, None


# ------------------------------------------------------------------ the calls
def _config(c, prec, batch):
    return sp.Config(c["nx"], c["ny"], c["nz"], lx=LX * c["box"], lz=LZ * c["box"], re=c["re"], dt=c["dt"], prec=prec,
                     max_batch=batch, lam_adv=c["lam_adv"])


def prepare(case, seed):
    kind, prec = case["kind"], _prec(case)
    U, X = _inputs(case, seed)
    s = {"case": case, "U": U, "X": X}
    if kind == "group":
        g = s["ctx"] = sp.Group([_config(c, prec, 1) for c in _members(case)])
        s["U"], s["X"], s["out"] = g.zeros(), g.zeros(), g.zeros()
        for i in range(g.n):
            g.member_view(s["U"], i).copy_(U[i])
            g.member_view(s["X"], i).copy_(X[i])
        return s
    if kind in ("pstep", "pjvp"):
        ctx = sp.Context(sp.PipeConfig(case["nr"], case["mt"], case["kz"], case["ntheta"], case["nz"], 2, case["alpha"],
                                       case["re"], case["dt"], prec, case["n_dir"]))
    else:
        ctx = sp.Context(_config(case, prec, case["n_dir"]))
    s["ctx"] = ctx
    s["out"] = ctx.zeros() if X is None else torch.zeros_like(X)
    if kind == "grad":
        s["U"] = U.requires_grad_(True)
    elif kind == "pjvp" or (kind == "jvp" and not case["rebase"]):
        ctx.sp_set_base(U)
    return s


def run(state):
    kind, ctx, U, X, out = state["case"]["kind"], state["ctx"], state["U"], state["X"], state["out"]
    if kind in ("step", "pstep"):
        return ctx.sp_step(U, out)
    if kind in ("jvp", "pjvp"):
        if state["case"].get("rebase"):
            ctx.sp_set_base(U)
        return ctx.sp_jvp(X, out)
    if kind == "grad":
        G = sp.StokesStep.apply(U, ctx)
        return {"G": G.detach(), "grad": torch.autograd.grad(G, U, X)[0]}
    if kind == "group":
        ctx.sp_group_set_base(U)
        return ctx.sp_group_jvp(X, out)
    V = out.copy_(U)  # the solver updates its guess in place
    rep = ctx.sp_newton_gmres(V, max_newton=1, max_krylov=state["case"]["krylov"])
    return {"U": V, "norm_F": rep["norm_F"], "actions": rep["total_jvps"]}


# ------------------------------------------------------------------ the work
def _couette_flops(c):
    """Flops of one step or tangent: nine plane transforms and the product at every wall-normal
    point, the Chebyshev transforms as fast transforms, a banded solve of each mode."""
    kx, kz, mx, mz, ny = _dims(c)
    grid = c["nx"] * c["nz"]
    return 9 * ny * 2.5 * grid * math.log2(grid) + 18 * ny * grid + 9 * mx * mz * 5 * ny * math.log2(
        ny) + 250 * mx * mz * ny


def work(case):
    kind = case["kind"]
    if kind == "group":
        mem = _members(case)
        states = sum(3 * m[2] * m[3] * m[4] * 16 for m in map(_dims, mem))
        return {"bytes": 3 * states, "flops": 2 * sum(map(_couette_flops, mem))}
    if kind in ("pstep", "pjvp"):
        mk, mt, nr = 2 * case["kz"] + 1, case["mt"] + 1, case["nr"]
        state = 3 * mk * mt * nr * 16 + 16
        grid = case["ntheta"] * case["nz"]
        one = 9 * nr * 2.5 * grid * math.log2(grid) + 18 * nr * grid + 1000 * mk * mt * nr
        return {"bytes": 2 * case["n_dir"] * state, "flops": case["n_dir"] * one}
    kx, kz, mx, mz, ny = _dims(case)
    state, one = 3 * mx * mz * ny * 16, _couette_flops(case)
    if kind == "step":
        return {"bytes": 2 * state, "flops": one}
    if kind == "grad":
        return {"bytes": 4 * state, "flops": 2 * one}
    if kind == "newton":  # every action reads and writes a state and is orthogonalised against the basis
        k = case["krylov"]
        return {"bytes": k * (k + 5) * state // 2, "flops": k * one + k * k * state / 4}
    again = 1 if case["rebase"] else 0
    return {"bytes": (2 * case["n_dir"] + again) * state, "flops": (case["n_dir"] + again) * one}


# ------------------------------------------------------------------ 64 bits
def _phys(a, nf, nh):
    """Fourier modes [..., full, half, n] -> real grid [..., n, nf, nh]."""
    k = a.shape[-3] // 2
    s = torch.zeros(a.shape[:-3] + (nf, nh // 2 + 1, a.shape[-1]), dtype=a.dtype, device=a.device)
    s[..., :k + 1, :a.shape[-2], :] = a[..., :k + 1, :, :]
    s[..., nf - k:, :a.shape[-2], :] = a[..., k + 1:, :, :]
    return torch.fft.irfft2(s.movedim(-1, -3), s=(nf, nh), norm="forward")


def _spec(f, k, mh):
    """Real grid [..., n, nf, nh] -> retained modes [..., 2k+1, mh, n]."""
    s = torch.fft.rfft2(f, norm="forward")[..., :mh].movedim(-3, -1)
    return torch.cat([s[..., :k + 1, :, :], s[..., s.shape[-3] - k:, :, :]], dim=-3)


def _cross(a, b):
    a, b = a.unbind(-4), b.unbind(-4)
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]], dim=-4)


class _Couette:
    """Plane Couette maps on batches of states [n, 3, MX, MZ, NY]."""

    def __init__(self, c):
        self.c = c
        self.kx, self.kz, self.mx, self.mz, self.ny = _dims(c)
        self.t, self.fwd, self.d = (m.to(torch.complex128) for m in _cheb(c["ny"]))
        k1, k3 = _waves(c)
        self.k1, self.k3 = k1, k3
        self.ik1, self.ik3 = 1j * k1[:, None, None], 1j * k3[None, :, None]
        self.y = torch.cos(math.pi * torch.arange(self.ny, dtype=torch.float64, device="cuda") / (self.ny - 1))

    def fields(self, a):
        u, v, w = a.unbind(1)
        du, dw = u @ self.d.T, w @ self.d.T
        six = torch.stack([u, v, w, dw - self.ik3 * v, self.ik3 * u - self.ik1 * w, self.ik1 * v - du], dim=1)
        return _phys(six @ self.t.T, self.c["nx"], self.c["nz"])

    def total(self, u):
        f = self.fields(_sym(u)[None])
        f[:, 0] += self.y[:, None, None]
        f[:, 5] -= 1.0
        return f

    def shifted(self):
        """Multiplication by y on Chebyshev coefficients (degrees above N dropped)."""
        n = self.ny
        s = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
        for q in range(1, n):
            s[q - 1, q] = 0.5
            s[q, q - 1] = 0.5 if q > 1 else 1.0
        return s

    def systems(self, pos, iz):
        """Dense tau systems of the modes (pos[i], iz[i]): unknowns u, v, w, p."""
        c, n1 = self.c, self.ny
        kx, kz = self.k1[pos][:, None, None], self.k3[iz][:, None, None]
        nu, eye = 1.0 / c["re"], torch.eye(n1, dtype=torch.complex128, device="cuda")
        h = (1.0 / c["dt"] + nu * (kx * kx + kz * kz)) * eye - nu * (self.d @ self.d)
        if c["lam_adv"]:
            h = h + 1j * kx * self.shifted()
        a = torch.zeros((len(pos), 4 * n1, 4 * n1), dtype=torch.complex128, device="cuda")
        m = n1 - 2
        for i, g in enumerate((1j * kx * eye, self.d.expand(len(pos), n1, n1), 1j * kz * eye)):
            a[:, i * m:(i + 1) * m, i * n1:(i + 1) * n1] = h[:, :m]
            a[:, i * m:(i + 1) * m, 3 * n1:] = g[:, :m]
            a[:, 3 * m + 2 * i, i * n1:(i + 1) * n1] = 1.0
            a[:, 3 * m + 2 * i + 1, i * n1:(i + 1) * n1:2] = 1.0
            a[:, 3 * m + 2 * i + 1, i * n1 + 1:(i + 1) * n1:2] = -1.0
            a[:, 3 * n1:, i * n1:(i + 1) * n1] = g if i != 1 else self.d
        if c["lam_adv"]:
            a[:, :m, n1:2 * n1] += eye[:m]
        return a

    def mean(self):
        n1, nu = self.ny, 1.0 / self.c["re"]
        a = torch.eye(n1, dtype=torch.complex128, device="cuda") / self.c["dt"] - nu * (self.d @ self.d)
        a[n1 - 2] = 1.0
        a[n1 - 1] = torch.tensor([(-1.0) ** q for q in range(n1)], device="cuda")
        return a

    def solve(self, f, adjoint=False):
        """Per-mode solves (or their conjugate transposes) for right-hand sides [n, 3, MX, MZ, NY].
        Without laminar advection the modes +-ix share a matrix up to the sign of u."""
        n, n1, m = f.shape[0], self.ny, self.ny - 2
        out = torch.zeros_like(f)
        fold = not self.c["lam_adv"]
        todo = [(p, i) for p in range(self.kx + 1 if fold else self.mx) for i in range(self.mz) if p or i]
        for at in range(0, len(todo), 256):
            pos, iz = (torch.tensor(v, device="cuda") for v in zip(*todo[at:at + 256]))
            sides = [(pos, 1.0)] + ([((self.mx - pos) % self.mx, -1.0)] if fold else [])
            rhs = []
            for q, sign in sides:
                g = f[:, :, q, iz].clone()                       # [n, 3, modes, NY]
                g[:, 0] *= sign
                full = torch.zeros((len(pos), 4 * n1, n), dtype=f.dtype, device="cuda")
                cols = (n1 if adjoint else m)
                full[:, :3 * cols] = g[..., :cols].permute(2, 1, 3, 0).reshape(len(pos), 3 * cols, n)
                rhs.append(full)
            a = self.systems(pos, iz)
            x = torch.linalg.solve(a.mH if adjoint else a, torch.cat(rhs, dim=2))
            for k, (q, sign) in enumerate(sides):
                rows = m if adjoint else n1
                g = x[:, :3 * rows, k * n:(k + 1) * n].reshape(len(pos), 3, rows, n).permute(3, 1, 0, 2).clone()
                g[:, 0] *= sign
                out[:, :, q, iz, :rows] = g
        a = self.mean()
        for comp in (0, 2):
            if adjoint:
                out[:, comp, 0, 0, :m] = torch.linalg.solve(a.mH, f[:, comp, 0, 0].T).T[:, :m]
            else:
                g = torch.zeros_like(f[:, comp, 0, 0])
                g[:, :m] = f[:, comp, 0, 0, :m]
                out[:, comp, 0, 0] = torch.linalg.solve(a, g.T).T
        return out

    def finish(self, a, prod):
        rhs = a / self.c["dt"] + _spec(prod, self.kx, self.mz) @ self.fwd.T
        if self.c["lam_adv"]:
            adv = self.ik1 * (a @ self.shifted().T)
            adv[:, 0] += a[:, 1]
            rhs = rhs + adv
        return _sym(self.solve(rhs) - a)

    def step(self, u):
        f = self.total(u)
        return self.finish(_sym(u)[None], _cross(f[:, :3], f[:, 3:]))[0]

    def jvp(self, u, x):
        base, out = self.total(u), []
        for at in range(0, x.shape[0], 64):
            a = _sym(x[at:at + 64])
            g = self.fields(a)
            out.append(self.finish(a, _cross(base[:, :3].expand_as(g[:, :3]), g[:, 3:]) + _cross(
                g[:, :3], base[:, 3:].expand_as(g[:, 3:]))))
        return torch.cat(out)

    def vjp(self, u, r):
        """Transpose of jvp in the plain inner product of the stored real and imaginary parts."""
        base, w = self.total(u), _weights(self.mz)
        rw = _sym(r[None])
        gs = self.solve(rw, adjoint=True)
        a = _phys((gs @ self.fwd) * (1.0 / w), self.c["nx"], self.c["nz"]) / (self.c["nx"] * self.c["nz"])
        six = torch.cat([_cross(base[:, 3:], a), _cross(a, base[:, :3])], dim=1)
        six = _spec(six, self.kx, self.mz) * (self.c["nx"] * self.c["nz"]) * w @ self.t
        gu, gv, gw, gx, gy, gz = six.unbind(1)
        m = torch.stack([gu - self.ik3 * gy - gz @ self.d, gv + self.ik3 * gx - self.ik1 * gz,
                         gw + gx @ self.d + self.ik1 * gy], dim=1)
        return (_sym(gs / self.c["dt"] + m) - rw)[0]


class _Pipe:
    """Pipe maps on batches of flat states (field [3, 2kz+1, mt+1, nr], then the speed)."""

    def __init__(self, c):
        self.c, nr = c, c["nr"]
        self.mk, self.mt = 2 * c["kz"] + 1, c["mt"] + 1
        self.k, self.m = c["alpha"] * _modes(c["kz"]), 2.0 * torch.arange(self.mt).double().cuda()
        r = np.cos(np.pi * np.arange(nr) / (2 * nr - 1))
        pts = np.concatenate([r, -r])
        der = np.zeros((2, 2, nr, nr))                            # [parity][order - 1]
        for i in range(nr):
            near = np.argsort(np.abs(pts - r[i]), kind="stable")[:9]
            h = np.max(np.abs(pts[near] - r[i]))
            van = np.linalg.inv(np.vander((pts[near] - r[i]) / h, 9, increasing=True).T)
            for o in (1, 2):
                for q, wt in zip(near, van[:, o] * math.factorial(o) / h ** o):
                    der[0, o - 1, i, q % nr] += wt
                    der[1, o - 1, i, q % nr] += wt if q < nr else -wt
        self.der = torch.from_numpy(der).cuda()
        self.r = torch.from_numpy(r).cuda()
        self.nu = 1.0 / c["re"]

    def split(self, s):
        shape = (s.shape[0], 3, self.mk, self.mt, self.c["nr"])
        return _sym(s[:, :-1].reshape(shape)), s[:, -1].real

    def d1(self, f, shift):
        par = (self.m.long() + shift) % 2                         # even m: every mode has the same parity
        return f @ self.der[int(par[0]), 0].T.to(f.dtype)

    def fields(self, a):
        ur, ut, uz = a.unbind(1)
        im, ik, r = 1j * self.m[None, :, None], 1j * self.k[:, None, None], self.r
        six = torch.stack([ur, ut, uz, im / r * uz - ik * ut, ik * ur - self.d1(uz, 0),
                           self.d1(ut, 1) + ut / r - im / r * ur], dim=1)
        return _phys(six, self.c["nz"], self.c["ntheta"])

    def total(self, a):
        f = self.fields(a)
        f[:, 2] += (1 - self.r ** 2)[:, None, None]
        f[:, 4] += (2 * self.r)[:, None, None]
        return f

    def lap(self, q, k, par):
        eye = torch.eye(self.c["nr"], dtype=torch.float64, device="cuda")
        d1, d2 = self.der[par]
        return d2 + d1 / self.r[:, None] - eye * ((q * q)[:, None, None] / self.r ** 2 + (k * k)[:, None, None])

    def solve(self, f):
        nr, n, lam = self.c["nr"], f.shape[0], 1.0 / self.c["dt"]
        r, eye = self.r, torch.eye(nr, dtype=torch.complex128, device="cuda")
        out = torch.zeros_like(f)
        todo = [(p, q) for p in range(self.mk) for q in range(self.mt) if p or q]
        for at in range(0, len(todo), 256):
            pos, half = (torch.tensor(v, device="cuda") for v in zip(*todo[at:at + 256]))
            m, k = self.m[half], self.k[pos]
            mm, kk, b = m[:, None, None].to(f.dtype), k[:, None, None].to(f.dtype), len(pos)
            dp, du = self.der[0, 0].to(f.dtype), self.der[1, 0].to(f.dtype)
            a = torch.zeros((b, 4 * nr, 4 * nr), dtype=f.dtype, device="cuda")
            grads = (dp - mm / r * eye, dp + mm / r * eye, 1j * kk * eye)
            for i, (q, par) in enumerate(((m + 1, 1), (m - 1, 1), (m, 0))):
                h = lam * eye - self.nu * self.lap(q, k, par)
                a[:, i * nr + 1:(i + 1) * nr, i * nr:(i + 1) * nr] = h[:, 1:]
                a[:, i * nr + 1:(i + 1) * nr, 3 * nr:] = grads[i].expand(b, nr, nr)[:, 1:]
                a[:, i * nr, i * nr] = 1.0
            a[:, 3 * nr + 1:, 3 * nr:] = self.lap(m, k, 0)[:, 1:].to(f.dtype)
            div = torch.cat([0.5 * (du + (1 + mm) / r * eye), 0.5 * (du + (1 - mm) / r * eye),
                             (1j * kk * eye).expand(b, nr, nr)], dim=2)
            a[:, 3 * nr, :3 * nr] = div[:, 0]
            g = f[:, :, pos, half].permute(2, 1, 3, 0)            # [modes, 3, nr, n]
            g = torch.stack([g[:, 0] + 1j * g[:, 1], g[:, 0] - 1j * g[:, 1], g[:, 2]], dim=1)
            rhs = torch.cat([g.reshape(b, 3 * nr, n), div @ g.reshape(b, 3 * nr, n)], dim=1)
            rhs[:, ::nr] = 0
            x = torch.linalg.solve(a, rhs)[:, :3 * nr].reshape(b, 3, nr, n)
            x = torch.stack([0.5 * (x[:, 0] + x[:, 1]), (x[:, 0] - x[:, 1]) / 2j, x[:, 2]], dim=1)
            out[:, :, pos, half] = x.permute(3, 1, 0, 2)
        for comp, q, par in ((1, 1.0, 1), (2, 0.0, 0)):
            z = torch.zeros(1, dtype=torch.float64, device="cuda")
            h = lam * eye - self.nu * self.lap(z + q, z, par)[0]
            h[0] = 0
            h[0, 0] = 1.0
            g = f[:, comp, 0, 0].clone()
            g[:, 0] = 0
            out[:, comp, 0, 0] = torch.linalg.solve(h, g.T).T
        return out

    def finish(self, a, prod, extra):
        rhs = a / self.c["dt"] + _spec(prod, self.c["kz"], self.mt) + extra
        return _sym(self.solve(rhs) - a)

    def ddz(self, a):
        return 1j * self.k[:, None, None] * a

    def flat(self, g, last):
        return torch.cat([g.reshape(g.shape[0], -1), last.to(g.dtype).reshape(-1, 1)], dim=1)

    def step(self, s):
        a, speed = self.split(s[None])
        f = self.total(a)
        return self.flat(self.finish(a, _cross(f[:, :3], f[:, 3:]), speed * self.ddz(a)), speed * 0)[0]

    def jvp(self, s, x):
        u, speed = self.split(s[None])
        a, ds = self.split(x)
        base, g = self.total(u), self.fields(a)
        prod = _cross(base[:, :3].expand_as(g[:, :3]), g[:, 3:]) + _cross(g[:, :3], base[:, 3:].expand_as(g[:, 3:]))
        out = self.finish(a, prod, speed * self.ddz(a) + ds[:, None, None, None, None] * self.ddz(u))
        phase = (_weights(self.mt) * (self.ddz(u).conj() * a).real).sum(dim=(1, 2, 3, 4))
        return self.flat(out, phase)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("group", "newton"):  # tens of thousands of dense systems; a path of many steps
        return None
    U, X = _inputs(case, seed)
    if kind in ("pstep", "pjvp"):
        p = _Pipe(case)
        return p.step(U) if kind == "pstep" else p.jvp(U, X)
    c = _Couette(case)
    if kind == "step":
        return c.step(U)
    if kind == "jvp":
        return c.jvp(U, X)
    return {"G": c.step(U), "grad": c.vjp(U, X)}
