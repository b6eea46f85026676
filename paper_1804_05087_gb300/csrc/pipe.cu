// Kernels of the pipe-flow step and tangent (the plane stage is k_xz of
// kernels.cu with the pipe's laminar table).
//   k_pvals : per Fourier mode, the six fields u_r, u_theta, u_z and the
//             vorticity at every radial point: omega_r = (i m/r) u_z - i k u_theta,
//             omega_theta = i k u_r - D1 u_z, omega_z = D1 u_theta + u_theta/r - (i m/r) u_r
//             (radial derivatives by the 9-point parity-aware stencils),
//             written plane-major (one radial point per plane).
//   k_psolve: per Fourier mode, the right-hand side u/dt + N + c du/dz (for the
//             tangent + dc dU/dz), rotation to u+- = u_r +- i u_theta and
//             u~_z = -i u_z, the per-mode Stokes problem by banded solves and one
//             influence coefficient (FP64), and G = u_new - u with a Hermitian output.
// Index conventions: position pos over the axial wavenumbers in FFT order
// (k = alpha kz), iz = m' (m = sym m').
#include "dev_util.h"
#include "sp_internal.h"

namespace {

constexpr int kTileP = 8;        // modes per k_pvals block
constexpr int kThreadsP = 256;

struct PArgs {
  const double* r;      // [NR], then the reciprocals [NR] (a division takes the FP64 pipe tenfold)
  const double* w1;     // [2][NR][9]
  const int* c1;        // [2][NR][9]
  const unsigned char* pb_fac;  // banded factors of the per-mode radial problems (plan_pipe.cpp)
  size_t pb_chunk;
  const double* pb_uh;  // [n_unique][3][NR]
  const double* pb_dinv;
  size_t sstride;       // complex values per state (field + speed)
  int Mm, MX, MZ, Kx, NR, n_unique, sms;
  double alpha, sym, inv_dt;
};

template <typename T>
__device__ __forceinline__ C2<T> cmk(double2 v) { return mk((T)v.x, (T)v.y); }

template <typename T>
__global__ void __launch_bounds__(kThreadsP) k_pvals(const double2* __restrict__ in, C2<T>* __restrict__ out,
                                                     PArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* su = reinterpret_cast<double2*>(smem_raw);  // [3][TM][NR]
  const int TM = kTileP, NR = a.NR, Mm = a.Mm;
  const int m0 = blockIdx.x * TM, dir = blockIdx.y;
  const double2* src = in + (size_t)dir * a.sstride;
  for (int idx = threadIdx.x; idx < 3 * TM * NR; idx += blockDim.x) {
    const int j = idx % NR, t = (idx / NR) % TM, c = idx / (NR * TM);
    const int m = m0 + t;
    su[idx] = m < Mm ? __ldg(src + ((size_t)c * Mm + m) * NR + j) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  C2<T>* o = out + (size_t)dir * 6 * NR * Mm;
  for (int idx = threadIdx.x; idx < TM * NR; idx += blockDim.x) {
    const int t = idx % TM, j = idx / TM;
    const int m = m0 + t;
    if (m >= Mm) continue;
    const int pos = m / a.MZ, iz = m - pos * a.MZ;
    const int kzi = pos <= a.Kx ? pos : pos - a.MX;
    const double k = a.alpha * kzi, mm = a.sym * iz;
    const double ir = __ldg(a.r + NR + j);
    const double2* ur = su + (0 * TM + t) * NR;
    const double2* ut = su + (1 * TM + t) * NR;
    const double2* uz = su + (2 * TM + t) * NR;
    // D1 of u_z (parity of m) and of u_theta (parity of m + 1)
    const int pz = ((int)mm) & 1, pt = pz ^ 1;
    double2 dz = make_double2(0.0, 0.0), dt = dz;
    for (int q = 0; q < 9; ++q) {
      const double wz = __ldg(a.w1 + ((size_t)pz * NR + j) * 9 + q);
      const int cz = __ldg(a.c1 + ((size_t)pz * NR + j) * 9 + q);
      const double wt = __ldg(a.w1 + ((size_t)pt * NR + j) * 9 + q);
      const int ct = __ldg(a.c1 + ((size_t)pt * NR + j) * 9 + q);
      dz.x += wz * uz[cz].x;
      dz.y += wz * uz[cz].y;
      dt.x += wt * ut[ct].x;
      dt.y += wt * ut[ct].y;
    }
    const double2 vr = ur[j], vt = ut[j], vz = uz[j];
    // i m/r u_z - i k u_theta
    const double2 orr = make_double2(-mm * ir * vz.y + k * vt.y, mm * ir * vz.x - k * vt.x);
    // i k u_r - D1 u_z
    const double2 ot = make_double2(-k * vr.y - dz.x, k * vr.x - dz.y);
    // D1 u_theta + u_theta/r - i m/r u_r
    const double2 oz = make_double2(dt.x + vt.x * ir + mm * ir * vr.y, dt.y + vt.y * ir - mm * ir * vr.x);
    const size_t base = (size_t)j * Mm + m;
    o[0 * (size_t)NR * Mm + base] = cmk<T>(vr);
    o[1 * (size_t)NR * Mm + base] = cmk<T>(vt);
    o[2 * (size_t)NR * Mm + base] = cmk<T>(vz);
    o[3 * (size_t)NR * Mm + base] = cmk<T>(orr);
    o[4 * (size_t)NR * Mm + base] = cmk<T>(ot);
    o[5 * (size_t)NR * Mm + base] = cmk<T>(oz);
  }
}

// Hermitian projection of entry (c, pos, iz, j) of a state
__device__ __forceinline__ double2 sym_load(const double2* s, int c, int pos, int iz, int j, const PArgs& a) {
  double2 v = __ldg(s + ((size_t)c * a.Mm + pos * a.MZ + iz) * a.NR + j);
  if (iz == 0) v = project(v, __ldg(s + ((size_t)c * a.Mm + (pos == 0 ? 0 : a.MX - pos) * a.MZ) * a.NR + j));
  return v;
}

// Banded solve of one real right-hand side in place (b: every second double, the real or the
// imaginary part of a complex vector in shared memory), with one matrix's factors from
// plan_pipe.cpp staged in shared memory: row interchanges and multipliers forward, then the upper
// band backward (two partial sums per row). NR > 0: the vector is held in registers and the loops
// are unrolled (the row interchange of step k is a select among rows k .. k + KL); NR = 0: any
// size, the vector stays in shared memory.
// (the unrolled form is one out-of-line function shared by every kernel that uses it)
template <int NR>
__device__ __noinline__ void band_solve_reg(double* b, const unsigned char* fac) {
  constexpr int KL = kPipeKL, KW = kPipeKW;
  const double* U = reinterpret_cast<const double*>(fac);
  const double* L = U + (size_t)NR * KW;
  const int* piv = reinterpret_cast<const int*>(L + (size_t)NR * KL);
  {
    double x[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) x[i] = b[2 * i];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      const int p = piv[k];
      double xk = x[k];
#pragma unroll
      for (int q = 1; q <= KL; ++q) {
        if (k + q < NR) {
          const bool sw = p == k + q;
          const double t = x[k + q];
          x[k + q] = sw ? x[k] : t;
          xk = sw ? t : xk;
        }
      }
      x[k] = xk;
#pragma unroll
      for (int q = 0; q < KL; ++q)
        if (k + 1 + q < NR) x[k + 1 + q] = fma(-L[k * KL + q], xk, x[k + 1 + q]);
    }
#pragma unroll
    for (int i = NR - 1; i >= 0; --i) {
      double s0 = x[i], s1 = 0.0;
#pragma unroll
      for (int q = 1; q < KW; ++q) {
        if (i + q < NR) {
          if (q & 1) s1 = fma(-U[i * KW + q], x[i + q], s1);
          else s0 = fma(-U[i * KW + q], x[i + q], s0);
        }
      }
      x[i] = (s0 + s1) * U[i * KW];
    }
#pragma unroll
    for (int i = 0; i < NR; ++i) b[2 * i] = x[i];
  }
}

template <int NR>
__device__ __forceinline__ void band_solve_d(double* b, const unsigned char* fac, int n) {
  constexpr int KL = kPipeKL, KW = kPipeKW;
  const double* U = reinterpret_cast<const double*>(fac);
  const double* L = U + (size_t)n * KW;
  const int* piv = reinterpret_cast<const int*>(L + (size_t)n * KL);
  if constexpr (NR > 0) {
    band_solve_reg<NR>(b, fac);
  } else {
    for (int k = 0; k < n; ++k) {
      const int p = piv[k];
      double bk = b[2 * k];
      if (p != k) {
        const double t = b[2 * p];
        b[2 * p] = bk;
        bk = t;
        b[2 * k] = bk;
      }
#pragma unroll
      for (int q = 0; q < KL; ++q)
        if (k + 1 + q < n) b[2 * (k + 1 + q)] -= L[k * KL + q] * bk;
    }
    for (int i = n - 1; i >= 0; --i) {
      double s0 = b[2 * i], s1 = 0.0;
#pragma unroll
      for (int q = 1; q < KW; ++q) {
        if (i + q < n) {
          if (q & 1) s1 = fma(-U[i * KW + q], b[2 * (i + q)], s1);
          else s0 = fma(-U[i * KW + q], b[2 * (i + q)], s0);
        }
      }
      b[2 * i] = (s0 + s1) * U[i * KW];
    }
  }
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// bounded wait on an mbarrier phase; false if the limit ran out
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t phase) {
  for (uint32_t it = 0; it < (1u << 26); ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Shared-memory vectors are NRP >= NR entries apart, NRP = 1 mod 8: the 16 vectors that the 32 lanes
// of a warp walk through (two lanes, real and imaginary part, per vector) then start 4 banks apart
// and a warp's 8-byte accesses take the minimum two wavefronts.
__host__ __device__ __forceinline__ int psolve_nrp(int NR) { return NR + ((9 - (NR & 7)) & 7); }

// Warps of a block. ND = 16: the velocity chains of 16 directions fill three warps, the pressure
// chains the fourth, so every scheduler's FP64 unit has one full warp of chains; ND = 1: two, for
// the parallel phases (one of them runs the chains).
__host__ __device__ constexpr int psolve_warps(int ND) { return ND >= 8 ? 4 : 2; }
__host__ __device__ constexpr int psolve_threads(int ND) { return 32 * psolve_warps(ND); }

__host__ __device__ __forceinline__ size_t psolve_smem(int ND, int NR, size_t chunk) {
  return 3 * chunk + (size_t)ND * 4 * psolve_nrp(NR) * 16;
}

// one bulk copy of a matrix's factors
__device__ __forceinline__ void copy_factor(unsigned char* dst, const unsigned char* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void expect_bytes(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// in3: [dir][3][NR][Mm] values of N (T); u: the states (step: the state itself, tangent: the
// directions); U0: the base state (tangent only); out: states. One block: one mode of ND directions.
// The Stokes problem of the mode is solved by banded solves (plan_pipe.cpp): the pressure p_f (Poisson,
// wall value zero), the three velocity components driven by f - grad p_f, and the influence
// coefficient a of the precomputed u_h from the wall continuity row. The stencil work (div_h f,
// grad p) runs over all threads, row by row in parallel; only the banded substitutions are serial,
// one thread per (direction, component, real/imaginary part), packed into as few warps as they fill:
// a scheduler's FP64 unit takes 64 cycles per instruction whatever the lanes, and a row costs about
// 20 of them. The factors come into shared memory by bulk TMA copies, u+ and u- beside the pressure's,
// u~z in the pressure's place once that is solved: three matrices instead of four, so that all modes of a
// single direction run at once (613 modes at Nr = 64; with two modes per block the last three blocks ran
// a second wave, 280 us). Every wait has an iteration limit, past which the block writes NaN.
template <typename T, bool TANGENT, int ND, int NRT>
__global__ void __launch_bounds__(psolve_threads(ND)) k_psolve(const C2<T>* __restrict__ in3,
                                                               const double2* __restrict__ u,
                                                               const double2* __restrict__ U0,
                                                               double2* __restrict__ out, PArgs a, int n_dir) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int NR = NRT > 0 ? NRT : a.NR, Mm = a.Mm, NRP = psolve_nrp(NR), n3 = 3 * NRP;
  const size_t chunk = a.pb_chunk;
  unsigned char* sfac = smem_raw;                                         // [3][chunk]: p then u~z, u+, u-
  double2* sf = reinterpret_cast<double2*>(smem_raw + 3 * chunk);         // [ND][3][NRP]
  double2* sp = sf + ND * n3;                                             // [ND][NRP] pressure
  __shared__ double s_alpha[ND][2];
  __shared__ __align__(8) uint64_t s_bar;
  const int mode = blockIdx.x, d0 = blockIdx.y * ND, nd = min(ND, n_dir - d0);
  const int tid = threadIdx.x, nt = blockDim.x;
  const uint32_t bar = smem_addr(&s_bar);
  int pos, iz;
  unique_mode(mode, a.Kx, a.MZ, &pos, &iz);
  const bool mean = pos == 0 && iz == 0;
  const int kzi = pos <= a.Kx ? pos : pos - a.MX;
  const double k = a.alpha * kzi, mm = a.sym * iz;
  const int pz = ((int)mm) & 1, pe = pz ^ 1;  // parity of u_z and p, of u_r and u_theta
  const double* wz = a.w1 + (size_t)pz * NR * 9;
  const double* we = a.w1 + (size_t)pe * NR * 9;
  const int* cz = a.c1 + (size_t)pz * NR * 9;
  const int* ce = a.c1 + (size_t)pe * NR * 9;
  const unsigned char* fac = a.pb_fac + (size_t)mode * 4 * chunk;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    expect_bytes(bar, (uint32_t)(3 * chunk));
    for (int q = 0; q < 3; ++q) copy_factor(sfac + q * chunk, fac + q * chunk, (uint32_t)chunk, bar);
  }
  // f = u/dt + N + speed terms, rotated to (f+, f-, f~z) = (f_r + i f_theta, f_r - i f_theta, -i f_z)
  for (int idx = tid; idx < nd * NR; idx += nt) {
    const int d = idx / NR, j = idx - d * NR, dir = d0 + d;
    const double2* us = u + (size_t)dir * a.sstride;
    const C2<T>* vin = in3 + (size_t)dir * 3 * NR * Mm;
    // speed terms: step c du/dz; tangent c0 du/dz + dc dU0/dz
    const double c_eff = TANGENT ? __ldg(U0 + a.sstride - 1).x : __ldg(us + a.sstride - 1).x;
    const double dc = TANGENT ? __ldg(us + a.sstride - 1).x : 0.0;
    double2 f[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 v = sym_load(us, c, pos, iz, j, a);
      const C2<T> nv = vin[((size_t)c * NR + j) * Mm + pos * a.MZ + iz];
      f[c] = make_double2(v.x * a.inv_dt + (double)nv.x - c_eff * k * v.y,
                          v.y * a.inv_dt + (double)nv.y + c_eff * k * v.x);
      if (TANGENT) {
        const double2 w = sym_load(U0, c, pos, iz, j, a);
        f[c].x -= dc * k * w.y;
        f[c].y += dc * k * w.x;
      }
      if (mean) f[c].y = 0.0;
    }
    double2* d3 = sf + d * n3;
    if (mean) {  // the mean mode keeps (f_r, f_theta, f_z)
      d3[j] = f[0];
      d3[NRP + j] = f[1];
      d3[2 * NRP + j] = f[2];
    } else {
      d3[j] = make_double2(f[0].x - f[1].y, f[0].y + f[1].x);
      d3[NRP + j] = make_double2(f[0].x + f[1].y, f[0].y - f[1].x);
      d3[2 * NRP + j] = make_double2(f[2].y, -f[2].x);
    }
  }
  __syncthreads();
  // pressure right-hand side: div_h f on the inner rows, wall value 0 (all rows in parallel)
  for (int idx = tid; idx < nd * NR; idx += nt) {
    const int d = idx / NR, i = idx - d * NR;
    double2 g = make_double2(0.0, 0.0);
    if (!mean && i > 0) {
      const double2* fp = sf + d * n3;
      const double2* fm = fp + NRP;
      const double2* fz = fp + 2 * NRP;
      double2 acc = make_double2(0.0, 0.0);
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const int col = __ldg(ce + i * 9 + q);
        const double w = __ldg(we + i * 9 + q);
        acc.x = fma(w, fp[col].x + fm[col].x, acc.x);
        acc.y = fma(w, fp[col].y + fm[col].y, acc.y);
      }
      const double ir = __ldg(a.r + NR + i);
      g.x = 0.5 * acc.x + 0.5 * ir * ((1.0 + mm) * fp[i].x + (1.0 - mm) * fm[i].x) - k * fz[i].x;
      g.y = 0.5 * acc.y + 0.5 * ir * ((1.0 + mm) * fp[i].y + (1.0 - mm) * fm[i].y) - k * fz[i].y;
    }
    sp[d * NRP + i] = g;
  }
  bool ok = mbar_wait_bounded(bar, 0);
  if (!ok) (void)mbar_wait_bounded(bar, 0);  // copies still in flight: a second limit before going on
  ok = __syncthreads_and(ok) != 0;            // the same decision in every thread of the block
  if (ok) {
    // The warp of the chains: one direction fills six lanes of one warp; blocks of one SM alternate
    // between their warps, so that the schedulers share the chains.
    constexpr int W = psolve_warps(ND);
    const int pt = ND >= 8 ? tid - 32 * (W - 1) : tid - 32 * ((blockIdx.x / (2 * a.sms)) & 1);
    const int vt = ND >= 8 ? tid : pt;
    // pressure solve: one task per (direction, part)
    if (pt >= 0 && pt < 2 * nd && !mean)
      band_solve_d<NRT>(reinterpret_cast<double*>(sp + (pt >> 1) * NRP) + (pt & 1), sfac, NR);
    __syncthreads();
    if (tid == 0 && !mean) {  // u~z takes the place of the pressure's factors
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      expect_bytes(bar, (uint32_t)chunk);
      copy_factor(sfac, fac + 3 * chunk, (uint32_t)chunk, bar);
    }
    // velocity right-hand sides f - grad p on the inner rows, no slip at the wall (parallel)
    for (int idx = tid; idx < nd * 3 * NR; idx += nt) {
      const int d = idx / (3 * NR), rem = idx - d * 3 * NR, comp = rem / NR, i = rem - comp * NR;
      double2& x = sf[d * n3 + comp * NRP + i];
      if (mean) {  // mean flow: u_r = 0, wall rows zero
        if (comp == 0 || i == 0) x = make_double2(0.0, 0.0);
        continue;
      }
      if (i == 0) {
        x = make_double2(0.0, 0.0);
        continue;
      }
      const double2* p = sp + d * NRP;
      double2 gp;
      if (comp == 2) {
        gp = make_double2(k * p[i].x, k * p[i].y);
      } else {
        double2 d1 = make_double2(0.0, 0.0);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
          const int col = __ldg(cz + i * 9 + q);
          const double w = __ldg(wz + i * 9 + q);
          d1.x = fma(w, p[col].x, d1.x);
          d1.y = fma(w, p[col].y, d1.y);
        }
        const double mr = mm * __ldg(a.r + NR + i);
        gp = comp == 0 ? make_double2(d1.x - mr * p[i].x, d1.y - mr * p[i].y)
                       : make_double2(d1.x + mr * p[i].x, d1.y + mr * p[i].y);
      }
      x.x -= gp.x;
      x.y -= gp.y;
    }
    if (!mean) {
      ok = mbar_wait_bounded(bar, 1);
      if (!ok) (void)mbar_wait_bounded(bar, 1);
    }
    ok = __syncthreads_and(ok) != 0;
    // velocity solves: one task per (direction, component, part)
    if (ok && vt >= 0 && vt < 6 * nd) {
      const int d = vt / 6, rem = vt - 6 * d, comp = rem >> 1, part = rem & 1;
      // buffers: u~z 0, u+ 1, u- 2; mean mode: u_theta 1, u_z 2
      const int buf = mean ? comp : (comp == 2 ? 0 : comp + 1);
      if (!(mean && comp == 0))
        band_solve_d<NRT>(reinterpret_cast<double*>(sf + d * n3 + comp * NRP) + part, sfac + buf * chunk, NR);
    }
    __syncthreads();
    // influence coefficient from the wall continuity row: 0.5 D1 (u+ + u-) at r = 1 vanishes
    if (tid < 2 * nd) {
      const int d = tid >> 1, part = tid & 1;
      double al = 0.0;
      if (!mean) {
        const double* up = reinterpret_cast<const double*>(sf + d * n3) + part;
        const double* um = up + 2 * NRP;
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
          const int col = __ldg(ce + q);
          s += __ldg(we + q) * (up[2 * col] + um[2 * col]);
        }
        al = -0.5 * s * __ldg(a.pb_dinv + mode);
      }
      s_alpha[d][part] = al;
    }
    __syncthreads();
  }
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  for (int idx = tid; idx < nd * NR; idx += nt) {
    const int d = idx / NR, j = idx - d * NR, dir = d0 + d;
    const double2* us = u + (size_t)dir * a.sstride;
    double2* dst = out + (size_t)dir * a.sstride;
    const double2* x = sf + d * n3;
    double2 vr, vt, vz;
    if (!ok) {
      vr = vt = vz = make_double2(nan, nan);
    } else if (mean) {
      vr = make_double2(0.0, 0.0);
      vt = make_double2(x[NRP + j].x, 0.0);
      vz = make_double2(x[2 * NRP + j].x, 0.0);
    } else {
      const double* h = a.pb_uh + (size_t)mode * 3 * NR + j;
      const double ax = s_alpha[d][0], ay = s_alpha[d][1];
      auto with = [&](int comp) {
        const double w = __ldg(h + comp * NR);
        const double2 v = x[comp * NRP + j];
        return make_double2(v.x + ax * w, v.y + ay * w);
      };
      const double2 up = with(0), um = with(1), uzt = with(2);
      vr = make_double2(0.5 * (up.x + um.x), 0.5 * (up.y + um.y));
      vt = make_double2(0.5 * (up.y - um.y), -0.5 * (up.x - um.x));  // (u+ - u-)/(2i)
      vz = make_double2(-uzt.y, uzt.x);                                // i u~z
    }
    const double2 res[3] = {vr, vt, vz};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 d2 = sym_load(us, c, pos, iz, j, a);
      double2 g = make_double2(res[c].x - d2.x, res[c].y - d2.y);
      if (mean) g.y = 0.0;
      dst[((size_t)c * Mm + pos * a.MZ + iz) * NR + j] = g;
      if (iz == 0 && pos != 0) dst[((size_t)c * Mm + (a.MX - pos) * a.MZ) * NR + j] = make_double2(g.x, -g.y);
    }
  }
  // the speed slot of a step is zero (no equation of its own); the tangent's
  // phase condition is written afterwards
  if (blockIdx.x == 0 && tid < nd) out[(size_t)(d0 + tid) * a.sstride + a.sstride - 1] = make_double2(0.0, 0.0);
}

// dzU = i k P(U) (P: Hermitian projection), speed slot zero
__global__ void k_pipe_dz(const double2* U, double2* dzU, PArgs a) {
  const size_t n = (size_t)3 * a.Mm * a.NR;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(e % a.NR);
    const int m = (int)((e / a.NR) % a.Mm);
    const int c = (int)(e / ((size_t)a.NR * a.Mm));
    const int pos = m / a.MZ, iz = m - pos * a.MZ;
    const int kzi = pos <= a.Kx ? pos : pos - a.MX;
    const double k = a.alpha * kzi;
    const double2 v = sym_load(U, c, pos, iz, j, a);
    dzU[e] = make_double2(-k * v.y, k * v.x);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) dzU[n] = make_double2(0.0, 0.0);
}

// partial sums of <dzU, du> (the speed slots included, weights w(m')), grid (nb, directions)
__global__ void __launch_bounds__(256) k_phase_partials(const double2* __restrict__ dz, const double2* __restrict__ du,
                                                        double* __restrict__ partials, PArgs a) {
  const double2* d = du + (size_t)blockIdx.y * a.sstride;
  double acc = 0.0;
  for (unsigned e = blockIdx.x * 256 + threadIdx.x; e < a.sstride; e += gridDim.x * 256) {
    const unsigned iz = (e / (unsigned)a.NR) % (unsigned)a.MZ;
    const double2 p = __ldg(dz + e), q = __ldg(d + e);
    const double t = fma(p.x, q.x, p.y * q.y);
    acc += iz == 0 ? t : 2.0 * t;
  }
  __shared__ double red[8];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) acc += red[w];
    partials[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = acc;
  }
}

// one warp per direction
__global__ void __launch_bounds__(128) k_phase_sum(const double* __restrict__ partials, int nb, double2* __restrict__ out,
                                                   size_t sstride, int n_dir) {
  const int d = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (d >= n_dir) return;
  double acc = 0.0;
  for (int b = lane; b < nb; b += 32) acc += partials[(size_t)d * nb + b];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) out[(size_t)(d + 1) * sstride - 1] = make_double2(acc, 0.0);
}

// seeded pipe state: A = streak part, B = poloidal part (both unscaled)
__global__ void k_pipe_seed(const double* streak, const double2* pol, int npoly, double2* A, double2* B, PArgs a) {
  const int m = blockIdx.x;  // stored mode index
  if (m >= a.Mm) return;
  const int pos = m / a.MZ, iz = m - pos * a.MZ;
  const int kzi = pos <= a.Kx ? pos : pos - a.MX;
  const double k = a.alpha * kzi;
  const int mm = (int)lround(a.sym) * iz;
  for (int j = threadIdx.x; j < a.NR; j += blockDim.x) {
    const double r = a.r[j], x = 1.0 - r * r;
    double2 zr = make_double2(0.0, 0.0), zt = zr, zz = zr, sz = zr;
    if (kzi == 0 && iz >= 1 && iz <= 3) {
      double rm = 1.0;
      for (int q = 0; q < mm; ++q) rm *= r;
      sz = make_double2(streak[iz] * x * rm, 0.0);
    }
    if (kzi != 0) {
      // phi = (1 - r^2)^3 r^m s(r), s = sum_n p_n r^(2n): phi', phi'' by the product rule
      double2 s = make_double2(0.0, 0.0), s1 = s, s2 = s;
      double rp = 1.0;  // r^(2n)
      for (int n = 0; n < npoly; ++n) {
        const double2 p = pol[((size_t)pos * a.MZ + iz) * npoly + n];
        const double e = 2.0 * n;
        const double d1 = n > 0 ? e * rp / r : 0.0;                  // d/dr r^(2n)
        const double d2 = n > 0 ? e * (e - 1.0) * rp / (r * r) : 0.0;  // d2/dr2 r^(2n)
        s.x += p.x * rp; s.y += p.y * rp;
        s1.x += p.x * d1; s1.y += p.y * d1;
        s2.x += p.x * d2; s2.y += p.y * d2;
        rp *= r * r;
      }
      double rm = 1.0;
      for (int q = 0; q < mm; ++q) rm *= r;
      // g = (1 - r^2)^3 r^m
      const double g = x * x * x * rm;
      const double g1 = -6.0 * r * x * x * rm + (mm > 0 ? mm * x * x * x * rm / r : 0.0);
      const double g2 = 24.0 * r * r * x * rm - 6.0 * x * x * rm - (mm > 0 ? 12.0 * mm * x * x * rm : 0.0) +
                        (mm > 1 ? mm * (mm - 1.0) * x * x * x * rm / (r * r) : 0.0);
      const double2 ph = make_double2(g * s.x, g * s.y);
      const double2 p1 = make_double2(g1 * s.x + g * s1.x, g1 * s.y + g * s1.y);
      const double2 p2 = make_double2(g2 * s.x + 2.0 * g1 * s1.x + g * s2.x, g2 * s.y + 2.0 * g1 * s1.y + g * s2.y);
      zr = make_double2(-k * p1.y, k * p1.x);                   // i k phi'
      zt = make_double2(-mm * k / r * ph.x, -mm * k / r * ph.y);  // -(m k / r) phi
      zz = make_double2(-(p2.x + p1.x / r - mm * mm * ph.x / (r * r)), -(p2.y + p1.y / r - mm * mm * ph.y / (r * r)));
    }
    const size_t e = (size_t)m * a.NR + j;
    A[0 * (size_t)a.Mm * a.NR + e] = make_double2(0.0, 0.0);
    A[1 * (size_t)a.Mm * a.NR + e] = make_double2(0.0, 0.0);
    A[2 * (size_t)a.Mm * a.NR + e] = sz;
    B[0 * (size_t)a.Mm * a.NR + e] = zr;
    B[1 * (size_t)a.Mm * a.NR + e] = zt;
    B[2 * (size_t)a.Mm * a.NR + e] = zz;
  }
  if (m == 0 && threadIdx.x == 0) {
    A[(size_t)3 * a.Mm * a.NR] = make_double2(0.0, 0.0);
    B[(size_t)3 * a.Mm * a.NR] = make_double2(0.0, 0.0);
  }
}

PArgs pargs(const sp_ctx* c) {
  PArgs a;
  a.r = c->yv;
  a.w1 = c->fd_w1;
  a.c1 = c->fd_c1;
  a.pb_fac = c->pb_fac;
  a.pb_chunk = c->pb_chunk;
  a.pb_uh = c->pb_uh;
  a.pb_dinv = c->pb_dinv;
  a.sstride = c->cplx_per_state;
  a.Mm = c->Mm; a.MX = c->MX; a.MZ = c->MZ; a.Kx = c->Kx; a.NR = c->NY; a.n_unique = c->n_unique; a.sms = c->sm_count;
  a.alpha = c->alpha; a.sym = c->beta; a.inv_dt = 1.0 / c->dt;
  return a;
}

}  // namespace

cudaError_t launch_pvals(const sp_ctx* c, bool fp32, const double* in, void* out6, int n_dir, cudaStream_t st) {
  PArgs a = pargs(c);
  dim3 grid((c->Mm + kTileP - 1) / kTileP, n_dir);
  const size_t sm = (size_t)3 * kTileP * c->NY * sizeof(double2);
  if (fp32) {
    cudaFuncSetAttribute(k_pvals<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_pvals<float><<<grid, kThreadsP, sm, st>>>(reinterpret_cast<const double2*>(in),
                                                reinterpret_cast<C2<float>*>(out6), a);
  } else {
    cudaFuncSetAttribute(k_pvals<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_pvals<double><<<grid, kThreadsP, sm, st>>>(reinterpret_cast<const double2*>(in),
                                                 reinterpret_cast<C2<double>*>(out6), a);
  }
  return cudaGetLastError();
}

cudaError_t launch_pipe_phase(const sp_ctx* c, const double* du, double* out, double* partials, int nb, int n_dir,
                              cudaStream_t st) {
  const PArgs a = pargs(c);
  k_phase_partials<<<dim3(nb, n_dir), 256, 0, st>>>(reinterpret_cast<const double2*>(c->dzU),
                                                    reinterpret_cast<const double2*>(du), partials, a);
  k_phase_sum<<<(n_dir + 3) / 4, 128, 0, st>>>(partials, nb, reinterpret_cast<double2*>(out), a.sstride, n_dir);
  return cudaGetLastError();
}

template <typename T, bool TG, int ND, int NRT>
static cudaError_t psolve_t(const sp_ctx* c, const PArgs& a, const void* in3, const double2* uu, const double2* U0,
                            double2* o, int n_dir, cudaStream_t st) {
  const size_t sm = psolve_smem(ND, c->NY, c->pb_chunk);
  auto kern = k_psolve<T, TG, ND, NRT>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  kern<<<dim3(c->n_unique, (n_dir + ND - 1) / ND), psolve_threads(ND), sm, st>>>(reinterpret_cast<const C2<T>*>(in3), uu, U0, o,
                                                                                a, n_dir);
  return cudaGetLastError();
}

// Directions per block: eight from two directions on, where their factors and vectors fit; sixteen (full warps
// of chains) where two such blocks share an SM and there are at least eight per SM. us with 1, 8 and 16, FP64:
// 613 modes of Nr = 64, 2 directions 273, 254, 362; 4: 445, 281, 389; 16: 1627, 566, 600; 24: 2467, 902, 874;
// 64: 6627, 2037, 1882; 163 modes of Nr = 32, 4: 86, 78, 78; 16: 281, 109, 123; 64: 962, 300, 294; 145 modes
// of Nr = 96, 2: 210, 207, 206; 16: 844, 262, 305; 64: 3359, 1037, 1174.
template <typename T, bool TG>
static cudaError_t psolve_nd(const sp_ctx* c, const PArgs& a, const void* in3, const double2* uu, const double2* U0,
                             double2* o, int n_dir, cudaStream_t st) {
  constexpr size_t kMax = 225 * 1024;
  // the grids that a block with one mode's four matrices holds (radial counts up to 235)
  if (4 * c->pb_chunk + (size_t)4 * psolve_nrp(c->NY) * 16 + (size_t)2 * c->NY * 9 * 12 > kMax) return cudaErrorInvalidValue;
  const bool r64 = c->NY == 64;
  const long long blocks16 = (long long)c->n_unique * ((n_dir + 15) / 16);
  if (n_dir > 16 && blocks16 >= 8LL * c->sm_count && psolve_smem(16, c->NY, c->pb_chunk) <= kMax / 2)
    return r64 ? psolve_t<T, TG, 16, 64>(c, a, in3, uu, U0, o, n_dir, st) : psolve_t<T, TG, 16, 0>(c, a, in3, uu, U0, o, n_dir, st);
  if (n_dir >= 2 && psolve_smem(8, c->NY, c->pb_chunk) <= kMax)
    return r64 ? psolve_t<T, TG, 8, 64>(c, a, in3, uu, U0, o, n_dir, st) : psolve_t<T, TG, 8, 0>(c, a, in3, uu, U0, o, n_dir, st);
  return r64 ? psolve_t<T, TG, 1, 64>(c, a, in3, uu, U0, o, n_dir, st) : psolve_t<T, TG, 1, 0>(c, a, in3, uu, U0, o, n_dir, st);
}

cudaError_t launch_psolve(const sp_ctx* c, bool fp32, bool tangent, const void* in3, const double* u, double* out,
                          int n_dir, cudaStream_t st) {
  PArgs a = pargs(c);
  const double2* uu = reinterpret_cast<const double2*>(u);
  const double2* U0 = reinterpret_cast<const double2*>(c->U0);
  double2* o = reinterpret_cast<double2*>(out);
  if (fp32) return tangent ? psolve_nd<float, true>(c, a, in3, uu, U0, o, n_dir, st)
                           : psolve_nd<float, false>(c, a, in3, uu, U0, o, n_dir, st);
  return tangent ? psolve_nd<double, true>(c, a, in3, uu, U0, o, n_dir, st)
                 : psolve_nd<double, false>(c, a, in3, uu, U0, o, n_dir, st);
}

cudaError_t launch_pipe_dz(const sp_ctx* c, const double* U, double* dzU, cudaStream_t st) {
  PArgs a = pargs(c);
  k_pipe_dz<<<256, 256, 0, st>>>(reinterpret_cast<const double2*>(U), reinterpret_cast<double2*>(dzU), a);
  return cudaGetLastError();
}

cudaError_t launch_pipe_seed(const sp_ctx* c, const double* streak, const double* pol, int npoly, double* A,
                             double* B, cudaStream_t st) {
  PArgs a = pargs(c);
  k_pipe_seed<<<c->Mm, 64, 0, st>>>(streak, reinterpret_cast<const double2*>(pol), npoly,
                                    reinterpret_cast<double2*>(A), reinterpret_cast<double2*>(B), a);
  return cudaGetLastError();
}
