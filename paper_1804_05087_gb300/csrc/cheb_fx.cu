// Chebyshev transforms of the FP64 step and tangent in 64-bit fixed point (Sec. 3.2: Chebyshev in y).
//
//   k_yinv_fx: per Fourier mode, coefficients of u, v, w -> values of u, v, w and of the vorticity at
//              the Gauss-Lobatto points (curl in spectral space), plane-major: the inputs and
//              outputs of k_yinv (kernels.cu).
//   k_rhs_fx : values of the product -> coefficients of the rows 0..N-2, plus u/dt: the right-hand
//              sides of the per-mode solves (k_chain, k_solve).
//
// Both are sums over the constants T_n(y_j) = cos(pi j n / N). An SM does 25 multiply-adds of 32-bit halves per
// clock but 1.7 in FP64 (fx_arith.h), and three of them make one term of a sum whose inputs share a scale.
// 48 x 65 x 48, 256 directions: k_yinv_fx 1.72 ms (FP64 4.05; its multiply-adds alone 1.09), k_rhs_fx 1.03 ms
// (FP64 2.39; 0.61). A column (one component of one mode) is scaled by its largest value, a point pair's sum
// by twice that (59 bits, after rounding up), and by its sum of moduli (62 bits, a bound of every result), and
// split as x = hi 2^28 + lo; the constants are 56-bit, split the same way. hi hi and hi lo + lo hi are summed
// in two 64-bit accumulators (both stay below 2^63 up to 129 terms, N <= 256); lo lo, below a quarter
// of a unit, is dropped. Derivatives: n^2 a_n, scaled as a column of its own, times T_n'(y_j) / n^2.
// Points y and -y share a table row: T_n(-y) = (-1)^n T_n(y), T_n'(-y) = -(-1)^n T_n'(y).
#include <algorithm>
#include <cmath>
#include <vector>

#include "dev_util.h"
#include "fx_arith.h"
#include "sp_internal.h"

namespace {

using namespace fx;

constexpr int kThreadsC = 256;
// modes per block: eight share the table loads best; four, when eight leave SMs without a block
constexpr int kModes = 8, kModesFew = 4;
// columns of a block's rows: u, v, w, Du, Dw (values: the three components) of every mode, padded
__host__ __device__ constexpr int stride_y(int tm) { return 5 * tm + 1; }
__host__ __device__ constexpr int stride_r(int tm) { return 3 * tm + 1; }
constexpr int kNotFinite = 1 << 28;             // exponent of a column with a non-finite input

__device__ __forceinline__ int4 halves2(i64 x, i64 y) {
  const int2 a = halves28(x), b = halves28(y);
  return make_int4(a.x, a.y, b.x, b.y);
}

struct Sum2 {  // complex columns
  Sum x, y;
  __device__ __forceinline__ void add(int4 v, int2 c) {
    x.add(v.x, v.y, c);
    y.add(v.z, v.w, c);
  }
};

__device__ __forceinline__ unsigned top_of(double2 v) {
  return max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
}
// round(v f 2^sh), f a small integer
__device__ __forceinline__ i64 from_double_times(double v, int sh, double f) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
  const double d = __hiloint2double(hi + sh * (1 << 20), __double2loint(v));
  return e != 0 && e + sh > 1000 ? __double2ll_rn(d * f) : 0;
}

__device__ __forceinline__ double unscale(i64 X, int sh) { return sh == kNotFinite ? nan("") : from_fixed(X, sh); }
__device__ __forceinline__ double2 unscale(i64 x, i64 y, int sh) { return make_double2(unscale(x, sh), unscale(y, sh)); }

// Tables of constants, 56-bit halves, each row padded to PH entries (even, zeros) so that two come
// with one load: values [NH][2][PH] (degrees 2 q + parity at q), derivatives [NH][2][PH], forward
// [NY][PH] (point j of row n at j). PH covers NH = N / 2 + 1 entries.
__host__ __device__ constexpr int tab_ph(int NY) { return (NY / 2 + 2) & ~1; }

struct YArgs {
  const double2* in;   // [dir][3][Mm][NY]
  double2* out;        // [dir][6][NY][Mm]
  const int2* tab;     // T_n(y_j), T_n'(y_j) / n^2 (ChebTab)
  int Mm, MZ, MX, Kx, NY, NH, jchunk;
  double alpha, beta;
};

// (bx, by, bz): mode tile, chunk of the half grid, direction. xs: [2 PH][stride_y]
template <int TM>
__device__ __forceinline__ void yinv_fx(const YArgs& a, int bx, int by, int bz, int4* xs, int (*sh)[TM]) {
  constexpr int ST = stride_y(TM), kWarps = kThreadsC / 32, RW = (3 * TM + kWarps - 1) / kWarps;
  const int NY = a.NY, N = NY - 1, Mm = a.Mm, m0 = bx * TM, PH = tab_ph(NY), rows = 2 * PH;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // one warp per (component, mode): the rows' loads first, kept in their own slots
  unsigned em[RW];
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    em[r] = 0;
    const int row = warp + r * kWarps, f = row / TM, m = m0 + row - f * TM;
    if (row >= 3 * TM) continue;
    const double2* src = a.in + (((size_t)bz * 3 + f) * Mm + m) * NY;
    for (int n = lane; n < rows; n += 32) {  // zeros past the last degree
      double2 v = make_double2(0.0, 0.0);
      if (m < Mm && n < NY) v = __ldg(src + n);
      em[r] = max(em[r], top_of(v));
      reinterpret_cast<double2*>(xs)[n * ST + row] = v;
    }
  }
  // scales, halves and derivative columns
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    const int row = warp + r * kWarps, f = row / TM, t = row - f * TM;
    if (row >= 3 * TM) continue;
    const int e = (int)(__reduce_max_sync(0xffffffffu, em[r]) >> 20);
    u64 s0 = 0, s2 = 0, t0 = 0, t2 = 0;  // sums and largest values of a_n and of n^2 a_n
    for (int n = lane; n < NY; n += 32) {
      const double2 v = reinterpret_cast<const double2*>(xs)[n * ST + row];
      const unsigned px = part_of(v.x, e), py = part_of(v.y, e), q = max(px, py);
      s0 += px + py;
      s2 += (u64)(n * n) * (px + py);
      t0 = max(t0, (u64)q);
      t2 = max(t2, (u64)(n * n) * q);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      t0 = max(t0, __shfl_xor_sync(0xffffffffu, t0, o));
      t2 = max(t2, __shfl_xor_sync(0xffffffffu, t2, o));
    }
    const int e0 = exponent_of(s0, t0, e), ed = exponent_of(s2, t2, e);
    const int g = f == 0 ? 3 : 4;  // derivative column of u and w
    if (lane == 0) {
      sh[f][t] = e == 0x7ff ? kNotFinite : e0;
      if (f != 1) sh[g][t] = e == 0x7ff ? kNotFinite : ed;
    }
    for (int n = lane; n < rows; n += 32) {
      int4* x = xs + n * ST;
      const double2 v = reinterpret_cast<const double2*>(x)[row];
      x[row] = halves2(from_double(v.x, e0), from_double(v.y, e0));
      if (f == 1) continue;
      const double n2 = (double)(n * n);
      x[g * TM + t] = n == 0 ? make_int4(0, 0, 0, 0) : halves2(from_double_times(v.x, ed, n2), from_double_times(v.y, ed, n2));
    }
  }
  __syncthreads();
  // two lanes per point pair (y, -y) of a mode: one sums the even degrees, one the odd; then each
  // forms the values of one of the two points
  const int j_lo = by * a.jchunk, j_hi = min(a.NH, j_lo + a.jchunk), items = 2 * TM * (j_hi - j_lo);
  const size_t NYMm = (size_t)NY * Mm;
  double2* o = a.out + (size_t)bz * 6 * NYMm;
  const int t = lane % TM, m = m0 + t;  // a lane keeps its mode
  double kx = 0.0, kz = 0.0;
  auto wave = [&] {
    const int pos = m / a.MZ, iz = m - pos * a.MZ;
    kx = a.alpha * (pos <= a.Kx ? pos : pos - a.MX);
    kz = a.beta * iz;
  };
  if (TM == kModes) wave();  // many items per lane: once; else it would delay the only sum
  for (int i0 = warp * 32; i0 < items; i0 += kThreadsC) {
    const int it = i0 + lane, odd = it / TM & 1, jh = min(j_lo + it / (2 * TM), j_hi - 1);
    Sum2 S[5];
    const int4* tr = reinterpret_cast<const int4*>(a.tab + (size_t)(2 * jh + odd) * PH);
    const int4* td = tr + (size_t)a.NH * PH;  // 2 NH rows of PH / 2 loads
    const int4* x = xs + odd * ST + t;
    for (int q = 0; q < PH / 2; ++q) {
      const int4 c = __ldg(tr + q), d = __ldg(td + q);
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        const int4 k = f < 3 ? c : d;
        S[f].add(x[f * TM], make_int2(k.x, k.y));
        S[f].add(x[2 * ST + f * TM], make_int2(k.z, k.w));
      }
      x += 4 * ST;
    }
    i64 vx[5], vy[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      const i64 mx = S[f].x.value(), my = S[f].y.value();
      const i64 px = __shfl_xor_sync(0xffffffffu, mx, TM), py = __shfl_xor_sync(0xffffffffu, my, TM);
      // even lane: E + O at jh; odd lane: values E - O, derivatives O - E at N - jh
      vx[f] = !odd ? mx + px : f < 3 ? px - mx : mx - px;
      vy[f] = !odd ? my + py : f < 3 ? py - my : my - py;
    }
    const int j = odd ? N - jh : jh;
    if (it >= items || m >= Mm || (odd && j == jh)) continue;
    if (TM != kModes) wave();
    double2 v[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) v[f] = unscale(vx[f], vy[f], sh[f][t]);
    double2* d = o + (size_t)j * Mm + m;
    d[0] = v[0];
    d[NYMm] = v[1];
    d[2 * NYMm] = v[2];
    // Dw - i kz v, i kz u - i kx w, i kx v - Du
    d[3 * NYMm] = make_double2(fma(kz, v[1].y, v[4].x), fma(-kz, v[1].x, v[4].y));
    d[4 * NYMm] = make_double2(fma(kx, v[2].y, -kz * v[0].y), fma(-kx, v[2].x, kz * v[0].x));
    d[5 * NYMm] = make_double2(-fma(kx, v[1].y, v[3].x), fma(kx, v[1].x, -v[3].y));
  }
}

template <int TM>
__global__ void __launch_bounds__(kThreadsC, 3) k_yinv_fx(const __grid_constant__ YArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int sh[5][TM];
  yinv_fx<TM>(a, blockIdx.x, blockIdx.y, blockIdx.z, reinterpret_cast<int4*>(smem), sh);
}

// ------------------------------------------------------------------ forward
struct RArgs {
  const double2* in3;  // [dir][3][NY][Mm]
  const double2* du;   // [dir][3][Mm][NY]
  double2* W;          // (u, d, row c (N-1) + n) at u su + d sd + row sn
  const int2* tab;
  long long su, sd, sn;
  int n_dir, n_unique, Mm, MX, MZ, Kx, NY, NH, rchunk;
  double inv_dt, c0, cn;  // 1 / N, 2 / N
};

template <int TM>
struct RShared {
  unsigned em[3 * TM];
  int sum[3 * TM];
  int sh[3 * TM];
  int pos[TM], iz[TM];
};

// (bx, by, bz): tile of solved modes, chunk of rows, direction. xs: [2 PH][stride_r]: the values, then
// the even parts of the point pairs (rows j < PH) and the odd parts (rows PH + j)
template <int TM>
__device__ __forceinline__ void rhs_fx(const RArgs& a, int bx, int by, int bz, int4* xs, RShared<TM>& s) {
  constexpr int ST = stride_r(TM);
  const int NY = a.NY, N = NY - 1, NH = a.NH, NR = N - 1, Mm = a.Mm, u0 = bx * TM, PH = tab_ph(NY);
  const int tid = threadIdx.x;
  if (tid < TM) {
    int pos = 0, iz = 0;
    if (u0 + tid < a.n_unique) unique_mode(u0 + tid, a.Kx, a.MZ, &pos, &iz);
    s.pos[tid] = pos;
    s.iz[tid] = iz;
  }
  if (tid < 3 * TM) {
    s.em[tid] = 0;
    s.sum[tid] = 0;
  }
  __syncthreads();
  // lanes take the modes fastest, then the points: value (c, j) of mode t into its own slot
  const int t = tid % TM, part = tid / TM;
  constexpr int nparts = kThreadsC / TM;
  const bool on = u0 + t < a.n_unique;
  const double2* src = a.in3 + (size_t)bz * 3 * NY * Mm + s.pos[t] * a.MZ + s.iz[t];
  double2* raw = reinterpret_cast<double2*>(xs);
  // the two points of a pair: slots j and PH + j
  auto slot = [&](int j) { return j < NH ? j : PH + N - j; };
  unsigned em[3] = {0, 0, 0};
#pragma unroll
  for (int c = 0; c < 3; ++c)
    for (int j = part; j < NY; j += nparts) {
      const double2 v = on ? __ldg(src + ((size_t)c * NY + j) * Mm) : make_double2(0.0, 0.0);
      em[c] = max(em[c], top_of(v));
      raw[slot(j) * ST + c * TM + t] = v;
    }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
#pragma unroll
    for (int o = TM; o < 32; o <<= 1) em[c] = max(em[c], __shfl_xor_sync(0xffffffffu, em[c], o));
    if ((tid & 31) < TM) atomicMax(&s.em[c * TM + t], em[c]);
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int e = (int)(s.em[c * TM + t] >> 20);
    int sum = 0;
    for (int j = part; j < NY; j += nparts) {
      const double2 v = raw[slot(j) * ST + c * TM + t];
      sum += part_of(v.x, e) + part_of(v.y, e);
    }
#pragma unroll
    for (int o = TM; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((tid & 31) < TM) atomicAdd(&s.sum[c * TM + t], sum);
  }
  __syncthreads();
  if (tid < 3 * TM) {
    const int e = (int)(s.em[tid] >> 20);
    s.sh[tid] = e == 0x7ff ? kNotFinite : exponent_of((u64)s.sum[tid], pair_top(s.em[tid]), e);
  }
  __syncthreads();
  // even and odd parts of the point pairs (j, N - j), in place; the end points enter with half weight
  for (int idx = part; idx < 3 * PH; idx += nparts) {
    const int c = idx / PH, j = idx - c * PH, col = c * TM + t;
    int4* x = xs + j * ST + col;
    int4* y = x + PH * ST;
    if (j >= NH) {
      *x = *y = make_int4(0, 0, 0, 0);
      continue;
    }
    const int sh = s.sh[col] == kNotFinite ? -2000 : s.sh[col];
    const double2 p = *reinterpret_cast<const double2*>(x);
    const i64 px = from_double(p.x, sh), py = from_double(p.y, sh);
    if (2 * j == N) {
      *x = halves2(px, py);
      *y = make_int4(0, 0, 0, 0);
    } else {
      const double2 q = *reinterpret_cast<const double2*>(y);
      const i64 qx = from_double(q.x, sh), qy = from_double(q.y, sh);
      const int d = j == 0 ? 1 : 0;
      *x = halves2((px + qx) >> d, (py + qy) >> d);
      *y = halves2((px - qx) >> d, (py - qy) >> d);
    }
  }
  __syncthreads();
  const int lo = by * a.rchunk, hi = min(NR, lo + a.rchunk);
  if (!on) return;
  const int pos = s.pos[t], iz = s.iz[t];
  const int mpos = pos == 0 ? 0 : a.MX - pos;
  const double2* dsrc = a.du + (size_t)bz * 3 * Mm * NY;
  const int ne = (NR + 1) / 2;  // even rows come first, so that a warp runs one trip count
  for (int r = lo + part; r < hi; r += nparts) {
    const int n = r < ne ? 2 * r : 2 * (r - ne) + 1, odd = n & 1;
    Sum2 S[3];
    const int4* x = xs + t + odd * PH * ST;
    const int4* tc = reinterpret_cast<const int4*>(a.tab + (size_t)n * PH);
    for (int q = 0; q < PH / 2; ++q) {
      const int4 c = __ldg(tc + q);
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        S[f].add(x[f * TM], make_int2(c.x, c.y));
        S[f].add(x[ST + f * TM], make_int2(c.z, c.w));
      }
      x += 2 * ST;
    }
    const double cn = n == 0 ? a.c0 : a.cn;  // 2 / (N cbar_n)
    double2 du[3], dm[3];
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      du[f] = __ldg(dsrc + ((size_t)f * Mm + pos * a.MZ + iz) * NY + n);
      if (iz == 0) dm[f] = __ldg(dsrc + ((size_t)f * Mm + mpos * a.MZ) * NY + n);
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      double2 d = du[f];
      if (iz == 0) d = project(d, dm[f]);
      const double2 v = unscale(S[f].x.value(), S[f].y.value(), s.sh[f * TM + t]);
      double2 g = make_double2(fma(cn, v.x, d.x * a.inv_dt), fma(cn, v.y, d.y * a.inv_dt));
      if (pos == 0 && iz == 0) g.y = 0.0;
      a.W[(u0 + t) * a.su + bz * a.sd + (long long)(f * NR + n) * a.sn] = g;
    }
  }
}

template <int TM>
__global__ void __launch_bounds__(kThreadsC, 3) k_rhs_fx(const __grid_constant__ RArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ RShared<TM> s;
  // directions fastest: with one direction per 16-byte column of W, the blocks that run together
  // fill its sectors
  rhs_fx<TM>(a, blockIdx.x / a.n_dir, blockIdx.y, blockIdx.x % a.n_dir, reinterpret_cast<int4*>(smem), s);
}

// ------------------------------------------------------------------ groups
struct GY {
  size_t off;  // offset (doubles) of the member's state in a group vector
  YArgs a;
  int gx;      // mode tiles of the member's launch
};
struct GR {
  size_t off;
  RArgs a;
  int gx;
};

__global__ void __launch_bounds__(kThreadsC, 3) k_yinv_fx_grp(const double* __restrict__ in, const GY* __restrict__ recs,
                                                              const int* __restrict__ inst, const int* __restrict__ first,
                                                              const int* __restrict__ active) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int sh[5][kModes];
  __shared__ GY r;
  const int i = inst[blockIdx.x];
  if (active && !active[i]) return;
  if (threadIdx.x == 0) {
    r = recs[i];
    r.a.in = reinterpret_cast<const double2*>(in + r.off);
  }
  __syncthreads();
  const int b = blockIdx.x - first[i];
  yinv_fx<kModes>(r.a, b % r.gx, b / r.gx, 0, reinterpret_cast<int4*>(smem), sh);
}

__global__ void __launch_bounds__(kThreadsC, 3) k_rhs_fx_grp(const double* __restrict__ du, const GR* __restrict__ recs,
                                                             const int* __restrict__ inst, const int* __restrict__ first,
                                                             const int* __restrict__ active) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ RShared<kModes> s;
  __shared__ GR r;
  const int i = inst[blockIdx.x];
  if (active && !active[i]) return;
  if (threadIdx.x == 0) {
    r = recs[i];
    r.a.du = reinterpret_cast<const double2*>(du + r.off);
  }
  __syncthreads();
  const int b = blockIdx.x - first[i];
  rhs_fx<kModes>(r.a, b % r.gx, b / r.gx, 0, reinterpret_cast<int4*>(smem), s);
}

size_t smem_y(const sp_ctx* c, int tm) { return (size_t)2 * tab_ph(c->NY) * stride_y(tm) * 16; }
size_t smem_r(const sp_ctx* c, int tm) { return (size_t)2 * tab_ph(c->NY) * stride_r(tm) * 16; }

// parts of the outputs of a mode tile: one block per tile when the tiles fill the GPU (each part
// scales the inputs again)
int parts_for(int tiles, int rows, int sms) {
  int p = 1;
  while (tiles * p < sms && rows > p * (kThreadsC / kModes) / 2) ++p;
  return p;
}

YArgs y_args(const sp_ctx* c, const void* in, void* out, int parts) {
  YArgs a;
  a.in = static_cast<const double2*>(in);
  a.out = static_cast<double2*>(out);
  a.tab = c->cheb_fx;
  a.Mm = c->Mm; a.MZ = c->MZ; a.MX = c->MX; a.Kx = c->Kx; a.NY = c->NY; a.NH = c->NH;
  a.jchunk = (c->NH + parts - 1) / parts;
  a.alpha = c->alpha;
  a.beta = c->beta;
  return a;
}

RArgs r_args(const sp_ctx* c, const void* in3, const void* du, void* W, int parts) {
  RArgs a;
  a.in3 = static_cast<const double2*>(in3);
  a.du = static_cast<const double2*>(du);
  a.W = static_cast<double2*>(W);
  a.tab = c->cheb_fx + (size_t)4 * c->NH * tab_ph(c->NY);
  a.su = 3LL * (c->N - 1);
  a.sd = a.su * c->n_unique;
  a.sn = 1;
  a.n_dir = 1;
  a.n_unique = c->n_unique;
  a.Mm = c->Mm; a.MX = c->MX; a.MZ = c->MZ; a.Kx = c->Kx; a.NY = c->NY; a.NH = c->NH;
  a.rchunk = (c->N - 1 + parts - 1) / parts;
  a.inv_dt = 1.0 / c->dt;
  a.c0 = 1.0 / c->N;
  a.cn = 2.0 / c->N;
  return a;
}

template <class R>
cudaError_t upload_grp(GrpKernel* k, const std::vector<R>& recs, const std::vector<int>& nblk, const int* order, size_t smem) {
  const int n = (int)recs.size();
  std::vector<int> inst, first(n, 0);
  for (int q = 0; q < n; ++q) {
    first[order[q]] = (int)inst.size();
    inst.insert(inst.end(), nblk[order[q]], order[q]);
  }
  k->blocks = (int)inst.size();
  k->smem = smem;
  cudaError_t e;
  if ((e = grp_upload(&k->recs, recs.data(), recs.size() * sizeof(R))) != cudaSuccess) return e;
  if ((e = grp_upload((void**)&k->inst, inst.data(), inst.size() * sizeof(int))) != cudaSuccess) return e;
  return grp_upload((void**)&k->first, first.data(), first.size() * sizeof(int));
}

}  // namespace

std::vector<int> cheb_fx_table(int NY) {
  const int N = NY - 1, NH = N / 2 + 1, PH = tab_ph(NY);
  std::vector<int> t(((size_t)4 * NH + NY) * PH * 2, 0);
  // cos(pi k / N) for k = 0 .. 2N - 1, exact at the multiples of a quarter turn
  std::vector<long double> cs(2 * N);
  for (int k = 0; k < 2 * N; ++k)
    cs[k] = k == 0 ? 1.0L : k == N ? -1.0L : 2 * k == N || 2 * k == 3 * N ? 0.0L
                                           : cosl(3.141592653589793238462643383279502884L * k / N);
  auto cosine = [&](long long k) { return cs[(k % (2 * N) + 2 * N) % (2 * N)]; };
  // sin(pi k / N) = cos(pi (2k - N) / 2N): from the table where N is even
  auto sine = [&](long long k) { return cosine(k - N / 2); };
  auto put = [&](size_t at, long double v) {
    const long long q = llrintl(v * 72057594037927936.0L);  // 2^56
    const long long hi = (q + (1 << 27)) >> 28;
    t[2 * at] = (int)hi;
    t[2 * at + 1] = (int)(q - hi * (1LL << 28));
  };
  for (int j = 0; j < NH; ++j)
    for (int n = 0; n < NY; ++n) {
      const size_t at = (size_t)(2 * j + (n & 1)) * PH + n / 2;
      put(at, cosine((long long)j * n));
      // T_n' / n^2 = sin(n s) / (n sin s), s = pi j / N
      put((size_t)2 * NH * PH + at, n == 0 ? 0.0L : j == 0 ? 1.0L : sine((long long)j * n) / (n * sine(j)));
      put((size_t)4 * NH * PH + (size_t)n * PH + j, cosine((long long)j * n));
    }
  return t;
}

template <int TM>
static cudaError_t launch_y(const sp_ctx* c, const double* in, void* out6, int n_dir, cudaStream_t st) {
  const int tiles = (c->Mm + TM - 1) / TM;
  const YArgs a = y_args(c, in, out6, parts_for(tiles * n_dir, c->NH, c->sm_count));
  const size_t sm = smem_y(c, TM);
  const cudaError_t e = cudaFuncSetAttribute(k_yinv_fx<TM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_yinv_fx<TM><<<dim3(tiles, (c->NH + a.jchunk - 1) / a.jchunk, n_dir), kThreadsC, sm, st>>>(a);
  return cudaGetLastError();
}

template <int TM>
static cudaError_t launch_r(const sp_ctx* c, const void* in3, const double* du, void* W, int n_dir, long long su,
                            long long sd, long long sn, cudaStream_t st) {
  const int tiles = (c->n_unique + TM - 1) / TM;
  RArgs a = r_args(c, in3, du, W, parts_for(tiles * n_dir, c->N - 1, c->sm_count));
  a.n_dir = n_dir;
  if (sn) {
    a.su = su;
    a.sd = sd;
    a.sn = sn;
  }
  const size_t sm = smem_r(c, TM);
  const cudaError_t e = cudaFuncSetAttribute(k_rhs_fx<TM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_rhs_fx<TM><<<dim3(n_dir * tiles, (c->N - 1 + a.rchunk - 1) / a.rchunk), kThreadsC, sm, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_yinv_fx(const sp_ctx* c, const double* in, void* out6, int n_dir, cudaStream_t st) {
  if ((c->Mm + kModes - 1) / kModes * n_dir >= c->sm_count) return launch_y<kModes>(c, in, out6, n_dir, st);
  return launch_y<kModesFew>(c, in, out6, n_dir, st);
}

cudaError_t launch_rhs_fx(const sp_ctx* c, const void* in3, const double* du, void* W, int n_dir, long long su,
                          long long sd, long long sn, cudaStream_t st) {
  if ((c->n_unique + kModes - 1) / kModes * n_dir >= c->sm_count)
    return launch_r<kModes>(c, in3, du, W, n_dir, su, sd, sn, st);
  return launch_r<kModesFew>(c, in3, du, W, n_dir, su, sd, sn, st);
}

cudaError_t grp_build_cheb_fx(GrpPlan* p, sp_ctx* const* mem, int n, const size_t* offs, const int* order) {
  int ty = 0, tr = 0;
  for (int m = 0; m < n; ++m) {
    ty += (mem[m]->Mm + kModes - 1) / kModes;
    tr += (mem[m]->n_unique + kModes - 1) / kModes;
  }
  std::vector<GY> ry(n);
  std::vector<GR> rr(n);
  std::vector<int> by(n), br(n);
  size_t sy = 0, sr = 0;
  for (int m = 0; m < n; ++m) {
    const sp_ctx* c = mem[m];
    ry[m].off = rr[m].off = offs[m];
    ry[m].a = y_args(c, nullptr, c->ws6, parts_for(ty, c->NH, c->sm_count));
    ry[m].gx = (c->Mm + kModes - 1) / kModes;
    by[m] = ry[m].gx * ((c->NH + ry[m].a.jchunk - 1) / ry[m].a.jchunk);
    rr[m].a = r_args(c, c->ws3, nullptr, c->ws6, parts_for(tr, c->N - 1, c->sm_count));
    rr[m].gx = (c->n_unique + kModes - 1) / kModes;
    br[m] = rr[m].gx * ((c->N - 1 + rr[m].a.rchunk - 1) / rr[m].a.rchunk);
    sy = std::max(sy, smem_y(c, kModes));
    sr = std::max(sr, smem_r(c, kModes));
  }
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_yinv_fx_grp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sy)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_rhs_fx_grp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sr)) != cudaSuccess) return e;
  if ((e = upload_grp(&p->yinv64, ry, by, order, sy)) != cudaSuccess) return e;
  return upload_grp(&p->rhs64, rr, br, order, sr);
}

cudaError_t grp_launch_yinv_fx(const GrpPlan& p, const double* in, const int* active, cudaStream_t st) {
  const GrpKernel& k = p.yinv64;
  k_yinv_fx_grp<<<k.blocks, kThreadsC, k.smem, st>>>(in, static_cast<const GY*>(k.recs), k.inst, k.first, active);
  return cudaGetLastError();
}
cudaError_t grp_launch_rhs_fx(const GrpPlan& p, const double* du, const int* active, cudaStream_t st) {
  const GrpKernel& k = p.rhs64;
  k_rhs_fx_grp<<<k.blocks, kThreadsC, k.smem, st>>>(du, static_cast<const GR*>(k.recs), k.inst, k.first, active);
  return cudaGetLastError();
}
