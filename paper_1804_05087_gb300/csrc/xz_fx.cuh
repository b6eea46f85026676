// Plane stage of the FP64 step, tangent and adjoint in 64-bit fixed point (same mathematics as k_xz
// in kernels.cu, pseudospectral products of Sec. 3.2): per wall-normal point j, inverse FFT along x
// of every (field, kz) column, c2r along z of pairs of x-rows, the pointwise product, r2c along z,
// forward FFT along x truncated to the retained modes. Values in and out are doubles; in between
// they are integers with one power-of-two scale per stage (fx_arith.h).
//
// Why integers: an SM does 25 multiply-adds of 32-bit halves and 56 additions of 64 bits per clock but 1.7 in
// FP64 (fx_arith.h), and a plane's transforms need no range, only precision. 48 x 65 x 48, 256 tangents:
// 12.57 ms in FP64 registers, 3.16 ms here, of which the multiply-adds alone are 0.68 (three per real product;
// the rest is shifts, carries, barriers and instruction fetch).
//
// Scales (every transformed value stays below 2^61). The x transforms of a field are scaled by the
// largest sum of moduli of its columns, the z transforms by that of its plane: bounds of every value
// they form, so that a rounding is 2^-60 of them. Every field has its own scale: v beside u near a
// wall, or v and w of a nearly streamwise-constant flow, keep their bits. At the product the values
// of one chunk of x-rows are shifted up to their field's largest magnitude there, and each term of an
// output component is shifted down to the component's coarsest exponent: a rounding is 2^-60 of the
// largest term. The products keep 32 fraction bits until their component's largest magnitude is known,
// and the rows that the r2c transforms leave carry an exponent per component and chunk, which the
// forward x transform brings to a common one. A plane with a non-finite input gives NaN.
//
// Transforms. Length N = N1 N2 with N1, N2 in {2, 3, 4, 6, 8, 9, 12}: N2 transforms of length N1
// in registers, a twiddle, N1 transforms of length N2, in place in shared memory. The inverse
// leaves element k = k1 + N1 k2 at slot k1 N2 + k2; the forward transform takes that order and
// runs the factors the other way round, so no pass reorders the data. Rows (x) are paired by slot.
#pragma once

#include "fx_arith.h"
#include "sp_internal.h"

namespace fxz {

using namespace fx;

constexpr int kThreads = 256;
constexpr int kPhaseIn = 1, kPhaseZ = 2, kPhaseOut = 4;
constexpr int kBadExp = 1 << 28;   // exponent that marks a non-finite base plane
constexpr int kMaxKz = 48;         // stored kz of a plane
constexpr int kMaxChunks = 72;     // chunks of row pairs per plane
constexpr int kMaxPairs = 72;      // row pairs of a plane

// one kernel per kind: the step and the base fields, the tangent, the adjoint
enum Kind { kStep, kTangent, kAdjoint };

struct Args {
  const double2* in;   // [dir][NIN][NY][Mm]
  double2* out;        // [dir][NOUT][NY][Mm]; null: no product (base fields only)
  int4* bfx;           // [NY][nx][nz][6] base fields (U_tot, Omega_tot), slot order, as halves (high,
                       // low): read by the tangent and the adjoint, written by the step (null: not)
  int* bmeta;          // [NY][12]: exponents, then bit lengths, of the base fields
  float* b32;          // [6][NY][nx][nz] and [6][NY][nz][nx] float base fields, written by the step
  float* b32t;         // (null: not)
  const double* lam;   // [NY][6] laminar U and Omega
  const int4* tw;      // [nx] then [nz]: cos, sin of 2 pi k / n as halves of 62-bit constants
  cx* G;               // split launches: [dir][NY][nx][6 MZ] between the phases
  int* gmeta;          // split launches: [dir][NY][meta_ints]
  int nx, nz, NY, Mm, MX, MZ, Kx, Kz;
  int n1x, n2x, n1z, n2z;
  Div dMZ, dnz, dn1z, dn2z, dn2x;
  int rp, nchunk;      // row pairs per chunk, chunks per plane
  int pin, pout;       // split launches: blocks per plane of the x transforms
  const int* active;   // split launches of a group member: device flag, 0 = do nothing (null: run)
};

// integers that a split call keeps per plane between its launches
__host__ __device__ constexpr size_t meta_ints(int nchunk) { return 13 + 12 * (size_t)nchunk; }

template <class F>
__device__ __forceinline__ void with_radix(int r, F f) {
  switch (r) {
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    case 8: f(std::integral_constant<int, 8>{}); break;
    case 9: f(std::integral_constant<int, 9>{}); break;
    default: f(std::integral_constant<int, 12>{}); break;
  }
}

struct Shared {
  unsigned emax[6];      // per field: largest high word of the inputs
  int sh[6];             // exponents of the z transforms: X = v 2^sh
  int up[6];             // bits that the x transforms are scaled finer
  int bad;               // a non-finite value in the plane
  unsigned orv[6];       // high words in use by the physical values of a chunk, per field
  unsigned orr[6];       // by the products, per output component
  unsigned ors[6];       // by the rows after r2c
  int ex[6];             // exponents of a chunk's products
  int ecom[6];           // exponents of the forward x transforms
  i64 lam[6];
  union {
    int col[6 * kMaxKz];  // sums of moduli of every column in units of 2^(emax exponent - 14)
    struct {
      short cexp[6][kMaxChunks];        // exponent and bit length of each chunk's rows after r2c
      signed char cbits[6][kMaxChunks];
      signed char lsh[6][kMaxPairs];    // shift of each row pair to the common exponent
    };
  };
};

// ceil(log2 n), n >= 2: bits that a sum of n terms can grow by
__host__ __device__ constexpr int growth(int n) {
  int b = 0;
  while ((1 << b) < n) ++b;
  return b;
}
// bit length of the magnitudes whose high words were or-ed (at least 32)
__device__ __forceinline__ int bits(unsigned o) { return 64 - __clz((int)o); }
__device__ __forceinline__ unsigned mag(i64 v) {
  const int h = (int)(v >> 32);
  return (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned mag(cx v) { return mag(v.x) | mag(v.y); }

// dst[i] |= v[i] over the block's threads (converged warps)
template <int N>
__device__ __forceinline__ void block_or(unsigned* dst, const unsigned (&v)[N]) {
  const int lane = threadIdx.x & 31;
  unsigned mine = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const unsigned t = __reduce_or_sync(0xffffffffu, v[i]);
    if (lane == i) mine = t;
  }
  if (lane < N) atomicOr(dst + lane, mine);
}
// v[f] |= o, f known at run time only
template <int N>
__device__ __forceinline__ void or_at(unsigned (&v)[N], int f, unsigned o) {
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i == f) v[i] |= o;
}

// exponents of the plane's fields. A few threads walk each column twice (the second time from the
// caches): the largest exponent, then the sums of moduli with 15-bit terms (integers, so that the
// result does not depend on the order). The laminar profile counts in the field it is added to.
__device__ __forceinline__ void plane_scale(const Args& a, Shared& s, const double2* in, size_t planeMm, int j,
                                            int nin, bool lam) {
  const int tid = threadIdx.x, ncol = nin * a.MZ;
  if (tid < 6) s.emax[tid] = 0;
  if (tid == 0) s.bad = 0;
  for (int i = tid; i < 6 * kMaxKz; i += kThreads) s.col[i] = 0;
  __syncthreads();
  auto top = [](double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; };
  const int per = max(1, kThreads / ncol), h0 = ncol >= kThreads ? 0 : tid / ncol;
  const int c0 = tid - h0 * ncol;
  if (h0 < per)
    for (int c = c0; c < ncol; c += kThreads) {
      const int f = quot(c, a.dMZ);
      const double2* p = in + f * planeMm + (c - f * a.MZ);
      unsigned t = 0;
      for (int q = h0; q < a.MX; q += per) {
        const double2 v = __ldg(p + q * a.MZ);
        t = max(t, max(top(v.x), top(v.y)));
      }
      atomicMax(&s.emax[f], t);
    }
  if (lam && tid < 6) atomicMax(&s.emax[tid], top(a.lam[j * 6 + tid]));
  __syncthreads();
  auto part = [&](double v, int e) -> int {
    const unsigned h = top(v);
    return (int)(((h & 0xfffffu) | 0x100000u) >> min(31, e - (int)(h >> 20) + 6)) + 1;
  };
  if (h0 < per)
    for (int c = c0; c < ncol; c += kThreads) {
      const int f = quot(c, a.dMZ), iz = c - f * a.MZ, e = (int)(s.emax[f] >> 20);
      const double2* p = in + f * planeMm + iz;
      int acc = 0;
      for (int q = h0; q < a.MX; q += per) {
        const double2 v = __ldg(p + q * a.MZ);
        acc += part(v.x, e) + part(v.y, e);
      }
      atomicAdd(&s.col[f * kMaxKz + iz], acc);
    }
  __syncthreads();
  static_assert(kThreads >= 6 * 32, "a warp per field");
  const int f = tid >> 5;
  if (f < nin) {
    const int e = (int)(s.emax[f] >> 20);
    int tot = 0, most = 0;
    for (int iz = tid & 31; iz < a.MZ; iz += 32) {
      const int v = s.col[f * kMaxKz + iz];
      tot += iz == 0 ? v : 2 * v;
      most = max(most, v);
    }
    tot = __reduce_add_sync(0xffffffffu, tot);
    most = __reduce_max_sync(0xffffffffu, most);
    if ((tid & 31) == 0) {
      if (lam) tot += part(a.lam[j * 6 + f], e);
      // sums of moduli <= tot 2^(e - 1023 - 14): 60 bits
      const int sh = 60 - (32 - __clz(tot) + e - 1037);
      s.sh[f] = sh;
      s.up[f] = __clz(most) - __clz(tot);
      if (e == 0x7ff) s.bad = 1;
      if (lam) s.lam[f] = from_double(a.lam[j * 6 + f], sh);
    }
  }
  __syncthreads();
}

// inverse x transforms of the columns [c0, c0 + nc) (column = field MZ + iz): X[slot][ldx], X
// column 0 = c0; the result goes to dst[slot * ldd + column]
template <Kind KIND>
__device__ __forceinline__ void x_inverse(const Args& a, const Shared& s, const int4* tw, const double2* in,
                                          size_t planeMm, int c0, int nc, cx* X, int ldx, cx* dst, int ldd) {
  const int N1 = a.n1x, N2 = a.n2x, nx = a.nx;
  const Div dnc = div_of(nc);
  with_radix(N1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < N2 * nc; idx += kThreads) {
      const int n2 = quot(idx, dnc), col = idx - n2 * nc;
      const int f = quot(c0 + col, a.dMZ), iz = c0 + col - f * a.MZ;
      // the adjoint's transposed forward transform halves the iz > 0 terms
      const int sh = s.sh[f] + s.up[f] - (KIND == kAdjoint && iz > 0 ? 1 : 0);
      const double2* p = in + f * planeMm + iz;
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) {
        const int e = k * N2 + n2;
        v[k] = {0, 0};
        if (e <= a.Kx || e >= nx - a.Kx) {
          const double2 d = __ldg(p + (e <= a.Kx ? e : e - nx + a.MX) * a.MZ);
          v[k] = {from_double(d.x, sh), from_double(d.y, sh)};
        }
      }
      dft<R, 1>(v);
      cx* x = X + n2 * ldx + col;
#pragma unroll
      for (int k = 0; k < R; ++k) x[k * N2 * ldx] = k == 0 ? v[0] : rot<1>(v[k], tw[n2 * k]);
    }
  });
  __syncthreads();
  with_radix(N2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < N1 * nc; idx += kThreads) {
      const int k1 = quot(idx, dnc), col = idx - k1 * nc;
      const cx* x = X + k1 * R * ldx + col;
      cx* d = dst + (size_t)(k1 * R) * ldd + c0 + col;
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) v[k] = x[k * ldx];
      dft<R, 1>(v);
#pragma unroll
      for (int k = 0; k < R; ++k) d[k * ldd] = v[k];
    }
  });
}

// forward x transforms of the output columns [c0, c0 + nc): rows from src[slot * lds + column],
// each brought from its chunk's exponent to the common one
template <Kind KIND>
__device__ __forceinline__ void x_forward(const Args& a, Shared& s, const int4* tw, const cx* src, int lds, int c0,
                                          int nc, cx* X, int ldx, double2* out, size_t planeMm, int j) {
  const int N1 = a.n1x, N2 = a.n2x, nx = a.nx;
  const Div dnc = div_of(nc);
  // common exponent per component (a warp each): the sums of the first pass stay below 2^61, the
  // second pass shifts its inputs by its own growth
  const int lg = 32 - __clz(N2 - 1);
  constexpr int nout = KIND == kAdjoint ? 6 : 3;
  if (const int f = threadIdx.x >> 5, lane = threadIdx.x & 31; f < nout) {
    int top = -(1 << 28);
    for (int q = lane; q < a.nchunk; q += 32) top = max(top, s.cbits[f][q] - s.cexp[f][q]);
    const int e = 60 - lg - __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) s.ecom[f] = e;
    for (int i = lane; i < nx / 2; i += 32) s.lsh[f][i] = (signed char)max(-62, min(e - s.cexp[f][i / a.rp], 63));
  }
  __syncthreads();
  with_radix(N2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < N1 * nc; idx += kThreads) {
      const int p = quot(idx, dnc), col = idx - p * nc;
      const signed char* ls = s.lsh[quot(c0 + col, a.dMZ)];
      const cx* g = src + (size_t)(p * R) * lds + c0 + col;
      cx* x = X + p * R * ldx + col;
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) {
        const int l = ls[(p * R + k) >> 1];
        v[k] = g[k * lds];
        if (l >= 0) v[k] = {shift(v[k].x, l), shift(v[k].y, l)};
        else v[k] = {shift_down(v[k].x, -l), shift_down(v[k].y, -l)};
      }
      dft<R, -1>(v);
#pragma unroll
      for (int k = 0; k < R; ++k) x[k * ldx] = k == 0 ? v[0] : rot<-1>(v[k], tw[p * k]);
    }
  });
  __syncthreads();
  const double inv = 1.0 / ((double)a.nx * (double)a.nz);
  const bool bad = s.bad || (KIND != kStep && a.bmeta[12 * j] == kBadExp);
  with_radix(N1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < N2 * nc; idx += kThreads) {
      const int kb = quot(idx, dnc), col = idx - kb * nc;
      const int f = quot(c0 + col, a.dMZ), iz = c0 + col - f * a.MZ;
      const cx* x = X + kb * ldx + col;
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) {
        v[k] = x[k * N2 * ldx];
        v[k] = {shift_down(v[k].x, growth(R)), shift_down(v[k].y, growth(R))};
      }
      dft<R, -1>(v);
      // the adjoint's transposed inverse transform doubles the iz > 0 terms
      const Scale sc = scale_of(bad ? nan("") : inv, s.ecom[f] - growth(R) - (KIND == kAdjoint && iz > 0 ? 1 : 0));
      double2* o = out + f * planeMm + iz;
#pragma unroll
      for (int k = 0; k < R; ++k) {
        const int e = k * N2 + kb;
        if (e > a.Kx && e < nx - a.Kx) continue;
        o[(e <= a.Kx ? e : e - nx + a.MX) * a.MZ] = make_double2(scaled(v[k].x, sc), scaled(v[k].y, sc));
      }
    }
  });
}

// The products: term t of output component t / per is an input field times another field (the step: a
// vorticity; else a base field); the first half of a component's terms is added, the second subtracted.
// i = c + 1, k = c + 2 (mod 3).
template <Kind KIND>
struct Terms;
template <>
struct Terms<kStep> {  // U_i Omega_k - U_k Omega_i
  static constexpr int per = 2, count = 6;
  static __device__ __forceinline__ constexpr int input(int t) { return (t / 2 + 1 + t % 2) % 3; }
  static __device__ __forceinline__ constexpr int other(int t) { return 3 + (t / 2 + 2 - t % 2) % 3; }
};
template <>
struct Terms<kTangent> {  // omega_k U_i + u_i Omega_k - omega_i U_k - u_k Omega_i
  static constexpr int per = 4, count = 12;
  static __device__ __forceinline__ constexpr int input(int t) {
    const int c = t / 4, i = (c + 1) % 3, k = (c + 2) % 3, q = t % 4;
    return q == 0 ? 3 + k : q == 1 ? i : q == 2 ? 3 + i : k;
  }
  static __device__ __forceinline__ constexpr int other(int t) {
    const int c = t / 4, i = (c + 1) % 3, k = (c + 2) % 3, q = t % 4;
    return q == 0 ? i : q == 1 ? 3 + k : q == 2 ? k : 3 + i;
  }
};
template <>
struct Terms<kAdjoint> {  // u* = Omega x a: a_k Omega_i - a_i Omega_k; omega* = a x U: a_i U_k - a_k U_i
  static constexpr int per = 2, count = 12;
  static __device__ __forceinline__ constexpr int input(int t) {
    const int c = t / 2 % 3;
    return (c + (t < 6 ? 2 - t % 2 : 1 + t % 2)) % 3;
  }
  static __device__ __forceinline__ constexpr int other(int t) {
    const int c = t / 2 % 3;
    return t < 6 ? 3 + (c + 1 + t % 2) % 3 : (c + 2 - t % 2) % 3;
  }
};

// products of two fixed-point values by halves: the sum's high part and its 32 fraction bits
struct Acc {
  i64 m = 0, h = 0;
  __device__ __forceinline__ void add(int2 p, int2 q) {
    m = wide(p.x, q.x, m);
    h = wide(p.x, q.y, wide(p.y, q.x, h));
  }
};

// z transforms and products of the row pairs of chunk q: rows src[slot * lds + field MZ + kz]
// in, the same layout out (in place when src = dst); Z: [rp][zf][n1z (n2z + 1)], zf fields of a
// pair: the values, over them the products, then their fractions
template <Kind KIND>
constexpr int kZf = KIND == kAdjoint ? 12 : 6;

template <Kind KIND>
__device__ __forceinline__ void z_chunk(const Args& a, Shared& s, const int4* tw, const cx* src, cx* dst, int lds,
                                        cx* Z, int q, int j) {
  constexpr int nin = KIND == kAdjoint ? 3 : 6, nout = KIND == kAdjoint ? 6 : 3, NF = kZf<KIND>;
  const int N1 = a.n1z, N2 = a.n2z, nz = a.nz, MZ = a.MZ, P = N2 + 1, ZF = N1 * P;
  const int q0 = q * a.rp, nq = min(a.rp, a.nx / 2 - q0);
  if (threadIdx.x < 6) s.orv[threadIdx.x] = s.orr[threadIdx.x] = s.ors[threadIdx.x] = 0;
  // c2r of the packed pair A + iB: spectrum A + iB at kz, conj(A) + i conj(B) at nz - kz
  with_radix(N1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < nq * nin * N2; idx += kThreads) {
      const int r = quot(idx, a.dn2z), n2 = idx - r * N2, qq = r / nin, f = r - qq * nin;
      const cx* A = src + (size_t)(2 * (q0 + qq)) * lds + f * MZ;
      const cx* B = A + lds;
      const int dn = s.up[f];
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) {
        const int e = k * N2 + n2, m = min(e, nz - e);
        v[k] = {0, 0};
        if (m <= a.Kz) {
          cx p = A[m], t = B[m];
          if (m == 0) p.y = t.y = 0;
          v[k] = m == e ? cx{p.x - t.y, p.y + t.x} : cx{p.x + t.y, t.x - p.y};
          v[k] = {shift_down(v[k].x, dn), shift_down(v[k].y, dn)};
        }
      }
      dft<R, 1>(v);
      cx* z = Z + (qq * NF + f) * ZF + n2;
#pragma unroll
      for (int k = 0; k < R; ++k) z[k * P] = k == 0 ? v[0] : rot<1>(v[k], tw[n2 * k]);
    }
  });
  __syncthreads();
  unsigned ov[nin] = {};
  with_radix(N2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < nq * nin * N1; idx += kThreads) {
      const int r = quot(idx, a.dn1z), k1 = idx - r * N1, qq = r / nin, f = r - qq * nin;
      cx* z = Z + (qq * NF + f) * ZF + k1 * P;
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) v[k] = z[k];
      dft<R, 1>(v);
      const i64 lam = KIND == kStep ? s.lam[f] : 0;
      unsigned o = 0;
#pragma unroll
      for (int k = 0; k < R; ++k) {
        if (KIND == kStep) v[k] = {v[k].x + lam, v[k].y + lam};
        o |= mag(v[k]);
        z[k] = v[k];
      }
      or_at(ov, f, o);
    }
  });
  __syncwarp();
  block_or(s.orv, ov);
  __syncthreads();
  // Products: shifts that use the bits left above the chunk's largest values, so that the results
  // stay below 2^(60 - lgz) and the first pass's sums of a packed pair below 2^61; the second pass
  // shifts its inputs by its own growth. Lane t of every warp takes term t: its factor of the inputs
  // at as many bits as its other factor (and their number per component) leaves, less what brings it to the
  // component's coarsest exponent.
  const int lgz = 32 - __clz(N2 - 1), lgb = 32 - __clz(N1 - 1);
  const int xa = KIND == kTangent ? 122 - lgz : 123 - lgz;  // bits of both factors
  const int x0 = min(60, xa / 2), x1 = min(60, xa - x0);    // the step's velocity and vorticity
  int down[Terms<KIND>::count];  // of a value of 60 bits
  {
    using TT = Terms<KIND>;
    const int lane = threadIdx.x & 31, t = min(lane, TT::count - 1), fx = TT::input(t), fb = TT::other(t);
    const int n = bits(s.orv[fx]);
    int most, eb;
    if (KIND == kStep) {
      most = x0;
      eb = s.sh[fb] + x1 - bits(s.orv[fb]);
    } else {
      eb = __ldg(a.bmeta + 12 * j + fb);
      most = min(60, xa - __ldg(a.bmeta + 12 * j + 6 + fb));
    }
    const int e = s.sh[fx] + most - n + eb;
    int least = min(e, __shfl_xor_sync(0xffffffffu, e, 1));
    if (TT::per == 4) least = min(least, __shfl_xor_sync(0xffffffffu, least, 2));
    const int d = min(60 - most + (e - least), 63);
#pragma unroll
    for (int i = 0; i < TT::count; ++i) down[i] = __shfl_sync(0xffffffffu, d, i);
    if (threadIdx.x < TT::count && lane % TT::per == 0) s.ex[lane / TT::per] = least - 63;
    if (KIND == kStep && a.bmeta && threadIdx.x < 6) atomicMax(a.bmeta + 12 * j + 6 + threadIdx.x, bits(s.orv[threadIdx.x]));
  }
  int full[nin];  // shifts of the inputs to 60 bits (the step's vorticity: to x1)
#pragma unroll
  for (int f = 0; f < nin; ++f) full[f] = (KIND == kStep && f >= 3 ? x1 : 60) - bits(s.orv[f]);
  unsigned pv[nout] = {};
  for (int idx = threadIdx.x; idx < nq * nz; idx += kThreads) {
    const int qq = quot(idx, a.dnz), zi = idx - qq * nz, z1 = quot(zi, a.dn2z);
    cx* z = Z + qq * NF * ZF + zi + z1;  // slot z1 (N2 + 1) + zi - z1 N2
    cx F[nin];
#pragma unroll
    for (int f = 0; f < nin; ++f) F[f] = z[f * ZF];
    const int slot0 = 2 * (q0 + qq);
    const size_t pt = ((size_t)j * a.nx + slot0) * nz + zi;  // point of the first row; second: + nz
    if (KIND == kStep) {
      if (a.bfx) {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int f = 0; f < 6; f += 2) {
            const i64 u = r ? F[f].y : F[f].x, v = r ? F[f + 1].y : F[f + 1].x;
            a.bfx[(pt + r * nz) * 3 + f / 2] = make_int4(half_hi(u), half_lo(u), half_hi(v), half_lo(v));
          }
      }
      if (a.b32) {
        const int zn = z1 + N1 * (zi - z1 * N2);
        const int sa = quot(slot0, a.dn2x), sb = quot(slot0 + 1, a.dn2x);
        const int xa = sa + a.n1x * (slot0 - sa * a.n2x), xb = sb + a.n1x * (slot0 + 1 - sb * a.n2x);
#pragma unroll
        for (int f = 0; f < 6; ++f) {
          const size_t o = ((size_t)f * a.NY + j) * a.nx * nz;
          const float va = s.bad ? nanf("") : (float)from_fixed(F[f].x, s.sh[f]);
          const float vb = s.bad ? nanf("") : (float)from_fixed(F[f].y, s.sh[f]);
          a.b32[o + xa * nz + zn] = va;
          a.b32[o + xb * nz + zn] = vb;
          a.b32t[o + zn * a.nx + xa] = va;
          a.b32t[o + zn * a.nx + xb] = vb;
        }
      }
      if (!a.out) continue;
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      // the shifted values and the halves of the base fields (the step: of the vorticity)
      i64 x[nin];
      int2 b[6];
#pragma unroll
      for (int f = 0; f < nin; ++f) x[f] = shift(r ? F[f].y : F[f].x, full[f]);
      if constexpr (KIND == kStep) {
#pragma unroll
        for (int f = 3; f < 6; ++f) b[f] = make_int2(half_hi(x[f]), half_lo(x[f]));
      } else {
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const int4 t = __ldg(a.bfx + (pt + r * nz) * 3 + f);
          b[2 * f] = make_int2(t.x, t.y);
          b[2 * f + 1] = make_int2(t.z, t.w);
        }
      }
      auto put = [&](int c, const Acc& p, const Acc& n) {
        const i64 h = p.h - n.h, v = p.m - n.m + (h >> 32);
        reinterpret_cast<int*>(z + (nout + c) * ZF)[r] = (int)h;  // fraction
        if (r) z[c * ZF].y = v;
        else z[c * ZF].x = v;
        pv[c] |= mag(v);
      };
      using TT = Terms<KIND>;
#pragma unroll
      for (int c = 0; c < nout; ++c) {
        Acc p, n;
#pragma unroll
        for (int q = 0; q < TT::per; ++q) {
          const int t = c * TT::per + q;
          const i64 v = x[TT::input(t)] >> down[t];
          (2 * q < TT::per ? p : n).add(make_int2(half_hi(v), half_lo(v)), b[TT::other(t)]);
        }
        put(c, p, n);
      }
    }
  }
  if (KIND == kStep && !a.out) {
    __syncthreads();
    return;
  }
  __syncwarp();
  block_or(s.orr, pv);
  __syncthreads();
  // r2c: input slot order, factors the other way round, natural order out; the products' fraction
  // bits fill what their largest magnitude leaves
  auto fraction = [&](int f) { return max(0, min(60 - lgz - bits(s.orr[f]), 31)); };
  with_radix(N2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < nq * nout * N1; idx += kThreads) {
      const int r = quot(idx, a.dn1z), p = idx - r * N1, qq = r / nout, f = r - qq * nout;
      cx* z = Z + (qq * NF + f) * ZF + p * P;
      const int fb = fraction(f);
      const u64 rnd = 1ull << (31 - fb);
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) {
        const uint2 fr = *reinterpret_cast<const uint2*>(z + nout * ZF + k);
        v[k] = z[k];
        v[k] = {(i64)((u64)v[k].x << fb) + (i64)((fr.x + rnd) >> (32 - fb)),
                (i64)((u64)v[k].y << fb) + (i64)((fr.y + rnd) >> (32 - fb))};
      }
      dft<R, -1>(v);
#pragma unroll
      for (int k = 0; k < R; ++k) z[k] = k == 0 ? v[0] : rot<-1>(v[k], tw[p * k]);
    }
  });
  __syncthreads();
  with_radix(N1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < nq * nout * N2; idx += kThreads) {
      const int r = quot(idx, a.dn2z), kb = idx - r * N2, qq = r / nout, f = r - qq * nout;
      cx* z = Z + (qq * NF + f) * ZF + kb;
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) v[k] = {shift_down(z[k * P].x, growth(R)), shift_down(z[k * P].y, growth(R))};
      dft<R, -1>(v);
#pragma unroll
      for (int k = 0; k < R; ++k) z[k * P] = v[k];
    }
  });
  __syncthreads();
  unsigned sv[nout] = {};
  // twice the two real rows' spectra: X(k) + conj X(-k) and (X(k) - conj X(-k)) / i
  for (int idx = threadIdx.x; idx < nq * nout * MZ; idx += kThreads) {
    const int r = quot(idx, a.dMZ), k = idx - r * MZ, qq = r / nout, f = r - qq * nout;
    const cx* z = Z + (qq * NF + f) * ZF;
    const int m = k == 0 ? 0 : nz - k;
    const cx u = z[k + quot(k, a.dn2z)], v = z[m + quot(m, a.dn2z)];
    cx* A = dst + (size_t)(2 * (q0 + qq)) * lds + f * MZ + k;
    const cx ra = {u.x + v.x, u.y - v.y}, rb = {u.y + v.y, v.x - u.x};
    A[0] = ra;
    A[lds] = rb;
    or_at(sv, f, mag(ra) | mag(rb));
  }
  __syncwarp();
  block_or(s.ors, sv);
  __syncthreads();
  if (const int f = threadIdx.x; f < nout) {
    s.cexp[f][q] = (short)max(-30000, min(s.ex[f] + fraction(f) - lgb, 30000));
    s.cbits[f][q] = (signed char)bits(s.ors[f]);
  }
}

// One plane. Fused (SPLIT = false): all phases, the plane in shared memory. SPLIT: one phase per
// launch, the plane in global memory between them; part = column block, row-pair chunk or column
// block of the output. The arithmetic does not depend on the choice.
template <Kind KIND, bool SPLIT>
__device__ __forceinline__ void plane(const Args& a, int phase, int part, int j, int dir, unsigned char* smem,
                                      Shared& s) {
  constexpr int nin = KIND == kAdjoint ? 3 : 6, nout = KIND == kAdjoint ? 6 : 3;
  int4* twx = reinterpret_cast<int4*>(smem);
  int4* twz = twx + a.nx;
  cx* X = reinterpret_cast<cx*>(twz + a.nz);
  for (int i = threadIdx.x; i < a.nx + a.nz; i += kThreads) twx[i] = __ldg(a.tw + i);
  const size_t planeMm = (size_t)a.NY * a.Mm;
  const double2* in = a.in + (size_t)dir * nin * planeMm + (size_t)j * a.Mm;
  double2* out = a.out + (size_t)dir * nout * planeMm + (size_t)j * a.Mm;
  const int RS = 6 * a.MZ;
  auto begin = [&]() {
    plane_scale(a, s, in, planeMm, j, nin, KIND == kStep);
    if (KIND == kStep && threadIdx.x == 0 && part == 0 && a.bmeta) {
      for (int f = 0; f < 6; ++f) {
        a.bmeta[12 * j + f] = f == 0 && s.bad ? kBadExp : s.sh[f];
        a.bmeta[12 * j + 6 + f] = 0;
      }
    }
  };
  if constexpr (!SPLIT) {
    cx* Z = X + (size_t)a.nx * RS;
    begin();
    x_inverse<KIND>(a, s, twx, in, planeMm, 0, nin * a.MZ, X, RS, X, RS);
    __syncthreads();
    for (int q = 0; q < a.nchunk; ++q) z_chunk<KIND>(a, s, twz, X, X, RS, Z, q, j);
    if (KIND == kStep && !a.out) return;
    __syncthreads();
    x_forward<KIND>(a, s, twx, X, RS, 0, nout * a.MZ, X, RS, out, planeMm, j);
  } else {
    cx* G = a.G + ((size_t)dir * a.NY + j) * a.nx * RS;
    int* meta = a.gmeta + ((size_t)dir * a.NY + j) * meta_ints(a.nchunk);
    if (phase == kPhaseIn) {
      begin();
      if (part == 0 && threadIdx.x < nin) {
        meta[threadIdx.x] = s.sh[threadIdx.x];
        meta[6 + threadIdx.x] = s.up[threadIdx.x];
        if (threadIdx.x == 0) meta[12] = s.bad;
      }
      const int ncol = nin * a.MZ, c0 = part * ncol / a.pin, nc = (part + 1) * ncol / a.pin - c0;
      x_inverse<KIND>(a, s, twx, in, planeMm, c0, nc, X, nc, G, RS);
    } else if (phase == kPhaseZ) {
      if (const int f = threadIdx.x; f < nin) {
        s.sh[f] = meta[f];
        s.up[f] = meta[6 + f];
        if (f == 0) s.bad = meta[12];
        if (KIND == kStep) s.lam[f] = from_double(a.lam[j * 6 + f], meta[f]);
      }
      __syncthreads();
      z_chunk<KIND>(a, s, twz, G, G, RS, X, part, j);
      if (const int f = threadIdx.x; f < nout) {  // the thread that wrote them
        meta[13 + f * a.nchunk + part] = s.cexp[f][part];
        meta[13 + (6 + f) * a.nchunk + part] = s.cbits[f][part];
      }
    } else {
      for (int i = threadIdx.x; i < nout * a.nchunk; i += kThreads) {
        const int f = i / a.nchunk, q = i - f * a.nchunk;
        s.cexp[f][q] = (short)meta[13 + i];
        s.cbits[f][q] = (signed char)meta[13 + 6 * a.nchunk + i];
      }
      if (threadIdx.x == 0) s.bad = meta[12];
      __syncthreads();
      const int ncol = nout * a.MZ, c0 = part * ncol / a.pout, nc = (part + 1) * ncol / a.pout - c0;
      x_forward<KIND>(a, s, twx, G, RS, c0, nc, X, nc, out, planeMm, j);
    }
  }
}

constexpr size_t kSmemMax = 227 * 1024 - sizeof(Shared) - sizeof(Args) - 64;

template <Kind KIND>
__global__ void __launch_bounds__(kThreads, 2) k_xz_fx(const __grid_constant__ Args a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared s;
  plane<KIND, false>(a, 0, 0, blockIdx.x, blockIdx.y, smem, s);
}

template <Kind KIND>
__global__ void __launch_bounds__(kThreads, 2) k_xz_fx_part(const __grid_constant__ Args a, int phase) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared s;
  if (a.active && !*a.active) return;
  plane<KIND, true>(a, phase, blockIdx.x, blockIdx.y, blockIdx.z, smem, s);
}

// Planes of several contexts: block b is plane b - first[inst[b]] of member inst[b]. mode: what a
// step launch leaves out of the member's record (XZ_STEP: no base fields, XZ_BASE: no product).
template <Kind KIND>
__global__ void __launch_bounds__(kThreads, 2) k_xz_fx_grp(const Args* __restrict__ recs, const int* __restrict__ inst,
                                                           const int* __restrict__ first,
                                                           const int* __restrict__ active, int mode) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared s;
  __shared__ Args a;
  const int i = inst[blockIdx.x];
  if (active && !active[i]) return;
  if (threadIdx.x == 0) {
    a = recs[i];
    if (KIND == kStep && mode == XZ_STEP) {
      a.bfx = nullptr;
      a.bmeta = nullptr;
      a.b32 = nullptr;
    }
    if (KIND == kStep && mode == XZ_BASE) a.out = nullptr;
  }
  __syncthreads();
  plane<KIND, false>(a, 0, 0, blockIdx.x - first[i], 0, smem, s);
}

// Launch of one kind: one block per plane (smem: shared memory of a block), or three launches with
// several blocks per plane
template <Kind KIND>
cudaError_t launch_kind(const Args& a, int n_dir, bool split, size_t smem, cudaStream_t st) {
  auto kern = k_xz_fx<KIND>;
  auto part = k_xz_fx_part<KIND>;
  if (!split) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(a.NY, n_dir), kThreads, smem, st>>>(a);
    return cudaGetLastError();
  }
  cudaError_t e = cudaFuncSetAttribute(part, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  part<<<dim3(a.pin, a.NY, n_dir), kThreads, smem, st>>>(a, kPhaseIn);
  part<<<dim3(a.nchunk, a.NY, n_dir), kThreads, smem, st>>>(a, kPhaseZ);
  if (KIND != kStep || a.out) part<<<dim3(a.pout, a.NY, n_dir), kThreads, smem, st>>>(a, kPhaseOut);
  return cudaGetLastError();
}
template <Kind KIND>
cudaError_t launch_kind_grp(const GrpKernel& k, const int* active, int mode, cudaStream_t st) {
  auto kern = k_xz_fx_grp<KIND>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
  if (e != cudaSuccess) return e;
  kern<<<k.blocks, kThreads, k.smem, st>>>(static_cast<const Args*>(k.recs), k.inst, k.first, active, mode);
  return cudaGetLastError();
}

// defined in xz_fx_{step,tangent,adjoint}.cu (one translation unit per kind)
cudaError_t launch_step(const Args& a, int n_dir, bool split, size_t smem, cudaStream_t st);
cudaError_t launch_tangent(const Args& a, int n_dir, bool split, size_t smem, cudaStream_t st);
cudaError_t launch_adjoint(const Args& a, int n_dir, bool split, size_t smem, cudaStream_t st);
cudaError_t launch_step_grp(const GrpKernel& k, const int* active, int mode, cudaStream_t st);
cudaError_t launch_tangent_grp(const GrpKernel& k, const int* active, int mode, cudaStream_t st);

}  // namespace fxz
