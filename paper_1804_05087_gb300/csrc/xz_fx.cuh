// Plane stage of the FP64 step, tangent and adjoint in 64-bit fixed point (same mathematics as k_xz
// in kernels.cu, pseudospectral products of Sec. 3.2): per wall-normal point j, inverse FFT along x
// of every (field, kz) column, c2r along z of pairs of x-rows, the pointwise product, r2c along z,
// forward FFT along x truncated to the retained modes. Values in and out are doubles; in between
// they are integers with one power-of-two scale per stage (fx_arith.h).
//
// Why integers: the FP64 pipe issues 2 operations per SM and clock, the integer pipes about 28 multiply-
// adds of 32-bit halves or 52 additions of 64 bits (measured), and a plane's transforms need no range,
// only precision. 48 x 65 x 48, 256 tangents: 12.57 ms in FP64 registers, 3.11 ms here.
//
// Scales (every transformed value stays below 2^61). The x transforms of a group of fields
// (velocity, vorticity) are scaled by the largest sum of moduli of a column, the z transforms by
// that of the plane: bounds of every value they form, so that a rounding is 2^-60 of them. At the
// product the values of one chunk of x-rows are shifted up to their largest magnitude; the products
// keep 32 fraction bits until their own largest magnitude is known, and the rows that the r2c
// transforms leave carry an exponent per chunk, which the forward x transform brings to a common
// one. Each pass loses only what its sums can grow by. A plane with a non-finite input gives NaN.
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
  int* bmeta;          // [NY][4]: exponents and bit lengths of the two groups of the base fields
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
__host__ __device__ constexpr size_t meta_ints(int nchunk) { return 5 + 4 * (size_t)nchunk; }

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
  unsigned emax[2];      // per group: largest high word of the inputs
  int col[6 * kMaxKz];   // sums of moduli of every column in units of 2^(emax exponent - 14)
  int sh[2];             // exponents of the z transforms per group: X = v 2^sh
  int up[2];             // bits that the x transforms are scaled finer
  int bad;               // a non-finite value in the plane
  unsigned orv[2];       // high words in use by the physical values of a chunk, per group
  unsigned orr[2];       // by the products, per output group
  unsigned ors[2];       // by the rows after r2c
  i64 lam[6];
  int cexp[2][kMaxChunks];   // exponent and bit length of each chunk's rows after r2c
  int cbits[2][kMaxChunks];
  int lsh[2][kMaxPairs];     // shift of each row pair to the common exponent
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

// *dst |= v over the block's threads (converged warps)
__device__ __forceinline__ void block_or(unsigned* dst, unsigned v) {
  v = __reduce_or_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) atomicOr(dst, v);
}

// exponents of the plane's inputs. A few threads walk each column twice (the second time from the
// caches): the largest exponent, then the sums of moduli with 15-bit terms (integers, so that the
// result does not depend on the order).
__device__ __forceinline__ void plane_scale(const Args& a, Shared& s, const double2* in, size_t planeMm, int j,
                                            int nin, bool lam) {
  const int tid = threadIdx.x, ncol = nin * a.MZ;
  if (tid < 2) s.emax[tid] = 0;
  for (int i = tid; i < 6 * kMaxKz; i += kThreads) s.col[i] = 0;
  __syncthreads();
  auto top = [](double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; };
  const int per = max(1, kThreads / ncol), h0 = ncol >= kThreads ? 0 : tid / ncol;
  const int c0 = tid - h0 * ncol;
  unsigned em[2] = {0, 0};
  if (h0 < per)
    for (int c = c0; c < ncol; c += kThreads) {
      const int f = quot(c, a.dMZ);
      const double2* p = in + f * planeMm + (c - f * a.MZ);
      unsigned t = 0;
      for (int q = h0; q < a.MX; q += per) {
        const double2 v = __ldg(p + q * a.MZ);
        t = max(t, max(top(v.x), top(v.y)));
      }
      if (f < 3) em[0] = max(em[0], t);
      else em[1] = max(em[1], t);
    }
  if (lam && tid < 6) {
    const unsigned t = top(a.lam[j * 6 + tid]);
    if (tid < 3) em[0] = max(em[0], t);
    else em[1] = max(em[1], t);
  }
  __syncwarp();
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const unsigned t = __reduce_max_sync(0xffffffffu, em[g]);
    if ((tid & 31) == 0) atomicMax(&s.emax[g], t);
  }
  __syncthreads();
  const int e0[2] = {(int)(s.emax[0] >> 20), (int)(s.emax[1] >> 20)};
  auto part = [&](double v, int e) -> int {
    const unsigned h = top(v);
    return (int)(((h & 0xfffffu) | 0x100000u) >> min(31, e - (int)(h >> 20) + 6)) + 1;
  };
  if (h0 < per)
    for (int c = c0; c < ncol; c += kThreads) {
      const int f = quot(c, a.dMZ), iz = c - f * a.MZ, e = f < 3 ? e0[0] : e0[1];
      const double2* p = in + f * planeMm + iz;
      int acc = 0;
      for (int q = h0; q < a.MX; q += per) {
        const double2 v = __ldg(p + q * a.MZ);
        acc += part(v.x, e) + part(v.y, e);
      }
      atomicAdd(&s.col[f * kMaxKz + iz], acc);
    }
  __syncthreads();
  if (tid < 32) {
    int big[2] = {1, 1}, bigc[2] = {1, 1};
    for (int f = 0; f < nin; ++f) {
      int tot = 0, most = 0;
      for (int iz = tid; iz < a.MZ; iz += 32) {
        const int v = s.col[f * kMaxKz + iz];
        tot += iz == 0 ? v : 2 * v;
        most = max(most, v);
      }
      tot = __reduce_add_sync(0xffffffffu, tot);
      most = __reduce_max_sync(0xffffffffu, most);
      const int g = f < 3 ? 0 : 1;
      if (lam) tot += part(a.lam[j * 6 + f], g ? e0[1] : e0[0]);
      big[g] = max(big[g], tot);
      bigc[g] = max(bigc[g], most);
    }
    if (tid == 0) {
      // sums of moduli <= big 2^(e0 - 1023 - 14): 60 bits
      for (int g = 0; g < 2; ++g) {
        s.sh[g] = 60 - (32 - __clz(big[g]) + e0[g] - 1037);
        s.up[g] = __clz(bigc[g]) - __clz(big[g]);
      }
      s.bad = e0[0] == 0x7ff || e0[1] == 0x7ff;
    }
    __syncwarp();
    if (lam && tid < 6) s.lam[tid] = from_double(a.lam[j * 6 + tid], s.sh[tid / 3]);
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
      const int g = f < 3 ? 0 : 1, sh = s.sh[g] + s.up[g] - (KIND == kAdjoint && iz > 0 ? 1 : 0);
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
  // common exponent per group: the sums of the first pass stay below 2^61, the second pass
  // shifts its inputs by its own growth
  const int lg = 32 - __clz(N2 - 1);
  int ecom[2];
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    int top = -(1 << 28);
    for (int q = 0; q < a.nchunk; ++q) top = max(top, s.cbits[g][q] - s.cexp[g][q]);
    ecom[g] = 60 - lg - top;
  }
  for (int i = threadIdx.x; i < nx / 2; i += kThreads) {
    const int q = i / a.rp;
    s.lsh[0][i] = ecom[0] - s.cexp[0][q];
    s.lsh[1][i] = ecom[1] - s.cexp[1][q];
  }
  __syncthreads();
  with_radix(N2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < N1 * nc; idx += kThreads) {
      const int p = quot(idx, dnc), col = idx - p * nc;
      const int* ls = s.lsh[KIND == kAdjoint && c0 + col >= 3 * a.MZ ? 1 : 0];
      const cx* g = src + (size_t)(p * R) * lds + c0 + col;
      cx* x = X + p * R * ldx + col;
      cx v[R];
#pragma unroll
      for (int k = 0; k < R; ++k) {
        const int l = ls[(p * R + k) >> 1];
        v[k] = g[k * lds];
        if (l >= 0) v[k] = {shift(v[k].x, l), shift(v[k].y, l)};
        else v[k] = {shift_down(v[k].x, min(-l, 62)), shift_down(v[k].y, min(-l, 62))};
      }
      dft<R, -1>(v);
#pragma unroll
      for (int k = 0; k < R; ++k) x[k * ldx] = k == 0 ? v[0] : rot<-1>(v[k], tw[p * k]);
    }
  });
  __syncthreads();
  const double inv = 1.0 / ((double)a.nx * (double)a.nz);
  const bool bad = s.bad || (KIND != kStep && a.bmeta[4 * j] == kBadExp);
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
      const Scale sc = scale_of(bad ? nan("") : inv,
                                (KIND == kAdjoint && f >= 3 ? ecom[1] : ecom[0]) - growth(R) -
                                    (KIND == kAdjoint && iz > 0 ? 1 : 0));
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
  if (threadIdx.x == 0) s.orv[0] = s.orv[1] = s.orr[0] = s.orr[1] = s.ors[0] = s.ors[1] = 0;
  // c2r of the packed pair A + iB: spectrum A + iB at kz, conj(A) + i conj(B) at nz - kz
  with_radix(N1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < nq * nin * N2; idx += kThreads) {
      const int r = quot(idx, a.dn2z), n2 = idx - r * N2, qq = r / nin, f = r - qq * nin;
      const cx* A = src + (size_t)(2 * (q0 + qq)) * lds + f * MZ;
      const cx* B = A + lds;
      const int dn = s.up[f < 3 ? 0 : 1];
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
  unsigned o0 = 0, o1 = 0;
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
      if (f < 3) o0 |= o;
      else o1 |= o;
    }
  });
  __syncwarp();
  block_or(&s.orv[0], o0);
  if (nin == 6) block_or(&s.orv[1], o1);
  __syncthreads();
  // products: shifts that use the bits left above the chunk's largest values, so that the results
  // stay below 2^(60 - lgz) and the first pass's sums of a packed pair below 2^61; the second
  // pass shifts its inputs by its own growth
  const int lgz = 32 - __clz(N2 - 1), lgb = 32 - __clz(N1 - 1);
  const int n0 = bits(s.orv[0]), n1 = bits(s.orv[1]);
  int l0 = 0, l1 = 0, ex0 = 0, ex1 = 0;
  if (KIND == kTangent) {
    const int4 bm = __ldg(reinterpret_cast<const int4*>(a.bmeta) + j);  // exponents, bits of (U, Omega)
    l1 = min(60, 122 - lgz - bm.z) - n1;
    l0 = min(60, 122 - lgz - bm.w) - n0;
    // omega x U and u x Omega at the smaller of their exponents
    const int e1 = s.sh[1] + l1 + bm.x, e0 = s.sh[0] + l0 + bm.y, e = min(e0, e1);
    l1 -= e1 - e;
    l0 -= e0 - e;
    ex0 = e - 63;
  } else if (KIND == kAdjoint) {
    const int4 bm = __ldg(reinterpret_cast<const int4*>(a.bmeta) + j);
    l0 = min(60, 123 - lgz - max(bm.z, bm.w)) - n0;
    ex0 = s.sh[0] + l0 + bm.y - 63;
    ex1 = s.sh[0] + l0 + bm.x - 63;
  } else {
    const int m = 123 - lgz, x0 = min(60, m / 2), x1 = min(60, m - x0);
    l0 = x0 - n0;
    l1 = x1 - n1;
    ex0 = s.sh[0] + l0 + s.sh[1] + l1 - 63;
    if (threadIdx.x == 0 && a.bmeta) {
      atomicMax(a.bmeta + 4 * j + 2, n0);
      atomicMax(a.bmeta + 4 * j + 3, n1);
    }
  }
  unsigned p0 = 0, p1 = 0;
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
        const double one = s.bad ? nan("") : 1.0;
        const Scale sc[2] = {scale_of(one, s.sh[0]), scale_of(one, s.sh[1])};
#pragma unroll
        for (int f = 0; f < 6; ++f) {
          const size_t o = ((size_t)f * a.NY + j) * a.nx * nz;
          const float va = (float)scaled(F[f].x, sc[f / 3]), vb = (float)scaled(F[f].y, sc[f / 3]);
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
      // halves of the shifted values and of the base fields
      int2 x[6], b[6];
#pragma unroll
      for (int f = 0; f < nin; ++f) {
        const i64 v = shift(r ? F[f].y : F[f].x, f < 3 ? l0 : l1);
        x[f] = make_int2(half_hi(v), half_lo(v));
      }
      if (KIND != kStep) {
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
        if (c < 3) p0 |= mag(v);
        else p1 |= mag(v);
      };
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int i = (c + 1) % 3, k = (c + 2) % 3;
        Acc p, n;
        if (KIND == kTangent) {  // U_tot x omega + u x Omega_tot
          p.add(x[3 + k], b[i]);
          p.add(x[i], b[3 + k]);
          n.add(x[3 + i], b[k]);
          n.add(x[k], b[3 + i]);
          put(c, p, n);
        } else if (KIND == kAdjoint) {  // u* = Omega_tot x a, omega* = a x U_tot
          p.add(x[k], b[3 + i]);
          n.add(x[i], b[3 + k]);
          put(c, p, n);
          Acc p2, n2;
          p2.add(x[i], b[k]);
          n2.add(x[k], b[i]);
          put(3 + c, p2, n2);
        } else {  // U_tot x Omega_tot
          p.add(x[i], x[3 + k]);
          n.add(x[k], x[3 + i]);
          put(c, p, n);
        }
      }
    }
  }
  if (KIND == kStep && !a.out) {
    __syncthreads();
    return;
  }
  __syncwarp();
  block_or(&s.orr[0], p0);
  if (nout == 6) block_or(&s.orr[1], p1);
  __syncthreads();
  // r2c: input slot order, factors the other way round, natural order out; the products' fraction
  // bits fill what their largest magnitude leaves
  const int f0 = max(0, min(60 - lgz - bits(s.orr[0]), 31)), f1 = max(0, min(60 - lgz - bits(s.orr[1]), 31));
  with_radix(N2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int idx = threadIdx.x; idx < nq * nout * N1; idx += kThreads) {
      const int r = quot(idx, a.dn1z), p = idx - r * N1, qq = r / nout, f = r - qq * nout;
      cx* z = Z + (qq * NF + f) * ZF + p * P;
      const int fb = f < 3 ? f0 : f1;
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
  p0 = p1 = 0;
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
    if (f < 3) p0 |= mag(ra) | mag(rb);
    else p1 |= mag(ra) | mag(rb);
  }
  __syncwarp();
  block_or(&s.ors[0], p0);
  if (nout == 6) block_or(&s.ors[1], p1);
  __syncthreads();
  if (threadIdx.x == 0) {
    s.cexp[0][q] = ex0 + f0 - lgb;
    s.cexp[1][q] = ex1 + f1 - lgb;
    s.cbits[0][q] = bits(s.ors[0]);
    s.cbits[1][q] = bits(s.ors[1]);
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
      a.bmeta[4 * j] = s.bad ? kBadExp : s.sh[0];
      a.bmeta[4 * j + 1] = s.sh[1];
      a.bmeta[4 * j + 2] = 0;
      a.bmeta[4 * j + 3] = 0;
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
      if (part == 0 && threadIdx.x == 0) {
        meta[0] = s.sh[0];
        meta[1] = s.sh[1];
        meta[2] = s.bad;
        meta[3] = s.up[0];
        meta[4] = s.up[1];
      }
      const int ncol = nin * a.MZ, c0 = part * ncol / a.pin, nc = (part + 1) * ncol / a.pin - c0;
      x_inverse<KIND>(a, s, twx, in, planeMm, c0, nc, X, nc, G, RS);
    } else if (phase == kPhaseZ) {
      if (threadIdx.x < 2) {
        s.sh[threadIdx.x] = meta[threadIdx.x];
        s.up[threadIdx.x] = meta[3 + threadIdx.x];
      }
      if (threadIdx.x == 0) s.bad = meta[2];
      if (KIND == kStep && threadIdx.x < 6) s.lam[threadIdx.x] = from_double(a.lam[j * 6 + threadIdx.x], meta[threadIdx.x / 3]);
      __syncthreads();
      z_chunk<KIND>(a, s, twz, G, G, RS, X, part, j);
      if (threadIdx.x == 0) {
        for (int g = 0; g < 2; ++g) {
          meta[5 + g * a.nchunk + part] = s.cexp[g][part];
          meta[5 + (2 + g) * a.nchunk + part] = s.cbits[g][part];
        }
      }
    } else {
      for (int i = threadIdx.x; i < 2 * a.nchunk; i += kThreads) {
        const int g = i >= a.nchunk, q = i - g * a.nchunk;
        s.cexp[g][q] = meta[5 + i];
        s.cbits[g][q] = meta[5 + 2 * a.nchunk + i];
      }
      if (threadIdx.x == 0) s.bad = meta[2];
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
