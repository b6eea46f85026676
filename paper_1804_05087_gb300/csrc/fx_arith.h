// 64-bit fixed-point complex arithmetic for the FP64 plane stage (xz_fx.cu).
//
// This GPU does 25 integer multiply-adds of 32 bits with a 64-bit sum and 56 64-bit additions per SM
// and clock against 1.7 FP64 ones (measured: lanes of mad.wide.s32, add.s64 and fma.f64 in loops of nothing
// else, each operand from the step before), so a transform whose values share one scale runs in
// integers: a value v is the integer X = v 2^sh, |X| < 2^61, with 62-bit constants. A
// constant multiplication is three multiply-adds of 32-bit halves.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

namespace fx {

using i64 = long long;
using u64 = unsigned long long;

struct __align__(16) cx {
  i64 x, y;
};

__host__ __device__ __forceinline__ cx operator+(cx a, cx b) { return {a.x + b.x, a.y + b.y}; }
__host__ __device__ __forceinline__ cx operator-(cx a, cx b) { return {a.x - b.x, a.y - b.y}; }

// v = hi 2^32 + lo with both halves signed
__host__ __device__ __forceinline__ int half_hi(i64 v) { return (int)((v + 0x80000000ll) >> 32); }
__host__ __device__ __forceinline__ int half_lo(i64 v) { return (int)v; }
// a b + c in one multiply-add (left to itself the compiler may split it into a product and two adds)
__host__ __device__ __forceinline__ i64 wide(int a, int b, i64 c) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (i64)a * b + c;
#endif
}

__host__ __device__ constexpr int const_hi(i64 c) { return (int)((c + 0x80000000ll) >> 32); }
__host__ __device__ constexpr int const_lo(i64 c) { return (int)(unsigned)(c & 0xffffffffll); }

constexpr i64 kRnd30 = 1ll << 29;

// x C / 2^62, |x| < 2^61, |C| <= 2^62, rounded (the product of the low halves, below one
// unit, is dropped)
template <i64 C>
__host__ __device__ __forceinline__ i64 mulc(i64 x) {
  constexpr int ch = const_hi(C), cl = const_lo(C);
  const int xh = half_hi(x), xl = half_lo(x);
  const i64 mid = wide(xl, ch, wide(xh, cl, kRnd30));
  return wide(xh * 4, ch, mid >> 30);
}

// v (c + i s): c, s in units of 2^-62 as halves (ch, cl, sh, sl); |c|, |s| <= 1, |v| < 2^61
__host__ __device__ __forceinline__ cx rot_parts(cx v, int ch, int cl, int sh, int sl) {
  const int xh = half_hi(v.x), xl = half_lo(v.x), yh = half_hi(v.y), yl = half_lo(v.y);
  const i64 mrp = wide(xl, ch, wide(xh, cl, kRnd30)), mrn = wide(yl, sh, (i64)yh * sl);
  const i64 mi = wide(yl, ch, wide(yh, cl, wide(xl, sh, wide(xh, sl, kRnd30))));
  const int x4 = xh * 4, y4 = yh * 4;
  cx r;
  r.x = wide(x4, ch, (mrp - mrn) >> 30) - (i64)y4 * sh;
  r.y = wide(x4, sh, wide(y4, ch, mi >> 30));
  return r;
}
// sign of the angle as a template argument: v exp(SGN i t) for a table entry (cos t, sin t)
template <int SGN>
__host__ __device__ __forceinline__ cx rot(cx v, int4 w) {
  if (SGN > 0) return rot_parts(v, w.x, w.y, w.z, w.w);
  // conj(conj(v) e^{it})
  const cx r = rot_parts({v.x, -v.y}, w.x, w.y, w.z, w.w);
  return {r.x, -r.y};
}
template <i64 C, i64 S>
__host__ __device__ __forceinline__ cx rotc(cx v) {
  return rot_parts(v, const_hi(C), const_lo(C), const_hi(S), const_lo(S));
}

// ------------------------------------------------------------ small transforms
// y_k = sum_n v_n exp(SGN 2 pi i n k / R), natural order in and out
constexpr i64 kSin60 = 3993837246235628775ll;  // sqrt(3)/2, 2^62
constexpr i64 kR2 = 3260954456333195553ll;     // sqrt(1/2)

__host__ __device__ __forceinline__ cx muli(cx v, int s) { return s > 0 ? cx{-v.y, v.x} : cx{v.y, -v.x}; }

template <int SGN>
__host__ __device__ __forceinline__ void dft2(cx& a, cx& b) {
  const cx t = a - b;
  a = a + b;
  b = t;
}
template <int SGN>
__host__ __device__ __forceinline__ void dft3(cx& a, cx& b, cx& c) {
  const cx t = b + c, d = b - c;
  const cx e = muli({mulc<kSin60>(d.x), mulc<kSin60>(d.y)}, SGN);
  const cx m = {a.x - (t.x >> 1), a.y - (t.y >> 1)};
  a = a + t;
  b = m + e;
  c = m - e;
}
template <int SGN>
__host__ __device__ __forceinline__ void dft4(cx& a, cx& b, cx& c, cx& d) {
  const cx p = a + c, q = a - c, r = b + d, s = muli(b - d, SGN);
  a = p + r;
  c = p - r;
  b = q + s;
  d = q - s;
}

template <int R, int SGN>
__host__ __device__ __forceinline__ void dft(cx (&v)[R]) {
  if constexpr (R == 2) {
    dft2<SGN>(v[0], v[1]);
  } else if constexpr (R == 3) {
    dft3<SGN>(v[0], v[1], v[2]);
  } else if constexpr (R == 4) {
    dft4<SGN>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 6) {  // 2 x 3, coprime: n = 3 a + 2 b (mod 6), k = a' mod 2, b' mod 3
    cx p[2][3];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) p[a][b] = v[(3 * a + 2 * b) % 6];
    dft3<SGN>(p[0][0], p[0][1], p[0][2]);
    dft3<SGN>(p[1][0], p[1][1], p[1][2]);
#pragma unroll
    for (int b = 0; b < 3; ++b) dft2<SGN>(p[0][b], p[1][b]);
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = p[k % 2][k % 3];
  } else if constexpr (R == 8) {  // even and odd elements, then eighth-turn twiddles
    cx e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<SGN>(e0, e1, e2, e3);
    dft4<SGN>(o0, o1, o2, o3);
    const cx s1 = o1 + muli(o1, SGN), s3 = muli(o3, SGN) - o3;
    o1 = {mulc<kR2>(s1.x), mulc<kR2>(s1.y)};
    o2 = muli(o2, SGN);
    o3 = {mulc<kR2>(s3.x), mulc<kR2>(s3.y)};
    v[0] = e0 + o0; v[4] = e0 - o0;
    v[1] = e1 + o1; v[5] = e1 - o1;
    v[2] = e2 + o2; v[6] = e2 - o2;
    v[3] = e3 + o3; v[7] = e3 - o3;
  } else if constexpr (R == 9) {  // 3 x 3 with ninth-turn twiddles (cos, sin of 40, 80, 160 degrees)
    constexpr i64 C1 = 3532756447825785444ll, S1 = 2964334632409774423ll * SGN;
    constexpr i64 C2 = 800810873071977681ll, S2 = 4541624145405292212ll * SGN;
    constexpr i64 C4 = -4333567320897763126ll, S4 = 1577289512995517789ll * SGN;
    cx p[3][3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
#pragma unroll
      for (int a = 0; a < 3; ++a) p[b][a] = v[3 * a + b];
      dft3<SGN>(p[b][0], p[b][1], p[b][2]);
    }
    p[1][1] = rotc<C1, S1>(p[1][1]);
    p[1][2] = rotc<C2, S2>(p[1][2]);
    p[2][1] = rotc<C2, S2>(p[2][1]);
    p[2][2] = rotc<C4, S4>(p[2][2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      dft3<SGN>(p[0][k], p[1][k], p[2][k]);
#pragma unroll
      for (int q = 0; q < 3; ++q) v[k + 3 * q] = p[q][k];
    }
  } else {  // 12 = 4 x 3, coprime: n = 3 a + 4 b (mod 12)
    static_assert(R == 12, "radix");
    cx p[4][3];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) p[a][b] = v[(3 * a + 4 * b) % 12];
#pragma unroll
    for (int a = 0; a < 4; ++a) dft3<SGN>(p[a][0], p[a][1], p[a][2]);
#pragma unroll
    for (int b = 0; b < 3; ++b) dft4<SGN>(p[0][b], p[1][b], p[2][b], p[3][b]);
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = p[k % 4][k % 3];
  }
}

// ------------------------------------------------------------ conversions
// words of a double, on either side
__host__ __device__ __forceinline__ unsigned high_word(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2hiint(v);
#else
  u64 b;
  std::memcpy(&b, &v, 8);
  return (unsigned)(b >> 32);
#endif
}
// v 2^sh by an addition to the exponent field
__host__ __device__ __forceinline__ double add_exponent(double v, int sh) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(__double2hiint(v) + sh * (1 << 20), __double2loint(v));
#else
  u64 b;
  std::memcpy(&b, &v, 8);
  b += (u64)(i64)sh << 52;
  std::memcpy(&v, &b, 8);
  return v;
#endif
}
__host__ __device__ __forceinline__ i64 round_double(double v) {
#ifdef __CUDA_ARCH__
  return __double2ll_rn(v);
#else
  return llrint(v);
#endif
}

// round(v 2^sh), |v| 2^sh < 2^61. One operation of the FP64 pipe, which the rest leaves idle; the
// scaling is an addition to the exponent field (values that it would take below 1 round to 0, as
// do subnormal v).
__host__ __device__ __forceinline__ i64 from_double(double v, int sh) {
  const int e = (int)(high_word(v) >> 20) & 0x7ff;
  const bool in = e != 0 && e + sh > 1000;
  return in ? round_double(add_exponent(v, sh)) : 0;
}

// X 2^-sh, integer operations only in the normal range (rounded to nearest)
__device__ __forceinline__ double to_double(i64 X, int sh) {
  if (X == 0) return 0.0;
  const u64 sign = X < 0 ? 0x8000000000000000ull : 0ull;
  u64 a = X < 0 ? (u64)-X : (u64)X;
  const int lz = __clzll(a);
  a <<= lz;
  const int ex = 1086 - lz - sh;  // biased exponent of the leading bit
  if (ex < 2 || ex > 2044) {
    const int h = sh / 2;
    return scalbn(scalbn((double)X, -h), h - sh);
  }
  const u64 m = (a >> 11) + ((a >> 10) & 1);  // implicit bit at 52 (a carry moves the exponent)
  return __longlong_as_double((i64)(sign | (((u64)(ex - 1) << 52) + m)));
}

// X 2^-sh: one operation of the FP64 pipe, the scaling on the exponent field
__device__ __forceinline__ double from_fixed(i64 X, int sh) {
  if (sh <= -900 || sh >= 900) return to_double(X, sh);
  return X == 0 ? 0.0 : add_exponent((double)X, -sh);
}

// X f 2^-sh by the FP64 pipe (scale = f 2^-sh where that is a normal number, see scale_of)
struct Scale {
  double s;
  double f;
  int sh;
  bool plain;
};
__device__ __forceinline__ Scale scale_of(double f, int sh) {
  Scale r;
  r.plain = sh > -900 && sh < 900;
  r.s = r.plain ? f * __hiloint2double((1023 - sh) << 20, 0) : 0.0;
  r.f = f;
  r.sh = sh;
  return r;
}
__device__ __forceinline__ double scaled(i64 X, const Scale& c) {
  if (c.plain) return (double)X * c.s;
  return c.f * to_double(X, c.sh);
}

// v 2^l rounded towards minus infinity
__device__ __forceinline__ i64 shift(i64 v, int l) {
  return l >= 0 ? (i64)((u64)v << min(l, 63)) : v >> min(-l, 63);
}
// v / 2^k rounded, 0 <= k <= 62
__device__ __forceinline__ i64 shift_down(i64 v, int k) { return (v + ((1ll << k) >> 1)) >> k; }

// ------------------------------------------------------------ columns of the Chebyshev transforms
// x = hi 2^28 + lo, both signed; |x| < 2^59 - 2^27, so that hi, which is rounded, stays below 2^31
__host__ __device__ __forceinline__ int2 halves28(i64 x) {
  const i64 hi = (x + (1 << 27)) >> 28;
  return int2{(int)hi, (int)(x - hi * (1 << 28))};
}
// sum of x c: c in units of 2^-56 as halves
struct Sum {
  i64 m = 0, h = 0;
  __host__ __device__ __forceinline__ void add(int xh, int xl, int2 c) {
    m = wide(xh, c.x, m);
    h = wide(xh, c.y, wide(xl, c.x, h));
  }
  __host__ __device__ __forceinline__ i64 value() const { return m + ((h + (1 << 27)) >> 28); }
};
constexpr int kSumBits = 62, kMaxBits = 59;  // bits of a column's sum of moduli and of its values
// |v| rounded up, in units of 2^(e - 1037), 15 bits or 2^15
__host__ __device__ __forceinline__ int part_of(double v, int e) {
  const unsigned h = high_word(v) & 0x7fffffffu;
  const int d = e - (int)(h >> 20) + 6;
  return (int)(((h & 0xfffffu) | 0x100000u) >> (d < 31 ? d : 31)) + 1;
}
// a bound of p + q of two values whose high words are at most em, in units of 2^(e - 1037): twice the
// part of the largest (2^16 where that is rounded up to a power of two, which takes a bit more)
__host__ __device__ __forceinline__ u64 pair_top(unsigned em) {
  return 2 * (u64)((((em & 0xfffffu) | 0x100000u) >> 6) + 1);
}
// exponent that scales values of at most top 2^(e - 1037), whose moduli sum to s 2^(e - 1037)
__host__ __device__ __forceinline__ int exponent_of(u64 s, u64 top, int e) {
#ifdef __CUDA_ARCH__
  const int bs = 64 - __clzll((i64)(s | 1)), bt = 64 - __clzll((i64)(top | 1));
#else
  const int bs = 64 - __builtin_clzll(s | 1), bt = 64 - __builtin_clzll(top | 1);
#endif
  const int a = kSumBits - bs, b = kMaxBits - bt;
  return (a < b ? a : b) - (e - 1037);
}

// n / d for n < 2^16 by a precomputed reciprocal
struct Div {
  unsigned d, m;
};
__host__ __device__ __forceinline__ Div div_of(unsigned d) { return {d, 0xffffffffu / d + 1}; }
__device__ __forceinline__ int quot(int n, Div v) { return (int)__umulhi((unsigned)n, v.m); }  // d >= 2
__device__ __forceinline__ int quot1(int n, Div v) { return v.d == 1 ? n : quot(n, v); }

}  // namespace fx
