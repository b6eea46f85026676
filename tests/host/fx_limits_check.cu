// Host check of the fixed-point transforms (fx_arith.h) at the kernels' bound: inputs whose moduli sum to
// 2^60 (that bounds every value a transform forms by 2^60.5), all in one element, in the odd ones, on the
// diagonals or evenly, and turned by table twiddles first. Prints, per radix and direction, the largest
// error against the same sum in long double, in units of the last place.
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>

#include "fx_arith.h"

using L = long double;
using C = std::complex<L>;
static const L kTau = 6.283185307179586476925286766559005768L;

static int4 twiddle(L t) {
  auto half = [](L v, int* hi, int* lo) {
    const long long q = llrintl(v * 4611686018427387904.0L);
    *lo = (int)(unsigned)(q & 0xffffffffLL);
    *hi = (int)((q - *lo) >> 32);
  };
  int4 w;
  half(cosl(t), &w.x, &w.y);
  half(sinl(t), &w.z, &w.w);
  return w;
}

template <int R, int S>
void one() {
  std::mt19937_64 g(R);
  L worst = 0;
  const L top = 1152921504606846976.0L - 64;  // 2^60
  for (int trial = 0; trial < 400; ++trial) {
    L share[R];
    L sum = 0;
    for (int i = 0; i < R; ++i) {
      const int style = trial % 4;
      share[i] = style == 0 ? (i == trial / 4 % R) : style == 1 ? (i & 1) : style == 2 ? 1 : (L)(g() % 1000 + 1);
      sum += share[i];
    }
    fx::cx v[R];
    C u[R];
    for (int i = 0; i < R; ++i) {
      const L t = kTau * (trial % 3 == 0 ? (L)(g() % 8) / 8 : (L)(g() % 4096) / 4096), m = top * share[i] / sum;
      v[i] = {(fx::i64)(m * cosl(t)), (fx::i64)(m * sinl(t))};
      u[i] = {(L)v[i].x, (L)v[i].y};
      if (trial & 1) {  // by a twiddle, as between the passes
        const L a = kTau * (g() % 144) / 144;
        v[i] = fx::rot<S>(v[i], twiddle(a));
        u[i] *= C(cosl(a), S * sinl(a));
      }
    }
    fx::dft<R, S>(v);
    for (int k = 0; k < R; ++k) {
      C s = 0;
      for (int n = 0; n < R; ++n) {
        const L t = kTau * (n * k % R) / R * S;
        s += u[n] * C(cosl(t), sinl(t));
      }
      worst = std::max(worst, std::abs(s - C((L)v[k].x, (L)v[k].y)));
    }
  }
  std::printf("%d %d %.3f\n", R, S, (double)worst);
}

int main() {
  one<2, 1>(); one<3, 1>(); one<4, 1>(); one<6, 1>(); one<8, 1>(); one<9, 1>(); one<12, 1>();
  one<2, -1>(); one<3, -1>(); one<4, -1>(); one<6, -1>(); one<8, -1>(); one<9, -1>(); one<12, -1>();
  return 0;
}
