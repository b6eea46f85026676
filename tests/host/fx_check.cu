// Host check of the fixed-point transforms (fx_arith.h): prints, per radix and direction, the largest
// error of a transform against the same sum in long double, in units of the last place.
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>

#include "fx_arith.h"

using L = long double;

template <int R, int S>
void one() {
  std::mt19937_64 g(R);
  L worst = 0;
  for (int trial = 0; trial < 200; ++trial) {
    fx::cx v[R];
    std::complex<L> u[R];
    for (int i = 0; i < R; ++i) {
      v[i] = {(fx::i64)(g() >> 8) - (1ll << 55), (fx::i64)(g() >> 8) - (1ll << 55)};
      u[i] = {(L)v[i].x, (L)v[i].y};
    }
    fx::dft<R, S>(v);
    for (int k = 0; k < R; ++k) {
      std::complex<L> s = 0;
      for (int n = 0; n < R; ++n) {
        const L t = 6.283185307179586476925286766559005768L * (n * k % R) / R * S;
        s += u[n] * std::complex<L>(cosl(t), sinl(t));
      }
      worst = std::max(worst, std::abs(s - std::complex<L>((L)v[k].x, (L)v[k].y)));
    }
  }
  std::printf("%d %d %.3f\n", R, S, (double)worst);
}

int main() {
  one<2, 1>(); one<3, 1>(); one<4, 1>(); one<6, 1>(); one<8, 1>(); one<9, 1>(); one<12, 1>();
  one<2, -1>(); one<3, -1>(); one<4, -1>(); one<6, -1>(); one<8, -1>(); one<9, -1>(); one<12, -1>();
  // quotients by a precomputed reciprocal
  for (unsigned d = 2; d < 4700; ++d) {
    const fx::Div v = fx::div_of(d);
    for (unsigned n = 0; n < 65536; n += 1 + n / 97)
      for (unsigned m : {n, n / d * d, n / d * d + d - 1})
        if (m < 65536 && (unsigned)(((unsigned long long)m * v.m) >> 32) != m / d) {
          std::printf("div %u / %u\n", m, d);
          return 1;
        }
  }
  return 0;
}
