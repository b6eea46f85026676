// Host check of the column arithmetic of the forward Chebyshev transform in fixed point (fx_arith.h,
// the steps of k_rhs_fx in cheb_fx.cu) against long double. Prints, per number of points, the largest
// error of a coefficient relative to the column's sum of moduli.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "fx_arith.h"

using L = long double;
static const L kPi = 3.141592653589793238462643383279502884L;

static int2 constant(L v) {  // 56 bits as halves
  const long long q = llrintl(v * 72057594037927936.0L), hi = (q + (1 << 27)) >> 28;
  return int2{(int)hi, (int)(q - hi * (1LL << 28))};
}

static double transform(const std::vector<double>& f, const std::vector<L>& cs) {
  const int N = (int)f.size() - 1, NH = N / 2 + 1;
  unsigned em = 0;
  for (double v : f) em = std::max(em, fx::high_word(v) & 0x7fffffffu);
  const int e = (int)(em >> 20);
  long long sum = 0;
  L mod = 0;
  for (double v : f) {
    sum += fx::part_of(v, e) + fx::part_of(0.0, e);
    mod += fabsl((L)v);
  }
  const int sh = fx::exponent_of((fx::u64)sum, fx::pair_top(em), e);
  std::vector<int2> even(NH), odd(NH);
  for (int j = 0; j < NH; ++j) {
    const fx::i64 p = fx::from_double(f[j], sh), q = fx::from_double(f[N - j], sh);
    const int d = j == 0 ? 1 : 0;
    even[j] = 2 * j == N ? fx::halves28(p) : fx::halves28((p + q) >> d);
    odd[j] = 2 * j == N ? int2{0, 0} : fx::halves28((p - q) >> d);
  }
  double worst = 0;
  for (int n = 0; n < N; ++n) {
    fx::Sum s;
    L ref = 0;
    for (int j = 0; j < NH; ++j) {
      const int2 x = n & 1 ? odd[j] : even[j];
      s.add(x.x, x.y, constant(cs[(long long)j * n % (2 * N)]));
    }
    for (int j = 0; j <= N; ++j) ref += (j == 0 || j == N ? 0.5L : 1.0L) * f[j] * cs[(long long)j * n % (2 * N)];
    worst = std::max(worst, (double)(fabsl(ldexpl((L)s.value(), -sh) - ref) / mod));
  }
  return worst;
}

int main() {
  std::mt19937_64 g(1);
  for (int ny = 5; ny <= 257; ny += ny < 17 ? 2 : 16) {
    const int N = ny - 1;
    std::vector<L> cs(2 * N);
    for (int k = 0; k < 2 * N; ++k) cs[k] = cosl(kPi * k / N);
    double worst = 0;
    // a pair at the edge of a power of two, equal and opposite, alone and beside other values
    for (double edge : {1.0 - ldexp(1.0, -53), 1.0 - 1e-12, 1.0 - 1e-10, 1.0 - ldexp(1.0, -15), 1.0, 0.7})
      for (double sign : {1.0, -1.0})
        for (double rest : {0.0, 1e-3, 0.3, 1.0})
          for (int j : {0, 1, N / 2 - 1, N / 2})
            for (int ex : {0, 300, -700}) {
              std::vector<double> f(ny);
              for (double& v : f) v = rest * ldexp((double)(long long)(g() >> 11), -53) * (g() & 1 ? 1 : -1);
              if (rest == 1.0)
                for (double& v : f) v = edge;
              f[j] = edge;
              f[N - j] = sign * edge;
              for (double& v : f) v = ldexp(v, ex);
              worst = std::max(worst, transform(f, cs));
            }
    std::printf("%d %.3e\n", ny, worst);
  }
  return 0;
}
