// Small device helpers shared by the kernel translation units.
#pragma once

#include <cuda_runtime.h>

// stored position (x index in FFT order) and kz index of solved mode u: all kz of ix >= 0, then kz >= 1 of
// ix < 0 (the others follow by Hermitian symmetry)
__device__ __forceinline__ void unique_mode(int u, int Kx, int MZ, int* pos, int* iz) {
  const int first = (Kx + 1) * MZ;
  if (u < first) {
    *pos = u / MZ;
    *iz = u - *pos * MZ;
  } else {
    const int v = u - first;
    *pos = Kx + 1 + v / (MZ - 1);
    *iz = 1 + v % (MZ - 1);
  }
}

// sum_c w[c * ws] x[c * xs] with four independent partial sums (real w, complex x):
// eight independent FMA chains per thread hide the FP64 latency
__device__ __forceinline__ double2 dot4(const double* __restrict__ w, int ws, const double2* x, int xs, int n) {
  double2 s0 = make_double2(0.0, 0.0), s1 = s0, s2 = s0, s3 = s0;
  int c = 0;
  for (; c + 4 <= n; c += 4) {
    const double w0 = __ldg(w + (size_t)c * ws), w1 = __ldg(w + (size_t)(c + 1) * ws),
                 w2 = __ldg(w + (size_t)(c + 2) * ws), w3 = __ldg(w + (size_t)(c + 3) * ws);
    const double2 x0 = x[c * xs], x1 = x[(c + 1) * xs], x2 = x[(c + 2) * xs], x3 = x[(c + 3) * xs];
    s0.x = fma(w0, x0.x, s0.x);
    s0.y = fma(w0, x0.y, s0.y);
    s1.x = fma(w1, x1.x, s1.x);
    s1.y = fma(w1, x1.y, s1.y);
    s2.x = fma(w2, x2.x, s2.x);
    s2.y = fma(w2, x2.y, s2.y);
    s3.x = fma(w3, x3.x, s3.x);
    s3.y = fma(w3, x3.y, s3.y);
  }
  for (; c < n; ++c) {
    const double w0 = __ldg(w + (size_t)c * ws);
    const double2 x0 = x[c * xs];
    s0.x = fma(w0, x0.x, s0.x);
    s0.y = fma(w0, x0.y, s0.y);
  }
  return make_double2((s0.x + s1.x) + (s2.x + s3.x), (s0.y + s1.y) + (s2.y + s3.y));
}


// sum_c w[c * ws] x[c] with complex w and x: the real and imaginary parts of each
// product go to separate partial sums, eight independent FMA chains per thread
__device__ __forceinline__ double2 cdot4(const double2* __restrict__ w, int ws, const double2* x, int n) {
  double2 s0 = make_double2(0.0, 0.0), s1 = s0, s2 = s0, s3 = s0;
  int c = 0;
  for (; c + 2 <= n; c += 2) {
    const double2 w0 = __ldg(w + (size_t)c * ws), w1 = __ldg(w + (size_t)(c + 1) * ws);
    const double2 x0 = x[c], x1 = x[c + 1];
    s0.x = fma(w0.x, x0.x, s0.x);
    s1.x = fma(-w0.y, x0.y, s1.x);
    s0.y = fma(w0.x, x0.y, s0.y);
    s1.y = fma(w0.y, x0.x, s1.y);
    s2.x = fma(w1.x, x1.x, s2.x);
    s3.x = fma(-w1.y, x1.y, s3.x);
    s2.y = fma(w1.x, x1.y, s2.y);
    s3.y = fma(w1.y, x1.x, s3.y);
  }
  if (c < n) {
    const double2 w0 = __ldg(w + (size_t)c * ws);
    const double2 x0 = x[c];
    s0.x = fma(w0.x, x0.x, s0.x);
    s1.x = fma(-w0.y, x0.y, s1.x);
    s0.y = fma(w0.x, x0.y, s0.y);
    s1.y = fma(w0.y, x0.x, s1.y);
  }
  return make_double2((s0.x + s1.x) + (s2.x + s3.x), (s0.y + s1.y) + (s2.y + s3.y));
}

// inclusive suffix sum over rows i < cnt of x(i), one warp, chunks of 32 from the top: put(i, sum)
template <class X, class Put>
__device__ __forceinline__ void suffix_scan(int cnt, X x, Put put) {
  const int lane = threadIdx.x & 31;
  double2 carry = make_double2(0.0, 0.0);
  for (int c0 = ((cnt - 1) >> 5) << 5; c0 >= 0; c0 -= 32) {
    const int i = c0 + lane;
    double2 s = i < cnt ? x(i) : make_double2(0.0, 0.0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double yx = __shfl_down_sync(0xffffffffu, s.x, o), yy = __shfl_down_sync(0xffffffffu, s.y, o);
      if (lane + o < 32) {
        s.x += yx;
        s.y += yy;
      }
    }
    s.x += carry.x;
    s.y += carry.y;
    if (i < cnt) put(i, s);
    carry = make_double2(__shfl_sync(0xffffffffu, s.x, 0), __shfl_sync(0xffffffffu, s.y, 0));
  }
}

// (double)f by integer operations: the conversion instruction takes a slot of the FP64 unit
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), e = (u >> 23) & 0xffu;
  unsigned m = u & 0x7fffffu, x = e + 896u;
  if (e == 0 || e == 255) {
    if (e == 255) {
      x = 2047;
    } else if (m == 0) {
      x = 0;
    } else {
      const int s = __clz(m) - 8;
      m = (m << s) & 0x7fffffu;
      x = 897 - s;
    }
  }
  return __hiloint2double((int)((u & 0x80000000u) | (x << 20) | (m >> 3)), (int)(m << 29));
}

// (v + conj w) / 2 with w the mirror mode's value. A call: the compiler predicates a short branch, and a
// predicated-off FP64 instruction still takes its slot of the FP64 unit
static __device__ __noinline__ double2 project(double2 v, double2 w) {
  return make_double2(0.5 * (v.x + w.x), 0.5 * (v.y - w.y));
}
