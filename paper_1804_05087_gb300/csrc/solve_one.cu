// Per-mode Stokes solve by the precomputed dense operators, one Fourier mode of one or a few directions
// per block: the step, single tangents and small batches (batches from kChainMinBatch directions take the
// O(N) chains, solve_chain.cu; laminar advection in L takes k_solve, kernels.cu). Same problem as
// k_solve: right-hand side u/dt + N, rotation along / across the wavevector, reduced right-hand side,
// v = V g and b = H f_b per parity, back-rotation, G = u_new - u (Sec. 2, Eq. befe; Sec. 3.2).
//
// A call with one direction is bound by latency: the FP64 unit of a warp scheduler takes 64 cycles
// per instruction, and four modes per block of 128 threads left 121 warps' worth of serial phases
// on 152 SMs. Here a block takes one mode with a thread per row of each operator (2 NY), the
// operators come into shared memory by one bulk copy that runs during the earlier phases, the suffix
// sums are warp scans, and wavenumbers and row indices are read, not computed. Several blocks share
// an SM, so that one block's scans overlap another's products. Measured at 48 x 65 x 48, one FP64
// direction: 55 us with four modes per block and loads inside the products, 28 us here. A batch is bound by
// FP64 instructions, whose idle lanes cost as much as busy ones, so there a block takes two or four
// directions of its mode (directions_of; threads: threads_of). k_solve_adj is the transposed solve, one
// direction per block.
#include <algorithm>
#include <cstdint>

#include "dev_util.h"
#include "sp_internal.h"

namespace {

struct OneArgs {
  const void* in;      // float: values [dir][3][NY][Mm]; double: right-hand sides [dir][mode][3][N - 1]
  const double2* du;   // [dir][3][Mm][NY]
  double2* out;
  const double* ops;   // [mode][op_stride]: V0, V1, H0, H1, column-major
  const double* wave;  // [mode][4]: kx, kz, 1/k, 0
  const float* cft;    // [NH][NY] forward transform (float), points fastest last
  const double* row;   // row indices 0, 1, ... as doubles
  int n_dir, n_unique, Mm, MX, MZ, Kx, NY, cv, rb0, rb1, off_v0, off_v1, off_h0, off_h1, op_stride, staged;
  double inv_dt;
};

__device__ __forceinline__ uint32_t smem_of(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void bulk_copy(double* dst, const double* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_of(dst)),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// one bulk copy of a mode's operators (one thread), and the wait for it (all threads): false when the
// limit runs out
__device__ __forceinline__ void stage_begin(double* dst, const double* op, uint32_t bytes, uint64_t* s_bar) {
  const uint32_t bar = smem_of(s_bar);
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  bulk_copy(dst, op, bytes, bar);
}
__device__ __forceinline__ bool stage_wait(uint64_t* s_bar) {
  const uint32_t bar = smem_of(s_bar);
  uint32_t done = 0;
  for (uint32_t it = 0; it < (1u << 25) && !done; ++it)  // the second half of the limit: the copy may be in flight
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(bar)
        : "memory");
  return done != 0;
}

// mode u of the directions dir0 to dir0 + D - 1 (as far as there are). Work items take the directions
// slowest, so that the last warp of a phase is filled by the next direction.
template <typename T, int D>
__device__ __forceinline__ void solve_one(const OneArgs& a, int u, int dir0, unsigned char* smem, uint64_t* s_bar) {
  const int NY = a.NY, N = NY - 1, NH = N / 2 + 1, NR = N - 1, Mm = a.Mm, MZ = a.MZ;
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, nw = nt >> 5;
  const int nd = D == 1 ? 1 : min(D, a.n_dir - dir0);
  double* sop = reinterpret_cast<double*>(smem);
  double2* sdu = reinterpret_cast<double2*>(sop + (a.staged ? a.op_stride : 0));  // [D][3][NY]
  double2* sfa = sdu + D * 3 * NY;  // [D][NR] -i f_a
  double2* sfb = sfa + D * NR;      // [D][NR] (mean mode: f_u)
  double2* srv = sfb + D * NR;      // [D][2][cv] reduced right-hand sides per parity
  double2* sfw = srv + D * 2 * a.cv;  // [D][3][NR] staged right-hand sides
  double2* sv = sfw + D * 3 * NR;   // [D][NY]
  double2* sb = sv + D * NY;        // [D][NY]
  double2* ss = sb + D * NY;        // [D][NY + 1] sums of p v_p over p >= n of the parity of n
  C2<T>* vals = reinterpret_cast<C2<T>*>(ss + D * (NY + 1));  // [D][3][NY] (float)
  // direction of item i, per items each; i becomes the item in it
  auto split = [&](int& i, int per) -> int {
    if constexpr (D == 1) return 0;
    int d = 0;
#pragma unroll
    for (int q = 1; q < D; ++q)
      if (i >= per) {
        i -= per;
        ++d;
      }
    return d;
  };
  int pos, iz;
  unique_mode(u, a.Kx, a.MZ, &pos, &iz);
  const bool mean = u == 0;
  const double* op = a.ops + (size_t)u * a.op_stride;
  if (a.staged && tid == 0) stage_begin(sop, op, (uint32_t)a.op_stride * 8, s_bar);
  const double kx = __ldg(a.wave + 4 * u), kz = __ldg(a.wave + 4 * u + 1), ik = __ldg(a.wave + 4 * u + 2);
  // input state (Hermitian-projected)
  const double2* dsrc = a.du + ((size_t)dir0 * 3 * Mm + pos * MZ + iz) * NY;
  const long long mir = pos == 0 ? 0 : (long long)(a.MX - 2 * pos) * MZ * NY;  // to the mirror mode
  for (int i = tid; i < nd * 3 * NY; i += nt) {
    const int c = i / NY;  // component of a direction: the directions follow one another
    const double2* p = dsrc + (size_t)c * Mm * NY + (i - c * NY);
    double2 v = __ldg(p);
    if (iz == 0) v = project(v, __ldg(p + mir));
    sdu[i] = v;
  }
  if constexpr (sizeof(T) == 8) {
    for (int d = 0; d < nd; ++d) {
      const double2* W = static_cast<const double2*>(a.in) + ((size_t)(dir0 + d) * a.n_unique + u) * 3 * NR;
      for (int i = tid; i < 3 * NR; i += nt) sfw[d * 3 * NR + i] = __ldg(W + i);
    }
    __syncthreads();
  } else {
    // forward transform of the values: even and odd parts of the point pairs, then one thread per row
    // (even rows first; the order of k_solve's sums)
    const C2<T>* vin = static_cast<const C2<T>*>(a.in) + (size_t)dir0 * 3 * NY * Mm + pos * MZ + iz;
    for (int i = tid; i < nd * 3 * NH; i += nt) {
      const int c = i / NH, j = i - c * NH;
      const C2<T> p = vin[((size_t)c * NY + j) * Mm], q = vin[((size_t)c * NY + N - j) * Mm];
      C2<T>* col = vals + c * NY;
      if (2 * j == N) {
        col[j] = p;
      } else {
        col[j] = p + q;
        col[N - j] = p - q;
      }
    }
    __syncthreads();
    const int ne = (NR + 1) / 2, even = nd * 3 * ne;
    for (int i = tid; i < nd * 3 * NR; i += nt) {
      const bool odd = i >= even;
      const int k = odd ? i - even : i, per = odd ? NR - ne : ne;
      const int c = k / per, n = 2 * (k - c * per) + (odd ? 1 : 0);
      const C2<T>* col = vals + c * NY;
      const float* cf = a.cft + n;
      C2<T> acc = mk((T)0, (T)0);
      if (!odd) {
        for (int j = 0; j < NH - 1; ++j) acc = acc + scl(col[j], __ldg(cf + j * NY));
        acc = acc + scl(col[NH - 1], __ldg(cf + (NH - 1) * NY));
      } else {
        for (int j = 0; j < NH - 1; ++j) acc = acc + scl(col[N - j], __ldg(cf + j * NY));
      }
      const double2 d = sdu[c * NY + n];
      double2 f = make_double2(fma(d.x, a.inv_dt, widen(acc.x)), fma(d.y, a.inv_dt, widen(acc.y)));
      if (mean) f.y = 0.0;
      sfw[c * NR + n] = f;
    }
    __syncthreads();
  }
  // rotation to the components along / across the wavevector
  for (int i = tid; i < nd * NR; i += nt) {
    int n = i;
    const int d = split(n, NR);
    const double2* fw = sfw + d * 3 * NR;
    const double2 fx = fw[n], fy = fw[NR + n], fz = fw[2 * NR + n];
    if (mean) {
      sfb[i] = fx;
      sfa[i] = fz;
      continue;
    }
    const double2 fa = make_double2((kx * fx.x + kz * fz.x) * ik, (kx * fx.y + kz * fz.y) * ik);
    sfb[i] = make_double2((-kz * fx.x + kx * fz.x) * ik, (-kz * fx.y + kx * fz.y) * ik);
    srv[d * 2 * a.cv + (n & 1) * a.cv + n / 2] = fy;
    sfa[i] = make_double2(fa.y, -fa.x);  // -i f_a
  }
  __syncthreads();
  // reduced right-hand side g_n = f_v,n - (2 / (c_n k)) sum over m > n, m + n odd, of m (-i f_a,m)
  if (!mean) {
    for (int q = warp; q < 2 * nd; q += nw) {
      const int P = q & 1;
      double2* g = srv + q * a.cv;
      const double2* fa = sfa + (q >> 1) * NR;
      suffix_scan(
          P == 0 ? a.rb0 : a.rb1,
          [&](int i) -> double2 {
            const int m = 2 * i + P + 1;
            if (m > N - 2) return make_double2(0.0, 0.0);
            const double w = __ldg(a.row + m);
            return make_double2(w * fa[m].x, w * fa[m].y);
          },
          [&](int i, double2 s) {
            const double f = (2 * i + P == 0 ? 1.0 : 2.0) * ik;
            g[i] = make_double2(g[i].x - f * s.x, g[i].y - f * s.y);
          });
    }
  }
  bool ok = true;
  if (a.staged) {
    ok = stage_wait(s_bar);
    op = sop;
  }
  ok = __syncthreads_and(ok) != 0;  // the limit ran out: NaN below
  // v = V g and b = H f_b: one row of one operator per thread
  const int nv0 = N / 2 + 1;
  for (int i = tid; i < nd * 2 * NY; i += nt) {
    int r = i;
    const int d = split(r, 2 * NY);
    const bool hel = r < NY;
    const int k = hel ? r : r - NY;
    const int Q = k < nv0 ? 0 : 1, row = Q == 0 ? k : k - nv0, n = 2 * row + Q;
    const int nrow = Q == 0 ? nv0 : NY - nv0, rb = Q == 0 ? a.rb0 : a.rb1;
    const double* H = op + (Q == 0 ? a.off_h0 : a.off_h1) + row;
    const double* V = op + (Q == 0 ? a.off_v0 : a.off_v1) + row;
    // mean flow: u and w from the Helmholtz operator, v = 0
    const double2* x = hel ? sfb + d * NR + Q : mean ? sfa + d * NR + Q : srv + (2 * d + Q) * a.cv;
    const double* M = hel || mean ? H : V;
    const int xs = hel || mean ? 2 : 1;
    double2 s[4] = {};
    int c = 0;
    for (; c + 4 <= rb; c += 4) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double w = M[(c + q) * nrow];
        const double2 y = x[(c + q) * xs];
        s[q].x = fma(w, y.x, s[q].x);
        s[q].y = fma(w, y.y, s[q].y);
      }
    }
    for (; c < rb; ++c) {
      const double w = M[c * nrow];
      const double2 y = x[c * xs];
      s[0].x = fma(w, y.x, s[0].x);
      s[0].y = fma(w, y.y, s[0].y);
    }
    (hel ? sb : sv)[d * NY + n] = make_double2((s[0].x + s[1].x) + (s[2].x + s[3].x), (s[0].y + s[1].y) + (s[2].y + s[3].y));
  }
  __syncthreads();
  // (D v)_n = (2 / c_n) sum over p > n, p + n odd, of p v_p
  if (!mean) {
    for (int q = warp; q < 2 * nd; q += nw) {
      const int P = q & 1;
      const double2* v = sv + (q >> 1) * NY;
      double2* to = ss + (q >> 1) * (NY + 1);
      suffix_scan(
          P == 0 ? nv0 : NY - nv0,
          [&](int i) -> double2 {
            const int p = 2 * i + P;
            const double w = __ldg(a.row + p);
            return make_double2(w * v[p].x, w * v[p].y);
          },
          [&](int i, double2 s) { to[2 * i + P] = s; });
    }
  }
  __syncthreads();
  // a = (i/k) D v, back-rotation, G = u_new - u, Hermitian output
  double2* dst = a.out + ((size_t)dir0 * 3 * Mm + pos * MZ + iz) * NY;
  for (int i = tid; i < nd * NY; i += nt) {
    int n = i;
    const int d = split(n, NY);
    double2 un, vn, wn;
    if (mean) {
      un = make_double2(sb[i].x, 0.0);
      wn = make_double2(sv[i].x, 0.0);
      vn = make_double2(0.0, 0.0);
    } else {
      double2 dv = make_double2(0.0, 0.0);
      if (n + 1 < NY) {
        const double2 sp = ss[d * (NY + 1) + n + 1];
        const double f = n == 0 ? 1.0 : 2.0;
        dv = make_double2(f * sp.x, f * sp.y);
      }
      const double2 an = make_double2(-dv.y * ik, dv.x * ik);  // (i/k) Dv
      const double2 bn = sb[i];
      un = make_double2((kx * an.x - kz * bn.x) * ik, (kx * an.y - kz * bn.y) * ik);
      wn = make_double2((kz * an.x + kx * bn.x) * ik, (kz * an.y + kx * bn.y) * ik);
      vn = sv[i];
    }
    const double2 res[3] = {un, vn, wn};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 e = sdu[(3 * d + c) * NY + n];
      double2 g = make_double2(res[c].x - e.x, res[c].y - e.y);
      if (mean) g.y = 0.0;
      if (!ok) g = make_double2(nan(""), nan(""));
      double2* o = dst + (size_t)(3 * d + c) * Mm * NY + n;
      *o = g;
      if (iz == 0 && pos != 0) o[mir] = make_double2(g.x, -g.y);
    }
  }
}

template <typename T, int D>
__global__ void __launch_bounds__(512) k_solve_one(const __grid_constant__ OneArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar;
  solve_one<T, D>(a, blockIdx.x, blockIdx.y * D, smem, &s_bar);
}

struct GOne {
  size_t off;  // offset (doubles) of the member's state in a group vector
  OneArgs a;
};

template <typename T>
__global__ void __launch_bounds__(512) k_solve_one_grp(const double* __restrict__ du, double* __restrict__ out,
                                                       const GOne* __restrict__ recs, const int* __restrict__ inst,
                                                       const int* __restrict__ first, const int* __restrict__ active) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ GOne r;
  const int i = inst[blockIdx.x];
  if (active && !active[i]) return;
  if (threadIdx.x == 0) {
    r = recs[i];
    r.a.du = reinterpret_cast<const double2*>(du + r.off);
    r.a.out = reinterpret_cast<double2*>(out + r.off);
  }
  __syncthreads();
  solve_one<T, 1>(r.a, blockIdx.x - first[i], 0, smem, &s_bar);
}

// out[4 i] = sum of x[xs j] over j <= i, in order; the first entry halved (c_0 = 2) where asked
__device__ __forceinline__ void prefix(const double* x, int xs, double* out, int cnt, bool half) {
  double s = 0.0, v = cnt > 0 ? x[0] : 0.0;
  if (half) v *= 0.5;
  for (int i = 0; i < cnt; ++i) {
    const double next = i + 1 < cnt ? x[(i + 1) * xs] : 0.0;  // before the store: `out` may be `x`
    s += v;
    out[4 * i] = s;
    v = next;
  }
}

// entries between columns in shared memory: a multiple of 4 puts the lanes of a warp on few banks
__host__ __device__ inline int col_stride(int nrow) { return nrow % 4 ? nrow : nrow + 2; }

// The transposed solve of the discrete adjoint, one mode of one direction per block: r' = P W r,
// f* = S^T r' (the transposed operators), out = f*/dt, vals = Cf^T f* at the Gauss-Lobatto points
// (float values feed the transposed plane stage in mixed precision).
//
// Bound by the FP64 unit, as the forward solve. With four modes per block of 128 threads the lanes of
// a product read columns of the operator in global memory (a stride of N/2 rows), the derivative sums
// ran on 8 threads and each multiplication of the float transform converted its factor again: 573 us
// at 96 x 97 x 96 against 162 us of the forward solve; 177 us now. The
// operators are staged as there and a thread takes one column (columns whose length is a multiple of 4
// are copied one by one, two entries apart, so that lanes meet in a bank by twos at most); f* is
// converted once. The prefix sums are serial, on four lanes (parity, part), and the fused products are
// written out: all feed values that mixed precision rounds to float, where a last bit of FP64 can turn
// into 6e-8.
template <typename T>
__global__ void __launch_bounds__(512) k_solve_adj(const __grid_constant__ OneArgs a, C2<T>* __restrict__ vals,
                                                   const T* __restrict__ cf, int weighted) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar;
  const int NY = a.NY, N = NY - 1, NH = N / 2 + 1, NR = N - 1, Mm = a.Mm, MZ = a.MZ;
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, nw = nt >> 5;
  const int u = blockIdx.x, dir = blockIdx.y;
  // column strides of the staged operators per parity
  const int st0 = a.staged ? col_stride(N / 2 + 1) : N / 2 + 1, st1 = a.staged ? col_stride(N / 2) : N / 2;
  double* sop = reinterpret_cast<double*>(smem);
  double2* sga = reinterpret_cast<double2*>(sop + (a.staged ? 2 * (a.rb0 * st0 + a.rb1 * st1) : 0));
  // sga: [NY] along k (mean mode: u), then its prefix sums
  double2* sgb = sga + NY;       // [NY] across k (mean mode: w)
  double2* sva = sgb + NY;       // [NY] v* = gv + D^T(-i ga / k)
  double2* srv = sva + NY;       // [2][cv] V^T v*
  double2* sfb = srv + 2 * a.cv; // [NR] H^T gb (mean mode: H^T gw)
  double2* sfa = sfb + NR;       // [NR] sums of f~_a* (mean mode: H^T gu)
  C2<T>* sf = reinterpret_cast<C2<T>*>(sfa + NR);  // [3][NR] f*
  int pos, iz;
  unique_mode(u, a.Kx, a.MZ, &pos, &iz);
  const bool mean = u == 0;
  const double* op = a.ops + (size_t)u * a.op_stride;
  const int v1 = a.staged ? a.rb0 * st0 : a.off_v1, h0 = a.staged ? v1 + a.rb1 * st1 : a.off_h0,
            h1 = a.staged ? h0 + a.rb0 * st0 : a.off_h1;
  if (a.staged && warp == 0) {
    const uint32_t bar = smem_of(&s_bar);
    if (tid == 0) {
      const uint32_t bytes = 16u * (uint32_t)(a.rb0 * (N / 2 + 1) + a.rb1 * (N / 2));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    }
    __syncwarp();
    for (int o = 0; o < 4; ++o) {
      const int Q = o & 1, nrow = Q ? N / 2 : N / 2 + 1, cols = Q ? a.rb1 : a.rb0, st = Q ? st1 : st0;
      const double* src = op + (o == 0 ? a.off_v0 : o == 1 ? a.off_v1 : o == 2 ? a.off_h0 : a.off_h1);
      double* to = sop + (o == 0 ? 0 : o == 1 ? v1 : o == 2 ? h0 : h1);
      if (st == nrow) {
        if (tid == 0 && cols > 0) bulk_copy(to, src, (uint32_t)(cols * nrow) * 8, bar);
      } else {
        for (int k = tid; k < cols; k += 32) bulk_copy(to + k * st, src + (size_t)k * nrow, (uint32_t)nrow * 8, bar);
      }
    }
  }
  const double kx = __ldg(a.wave + 4 * u), kz = __ldg(a.wave + 4 * u + 1), ik = __ldg(a.wave + 4 * u + 2);
  const size_t comp = (size_t)Mm * NY;
  const size_t at = (size_t)dir * 3 * comp + ((size_t)pos * MZ + iz) * NY;
  const long long mir = pos == 0 ? 0 : (long long)(a.MX - 2 * pos) * MZ * NY;  // to the mirror mode
  // r' = P W r, rotated to the components along / across the wavevector
  for (int n = tid; n < NY; n += nt) {
    double2 g[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2* p = a.du + at + c * comp + n;
      double2 v = __ldg(p);
      if (iz == 0) {
        const double2 w = __ldg(p + mir);
        v = make_double2(0.5 * (v.x + w.x), 0.5 * (v.y - w.y));
      } else if (weighted) {
        v = make_double2(2.0 * v.x, 2.0 * v.y);
      }
      g[c] = v;
    }
    sga[n] = mean ? g[0] : make_double2(fma(kx, g[0].x, kz * g[2].x) * ik, fma(kx, g[0].y, kz * g[2].y) * ik);
    sgb[n] = mean ? g[2] : make_double2(fma(kx, g[2].x, -kz * g[0].x) * ik, fma(kx, g[2].y, -kz * g[0].y) * ik);
    sva[n] = g[1];
  }
  __syncthreads();
  // a = (i/k) D v  =>  v* = gv + D^T (-i ga / k); (D^T x)_n = sum_{m<n, m+n odd} (2n/c_m) x_m: the sums
  // over the rows m = 2i + Q of each parity, in place
  if (!mean) {
    if (tid < 4) prefix(reinterpret_cast<double*>(sga + (tid >> 1)) + (tid & 1), 4,
                        reinterpret_cast<double*>(sga + (tid >> 1)) + (tid & 1), (NY - (tid >> 1) + 1) / 2, tid < 2);
    __syncthreads();
    for (int n = 1 + tid; n < NY; n += nt) {
      const double f = 2.0 * __ldg(a.row + n) * ik;
      const double2 gv = sva[n], s = sga[n - 1];
      // -i ga / k: (x + i y) * (-i) = y - i x
      sva[n] = make_double2(gv.x + f * s.y, gv.y - f * s.x);
    }
  }
  bool ok = true;
  if (a.staged) {
    ok = stage_wait(&s_bar);
    op = sop;
  }
  ok = __syncthreads_and(ok) != 0;  // the limit ran out: NaN below
  // columns of V_P (adjoint of g) and of H_Q: one per thread
  for (int i = tid; i < 2 * NR; i += nt) {
    const bool hel = i >= NR;
    const int k = hel ? i - NR : i;
    const int Q = k < a.rb0 ? 0 : 1, col = Q == 0 ? k : k - a.rb0;
    const int nrow = Q == 0 ? N / 2 + 1 : N / 2;
    const bool isH = hel || mean;
    const double* M = op + (isH ? (Q == 0 ? h0 : h1) : (Q == 0 ? a.off_v0 : v1)) + (size_t)col * (Q == 0 ? st0 : st1);
    const double2* x = (hel ? sgb : mean ? sga : sva) + Q;
    double2 p[4] = {};
    int c = 0;
    for (; c + 4 <= nrow; c += 4) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double w = M[c + q];
        const double2 y = x[2 * (c + q)];
        p[q].x = fma(w, y.x, p[q].x);
        p[q].y = fma(w, y.y, p[q].y);
      }
    }
    for (; c < nrow; ++c) {
      const double w = M[c];
      const double2 y = x[2 * c];
      p[0].x = fma(w, y.x, p[0].x);
      p[0].y = fma(w, y.y, p[0].y);
    }
    const double2 s = make_double2((p[0].x + p[1].x) + (p[2].x + p[3].x), (p[0].y + p[1].y) + (p[2].y + p[3].y));
    if (hel) sfb[2 * col + Q] = s;
    else if (mean) sfa[2 * col + Q] = s;
    else srv[Q * a.cv + col] = s;
  }
  __syncthreads();
  // g = f_v - (1/k) D f~_a  =>  f_v* = g*, f~_a*,m = -(2m/k) sum_{n < m, n + m odd} g*_n / c_n: the sums
  if (!mean) {
    if (tid < 4) prefix(reinterpret_cast<double*>(srv + (tid >> 1) * a.cv) + (tid & 1), 2,
                        reinterpret_cast<double*>(sfa + (tid >> 1) + 1) + (tid & 1), min(tid < 2 ? a.rb0 : a.rb1, (NR - (tid >> 1)) / 2), tid < 2);
    if (tid == 4) sfa[0] = make_double2(0.0, 0.0);  // no rows below
  }
  __syncthreads();
  // f* per component, out = f*/dt (rows N-1, N zero), mirrored for iz = 0
  double2* dst = a.out + at;
  for (int n = tid; n < NY; n += nt) {
    double2 f[3] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    if (n < NR) {
      if (mean) {
        f[0].x = sfa[n].x;
        f[2].x = sfb[n].x;
      } else {
        f[1] = srv[(n & 1) * a.cv + (n >> 1)];
        const double g = -2.0 * __ldg(a.row + n) * ik;
        const double2 S = sfa[n], t = make_double2(g * S.x, g * S.y), fb = sfb[n];
        const double2 fa = make_double2(-t.y, t.x);  // f_a* = i f~_a*
        f[0] = make_double2(fma(kx, fa.x, -kz * fb.x) * ik, fma(kx, fa.y, -kz * fb.y) * ik);
        f[2] = make_double2(fma(kx, fb.x, kz * fa.x) * ik, fma(kx, fb.y, kz * fa.y) * ik);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (!ok) f[c] = make_double2(nan(""), nan(""));
        sf[c * NR + n] = mk((T)f[c].x, (T)f[c].y);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 v = make_double2(f[c].x * a.inv_dt, f[c].y * a.inv_dt);
      double2* o = dst + c * comp + n;
      *o = v;
      if (iz == 0 && pos != 0) o[mir] = make_double2(v.x, -v.y);
    }
  }
  __syncthreads();
  // vals = Cf^T f*: sum_n Cf[n][j] f*_n with Cf[n][N-j] = (-1)^n Cf[n][j]; the even rows of a point pair
  // on one lane, the odd rows on the next
  C2<T>* vdst = vals + (size_t)dir * 3 * NY * Mm + pos * MZ + iz;
  const int vmir = (a.MX - 2 * pos) * MZ;
  for (int i0 = warp * 32; i0 < 6 * NH; i0 += nw * 32) {
    const int i = i0 + (tid & 31), q = min(i >> 1, 3 * NH - 1), par = i & 1;
    const int c = q / NH, jh = q - c * NH;
    C2<T> s = mk((T)0, (T)0);
    const C2<T>* f = sf + c * NR;
    for (int n = par; n < NR; n += 2) s = s + scl(f[n], __ldg(cf + (size_t)n * NH + jh));
    const C2<T> o = mk(__shfl_xor_sync(0xffffffffu, s.x, 1), __shfl_xor_sync(0xffffffffu, s.y, 1));
    const int j = par ? N - jh : jh;
    if (i >= 6 * NH || (par && j == jh)) continue;
    const C2<T> v = par ? o - s : s + o;
    C2<T>* p = vdst + ((size_t)c * NY + j) * Mm;
    *p = v;
    if (iz == 0 && pos != 0) p[vmir] = conj2(v);
  }
}

// operators in shared memory up to this size (N <= 104); larger ones are read in place
constexpr size_t kStageBytes = 100 * 1024;

size_t one_smem(const sp_ctx* c, int esize, int D = 1) {
  const size_t ops = (size_t)c->op_stride * 8 <= kStageBytes ? (size_t)c->op_stride * 8 : 0;
  const size_t NY = c->NY, NR = c->N - 1;
  return ops + D * (16 * (3 * NY + 2 * NR + 2 * c->cv + 3 * NR + 3 * NY + 1) + (esize == 4 ? 3 * NY * 8 + 8 : 0));
}

OneArgs one_args(const sp_ctx* c, const void* in, const double* du, double* out) {
  OneArgs a;
  a.in = in;
  a.du = reinterpret_cast<const double2*>(du);
  a.out = reinterpret_cast<double2*>(out);
  a.ops = c->ops;
  a.wave = c->wave;
  a.cft = c->cft_f;
  a.row = c->rowidx;
  a.n_dir = 1;
  a.n_unique = c->n_unique;
  a.Mm = c->Mm; a.MX = c->MX; a.MZ = c->MZ; a.Kx = c->Kx; a.NY = c->NY;
  a.cv = c->cv; a.rb0 = c->rb0; a.rb1 = c->rb1;
  a.off_v0 = c->off_v0; a.off_v1 = c->off_v1; a.off_h0 = c->off_h0; a.off_h1 = c->off_h1;
  a.op_stride = c->op_stride;
  a.staged = (size_t)c->op_stride * 8 <= kStageBytes;
  a.inv_dt = 1.0 / c->dt;
  return a;
}

}  // namespace

// Threads of a block: one per row of the two operators of every direction (shape 0; in equal rounds past
// 512), or a fixed number. us with 224, 288 and 352 threads, two directions of 48 x 81 x 48, 31 mixed ones:
// 823, 770, 676.
static int threads_of(const sp_ctx* c, int shape, int D) {
  const int all = 2 * c->NY * D, rounds = (all + 511) / 512;
  const int rows = D == 1 ? std::min((all + 31) / 32 * 32, 512) : ((all + rounds - 1) / rounds + 31) / 32 * 32;
  const int fixed[SP_TUNE_MAX] = {rows, 64, 96, 128, 192, 256, 384, 512};
  return fixed[shape];
}
int solve_one_threads(const sp_ctx* c, int shape) { return threads_of(c, shape, 1); }

// Directions of a block. With one, a phase's last warp is partly filled (70 rows on 96 lanes at 35 points) and
// the operators are staged for every direction; with several, a call of few blocks leaves SMs idle. us per
// solve with 1, 2 and 4 directions, mixed: 48 x 35 x 48, 4 directions 41, 37, 37; 8: 68, 60, 60; 31: 238, 207,
// 195; 48 x 65 x 48, 3: 70, 64, 72; 31: 612, 518, 535; 24 x 25 x 24 (113 modes), 8: 16.5, 16.4, 19.4; 12: 20.6,
// 22.6, 24.7; 31: 45.5, 45.1, 49.6. So two from nine blocks per SM, four for short columns from 36; and both
// only where two blocks share an SM.
static int directions_of(const sp_ctx* c, int n_dir, int esize) {
  const long long blocks = (long long)c->n_unique * n_dir, sms = c->sm_count;
  if (n_dir >= 4 && blocks >= 36 * sms && 8 * c->NY <= 288 && one_smem(c, esize, 4) <= 112 * 1024) return 4;
  return n_dir >= 2 && blocks >= 9 * sms && one_smem(c, esize, 2) <= 112 * 1024 ? 2 : 1;
}

template <typename T>
static cudaError_t launch_one(const sp_ctx* c, const OneArgs& a, int shape, int D, cudaStream_t st) {
  const size_t sm = one_smem(c, sizeof(T), D);
  auto kern = D == 1 ? k_solve_one<T, 1> : D == 2 ? k_solve_one<T, 2> : k_solve_one<T, 4>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  kern<<<dim3(c->n_unique, (a.n_dir + D - 1) / D), threads_of(c, shape, D), sm, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_solve_one(const sp_ctx* c, bool fp32, const void* in, const double* du, double* out, int n_dir,
                             int shape, cudaStream_t st) {
  OneArgs a = one_args(c, in, du, out);
  a.n_dir = n_dir;
  const int D = directions_of(c, n_dir, fp32 ? 4 : 8);
  return fp32 ? launch_one<float>(c, a, shape, D, st) : launch_one<double>(c, a, shape, D, st);
}

cudaError_t grp_build_solve_one(GrpKernel* k, sp_ctx* const* mem, int n, const size_t* offs, const int* order, int esize) {
  std::vector<GOne> recs(n);
  std::vector<int> inst, first(n, 0);
  size_t smem = 0;
  for (int q = 0; q < n; ++q) {
    const int m = order[q];
    const sp_ctx* c = mem[m];
    recs[m].off = offs[m];
    recs[m].a = one_args(c, esize == 8 ? c->ws6 : c->ws3, nullptr, nullptr);
    first[m] = (int)inst.size();
    inst.insert(inst.end(), c->n_unique, m);
    smem = std::max(smem, one_smem(c, esize));
    k->threads = std::max(k->threads, solve_one_threads(c, 0));
  }
  cudaError_t e = esize == 8 ? cudaFuncSetAttribute(k_solve_one_grp<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                             : cudaFuncSetAttribute(k_solve_one_grp<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k->blocks = (int)inst.size();
  k->smem = smem;
  if ((e = grp_upload(&k->recs, recs.data(), recs.size() * sizeof(GOne))) != cudaSuccess) return e;
  if ((e = grp_upload((void**)&k->inst, inst.data(), inst.size() * sizeof(int))) != cudaSuccess) return e;
  return grp_upload((void**)&k->first, first.data(), first.size() * sizeof(int));
}

cudaError_t grp_launch_solve_one(const GrpKernel& k, bool fp32, const double* du, double* out, const int* active, cudaStream_t st) {
  auto kern = fp32 ? k_solve_one_grp<float> : k_solve_one_grp<double>;
  kern<<<k.blocks, k.threads, k.smem, st>>>(du, out, static_cast<const GOne*>(k.recs), k.inst, k.first, active);
  return cudaGetLastError();
}

cudaError_t launch_solve_adj(const sp_ctx* c, bool fp32, const double* r, double* out, void* vals3, int n_dir,
                             bool weighted, cudaStream_t st) {
  const OneArgs a = one_args(c, nullptr, r, out);
  const size_t NY = c->NY, NR = c->N - 1;
  const size_t ops = a.staged ? 16 * ((size_t)c->rb0 * col_stride(c->N / 2 + 1) + (size_t)c->rb1 * col_stride(c->N / 2)) : 0;
  const size_t sm = ops + 16 * (3 * NY + 2 * c->cv + 2 * NR) + (fp32 ? 8 : 16) * 3 * NR;
  const dim3 grid(c->n_unique, n_dir);
  const int th = solve_one_threads(c, 0);
  const void* kern = fp32 ? (const void*)k_solve_adj<float> : (const void*)k_solve_adj<double>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  if (fp32)
    k_solve_adj<float><<<grid, th, sm, st>>>(a, static_cast<C2<float>*>(vals3), c->Cfh_f, weighted ? 1 : 0);
  else
    k_solve_adj<double><<<grid, th, sm, st>>>(a, static_cast<C2<double>*>(vals3), c->Cfh, weighted ? 1 : 0);
  return cudaGetLastError();
}
