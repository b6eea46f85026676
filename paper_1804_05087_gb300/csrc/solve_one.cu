// Per-mode Stokes solve by the precomputed dense operators, one Fourier mode of one direction per
// block: the step, single tangents and small batches (batches from kChainMinBatch directions take the
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
// direction: 55 us with four modes per block and loads inside the products, see the rule in
// sp_solve_shapes for the threads.
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
  int n_unique, Mm, MX, MZ, Kx, NY, cv, rb0, rb1, off_v0, off_v1, off_h0, off_h1, op_stride, staged;
  double inv_dt;
};

__device__ __forceinline__ uint32_t smem_of(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// mode u of direction dir
template <typename T>
__device__ __forceinline__ void solve_one(const OneArgs& a, int u, int dir, unsigned char* smem, uint64_t* s_bar) {
  const int NY = a.NY, N = NY - 1, NH = N / 2 + 1, NR = N - 1, Mm = a.Mm, MZ = a.MZ;
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, nw = nt >> 5;
  double* sop = reinterpret_cast<double*>(smem);
  double2* sdu = reinterpret_cast<double2*>(sop + (a.staged ? a.op_stride : 0));  // [3][NY]
  double2* sfa = sdu + 3 * NY;  // [NR] -i f_a
  double2* sfb = sfa + NR;      // [NR] (mean mode: f_u)
  double2* srv = sfb + NR;      // [2][cv] reduced right-hand sides per parity
  double2* sfw = srv + 2 * a.cv;  // [NR] mean mode: f_w; float: staged right-hand sides
  double2* sv = sfw + 3 * NR;   // [NY]
  double2* sb = sv + NY;        // [NY]
  double2* ss = sb + NY;        // [NY + 1] sums of p v_p over p >= n of the parity of n
  C2<T>* vals = reinterpret_cast<C2<T>*>(ss + NY + 1);  // [3][NY] (float)
  const uint32_t bar = smem_of(s_bar);
  int pos, iz;
  {
    const int first = (a.Kx + 1) * MZ;
    if (u < first) {
      pos = u / MZ;
      iz = u - pos * MZ;
    } else {
      const int v = u - first;
      pos = a.Kx + 1 + v / (MZ - 1);
      iz = 1 + v % (MZ - 1);
    }
  }
  const bool mean = u == 0;
  const double* op = a.ops + (size_t)u * a.op_stride;
  if (a.staged && tid == 0) {
    const uint32_t bytes = (uint32_t)a.op_stride * 8;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_of(sop)),
                 "l"(op), "r"(bytes), "r"(bar)
                 : "memory");
  }
  const double kx = __ldg(a.wave + 4 * u), kz = __ldg(a.wave + 4 * u + 1), ik = __ldg(a.wave + 4 * u + 2);
  // input state (Hermitian-projected)
  const double2* dsrc = a.du + ((size_t)dir * 3 * Mm + pos * MZ + iz) * NY;
  const long long mir = pos == 0 ? 0 : (long long)(a.MX - 2 * pos) * MZ * NY;  // to the mirror mode
  for (int i = tid; i < 3 * NY; i += nt) {
    const int c = i / NY;
    const double2* p = dsrc + (size_t)c * Mm * NY + (i - c * NY);
    double2 v = __ldg(p);
    if (iz == 0) {
      const double2 w = __ldg(p + mir);
      v = make_double2(0.5 * (v.x + w.x), 0.5 * (v.y - w.y));
    }
    sdu[i] = v;
  }
  if constexpr (sizeof(T) == 8) {
    const double2* W = static_cast<const double2*>(a.in) + ((size_t)dir * a.n_unique + u) * 3 * NR;
    for (int i = tid; i < 3 * NR; i += nt) sfw[i] = __ldg(W + i);
    __syncthreads();
  } else {
    // forward transform of the values: even and odd parts of the point pairs, then one thread per row
    // (even rows first; the order of k_solve's sums)
    const C2<T>* vin = static_cast<const C2<T>*>(a.in) + (size_t)dir * 3 * NY * Mm + pos * MZ + iz;
    for (int i = tid; i < 3 * NH; i += nt) {
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
    const int ne = (NR + 1) / 2;
    for (int i = tid; i < 3 * NR; i += nt) {
      const bool odd = i >= 3 * ne;
      const int k = odd ? i - 3 * ne : i, per = odd ? NR - ne : ne;
      const int c = k / per, n = 2 * (k - c * per) + (odd ? 1 : 0);
      const C2<T>* col = vals + c * NY;
      const float* cf = a.cft + n;
      C2<T> acc = mk((T)0, (T)0);
      if (!odd) {
        for (int j = 0; j < NH - 1; ++j) acc = acc + scl(col[j], (T)__ldg(cf + j * NY));
        acc = acc + scl(col[NH - 1], (T)__ldg(cf + (NH - 1) * NY));
      } else {
        for (int j = 0; j < NH - 1; ++j) acc = acc + scl(col[N - j], (T)__ldg(cf + j * NY));
      }
      const double2 d = sdu[c * NY + n];
      double2 f = make_double2((double)acc.x + d.x * a.inv_dt, (double)acc.y + d.y * a.inv_dt);
      if (mean) f.y = 0.0;
      sfw[c * NR + n] = f;
    }
    __syncthreads();
  }
  // rotation to the components along / across the wavevector
  for (int n = tid; n < NR; n += nt) {
    const double2 fx = sfw[n], fy = sfw[NR + n], fz = sfw[2 * NR + n];
    if (mean) {
      sfb[n] = fx;
      sfa[n] = fz;
      continue;
    }
    const double2 fa = make_double2((kx * fx.x + kz * fz.x) * ik, (kx * fx.y + kz * fz.y) * ik);
    sfb[n] = make_double2((-kz * fx.x + kx * fz.x) * ik, (-kz * fx.y + kx * fz.y) * ik);
    srv[(n & 1) * a.cv + n / 2] = fy;
    sfa[n] = make_double2(fa.y, -fa.x);  // -i f_a
  }
  __syncthreads();
  // reduced right-hand side g_n = f_v,n - (2 / (c_n k)) sum over m > n, m + n odd, of m (-i f_a,m)
  if (!mean) {
    for (int P = warp; P < 2; P += nw) {
      double2* g = srv + P * a.cv;
      suffix_scan(
          P == 0 ? a.rb0 : a.rb1,
          [&](int i) -> double2 {
            const int m = 2 * i + P + 1;
            if (m > N - 2) return make_double2(0.0, 0.0);
            const double w = __ldg(a.row + m);
            return make_double2(w * sfa[m].x, w * sfa[m].y);
          },
          [&](int i, double2 s) {
            const double f = (2 * i + P == 0 ? 1.0 : 2.0) * ik;
            g[i] = make_double2(g[i].x - f * s.x, g[i].y - f * s.y);
          });
    }
  }
  bool ok = true;
  if (a.staged) {
    uint32_t done = 0;
    for (uint32_t it = 0; it < (1u << 25) && !done; ++it)  // the second half of the limit: the copy may be in flight
      asm volatile(
          "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
          : "=r"(done)
          : "r"(bar)
          : "memory");
    ok = done != 0;
    op = sop;
  }
  ok = __syncthreads_and(ok) != 0;  // the limit ran out: NaN below
  // v = V g and b = H f_b: one row of one operator per thread
  const int nv0 = N / 2 + 1;
  for (int i = tid; i < 2 * NY; i += nt) {
    const bool hel = i < NY;
    const int k = hel ? i : i - NY;
    const int Q = k < nv0 ? 0 : 1, row = Q == 0 ? k : k - nv0, n = 2 * row + Q;
    const int nrow = Q == 0 ? nv0 : NY - nv0, rb = Q == 0 ? a.rb0 : a.rb1;
    const double* H = op + (Q == 0 ? a.off_h0 : a.off_h1) + row;
    const double* V = op + (Q == 0 ? a.off_v0 : a.off_v1) + row;
    // mean flow: u and w from the Helmholtz operator, v = 0
    const double2* x = hel ? sfb + Q : mean ? sfa + Q : srv + Q * a.cv;
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
    (hel ? sb : sv)[n] = make_double2((s[0].x + s[1].x) + (s[2].x + s[3].x), (s[0].y + s[1].y) + (s[2].y + s[3].y));
  }
  __syncthreads();
  // (D v)_n = (2 / c_n) sum over p > n, p + n odd, of p v_p
  if (!mean) {
    for (int P = warp; P < 2; P += nw)
      suffix_scan(
          P == 0 ? nv0 : NY - nv0,
          [&](int i) -> double2 {
            const int p = 2 * i + P;
            const double w = __ldg(a.row + p);
            return make_double2(w * sv[p].x, w * sv[p].y);
          },
          [&](int i, double2 s) { ss[2 * i + P] = s; });
  }
  __syncthreads();
  // a = (i/k) D v, back-rotation, G = u_new - u, Hermitian output
  double2* dst = a.out + ((size_t)dir * 3 * Mm + pos * MZ + iz) * NY;
  for (int n = tid; n < NY; n += nt) {
    double2 un, vn, wn;
    if (mean) {
      un = make_double2(sb[n].x, 0.0);
      wn = make_double2(sv[n].x, 0.0);
      vn = make_double2(0.0, 0.0);
    } else {
      double2 dv = make_double2(0.0, 0.0);
      if (n + 1 < NY) {
        const double2 sp = ss[n + 1];
        const double f = n == 0 ? 1.0 : 2.0;
        dv = make_double2(f * sp.x, f * sp.y);
      }
      const double2 an = make_double2(-dv.y * ik, dv.x * ik);  // (i/k) Dv
      const double2 bn = sb[n];
      un = make_double2((kx * an.x - kz * bn.x) * ik, (kx * an.y - kz * bn.y) * ik);
      wn = make_double2((kz * an.x + kx * bn.x) * ik, (kz * an.y + kx * bn.y) * ik);
      vn = sv[n];
    }
    const double2 res[3] = {un, vn, wn};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 d = sdu[c * NY + n];
      double2 g = make_double2(res[c].x - d.x, res[c].y - d.y);
      if (mean) g.y = 0.0;
      if (!ok) g = make_double2(nan(""), nan(""));
      double2* o = dst + (size_t)c * Mm * NY + n;
      *o = g;
      if (iz == 0 && pos != 0) o[mir] = make_double2(g.x, -g.y);
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(512) k_solve_one(const __grid_constant__ OneArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar;
  solve_one<T>(a, blockIdx.x, blockIdx.y, smem, &s_bar);
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
  solve_one<T>(r.a, blockIdx.x - first[i], 0, smem, &s_bar);
}

// operators in shared memory up to this size (N <= 104); larger ones are read in place
constexpr size_t kStageBytes = 100 * 1024;

size_t one_smem(const sp_ctx* c, int esize) {
  const size_t ops = (size_t)c->op_stride * 8 <= kStageBytes ? (size_t)c->op_stride * 8 : 0;
  const size_t NY = c->NY, NR = c->N - 1;
  return ops + 16 * (3 * NY + 2 * NR + 2 * c->cv + 3 * NR + 3 * NY + 1) + (esize == 4 ? 3 * NY * 8 + 8 : 0);
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

// threads of a block: one per row of the two operators (shape 0), or a fixed number
int solve_one_threads(const sp_ctx* c, int shape) {
  const int rows = std::min((2 * c->NY + 31) / 32 * 32, 512);
  const int fixed[SP_TUNE_MAX] = {rows, 64, 96, 128, 192, 256, 384, 512};
  return fixed[shape];
}

cudaError_t launch_solve_one(const sp_ctx* c, bool fp32, const void* in, const double* du, double* out, int n_dir,
                             int shape, cudaStream_t st) {
  const OneArgs a = one_args(c, in, du, out);
  const size_t sm = one_smem(c, fp32 ? 4 : 8);
  auto kern = fp32 ? k_solve_one<float> : k_solve_one<double>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  kern<<<dim3(c->n_unique, n_dir), solve_one_threads(c, shape), sm, st>>>(a);
  return cudaGetLastError();
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
