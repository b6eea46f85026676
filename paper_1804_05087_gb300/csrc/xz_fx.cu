// Launches of the fixed-point plane stage (xz_fx.cuh): one block per plane, or three launches
// with several blocks per plane.
#include <algorithm>
#include <cmath>
#include <vector>

#include "xz_fx.cuh"

namespace {

using namespace fxz;

// N = N1 N2 with both factors in {2, 3, 4, 6, 8, 9, 12}, as equal as possible, N1 <= N2
bool factor(int n, int* n1, int* n2) {
  for (int p : {12, 9, 8, 6, 4, 3, 2}) {
    if (p * p > n || n % p) continue;
    const int q = n / p;
    for (int r : {2, 3, 4, 6, 8, 9, 12})
      if (r == q) {
        *n1 = p;
        *n2 = q;
        return true;
      }
  }
  return false;
}

size_t tw_bytes(const sp_ctx* c) { return (size_t)(c->nx + c->nz) * 16; }
// z buffer of rp row pairs: six fields (the adjoint: six outputs and their fractions)
int z_fields(int mode) { return mode == XZ_ADJOINT ? 12 : 6; }
size_t chunk_bytes(const sp_ctx* c, int rp, int fields) {
  return (size_t)rp * fields * c->fx_n1z * (c->fx_n2z + 1) * 16;
}
size_t plane_bytes(const sp_ctx* c) { return (size_t)c->nx * 6 * c->MZ * 16; }
// row pairs per chunk: z buffers of about 34 KB, which leave two blocks of 48 x 48 planes on an SM (us with 24,
// 34 and 48 KB: 256 tangents of 48 x 65 x 48 3460, 3157, 4670; 32 of 64 x 65 x 64 1377, 1160, 1125; one of
// 36 x 45 x 24 26.8, 26.8, 24.6)
int chunk_rows(const sp_ctx* c, int mode) {
  return std::max(1, std::min(c->nx / 2, (int)(34 * 1024 / chunk_bytes(c, 1, z_fields(mode)))));
}
size_t fused_smem(const sp_ctx* c, int mode) {
  return tw_bytes(c) + plane_bytes(c) + chunk_bytes(c, chunk_rows(c, mode), z_fields(mode));
}

// blocks per plane of a split x transform: about 24 KB of staging each (every block scans the plane for its
// scales; us of the three launches with 12, 24 and 48 KB, one tangent: 48 x 65 x 48 41, 35, 39; 64 x 65 x 64
// 82, 66, 58; 96 x 97 x 96 282, 196, 156: large planes would take larger parts)
int split_parts(const sp_ctx* c, int ncol) {
  const int most = std::max(8, (int)(24576 / (16 * c->nx)));
  return (ncol + most - 1) / most;
}

Args make_args(const sp_ctx* c, int mode, const void* in, void* out) {
  Args a;
  a.in = reinterpret_cast<const double2*>(in);
  a.out = mode == XZ_BASE ? nullptr : reinterpret_cast<double2*>(out);
  a.bfx = reinterpret_cast<int4*>(c->base_fx);
  const bool keep = mode != XZ_STEP;  // XZ_STEP: a step without a new linearisation point
  if (!keep) a.bfx = nullptr;
  a.bmeta = keep ? c->base_meta : nullptr;
  a.b32 = keep && c->cfg.prec == SP_MIXED ? c->base32 : nullptr;
  a.b32t = c->base32t;
  a.active = nullptr;
  a.lam = c->lam6;
  a.tw = c->fx_tw;
  a.G = reinterpret_cast<cx*>(c->fx_G);
  a.gmeta = c->fx_gmeta;
  a.nx = c->nx; a.nz = c->nz; a.NY = c->NY; a.Mm = c->Mm; a.MX = c->MX; a.MZ = c->MZ; a.Kx = c->Kx; a.Kz = c->Kz;
  a.n1x = c->fx_n1x; a.n2x = c->fx_n2x; a.n1z = c->fx_n1z; a.n2z = c->fx_n2z;
  a.rp = chunk_rows(c, mode);
  a.nchunk = (c->nx / 2 + a.rp - 1) / a.rp;
  a.dMZ = div_of(c->MZ);
  a.dnz = div_of(c->nz);
  a.dn1z = div_of(a.n1z);
  a.dn2z = div_of(a.n2z);
  a.dn2x = div_of(a.n2x);
  const int nin = mode == XZ_ADJOINT ? 3 : 6;
  a.pin = split_parts(c, nin * c->MZ);
  a.pout = split_parts(c, (9 - nin) * c->MZ);
  return a;
}

// Three launches with several blocks per plane instead of one block per plane: planes that do not
// fit on chip, and large planes that fill less than two thirds of the SMs. Measured (us of a tangent, one
// block | several): 48 x 48, 65 planes 51 | 35; 97: 51 | 45; 113: 51 | 55; 260: 60 | 89; 64 x 64, 65 planes
// 84 | 66; 97: 83 | 74; 113: 84 | 92; 32 x 32, 49 planes 27 | 31; 36 x 24, 45 planes 27 | 31; 16 x 16, 33 planes
// 12.5 | 23.
bool use_split(const sp_ctx* c, int mode, int n_dir) {
  if (fused_smem(c, mode) > kSmemMax) return true;
  return c->nx * c->nz > 1600 && 3LL * c->NY * n_dir < 2LL * c->sm_count;
}

}  // namespace

sp_status sp_fx_setup(sp_ctx* c) {
  if (!factor(c->nx, &c->fx_n1x, &c->fx_n2x) || !factor(c->nz, &c->fx_n1z, &c->fx_n2z)) return SP_OK;
  if (c->MZ > kMaxKz || c->nx / 2 > kMaxPairs) return SP_OK;
  const int rp = chunk_rows(c, XZ_ADJOINT), chunks = (c->nx / 2 + rp - 1) / rp;
  if (chunks > kMaxChunks) return SP_OK;
  std::vector<int4> tw(c->nx + c->nz);
  auto half = [](long double v, int* hi, int* lo) {
    const long long q = llrintl(v * 4611686018427387904.0L);  // 2^62
    *lo = (int)(unsigned)(q & 0xffffffffLL);
    *hi = (int)((q - *lo) >> 32);
  };
  const long double tau = 6.283185307179586476925286766559005768L;
  for (int d = 0, n = c->nx; d < 2; ++d, n = c->nz)
    for (int k = 0; k < n; ++k) {
      int4& t = tw[d * c->nx + k];
      // quarter turns are exact
      long double co = cosl(tau * k / n), si = sinl(tau * k / n);
      if (4 * k % n == 0) {
        const int r = 4 * k / n;
        co = r == 0 ? 1.0L : r == 2 ? -1.0L : 0.0L;
        si = r == 1 ? 1.0L : r == 3 ? -1.0L : 0.0L;
      }
      half(co, &t.x, &t.y);
      half(si, &t.z, &t.w);
    }
  const size_t nxz = (size_t)c->nx * c->nz;
  // planes of the largest split call
  int split_dirs = 0;
  for (int d = c->cfg.max_batch; d >= 1 && !split_dirs; --d)
    if (use_split(c, XZ_TANGENT, d) || use_split(c, XZ_ADJOINT, d)) split_dirs = d;
  const size_t nplanes = std::max<size_t>((size_t)c->NY * split_dirs, 1);
  const size_t meta = meta_ints(chunks);  // the adjoint has the most chunks
  bool ok = cudaMalloc((void**)&c->fx_tw, tw.size() * 16) == cudaSuccess &&
            cudaMemcpy(c->fx_tw, tw.data(), tw.size() * 16, cudaMemcpyHostToDevice) == cudaSuccess &&
            cudaMalloc(&c->fx_G, nplanes * plane_bytes(c)) == cudaSuccess &&
            cudaMalloc((void**)&c->fx_gmeta, nplanes * meta * 4) == cudaSuccess;
  if (ok && c->cfg.prec == SP_FP64)
    ok = cudaMalloc((void**)&c->base_fx, (size_t)6 * c->NY * nxz * 8 + (size_t)c->NY * 48) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    return SP_ENOMEM;
  }
  if (c->base_fx) c->base_meta = reinterpret_cast<int*>(c->base_fx + (size_t)6 * c->NY * nxz);
  c->use_fx = 1;
  return SP_OK;
}

static cudaError_t launch_args(const sp_ctx* c, const Args& a, int mode, int n_dir, bool split, cudaStream_t st) {
  size_t smem = fused_smem(c, mode);
  if (split) {
    const int nin = mode == XZ_ADJOINT ? 3 : 6, ci = nin * c->MZ, co = (9 - nin) * c->MZ;
    const size_t cols = std::max((ci + a.pin - 1) / a.pin, (co + a.pout - 1) / a.pout);
    smem = tw_bytes(c) + std::max((size_t)c->nx * cols * 16, chunk_bytes(c, a.rp, z_fields(mode)));
  }
  if (mode == XZ_TANGENT) return launch_tangent(a, n_dir, split, smem, st);
  if (mode == XZ_ADJOINT) return launch_adjoint(a, n_dir, split, smem, st);
  return launch_step(a, n_dir, split, smem, st);
}

cudaError_t launch_xz_fx(const sp_ctx* c, int mode, const void* in, void* out, int n_dir, cudaStream_t st) {
  return launch_args(c, make_args(c, mode, in, out), mode, n_dir, use_split(c, mode, n_dir), st);
}

cudaError_t launch_xz_fx_apart(const sp_ctx* c, int mode, const void* in, void* out, void* scratch, size_t bytes,
                               cudaStream_t st) {
  Args a = make_args(c, mode, in, out);
  const bool split = fused_smem(c, mode) > kSmemMax;
  const size_t planes = (size_t)c->NY * plane_bytes(c);
  if (split && planes + c->NY * meta_ints(a.nchunk) * 4 <= bytes) {
    a.G = static_cast<cx*>(scratch);
    a.gmeta = reinterpret_cast<int*>(static_cast<unsigned char*>(scratch) + planes);
  }
  return launch_args(c, a, mode, 1, split, st);
}

// ------------------------------------------------------------------ groups
// Members in two classes by shared memory, so that small planes keep two blocks per SM beside large
// ones; members whose plane does not fit on chip run their own split launches.
cudaError_t grp_build_xz_fx(GrpPlan* p, sp_ctx* const* mem, int n, const int* order) {
  std::vector<Args> recs(n);
  for (int m = 0; m < n; ++m)
    if (mem[m]->use_fx) recs[m] = make_args(mem[m], XZ_STEP_BASE, mem[m]->ws6, mem[m]->ws3);
  for (int cls = 0; cls < 2; ++cls) {
    std::vector<int> inst, first(n, 0);
    size_t smem = 0;
    for (int q = 0; q < n; ++q) {
      const sp_ctx* c = mem[order[q]];
      const size_t need = c->use_fx ? fused_smem(c, XZ_TANGENT) : 0;
      if (!c->use_fx || need > kSmemMax || (need > kSmemMax / 2) != (cls == 0)) continue;
      first[order[q]] = (int)inst.size();
      for (int b = 0; b < c->NY; ++b) inst.push_back(order[q]);
      smem = std::max(smem, need);
    }
    GrpKernel& k = p->fx[cls];
    k.blocks = (int)inst.size();
    k.smem = smem;
    if (inst.empty()) continue;
    cudaError_t e;
    if ((e = grp_upload(&k.recs, recs.data(), recs.size() * sizeof(Args))) != cudaSuccess) return e;
    if ((e = grp_upload((void**)&k.inst, inst.data(), inst.size() * sizeof(int))) != cudaSuccess) return e;
    if ((e = grp_upload((void**)&k.first, first.data(), first.size() * sizeof(int))) != cudaSuccess) return e;
  }
  p->fx_own.clear();
  for (int m = 0; m < n; ++m)
    if (mem[m]->use_fx && fused_smem(mem[m], XZ_TANGENT) > kSmemMax) p->fx_own.push_back({m, mem[m]});
  return cudaSuccess;
}

cudaError_t grp_launch_xz_fx(const GrpPlan& p, int mode, const int* active, cudaStream_t st) {
  for (const auto& own : p.fx_own) {
    const sp_ctx* c = own.second;
    Args a = make_args(c, mode, c->ws6, c->ws3);
    a.active = active ? active + own.first : nullptr;
    const cudaError_t e = launch_args(c, a, mode, 1, true, st);
    if (e != cudaSuccess) return e;
  }
  for (const GrpKernel& k : p.fx) {
    if (k.blocks == 0) continue;
    const cudaError_t e = mode == XZ_TANGENT ? launch_tangent_grp(k, active, mode, st) : launch_step_grp(k, active, mode, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
