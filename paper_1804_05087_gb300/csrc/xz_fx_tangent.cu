// Fixed-point plane stage (xz_fx.cuh): kernels of one kind.
#include "xz_fx.cuh"

namespace fxz {

cudaError_t launch_tangent(const Args& a, int n_dir, bool split, size_t smem, cudaStream_t st) {
  return launch_kind<kTangent>(a, n_dir, split, smem, st);
}

cudaError_t launch_tangent_grp(const GrpKernel& k, const int* active, int mode, cudaStream_t st) {
  return launch_kind_grp<kTangent>(k, active, mode, st);
}

}  // namespace fxz
