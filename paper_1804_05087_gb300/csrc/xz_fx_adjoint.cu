// Fixed-point plane stage (xz_fx.cuh): kernels of one kind.
#include "xz_fx.cuh"

namespace fxz {

cudaError_t launch_adjoint(const Args& a, int n_dir, bool split, size_t smem, cudaStream_t st) {
  return launch_kind<kAdjoint>(a, n_dir, split, smem, st);
}

}  // namespace fxz
