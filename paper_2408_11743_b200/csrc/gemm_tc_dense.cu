// The dense 4-bit instances of the tcgen05 kernel.
#include "gemm_tc.cuh"

namespace marlin_b200 {
namespace tc {

cudaError_t launch_dense(int nt, int mpad, int scale, const GemmParams& p, cudaStream_t stream) {
  if (scale == kDeferred) return launch_mpad<1, kDeferred, kFmtDense4>(mpad, p, stream);
  return nt == 1 ? launch_scale<1, kFmtDense4>(mpad, scale, p, stream) : launch_scale<2, kFmtDense4>(mpad, scale, p, stream);
}

}  // namespace tc
}  // namespace marlin_b200
