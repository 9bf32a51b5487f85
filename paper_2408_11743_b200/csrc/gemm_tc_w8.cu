// The 8-bit instances of the tcgen05 kernel.
#include "gemm_tc.cuh"

namespace marlin_b200 {
namespace tc {

cudaError_t launch_w8(int nt, int mpad, int scale, const GemmParams& p, cudaStream_t stream) {
  return nt == 1 ? launch_scale<1, kFmtDense8>(mpad, scale, p, stream) : launch_scale<2, kFmtDense8>(mpad, scale, p, stream);
}

}  // namespace tc
}  // namespace marlin_b200
