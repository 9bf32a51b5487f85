// The 2:4 instances of the tcgen05 kernel (tcgen05.mma.sp on the wide layout).
#include "gemm_tc.cuh"

namespace marlin_b200 {
namespace tc {

cudaError_t launch_sparse(int nt, int mpad, int scale, const GemmParams& p, cudaStream_t stream) {
  return nt == 1 ? launch_scale<1, kFmtSparse4>(mpad, scale, p, stream) : launch_scale<2, kFmtSparse4>(mpad, scale, p, stream);
}

}  // namespace tc
}  // namespace marlin_b200
