// Host side of the tcgen05 kernel: tile, partition and instance for a call.
#include "gemm_tc.cuh"
#include "tc_plan.h"

namespace marlin_b200 {

int tc_max_rows(int K, int N, int sm_count) {
  // the device's 32-bit stripe arithmetic: slabs * tiles * k-blocks * workers stays below 2^31, with the smallest slab
  // (64 rows) and tile (128 columns)
  const long long per_slab = (long long)((N + 127) / 128) * (K / kTileK) * (sm_count < kMaxWorkers ? sm_count : kMaxWorkers);
  long long slabs = ((1ll << 31) - 1) / per_slab;
  if (slabs < 1) slabs = 1;
  if (slabs > (1 << 16)) slabs = 1 << 16;
  return (int)slabs * 64;
}

size_t tc_slot_bytes(int M, int K, int N) {
  // two slots of the widest tile per worker; no more workers than units
  const int mpad = tc_mpad(M);
  const long long slabs = (M + 63) / 64, units = (long long)((N + 127) / 128) * (K / kTileK) * slabs;
  const long long workers = units < kMaxWorkers ? units : kMaxWorkers;
  return (size_t)2 * workers * 256 * mpad * sizeof(float);
}

cudaError_t launch_gemm_tc(GemmParams p, int sm_count, bool sparse24, bool w8, cudaStream_t stream) {
  const int scale = !p.grouped ? tc::kPerColumn : (p.sub_groups > 1 ? tc::kInLoopSub : (p.N % 256 ? tc::kDeferred : tc::kInLoop));
  const int mpad = tc_mpad(p.M);
  // above mpad rows the layer is replicated in the unit numbering, once per slab of rows (Section 3.4, last
  // paragraph): one launch, its stripes running over (column tile, slab, k-block)
  p.slabs = (uint32_t)((p.M + mpad - 1) / mpad);
  const int format = w8 ? kTcDense8 : sparse24 ? kTcSparse4 : scale == tc::kDeferred ? kTcDeferred4 : p.zq ? kTcZero4 : kTcDense4;
  const TcPlan best = plan_tc(format, p.M, (int)p.kb, p.N, sm_count, kMaxWorkers);
  p.ncols = (int)best.ncols;
  p.units = (uint32_t)(best.ncols * (long long)p.kb);
  p.workers = (uint32_t)best.workers;
  p.split = (uint32_t)best.split;
  p.cluster = (uint32_t)best.cluster;
  p.whole = best.whole ? 1u : 0u;
  const int nt = best.nt;
  p.slab_rows = (uint32_t)tc_slab_rows(format, p.M, nt);
  if (w8) return tc::launch_w8(nt, mpad, scale, p, stream);
  if (sparse24) return tc::launch_sparse(nt, mpad, scale, p, stream);
  return tc::launch_dense(nt, mpad, scale, p, stream);
}

}  // namespace marlin_b200
