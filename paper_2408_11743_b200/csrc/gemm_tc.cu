// Host side of the tcgen05 kernel: tile, partition and instance for a call.
#include "gemm_tc.cuh"

namespace marlin_b200 {

namespace {

int tc_mpad(int m) { return m <= 32 ? 32 : (m <= 64 ? 64 : 128); }

struct TcPlan {
  int nt;                     // 128-column UMMA tiles per CTA
  long long ncols, workers;   // (column tile, slab) pairs; CTAs
  int split, cluster;         // k-ranges per tile (0: stripes over all units); CTAs per cluster
  bool whole;                 // stripes cut at tile boundaries
  double cost;                // us
};

// The best partition with tiles of 128 nt columns, by a cost in microseconds fitted to measured launch times (launches one behind
// the other).  A k-block costs a CTA 0.30 us with 128 columns and 0.43 with 256 (0.55 at 64 rows; 0.33 and 0.66 at 128, where the MMAs
// take part): up to 64 rows less its weights than the waits between the warps.  The exchange of partial tiles between the CTAs of
// a tile costs 0.5 us + 5 us per 128 KB; clusters of more than four CTAs are slower to place (0.3 to 1.6 us); a second
// round through the workspace (several clusters per tile) costs 1.6 us and half of the exchange again; with stripes one CTA
// reads every contributor's partial tile.  A grid of at most half of the SMs lets the next launch start beside it: 1.8 us.
// Measured on B200 (256 / 128 columns): 8192 x 8192 13.5 / 14.4 us at 32 rows, 15.9 / 15.4 at 64, 22.4 / 18.6 at 128;
// 4096 x 4096 at 17 rows 9.2 with eight k-ranges of 256 columns, 7.8 with six, 7.0 with four, 7.3 with four of 128 columns; at 100
// rows 13.3 / 10.2; 28672 x 8192 25 / 32 us at 17 rows; 4096 x 22016 29 / 27 us at 100 rows.
TcPlan plan_tile(int nt, int scale, int rows, int slabs, int kb, int N, int sm_count, double per_kb) {
  TcPlan best{};
  const long long sms = sm_count < kMaxWorkers ? sm_count : kMaxWorkers;
  const long long ncols = (long long)((N + 128 * nt - 1) / (128 * nt)) * slabs, units = ncols * kb;
  double u = per_kb * (nt == 1 ? (rows > 64 ? (scale == tc::kDeferred ? 0.50 : 0.33) : rows > 32 && scale == tc::kDeferred ? 0.40 : 0.30)
                                     : (rows > 64 ? 0.66 : rows > 32 ? 0.55 : 0.43));
  // Several slabs: a 128-column tile fetches the activations of a k-block for half as many MMAs as a 256-column one.  That tells where
  // the MMAs are short (2:4: 3634 x 10112 x 4864 265 us with 128 columns, 186 with 256; 1024 x 8192 x 8192 83 / 70; but 512 x
  // 4096 x 11008 32 / 42, whose 256-column tiles divide the SMs badly), and where the activations outgrow the L2's nearer
  // half (4-bit, 3634 x 10112 x 4864: 350 / 304 us; 2048 x 4096 x 22016: 293 / 309).
  if (slabs > 1 && per_kb < 1.0) u = nt == 1 ? 0.34 : 0.56;
  if (slabs > 1 && per_kb >= 1.0 && nt == 1 && (double)slabs * rows * kb * 256.0 > 48e6) u *= 1.2;
  const double fixed = per_kb < 1.0 && nt == 1 ? 0.6 : 0.0;  // (2:4: three copies per k-block instead of two)
  const double exchange = 0.5 + 5.0 * rows / 128 * nt / 2;
  const char* e = getenv("MARLIN_B200_TC_SPLIT");    // tuning knob: 0 forces stripes, 1.. = that many k-ranges per tile
  const char* c = getenv("MARLIN_B200_TC_CLUSTER");  // tuning knob: largest cluster (0: none)
  const int forced = e ? atoi(e) : -1, max_cluster = c ? atoi(c) : 8;
  auto take = [&](long long workers, int split, int cluster, bool whole, double cost) {
    cost += fixed - (2 * workers <= sms ? 1.8 : 0.0);
    if (best.nt && cost >= best.cost) return;
    best = TcPlan{nt, ncols, workers, split, cluster, whole, cost};
  };
  // tiles cut into S k-ranges, S CTAs of as many as possible per cluster (all clusters have to be resident at once; the
  // numbers are what the occupancy query returns on a B200 for CTAs that fill an SM)
  static const int resident[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
  for (long long S = 1; S * ncols <= sms && S <= kb && forced != 0; ++S) {
    if (forced > 0 && S != forced && forced * ncols <= sms && forced <= kb) continue;
    int cs = 1;
    for (int d = 2; d <= 8 && d <= max_cluster; ++d)
      if (S % d == 0 && S * ncols <= (long long)resident[d] * d) cs = d;
    const long long n = (kb + S - 1) / S;
    static const double placing[9] = {0, 0, 0, 0, 0, 0.3, 0.45, 1.5, 1.6};
    const double fix = S == 1    ? 0.0
                       : cs == 1 ? exchange * (0.5 + 0.7 * (double)S)
                                 : exchange + placing[cs] + (S > cs ? 1.6 + exchange * (0.4 + 0.1 * (double)(S / cs)) : 0.0);
    take(S * ncols, (int)S, cs, false, u * (double)n + fix);
  }
  // even stripes over all units (the paper's form)
  const long long workers = units < sms ? units : sms;
  if (forced <= 0 || !best.nt) {
    const double n = (double)units / (double)workers;
    const double contributors = (double)workers / (double)ncols + 1.0;
    // (2:4 with several slabs: 218 us in stripes, 186 with whole tiles, 3634 x 10112 x 4864)
    take(workers, 0, 0, false, u * (slabs > 1 && per_kb < 1.0 ? 1.3 : 1.0) * n + exchange * (0.5 + 0.7 * (contributors < 2.0 ? 2.0 : contributors)));
  }
  // stripes cut at tile boundaries: nothing is shared
  if (forced < 0 && ncols >= workers) take(workers, 0, 0, true, u * (double)((ncols + workers - 1) / workers * kb));
  return best;
}

}  // namespace

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
  // columns per tile: 128 or 256 (deferred scales: 128)
  const bool choice = scale != tc::kDeferred;
  const char* tile = getenv("MARLIN_B200_TC_TILE");  // tuning knob: 128 or 256 columns per tile, where there is a choice
  TcPlan best{};
  for (int nt = 1; nt <= 2; ++nt) {
    if (choice ? (tile && (atoi(tile) == 128) != (nt == 1)) : nt != 1) continue;
    const TcPlan c = plan_tile(nt, scale, p.M < mpad ? p.M : mpad, (int)p.slabs, (int)p.kb, p.N, sm_count, sparse24 ? 0.65 : w8 ? 1.25 : 1.0);
    if (!best.nt || c.cost < best.cost) best = c;
  }
  p.ncols = (int)best.ncols;
  p.units = (uint32_t)(best.ncols * (long long)p.kb);
  p.workers = (uint32_t)best.workers;
  p.split = (uint32_t)best.split;
  p.cluster = (uint32_t)best.cluster;
  p.whole = best.whole ? 1u : 0u;
  const int nt = best.nt;
  if (w8) return tc::launch_w8(nt, mpad, scale, p, stream);
  if (sparse24) return tc::launch_sparse(nt, mpad, scale, p, stream);
  return tc::launch_dense(nt, mpad, scale, p, stream);
}

}  // namespace marlin_b200
