// Tile and partition of the warp-level kernel (gemm_dense.cu) for a launch.  Host arithmetic alone, without CUDA, so that it can be
// compiled and checked by itself.
#pragma once
#include <stdint.h>
#include <stdlib.h>

#ifdef __CUDACC__
#define MARLIN_HOST_DEVICE __host__ __device__
#else
#define MARLIN_HOST_DEVICE
#endif

namespace marlin_b200 {

constexpr int kPlanChunk = 64;  // columns of a chunk
// Twelve consumer warps (three per scheduler, 152 registers each: the 8-row instances need no more; the 16-row ones
// would spill) hide more of the latency of the conversion -> MMA chains: the loop runs about 10 % faster.  The plan
// takes them where that shows in the launch time.
constexpr int kNarrowConsumerWarps = 8, kWideConsumerWarps = 12;

struct DensePartition {
  int nw;       // chunks per stage; column tile = 64 * nw
  int ncols;    // column tiles
  int split;    // 0: even stripes over all units; S > 0: teams of S CTAs, each with consecutive column tiles of its own
  int teams;    // number of teams (ncols: a column tile each, cut into S k-ranges)
  int workers;  // CTAs
  int cw;       // consumer warps
};

// Teams of S workers, C of them: the first ncols % C teams own ncols / C + 1 column tiles, the others
// ncols / C, one team after the other; the workers of a team have even stripes over its k-blocks.  With C = ncols every
// tile is cut into S k-ranges.
MARLIN_HOST_DEVICE inline uint32_t team_first_tile(uint32_t t, uint32_t tiles, uint32_t extra) {
  return t * tiles + (t < extra ? t : extra);
}

// mb: blocks of eight rows (1, 2); teams_too: what a launch takes (teams of any form); otherwise the best of even stripes and of one
// column tile per team
inline DensePartition plan_dense(int mb, bool sparse, int kb, int N, long long max_workers, bool teams_too) {
  // Partition (Section 3.4 "Striped Partitioning", adapted).  Two forms.  Tile-aligned: every column tile
  // is cut into S equal k-ranges, one per CTA, so that all CTAs do the same work and run the fix-up once
  // (S = 1: not at all), with the tile width (64, 128 or 256 columns) that suits the shape.  Even stripes
  // over all units (the paper's form, 128-column tiles): every SM is busy to the end, but a CTA whose
  // stripe crosses a tile boundary pays the fix-up twice and finishes microseconds after the others.
  // A cost in microseconds picks between them: a least-squares fit (relative error) to the launch times measured
  // on B200 for every candidate on 36 layer shapes (K, N from 2048 to 28672), at one row and at sixteen.  Up to
  // eight rows: 2.33 fixed, the chunks of the longest CTA at 0.121 (64-column tiles), 0.099 (128 columns; 0.096
  // with twelve consumer warps) or 0.105 (256 columns) each, the cluster fix-up at 0 / 0.36 / 0.68 by tile width
  // plus 0.137 per CTA of the tile (1.11 more through the workspace, above eight CTAs), 4.14 for the late finishers
  // of even stripes: the pick is within 3 % of the fastest candidate on all 36 shapes (0.1 % on average).  Sixteen
  // rows (twice the MMAs per chunk, a ring of fewer and larger stages) have constants of their own and leave out
  // split 256-column tiles, whose times the linear model does not follow (0.3 % on average, at most 5 %).
  int forced_nw = 0;
  if (const char* e = getenv("MARLIN_B200_NW")) { int v = atoi(e); if (v == 1 || v == 2 || v == 4) forced_nw = v; }
  bool allow_split = true;
  if (const char* e = getenv("MARLIN_B200_SPLIT")) allow_split = atoi(e) != 0;
  int want_cw = 0;  // MARLIN_B200_CW: tuning knob, 8 or 12
  if (const char* e = getenv("MARLIN_B200_CW")) want_cw = atoi(e);
  // twelve consumer warps: 128-column tiles from 16 stages per CTA on (see the end)
  auto wide_pays = [&](int nw_, long long n) { return mb == 1 && nw_ == 2 && n >= 16 && !sparse; };
  auto chunk_us = [&](int nw_, long long n) {
    if (mb != 1) return nw_ == 1 ? 0.1536 : nw_ == 4 ? 0.1424 : 0.1303;
    const bool wide = want_cw == kWideConsumerWarps || (want_cw != kNarrowConsumerWarps && wide_pays(nw_, n));
    return nw_ == 1 ? 0.1213 : nw_ == 4 ? 0.1051 : (wide ? 0.0964 : 0.0991);
  };
  const double base_us = mb == 1 ? 2.33 : 2.55, even_us = mb == 1 ? 4.14 : 4.62;
  auto fixup_us = [&](int nw_, long long S) {
    if (S <= 1) return 0.0;
    if (mb == 1) return (nw_ == 1 ? 0.0 : nw_ == 2 ? 0.36 : 0.68) + 0.137 * (double)S + (S > 8 ? 1.11 : 0.0);
    return (nw_ == 1 ? -0.34 : nw_ == 2 ? 0.0 : 0.89) + 0.268 * (double)S + (S > 8 ? 0.51 : 0.0);
  };
  int even_nw = forced_nw ? forced_nw : 2;
  while (even_nw > 1 && N % (kPlanChunk * even_nw)) even_nw >>= 1;
  const long long even_units = (long long)(N / (kPlanChunk * even_nw)) * kb;
  const long long even_workers = even_units < max_workers ? even_units : max_workers;
  const long long even_n = (even_units + even_workers - 1) / even_workers;
  double best = base_us + even_us + chunk_us(even_nw, even_n) * (double)(even_n * even_nw);
  int nw = even_nw, split = 0;
  // The stripes of the paper or the tile-aligned form, with the most CTAs; what a launch takes in their place comes below.
  long long teams = 0;
  for (int cand = 1; cand <= 4 && allow_split; cand *= 2) {
    if (forced_nw && cand != forced_nw) continue;
    if (N % (kPlanChunk * cand)) continue;
    const long long ncols = N / (kPlanChunk * cand);
    long long S = max_workers / ncols;
    if (S > kb) S = kb;
    if (S < 1) continue;
    const long long stages_per_cta = (kb + S - 1) / S;
    if (mb != 1 && cand == 4 && S > 1 && !forced_nw) continue;
    const double cost = base_us + chunk_us(cand, stages_per_cta) * (double)(stages_per_cta * cand) + fixup_us(cand, S);
    if (cost < best) { nw = cand; split = (int)S; teams = ncols; best = cost; }
  }
  // Teams of S CTAs, each with consecutive column tiles of its own: one tile (tile-aligned: any S), or several, cut evenly
  // between two CTAs (whole tiles for S = 1), where no number of k-ranges uses the SMs well.  With more than two CTAs per
  // team several tiles gain as much in a chain of equal launches, but clusters of three behind clusters of four leave SMs in
  // pieces that the next ones do not fit: a wave more (gate_up 22016 columns, then down, one row: 29.9 us against 20.4 with
  // pairs and 21.7 with even stripes).
  // A grid of at most half of the SMs lets the next launch start beside it: 8192 x 1024 at one row 5.5 us with nine k-ranges,
  // 4.1 with four (64 CTAs); 1024 x 1024 4.6 with eight, 3.0 with two.  Clusters of seven and eight start late.  Clusters that
  // do not fit at once (`resident`: what the occupancy query returns on a B200) exchange through the workspace.
  static const int resident[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
  if (teams_too && allow_split) {
    double best_us = base_us + even_us + chunk_us(even_nw, even_n) * (double)(even_n * even_nw);
    nw = even_nw;
    split = 0;
    for (int cand = 1; cand <= 4; cand *= 2) {
      if (forced_nw && cand != forced_nw) continue;
      if (N % (kPlanChunk * cand)) continue;
      const long long ncols = N / (kPlanChunk * cand);
      for (long long S = 1; S <= kb && S <= max_workers; ++S) {
        if (S > 2 && S * ncols > max_workers) break;
        const long long per = max_workers / S, T = (ncols + per - 1) / per;  // column tiles of a team
        const long long C = (ncols + T - 1) / T;
        const long long stages_per_cta = (T * kb + S - 1) / S;
        if (mb != 1 && cand == 4 && S > 1 && !forced_nw) continue;
        double cost = base_us + chunk_us(cand, stages_per_cta) * (double)(stages_per_cta * cand) + fixup_us(cand, S);
        if (T > 1) cost += (mb == 1 ? 0.5 : 0.65) + 0.25 * (double)T;
        if (mb == 1 && cand == 4 && S > 1) cost += 0.47;
        if (S > 1 && S <= 8 && C > resident[S]) cost += 1.5;
        if (2 * S * C <= max_workers) cost -= mb == 1 ? 0.75 : 0.5;
        else if (S >= 7 && S <= 8) cost += mb == 1 ? 0.5 : 0.25;
        if (cost < best_us) { nw = cand; split = (int)S; teams = C; best_us = cost; }
      }
    }
  }
  DensePartition p;
  p.nw = nw;
  p.ncols = N / (kPlanChunk * nw);
  const long long units = (long long)p.ncols * kb;
  p.split = split;
  p.teams = split ? (int)teams : p.ncols;
  long long workers = split ? (long long)split * teams : max_workers;
  if (workers > units) workers = units;
  p.workers = (int)workers;
  // Consumer warps: twelve for 128-column tiles (nw = 2) from 16 stages per CTA on.  Measured on B200 over 42 layer
  // shapes (K, N from 2048 to 28672, one row): with 128-column tiles twelve warps are 5.5-7.7 % faster at every
  // shape from 16 stages per CTA up; with 64-column tiles they are 3-5 % slower (the ring, capped at 32 stages, holds
  // only two rounds of twelve stages, too few to cover the refill latency); with 256-column tiles it makes no
  // difference; the 2:4 instance gains nothing.
  p.cw = kNarrowConsumerWarps;
  if (mb == 1) {
    const long long n = (units + workers - 1) / workers;
    if (want_cw == kWideConsumerWarps || (want_cw != kNarrowConsumerWarps && wide_pays(nw, n))) p.cw = kWideConsumerWarps;
  }
  return p;
}

}  // namespace marlin_b200
