// Tile and partition of the tcgen05 kernel (gemm_tc.cuh) for a call.  Host arithmetic alone, without CUDA, so that it can be
// compiled and checked by itself.
#pragma once
#include <stdlib.h>

namespace marlin_b200 {

// how the weights reach the MMAs, as far as the cost of a k-block goes
enum TcFormat { kTcDense4 = 0, kTcSparse4 = 1, kTcDense8 = 2, kTcDeferred4 = 3, kTcZero4 = 4 };

// the kernel's instance: the most rows that a slab of it has
inline int tc_mpad(int m) { return m <= 32 ? 32 : (m <= 64 ? 64 : 128); }

// Rows of a slab, the MMA's N.  From 65 rows on a batch is cut into equal slabs, in units of 16 rows: what MMAs, copies and read-out cost goes with the
// rows of a slab, so 130 rows are two slabs of 80, not of 128 (8192 x 8192 at 130 rows 25.1 us so, 24.1 now; 4096 x 22016 at 100 rows
// 25.6 / 24.6; 2:4, 4096 x 4096 at 300 rows 12.6 / 12.2).  Up to 16 rows on tiles of 256 columns a slab has 16 (28672 x 8192 with one scale per
// column 25.6 us with 32, 25.3 so; 2:4, 8192 x 8192 at four rows 10.3 / 9.7).  The others are as high as the instance: rows that the issuer has
// to read at run time, or two loops for two heights, cost what the smaller MMAs give or more (4096 x 4096 at 24 rows 7.44 us with loops for 16 and
// 32 rows, 7.22 with one; at 48 rows 7.64 and no change).  With deferred scales the round trip of the accumulators bounds the loop, and
// rows at run time make it longer at every height (128 rows of 4096 x 5504 12.2 us, 12.6 with the same rows at run time).
constexpr bool tc_fixed_rows(bool deferred, int mpad, int nt) { return deferred || mpad == 64 || (mpad == 32 && nt == 1); }
inline int tc_slab_rows(int format, int m, int nt) {
  const int mpad = tc_mpad(m), slabs = (m + mpad - 1) / mpad;
  return tc_fixed_rows(format == kTcDeferred4, mpad, nt) ? mpad : ((m + slabs - 1) / slabs + 15) / 16 * 16;
}

struct TcPlan {
  int nt;                     // 128-column UMMA tiles per CTA
  long long ncols, workers;   // (column tile, slab) pairs; CTAs
  int split, cluster;         // k-ranges per tile (0: stripes over all units); CTAs per cluster
  bool whole;                 // stripes cut at tile boundaries
  double cost;                // us
};

// The best partition with tiles of 128 nt columns, by a cost in microseconds.
//
// Up to three forms: every tile cut into S k-ranges, one per CTA; even stripes over all (tile, k-block) units, the paper's form;
// and, with at least as many tiles as CTAs, whole tiles, which share nothing.  A CTA costs
//     start + k-blocks x (cost of one, by format, tile width and rows) x (1 + load x share of the SMs in use)
//   + read-out x tiles + exchange of the partial tiles.
// The MMAs of a tile wait while the accumulators of the one before are read out, hence the term per tile.  "load" is what CTAs
// cost one another: the L2 and, in 8-bit layers, the DRAM.  Clusters of more than two CTAs take longer to place; several clusters per
// tile meet a second time through the workspace; without clusters the last CTA reads every partial tile.  A grid of
// at most half of the SMs lets the next launch start beside it.  Activations of more than 40 MB outgrow the L2 where CTAs with narrow
// tiles are in different places of K.
//
// The constants are a fit to launch times on B200 (launches one behind the other, from 64 rows on for 60 ms and more, so
// that the power limit has its say: a 256-column tile reads the activations half as often, 8-bit, 2300 x 8192 x 8192 310 us against 352) of
// every candidate on 1220 (layer, rows) pairs: 4-bit with groups of 128, 64 and 32 rows and with one scale, 2:4, 8-bit and deferred
// scales, K and N from 1024 to 28672, 1 to 4096 rows.  The candidate it picked was on average 0.6 % slower than the
// fastest one and more than 5 % on 36 pairs.  The end of a launch (read-out by 16 warps, exchange in units of eight rows, sums of stripes) and the
// slabs have become faster since, the constants are those from before: of 95 pairs timed on the kernel as it is, the pick is 1.4 % slower on
// average, more than 5 % on nine (zero points, 49 x 8192 x 22272: 51 us in whole tiles, 38 in stripes; 22 x 4096 x 22016 18.5 / 16.8; 2:4, 1 x 4096 x
// 22016 13.1 / 12.2).  The constants before it (from about a dozen shapes, nothing per tile, the 8-bit ones
// scaled from 4-bit, 1.8 us for a small grid) missed by 2.6 % and, by more than 5 %, on 212 of 1198: 28672 x 8192 at 48 rows
// 46 us, 35 now (256 columns and four k-ranges instead of 128 and two); 8-bit at 256 rows 145 / 113; 2:4, 1024 x 14336 at 128 rows
// 11.5 / 8.0; 4096 x 22016 at 64 rows 18.5 / 14.4.  Zero points, whose conversion is longer, have k-blocks of their own: with those
// of 4-bit the pick is 1.6 % above the fastest on 76 pairs above 128 rows, 0.7 % so (200 x 5120 x 13824 42.3 us, 38.8 now).  Up to 32 rows the constants of 2:4 and zero points and the read-out come from
// another 200 pairs (2:4, 4096 x 22016 at one row 14.7 us with one k-range per tile, 12.5 in even stripes).
inline TcPlan plan_tc_tile(int nt, int format, int rows, int slabs, int kb, int N, int sm_count, int max_workers) {
  TcPlan best{};
  const long long sms = sm_count < max_workers ? sm_count : max_workers;
  const long long ncols = (long long)((N + 128 * nt - 1) / (128 * nt)) * slabs, units = ncols * kb;
  const int mpad = tc_mpad(rows), mi = mpad == 32 ? 0 : mpad == 64 ? 1 : 2;
  // [format][tiles][32, 64, 128 rows]
  static const double k_block[5][2][3] = {{{0.252, 0.291, 0.348}, {0.363, 0.431, 0.639}},
                                          {{0.254, 0.296, 0.254}, {0.250, 0.332, 0.373}},
                                          {{0.214, 0.280, 0.352}, {0.354, 0.487, 0.639}},
                                          {{0.349, 0.504, 0.714}, {0.349, 0.504, 0.714}},
                                          {{0.288, 0.341, 0.370}, {0.454, 0.553, 0.826}}};
  static const double load[5] = {0.152, 0.069, 0.415, 0.0, 0.087};
  static const double read_out[2][3] = {{1.00, 0.53, 1.80}, {1.70, 1.36, 3.35}};
  const double start = 2.09;
  const double tile = read_out[nt - 1][mi] * (rows < mpad / 4 ? 0.25 : (double)rows / mpad);
  const double exchange = 1.04 + 3.70 * rows / 128 * nt;
  auto per_k_block = [&](long long workers) { return k_block[format][nt - 1][mi] * (1.0 + load[format] * (double)workers / (double)sms); };
  const char* e = getenv("MARLIN_B200_TC_SPLIT");    // tuning knob: 0 forces stripes, 1.. = that many k-ranges per tile
  const char* c = getenv("MARLIN_B200_TC_CLUSTER");  // tuning knob: largest cluster (0: none)
  const int forced = e ? atoi(e) : -1, max_cluster = c ? atoi(c) : 8;
  auto take = [&](long long workers, int split, int cluster, bool whole, double cost) {
    cost += start - (2 * workers <= sms ? (mi == 0 ? 0.63 : 0.45) : 0.0);
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
    static const double placing[9] = {0, 0, 0.13, 0.82, 0.56, 1.29, 1.13, 1.60, 1.40};
    // large clusters that fill all places of their size start later: 22 of six, 4096 x 2752 with deferred scales at 24 rows 7.1 us
    // (of four 6.8), groups of 64 rows, 4096 x 5632 at two rows 8.5 (8.0)
    const bool tight = cs >= 5 && 10 * (S * ncols / cs) > 9 * resident[cs];
    const double fix = S == 1    ? tile
                       : cs == 1 ? exchange * (1.43 + 0.227 * (double)S)
                                 : exchange + placing[cs] + (tight ? 0.45 : 0.0) + (S > cs ? 1.46 + exchange * 0.204 * (double)(S / cs) : 0.0);
    take(S * ncols, (int)S, cs, false, per_k_block(S * ncols) * (double)n + fix);
  }
  const long long workers = units < sms ? units : sms;
  if (forced <= 0 || !best.nt) {
    const double n = (double)units / (double)workers, tiles = n / kb;
    double contributors = (double)workers / (double)ncols + 1.0;
    if (contributors < 2.0) contributors = 2.0;
    double far = 0.0;
    if (slabs > 1 && nt == 1) {
      far = ((double)slabs * rows * kb * 256.0 - 40e6) / 40e6;
      far = far < 0.0 ? 0.0 : far > 1.0 ? 1.0 : far;
    }
    take(workers, 0, 0, false,
         per_k_block(workers) * 1.113 * (1.0 + 0.16 * far) * n + tile * (tiles > 1.0 ? tiles - 1.0 : 0.0) + exchange * (2.03 + 0.222 * contributors));
  }
  if (forced < 0 && ncols >= workers) {
    const double tiles = (double)((ncols + workers - 1) / workers);
    take(workers, 0, 0, true, per_k_block(workers) * tiles * kb + tile * tiles);
  }
  return best;
}

// M rows on a layer of N columns and kb k-blocks; deferred scales have tiles of 128 columns alone
inline TcPlan plan_tc(int format, int M, int kb, int N, int sm_count, int max_workers) {
  const int mpad = tc_mpad(M), slabs = (M + mpad - 1) / mpad;
  const int rows = slabs == 1 ? M : tc_slab_rows(format, M, 1);  // (several slabs: the same with both tile widths)
  const char* columns = getenv("MARLIN_B200_TC_TILE");  // tuning knob: 128 or 256 columns per tile, where there is a choice
  TcPlan best{};
  for (int nt = 1; nt <= 2; ++nt) {
    if (format == kTcDeferred4 ? nt != 1 : (columns && (atoi(columns) == 128) != (nt == 1))) continue;
    const TcPlan p = plan_tc_tile(nt, format, rows, slabs, kb, N, sm_count, max_workers);
    if (!best.nt || p.cost < best.cost) best = p;
  }
  return best;
}

}  // namespace marlin_b200
