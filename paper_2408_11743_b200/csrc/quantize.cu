// Data-free quantiser in front of marlin_pack: fp16 weights -> 4-bit codes and fp16 group scales, round to nearest
// with a per-group search for the clipping threshold (Section 3.5 (a): group scales picked by searching for the
// best group-wise clipping thresholds; the grid is the symmetric one of Section 3.4, W ~ (q - 8) * s).
//
// Per group of G consecutive rows of one column:
//   a   = max |w|
//   r_t = 1 - t / n_grid,  t = 0 .. n_candidates - 1         (t = 0: no clipping)
//   s_t = fp16((a * r_t) * (2 / 15))                          (15 steps across [-a r, a r]; never zero)
//   q_i = clamp(round_half_even(w_i * (1 / s_t)), -8, 7) + 8
//   e_t = sum_i (w_i - (q_i - 8) s_t)^2, summed in the order i = 0 .. G - 1
// and the first candidate with the least e_t wins.  Codes and the winner are integers decided by fp32 arithmetic,
// so every operation is spelled out with its rounding (single IEEE operations, fused multiply-add where written):
// the same inputs give the same codes on every run and on any implementation that follows these lines.
//
// The order of the sums is fixed along the rows of a group, but nothing orders groups, columns or candidates: those are
// what runs in parallel.
//   - Groups of 32, 64 or 128 rows: one thread owns one (group, column) and holds its rows in registers, one read of W.
//   - Longer groups (up to one scale per column): three launches.  Column maxima in parts of 128 rows; then the search
//     with one thread per column and one or two candidates, so that the serial sum over the rows runs for all candidates at
//     once; then the codes, parallel over the rows.  (One thread per column, which re-read the group once per candidate,
//     left the chip idle on such layers: 4096 x 4096 with one scale per column took 7.96 ms.)
// Only |w_i - (q_i - 8) s_t| enters e_t, and that leaves the search a freedom: where w_i / s_t lies half way between two codes both
// give the same magnitude, s_t / 2, exactly (fp16 w and s: the difference is exact in fp32).  Where it does not, it is at least 2^-13
// away from half way (w = W 2^a, s = S 2^b with integers W, S < 2^11 and |w| >= s / 2: 2 w - (2 k + 1) s is a multiple of 2^(b-1), and is
// divided by 2 s < 2^(b+12)), so any arithmetic with less error finds the same code.  The search therefore clamps for free: with
//   u = sat(w / (15 s) + 8 / 15),   q = round(15 u)        (error below 2^-18 codes)
// the saturation of the first fma to [0, 1] is the clamp to [0, 15].  The codes themselves are made as written above.
// Bound: the fp32 pipe, five operations per weight and candidate (u, two for the rounding, two for the error), most of them issued in
// pairs (fma.rn.f32x2 and the like: the same IEEE operations, half the instructions); no conversions to integers, no comparisons.
// Measured with ten candidates, before (clamp by two comparisons) and now: 4096 x 11008, groups of 128: 114 / 99 us; one scale per column,
// 4096 x 4096: 99 / 85, 8192 x 1024: 163 / 134.
#include "device_utils.cuh"
#include "marlin_internal.cuh"

namespace marlin_b200 {
namespace {

__device__ __forceinline__ float load_w(const uint16_t* p) { return __half2float(__ushort_as_half(__ldg(p))); }

// Rounding half to even by adding 1.5 * 2^23: in [2^23, 2^24) the spacing of fp32 is one, so the sum rounds x to an
// integer q, which sits in the low bits of its representation.  Clamping to [-8, 7] first gives the same integer
// as clamping the rounded value (both ends are integers and rounding is monotone).
constexpr float kRoundMagic = 12582912.f;
// Here the integer comes with the bits of the magic number; of eight of them, put together by multiplications by 16, those are taken
// off at the end, and 8 is added to each.
__device__ __forceinline__ uint32_t code_bits(float w, float inv) {
  const float x = fminf(fmaxf(__fmul_rn(w, inv), -8.f), 7.f);
  return __float_as_uint(__fadd_rn(x, kRoundMagic));
}
constexpr uint32_t kMagicBits = 0x4b400000u, kEightMagicBits = (kMagicBits - 8u) * 0x11111111u;

// the search's u (see the top)
__device__ __forceinline__ float unit_of(float w, float inv15) {
  float u;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(u) : "f"(w), "f"(inv15), "f"(8.f / 15.f));
  return u;
}

// candidate t: fp16 scale bits, the scale and a fifteenth of its reciprocal
__device__ __forceinline__ uint16_t candidate_scale(float a, int t, int n_grid, float& s, float& inv15) {
  const float two_fifteenths = __fdiv_rn(2.f, 15.f);
  const float r = __fsub_rn(1.f, __fdiv_rn((float)t, (float)n_grid));
  uint16_t sh = __half_as_ushort(__float2half_rn(__fmul_rn(__fmul_rn(a, r), two_fifteenths)));
  if (sh == 0) sh = 1;  // a scale that rounds to zero: the smallest positive fp16
  s = __half2float(__ushort_as_half(sh));
  inv15 = __fmul_rn(__fdiv_rn(1.f, s), 1.f / 15.f);
  return sh;
}

// Groups of 32, 64 or 128 rows: the rows of a group in registers, two per register pair.
template <int GC>
__global__ void __launch_bounds__(128)
quantize_rtn_cached_kernel(const uint16_t* __restrict__ W, uint32_t* __restrict__ q_kpacked, uint16_t* __restrict__ scales,
                           int K, int N, int n_grid, int n_candidates) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const int g = blockIdx.y;
  if (n >= N) return;
  const uint16_t* wp = W + (size_t)g * GC * N + n;
  f32x2 w[GC / 2];
  float a = 0.f;
#pragma unroll
  for (int i = 0; i < GC / 2; ++i) {
    const float lo = load_w(wp + (size_t)(2 * i) * N), hi = load_w(wp + (size_t)(2 * i + 1) * N);
    w[i] = pack2(lo, hi);
    a = fmaxf(a, fmaxf(fabsf(lo), fabsf(hi)));
  }
  const f32x2 magic = pack2(kRoundMagic, kRoundMagic), minus_magic8 = pack2(-kRoundMagic - 8.f, -kRoundMagic - 8.f);
  const f32x2 fifteen = pack2(15.f, 15.f);
  float best_err = __int_as_float(0x7f800000);  // +inf
  uint16_t best_s = 1;
  if (n_candidates & 1) {
    float s, inv15, err = 0.f;
    const uint16_t sh = candidate_scale(a, 0, n_grid, s, inv15);
#pragma unroll
    for (int i = 0; i < GC; ++i) {
      float lo, hi;
      unpack2(w[i / 2], lo, hi);
      const float x = i % 2 ? hi : lo;
      const float q = __fsub_rn(__fmaf_rn(unit_of(x, inv15), 15.f, kRoundMagic), kRoundMagic + 8.f);
      const float d = __fmaf_rn(-q, s, x);
      err = __fmaf_rn(d, d, err);
    }
    if (err < best_err) {
      best_err = err;
      best_s = sh;
    }
  }
  // two candidates at a time, in the halves of a register pair
#pragma unroll 1
  for (int t = n_candidates & 1; t < n_candidates; t += 2) {
    float s[2], inv15[2], e[2];
    uint16_t sh[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) sh[c] = candidate_scale(a, t + c, n_grid, s[c], inv15[c]);
    f32x2 err = pack2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < GC; ++i) {  // in row order
      float lo, hi, q[2];
      unpack2(w[i / 2], lo, hi);
      const float x = i % 2 ? hi : lo;
      const f32x2 y = fma2(pack2(unit_of(x, inv15[0]), unit_of(x, inv15[1])), fifteen, magic);  // magic + q + 8
      unpack2(add2(y, minus_magic8), q[0], q[1]);
      const f32x2 d = pack2(__fmaf_rn(-q[0], s[0], x), __fmaf_rn(-q[1], s[1], x));
      err = fma2(d, d, err);
    }
    unpack2(err, e[0], e[1]);
#pragma unroll
    for (int c = 0; c < 2; ++c)
      if (e[c] < best_err) {
        best_err = e[c];
        best_s = sh[c];
      }
  }
  const float s = __half2float(__ushort_as_half(best_s));
  const float inv = __fdiv_rn(1.f, s);
  scales[(size_t)g * N + n] = best_s;
  // canonical code words: nibble j of word (k / 8, n) = code of row 8 * (k / 8) + j
#pragma unroll
  for (int i8 = 0; i8 < GC / 8; ++i8) {
    uint32_t word = 0;
#pragma unroll
    for (int j = 3; j >= 0; --j) {
      float lo, hi;
      unpack2(w[4 * i8 + j], lo, hi);
      word = 16u * word + code_bits(hi, inv);
      word = 16u * word + code_bits(lo, inv);
    }
    q_kpacked[((size_t)g * (GC / 8) + i8) * N + n] = word - kEightMagicBits;
  }
}

// ---- groups longer than 128 rows ---------------------------------------------------------------------------------
constexpr int kPartRows = 128;  // rows of one part of a column maximum

// Largest magnitudes of 128 rows of every column, as fp16 bits (a magnitude of an fp16 value is one).  They are left in the
// first code row of those rows (16 rows of words per part), which quantize_encode_kernel overwrites at the end.
__global__ void __launch_bounds__(128)
quantize_max_kernel(const uint16_t* __restrict__ W, uint32_t* __restrict__ q_kpacked, int N) {
  const int n2 = blockIdx.x * blockDim.x + threadIdx.x;  // pair of columns
  const int part = blockIdx.y;
  if (2 * n2 >= N) return;
  const uint32_t* w = reinterpret_cast<const uint32_t*>(W + (size_t)part * kPartRows * N) + n2;
  // magnitudes of fp16 values order like their bits without the sign
  uint32_t m = 0;
#pragma unroll 32
  for (int i = 0; i < kPartRows; ++i) m = __vmaxu2(m, __ldg(w + (size_t)i * (N / 2)) & 0x7fff7fffu);
  reinterpret_cast<uint2*>(q_kpacked + (size_t)part * (kPartRows / 8) * N)[n2] = make_uint2(m & 0xffffu, m >> 16);
}

// The search: lane = column, rows in order, a warp one candidate or a pair of them.  The rows come through a ring of shared-memory tiles
// (64 rows x 32 columns, three tiles ahead): with few warps per scheduler nothing else hides the latency of the L2.
constexpr int kSearchCols = 32, kSearchMinWarps = 8, kSearchMaxWarps = 16, kSearchRows = 64, kSearchTiles = 4;
typedef uint16_t SearchRing[kSearchTiles][kSearchRows][kSearchCols];
// asks for tile `tile` of the columns from w on, if it is one; one group of copies per call, empty ones too
__device__ __forceinline__ void fetch_tile(SearchRing& ring, const uint16_t* w, int N, int tile, int tiles) {
  if (tile < tiles) {
    for (int v = threadIdx.x; v < kSearchRows * 4; v += blockDim.x) {
      const int row = v >> 2, part = v & 3;
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&ring[tile % kSearchTiles][row][8 * part]);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(w + ((size_t)tile * kSearchRows + row) * N + 8 * part)
                   : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// the largest weight of a group, from the maxima of its parts
__device__ __forceinline__ float group_max(const uint32_t* q_kpacked, int N, int G, int g, int n) {
  uint32_t amax = 0;
  for (int part = 0; part < G / kPartRows; ++part)
    amax = max(amax, __ldg(q_kpacked + ((size_t)g * (G / kPartRows) + part) * (kPartRows / 8) * N + n));
  return __half2float(__ushort_as_half((uint16_t)amax));
}

// Warp = PER candidates (in the halves of a register pair), rows straight out of the ring.
template <int PER>
__global__ void __launch_bounds__(kSearchCols * kSearchMaxWarps)
quantize_search_direct_kernel(const uint16_t* __restrict__ W, const uint32_t* __restrict__ q_kpacked, uint16_t* __restrict__ scales,
                              int N, int G, int n_grid, int n_candidates) {
  __shared__ __align__(16) SearchRing ring;
  __shared__ float errs[PER * kSearchMaxWarps][kSearchCols];
  __shared__ uint16_t cands[PER * kSearchMaxWarps][kSearchCols];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int n = blockIdx.x * kSearchCols + lane;
  const int g = blockIdx.y;
  const uint16_t* w = W + (size_t)g * G * N + blockIdx.x * kSearchCols;
  const int tiles = G / kSearchRows;  // G is a multiple of 128
  const float a = group_max(q_kpacked, N, G, g, n);
  const f32x2 magic = pack2(kRoundMagic, kRoundMagic), minus_magic8 = pack2(-kRoundMagic - 8.f, -kRoundMagic - 8.f);
  const f32x2 fifteen = pack2(15.f, 15.f);
  float best_err = __int_as_float(0x7f800000);
  uint16_t best_s = 1;
  for (int t0 = 0; t0 < n_candidates; t0 += PER * warps) {
    // (slots past the last candidate repeat it)
    float s[PER], inv15[PER], err[PER];
#pragma unroll
    for (int c = 0; c < PER; ++c) {
      cands[PER * warp + c][lane] = candidate_scale(a, min(t0 + PER * warp + c, n_candidates - 1), n_grid, s[c], inv15[c]);
      err[c] = 0.f;
    }
    f32x2 err2 = pack2(0.f, 0.f);
    for (int i = 0; i < kSearchTiles - 1; ++i) fetch_tile(ring, w, N, i, tiles);
    for (int tile = 0; tile < tiles; ++tile) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kSearchTiles - 2) : "memory");
      __syncthreads();  // this tile has landed for everybody, and everybody has left the one before it
      fetch_tile(ring, w, N, tile + kSearchTiles - 1, tiles);
      const uint16_t* rows = &ring[tile % kSearchTiles][0][lane];
#pragma unroll 16
      for (int i = 0; i < kSearchRows; ++i) {
        const float x = __half2float(__ushort_as_half(rows[i * kSearchCols]));
        if constexpr (PER == 2) {
          float q[2];
          const f32x2 y = fma2(pack2(unit_of(x, inv15[0]), unit_of(x, inv15[1])), fifteen, magic);  // magic + q + 8
          unpack2(add2(y, minus_magic8), q[0], q[1]);
          const f32x2 d = pack2(__fmaf_rn(-q[0], s[0], x), __fmaf_rn(-q[1], s[1], x));
          err2 = fma2(d, d, err2);
        } else {
          const float q = __fsub_rn(__fmaf_rn(unit_of(x, inv15[0]), 15.f, kRoundMagic), kRoundMagic + 8.f);
          const float d = __fmaf_rn(-q, s[0], x);
          err[0] = __fmaf_rn(d, d, err[0]);
        }
      }
    }
    if constexpr (PER == 2) unpack2(err2, err[0], err[1]);
#pragma unroll
    for (int c = 0; c < PER; ++c) errs[PER * warp + c][lane] = err[c];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
      // in candidate order, the first one on ties
      for (int c = 0; c < PER * warps && t0 + c < n_candidates; ++c)
        if (errs[c][lane] < best_err) {
          best_err = errs[c][lane];
          best_s = cands[c][lane];
        }
    }
    __syncthreads();
  }
  if (warp == 0) scales[(size_t)g * N + n] = best_s;
}

// Warp = one candidate; a tile is turned into fp32 pairs of rows once for all candidates, one tile ahead of the sums.  IDLE: warps without
// a candidate fetch and widen only (else they repeat the last one: a branch around the sums takes 6 % longer).
template <bool IDLE>
__global__ void __launch_bounds__(kSearchCols * kSearchMaxWarps)
quantize_search_kernel(const uint16_t* __restrict__ W, const uint32_t* __restrict__ q_kpacked, uint16_t* __restrict__ scales,
                       int N, int G, int n_grid, int n_candidates) {
  __shared__ __align__(16) SearchRing ring;
  __shared__ f32x2 pairs[2][kSearchRows / 2][kSearchCols];
  __shared__ float errs[kSearchMaxWarps][kSearchCols];
  __shared__ uint16_t cands[kSearchMaxWarps][kSearchCols];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int n = blockIdx.x * kSearchCols + lane;
  const int g = blockIdx.y;
  const uint16_t* w = W + (size_t)g * G * N + blockIdx.x * kSearchCols;
  const int tiles = G / kSearchRows;  // G is a multiple of 128
  auto fetch = [&](int tile) { fetch_tile(ring, w, N, tile, tiles); };
  // rows of a tile from 16 to 32 bits, in two steps: loads into registers, and later their way into `pairs`
  constexpr int kWiden = kSearchRows / 2 / kSearchMinWarps;
  uint16_t wide[kWiden][2];
  auto widen_load = [&](int tile) {
#pragma unroll
    for (int i = 0; i < kWiden; ++i) {
      const int r2 = warp + i * warps;
      if (r2 < kSearchRows / 2) {
        wide[i][0] = ring[tile % kSearchTiles][2 * r2][lane];
        wide[i][1] = ring[tile % kSearchTiles][2 * r2 + 1][lane];
      }
    }
  };
  auto widen_store = [&](int tile) {
#pragma unroll
    for (int i = 0; i < kWiden; ++i) {
      const int r2 = warp + i * warps;
      if (r2 < kSearchRows / 2)
        pairs[tile & 1][r2][lane] = pack2(__half2float(__ushort_as_half(wide[i][0])), __half2float(__ushort_as_half(wide[i][1])));
    }
  };
  const float a = group_max(q_kpacked, N, G, g, n);
  const f32x2 magic = pack2(kRoundMagic, kRoundMagic), magic8 = pack2(kRoundMagic + 8.f, kRoundMagic + 8.f);
  const f32x2 minus1 = pack2(-1.f, -1.f), fifteen = pack2(15.f, 15.f);
  float best_err = __int_as_float(0x7f800000);
  uint16_t best_s = 1;
  for (int t0 = 0; t0 < n_candidates; t0 += warps) {
    const bool mine = !IDLE || t0 + warp < n_candidates;
    constexpr int B = 4;
    float s, inv15, err = 0.f, d[2 * B];
#pragma unroll
    for (int i = 0; i < 2 * B; ++i) d[i] = 0.f;
    cands[warp][lane] = candidate_scale(a, min(t0 + warp, n_candidates - 1), n_grid, s, inv15);
    const f32x2 s2 = pack2(s, s);
    for (int i = 0; i < kSearchTiles - 1; ++i) fetch(i);
    asm volatile("cp.async.wait_group %0;" ::"n"(kSearchTiles - 2) : "memory");
    __syncthreads();
    widen_load(0);
    widen_store(0);
    for (int tile = 0; tile < tiles; ++tile) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kSearchTiles - 3) : "memory");
      // this tile's pairs are there, the next tile has landed for everybody, and everybody has left the pairs of the tile before
      __syncthreads();
      if (tile + 1 < tiles) widen_load(tile + 1);
      fetch(tile + kSearchTiles - 1);
      const f32x2* rows = &pairs[tile & 1][0][lane];
      // Four pairs at a time, each operation for all of them, the next four already on their way and the squares of the four
      // before (a chain, in row order) in between: with two or three warps per scheduler one after the other would wait for itself
      // (two, four, eight at a time: 91, 85, 85 us for 4096 x 4096 with one scale per column; 167, 157, 169 for 4096 x 11008 in groups of 256).
      if (mine) {
        f32x2 next[B];
#pragma unroll
        for (int i = 0; i < B; ++i) next[i] = rows[i * kSearchCols];
#pragma unroll
        for (int i0 = 0; i0 < kSearchRows / 2; i0 += B) {
          f32x2 ww[B], y[B];
          float u[2 * B];
#pragma unroll
          for (int i = 0; i < B; ++i) {
            ww[i] = next[i];
            if (i0 + B < kSearchRows / 2) next[i] = rows[(i0 + B + i) * kSearchCols];
          }
#pragma unroll
          for (int i = 0; i < B; ++i) {
            float lo, hi;
            unpack2(ww[i], lo, hi);
            u[2 * i] = unit_of(lo, inv15);
            u[2 * i + 1] = unit_of(hi, inv15);
            err = __fmaf_rn(d[i], d[i], err);
          }
#pragma unroll
          for (int i = 0; i < B; ++i) {
            y[i] = fma2(pack2(u[2 * i], u[2 * i + 1]), fifteen, magic);  // magic + q + 8
            err = __fmaf_rn(d[B + i], d[B + i], err);
          }
#pragma unroll
          for (int i = 0; i < B; ++i) y[i] = fma2(y[i], minus1, magic8);  // -q, exactly
#pragma unroll
          for (int i = 0; i < B; ++i) unpack2(fma2(y[i], s2, ww[i]), d[2 * i], d[2 * i + 1]);
        }
      }
      if (tile + 1 < tiles) widen_store(tile + 1);
    }
#pragma unroll
    for (int i = 0; i < 2 * B; ++i) err = __fmaf_rn(d[i], d[i], err);
    errs[warp][lane] = err;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
      // in candidate order, the first one on ties
      for (int c = 0; c < warps && t0 + c < n_candidates; ++c)
        if (errs[c][lane] < best_err) {
          best_err = errs[c][lane];
          best_s = cands[c][lane];
        }
    }
    __syncthreads();
  }
  if (warp == 0) scales[(size_t)g * N + n] = best_s;
}

// Codes with the chosen scales: a thread owns two columns of eight rows.
__global__ void __launch_bounds__(128)
quantize_encode_kernel(const uint16_t* __restrict__ W, uint32_t* __restrict__ q_kpacked, const uint16_t* __restrict__ scales,
                       int N, int G, int first_row) {
  const int n2 = blockIdx.x * blockDim.x + threadIdx.x;
  const int k8 = first_row + blockIdx.y;
  if (2 * n2 >= N) return;
  const uint32_t* w = reinterpret_cast<const uint32_t*>(W + (size_t)k8 * 8 * N) + n2;
  uint32_t rows[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) rows[j] = __ldg(w + (size_t)j * (N / 2));
  const uint32_t sh = __ldg(reinterpret_cast<const uint32_t*>(scales + (size_t)(8 * k8 / G) * N) + n2);
  const float inv0 = __fdiv_rn(1.f, __half2float(__ushort_as_half((uint16_t)(sh & 0xffffu))));
  const float inv1 = __fdiv_rn(1.f, __half2float(__ushort_as_half((uint16_t)(sh >> 16))));
  uint2 word = make_uint2(0, 0);
#pragma unroll
  for (int j = 7; j >= 0; --j) {
    word.x = 16u * word.x + code_bits(__half2float(__ushort_as_half((uint16_t)(rows[j] & 0xffffu))), inv0);
    word.y = 16u * word.y + code_bits(__half2float(__ushort_as_half((uint16_t)(rows[j] >> 16))), inv1);
  }
  word.x -= kEightMagicBits;
  word.y -= kEightMagicBits;
  reinterpret_cast<uint2*>(q_kpacked + (size_t)k8 * N)[n2] = word;
}

}  // namespace

cudaError_t launch_quantize_rtn(const uint16_t* W, uint32_t* q_kpacked, uint16_t* scales, int K, int N, int G, int n_grid,
                                int n_candidates, cudaStream_t stream) {
  const int threads = N % 128 == 0 ? 128 : 64;
  dim3 grid((unsigned)(N / threads), (unsigned)(K / G));
  if (G == 128) {
    quantize_rtn_cached_kernel<128><<<grid, threads, 0, stream>>>(W, q_kpacked, scales, K, N, n_grid, n_candidates);
  } else if (G == 64) {
    quantize_rtn_cached_kernel<64><<<grid, threads, 0, stream>>>(W, q_kpacked, scales, K, N, n_grid, n_candidates);
  } else if (G == 32) {
    quantize_rtn_cached_kernel<32><<<grid, threads, 0, stream>>>(W, q_kpacked, scales, K, N, n_grid, n_candidates);
  } else {
    const unsigned pairs = (unsigned)((N / 2 + 127) / 128);
    quantize_max_kernel<<<dim3(pairs, (unsigned)(K / kPartRows)), 128, 0, stream>>>(W, q_kpacked, N);
    const dim3 blocks((unsigned)(N / kSearchCols), (unsigned)(K / G));
    // Pairs of candidates straight out of the ring take fewer instructions; single ones on widened rows spread over more warps and
    // shorten the chains, as long as one round of warps takes them and few blocks share an SM.  Of 9 to 12 candidates the fullest of the
    // four schedulers has four in pairs and three of single ones, of 13 to 16 four either way.  Measured, pairs / single, us: 4096 x 4096 with
    // one scale per column (128 blocks) 8, 10, 16, 17 candidates 88.6 / 70.2, 102.9 / 84.5, 102.9 / 100.9, 127 / 141; 8192 x 1024 in groups of 1024
    // (256) 50.3 / 45.5, 53.8 / 55.8 (10, 16); 4096 x 2048 in groups of 256 (1024) 35.3 / 35.3, 41.3 / 39.4, 49.6 / 51.7 (8, 10, 16); 4096 x 4096
    // in groups of 256 (2048) 64.0 / 66.0 (10); 4096 x 11008 (5504) 80.6 / 134, 92.9 / 134, 150 / 156, 246 / 263 (1, 4, 10, 20).
    const long long all = (long long)blocks.x * blocks.y;
    const bool single = n_candidates <= kSearchMaxWarps && (all < 2 * 148 || (all < 2048 && n_candidates > 8 && n_candidates <= 12));
    if (single && n_candidates > 4) {
      const int warps = n_candidates < kSearchMinWarps ? kSearchMinWarps : n_candidates;
      quantize_search_kernel<false><<<blocks, kSearchCols * warps, 0, stream>>>(W, q_kpacked, scales, N, G, n_grid, n_candidates);
    } else if (single) {
      // (up to four candidates: eight warps of which some have none, 64 us on 128 blocks and 30 to 33 on 256; all eight adding 70 and 39)
      quantize_search_kernel<true><<<blocks, kSearchCols * kSearchMinWarps, 0, stream>>>(W, q_kpacked, scales, N, G, n_grid, n_candidates);
    } else if (n_candidates == 1) {
      quantize_search_direct_kernel<1><<<blocks, kSearchCols, 0, stream>>>(W, q_kpacked, scales, N, G, n_grid, n_candidates);
    } else {
      // rounds of equal size
      const int pairs_all = (n_candidates + 1) / 2, rounds = (pairs_all + kSearchMaxWarps - 1) / kSearchMaxWarps;
      quantize_search_direct_kernel<2><<<blocks, kSearchCols * ((pairs_all + rounds - 1) / rounds), 0, stream>>>(W, q_kpacked, scales, N, G,
                                                                                                               n_grid, n_candidates);
    }
    // one grid row per eight rows of W: up to 2^20 / 8, above the limit of grid.y, so the rows go on in slices of it
    constexpr int kSlice = 32768;
    for (int r0 = 0; r0 < K / 8; r0 += kSlice) {
      const int rows = K / 8 - r0 < kSlice ? K / 8 - r0 : kSlice;
      quantize_encode_kernel<<<dim3(pairs, (unsigned)rows), 128, 0, stream>>>(W, q_kpacked, scales, N, G, r0);
    }
  }
  return cudaGetLastError();
}

}  // namespace marlin_b200
