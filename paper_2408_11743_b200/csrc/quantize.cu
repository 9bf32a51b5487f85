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
//     with one thread per (column, pair of candidates), so that the serial sum over the rows runs for all candidates at
//     once; then the codes, parallel over the rows.  (One thread per column, which re-read the group once per candidate,
//     left the chip idle on such layers: 4096 x 4096 with one scale per column took 7.96 ms; 100 us now.)
// Bound: the fp32 pipe.  Per weight and candidate there are five operations on it (product, two for the rounding, two
// for the error) and two comparisons beside it; rintf() would be a conversion instruction at an eighth of the rate, and
// was what bounded this file before.  The operations are issued on pairs (fma.rn.f32x2 and the like: the same
// IEEE operations, half the instructions).
#include "device_utils.cuh"
#include "marlin_internal.cuh"

namespace marlin_b200 {
namespace {

__device__ __forceinline__ float load_w(const uint16_t* p) { return __half2float(__ushort_as_half(__ldg(p))); }

__device__ __forceinline__ f32x2 clamp2(f32x2 x) {
  float lo, hi;
  unpack2(x, lo, hi);
  return pack2(fminf(fmaxf(lo, -8.f), 7.f), fminf(fmaxf(hi, -8.f), 7.f));
}

// Rounding half to even by adding 1.5 * 2^23: in [2^23, 2^24) the spacing of fp32 is one, so the sum rounds x to an
// integer q, which sits in the low bits of its representation.  Clamping to [-8, 7] first gives the same integer
// as clamping the rounded value (both ends are integers and rounding is monotone).
constexpr float kRoundMagic = 12582912.f;
__device__ __forceinline__ uint32_t code_of(float w, float inv) {
  const float x = fminf(fmaxf(__fmul_rn(w, inv), -8.f), 7.f);
  return (__float_as_uint(__fadd_rn(x, kRoundMagic)) + 8u) & 15u;  // q + 8, q = -8 .. 7
}

// candidate t: fp16 scale bits, the scale and its reciprocal
__device__ __forceinline__ uint16_t candidate_scale(float a, int t, int n_grid, float& s, float& inv) {
  const float two_fifteenths = __fdiv_rn(2.f, 15.f);
  const float r = __fsub_rn(1.f, __fdiv_rn((float)t, (float)n_grid));
  uint16_t sh = __half_as_ushort(__float2half_rn(__fmul_rn(__fmul_rn(a, r), two_fifteenths)));
  if (sh == 0) sh = 1;  // a scale that rounds to zero: the smallest positive fp16
  s = __half2float(__ushort_as_half(sh));
  inv = __fdiv_rn(1.f, s);
  return sh;
}

// Groups of 32, 64 or 128 rows: the rows of a group in registers, two per register pair.
// 4096 x 11008, groups of 128, ten candidates: 118 us (140 with rintf and without the pairs), both pipes about 60 % busy.
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
  const f32x2 magic = pack2(kRoundMagic, kRoundMagic), minus1 = pack2(-1.f, -1.f);
  float best_err = __int_as_float(0x7f800000);  // +inf
  uint16_t best_s = 1;
#pragma unroll 1
  for (int t = 0; t < n_candidates; ++t) {
    float s, inv;
    const uint16_t sh = candidate_scale(a, t, n_grid, s, inv);
    const f32x2 s2 = pack2(s, s), inv2 = pack2(inv, inv);
    float err = 0.f;
#pragma unroll
    for (int i = 0; i < GC / 2; ++i) {
      const f32x2 y = add2(clamp2(mul2(w[i], inv2)), magic);
      const f32x2 d = fma2(fma2(y, minus1, magic), s2, w[i]);  // w - q s: magic - y = -q exactly
      float d0, d1;
      unpack2(d, d0, d1);
      err = __fmaf_rn(d0, d0, err);  // in row order
      err = __fmaf_rn(d1, d1, err);
    }
    if (err < best_err) {
      best_err = err;
      best_s = sh;
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
    for (int j = 0; j < 4; ++j) {
      float lo, hi;
      unpack2(w[4 * i8 + j], lo, hi);
      word |= (code_of(lo, inv) << (8 * j)) | (code_of(hi, inv) << (8 * j + 4));
    }
    q_kpacked[((size_t)g * (GC / 8) + i8) * N + n] = word;
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

// The search: lane = column, warp = one candidate or (PAIRS) two of them in a register pair, rows in order.  The rows
// come through a ring of shared-memory tiles (64 rows x 32 columns, three tiles ahead): with few warps per scheduler
// nothing else hides the latency of the L2 (loading sixteen rows ahead into registers instead left the schedulers idle
// four cycles in five).
constexpr int kSearchCols = 32, kSearchMaxWarps = 16, kSearchRows = 64, kSearchTiles = 4;
template <bool PAIRS>
__global__ void __launch_bounds__(kSearchCols * kSearchMaxWarps)
quantize_search_kernel(const uint16_t* __restrict__ W, const uint32_t* __restrict__ q_kpacked, uint16_t* __restrict__ scales,
                       int N, int G, int n_grid, int n_candidates) {
  constexpr int PER = PAIRS ? 2 : 1;  // candidates of a warp
  __shared__ __align__(16) uint16_t ring[kSearchTiles][kSearchRows][kSearchCols];
  __shared__ float errs[PER * kSearchMaxWarps][kSearchCols];
  __shared__ uint16_t cands[PER * kSearchMaxWarps][kSearchCols];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int n = blockIdx.x * kSearchCols + lane;
  const int g = blockIdx.y;
  const uint16_t* w = W + (size_t)g * G * N + blockIdx.x * kSearchCols;
  const int tiles = G / kSearchRows;  // G is a multiple of 128
  auto fetch = [&](int tile) {
    if (tile < tiles) {
      for (int v = threadIdx.x; v < kSearchRows * 4; v += blockDim.x) {
        const int row = v >> 2, part = v & 3;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&ring[tile % kSearchTiles][row][8 * part]);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst),
                     "l"(w + ((size_t)tile * kSearchRows + row) * N + 8 * part)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");  // one group per call, empty ones too
  };
  uint32_t amax = 0;
  for (int part = 0; part < G / kPartRows; ++part)
    amax = max(amax, __ldg(q_kpacked + ((size_t)g * (G / kPartRows) + part) * (kPartRows / 8) * N + n));
  const float a = __half2float(__ushort_as_half((uint16_t)amax));
  const f32x2 magic = pack2(kRoundMagic, kRoundMagic), minus1 = pack2(-1.f, -1.f);
  float best_err = __int_as_float(0x7f800000);
  uint16_t best_s = 1;
  for (int t0 = 0; t0 < n_candidates; t0 += PER * warps) {
    // (slots past the last candidate repeat it)
    float s[PER], inv[PER], err[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      cands[PER * warp + e][lane] =
          candidate_scale(a, min(t0 + PER * warp + e, n_candidates - 1), n_grid, s[e], inv[e]);
      err[e] = 0.f;
    }
    const f32x2 s2 = pack2(s[0], s[PER - 1]), inv2 = pack2(inv[0], inv[PER - 1]);
    f32x2 err2 = pack2(0.f, 0.f);
    for (int i = 0; i < kSearchTiles - 1; ++i) fetch(i);
    for (int tile = 0; tile < tiles; ++tile) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kSearchTiles - 2) : "memory");
      __syncthreads();  // this tile has landed for everybody, and everybody has left the one before it
      fetch(tile + kSearchTiles - 1);
      const uint16_t* rows = &ring[tile % kSearchTiles][0][lane];
#pragma unroll 16
      for (int i = 0; i < kSearchRows; ++i) {
        const float wi = __half2float(__ushort_as_half(rows[i * kSearchCols]));
        if constexpr (PAIRS) {
          const f32x2 ww = pack2(wi, wi);
          const f32x2 y = add2(clamp2(mul2(ww, inv2)), magic);
          const f32x2 d = fma2(fma2(y, minus1, magic), s2, ww);
          err2 = fma2(d, d, err2);
        } else {
          const float x = fminf(fmaxf(__fmul_rn(wi, inv[0]), -8.f), 7.f);
          const float q = __fsub_rn(__fadd_rn(x, kRoundMagic), kRoundMagic);
          const float d = __fmaf_rn(-q, s[0], wi);
          err[0] = __fmaf_rn(d, d, err[0]);
        }
      }
    }
    if constexpr (PAIRS) unpack2(err2, err[0], err[PER - 1]);
#pragma unroll
    for (int e = 0; e < PER; ++e) errs[PER * warp + e][lane] = err[e];
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
  for (int j = 0; j < 8; ++j) {
    word.x |= code_of(__half2float(__ushort_as_half((uint16_t)(rows[j] & 0xffffu))), inv0) << (4 * j);
    word.y |= code_of(__half2float(__ushort_as_half((uint16_t)(rows[j] >> 16))), inv1) << (4 * j);
  }
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
    // Pairs of candidates need fewer instructions, single ones give twice the warps: with less than two warps of pairs
    // per scheduler the latter is faster (4096 x 4096, one scale per column, 640 warps of pairs: 80 us against 97 for the
    // search; 4096 x 11008, groups of 256, 27520 of them: 218 us against 184 for the whole conversion).
    const dim3 blocks((unsigned)(N / kSearchCols), (unsigned)(K / G));
    const int singles = n_candidates < kSearchMaxWarps ? n_candidates : kSearchMaxWarps;
    const int pairs_of = (n_candidates + 1) / 2 < kSearchMaxWarps ? (n_candidates + 1) / 2 : kSearchMaxWarps;
    if ((long long)blocks.x * blocks.y * pairs_of < 148 * 4 * 2)
      quantize_search_kernel<false><<<blocks, kSearchCols * singles, 0, stream>>>(W, q_kpacked, scales, N, G, n_grid, n_candidates);
    else
      quantize_search_kernel<true><<<blocks, kSearchCols * pairs_of, 0, stream>>>(W, q_kpacked, scales, N, G, n_grid, n_candidates);
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
