// Offline re-layout of the dense W4A16 weights and scales (and its inverse).
//
// The paper reshuffles the static weight matrix once so that every thread's 16-byte load holds
// exactly the codes of its tensor-core fragments and so that a tile is one contiguous run of memory
// (Section 3.4, "Maximizing Loading Bandwidth" and "Dequantization and Tensor Cores").  The order
// used here is this library's own:
//
//   One 4096-byte chunk holds the codes of 128 rows (k-block kb = k / 128) x 64 columns (nb = n / 64).
//   Chunks are ordered by "super-columns" of four chunks (256 columns): inside super-column sc = nb / 4
//   the k-blocks follow one another, each with its cs chunks side by side (cs = 4, or the 1..3 chunks
//   left over in the last super-column when N is not a multiple of 256):
//     chunk index = sc * 4 * (K/128) + kb * cs + (nb % 4)
//   so the weights a CTA streams for a 256-column tile are one contiguous run of memory, k-block after
//   k-block, and one k-block of a tile is a single 16 KB bulk copy.
//   Inside a chunk, 16-byte vector number v = (2*j + b) * 32 + 4*g + slot holds 32 codes of ONE column:
//     column n = 64*nb + 16*j + 8*b + g        (g = 0..7; slot = (c + g/2) % 4, c = 0..3)
//     rows   k = 128*kb + {16*c .. 16*c + 15} and 128*kb + 64 + {16*c .. 16*c + 15}
//   (the four vectors of a column are rotated by g/2 so that the threads of the tcgen05 kernel, one column each
//   and 64 bytes apart, hit different banks when they all read their vector of the same c)
//   word w of the vector (w = 2*h + u) holds rows 128*kb + 64*h + 16*c + 8*u + o, o = 0..7, with
//   row offset o in nibble (o >> 1) + 4*(o & 1): one AND+OR pulls out the two codes of rows (2i, 2i+1).
//   Two readers use this order:
//     - the warp-level MMA kernel: lane (g, c) reads the vectors (slot as above) of columns g and g + 8 of a 16-column
//       block; one word of each gives the A-operand registers of two m16n8k16 steps (weights on the
//       16-wide side), and the lane's activations for its rows are 16 contiguous fp16 per 64-row half;
//     - the tcgen05 kernel: a thread owns one column and reads its four vectors (c = 0..3), i.e. all
//       128 rows of the k-block, dequantises and stores them to tensor memory in row order.
//   scales: inside every run of 64 columns, position 8*g + 2*j + b holds column 16*j + 8*b + g,
//   so that the 8 scales a thread needs are one 16-byte load.  Groups of 128 rows and more keep the row order
//   [K/G][N].  Groups of 64 or 32 rows (N a multiple of 256) are stored per k-block and 256-column tile,
//   [K/128][N/256][128/G][256], so that the two or four rows a k-block needs are one contiguous copy.
#include "marlin_internal.cuh"

namespace marlin_b200 {
namespace {

// chunk index <-> (kb, nb)
__device__ __forceinline__ long long chunk_index(int kb, int nb, int KB, int nb64) {
  int sc = nb >> 2;
  int cs = min(4, nb64 - 4 * sc);
  return (long long)sc * 4 * KB + (long long)kb * cs + (nb & 3);
}
__device__ __forceinline__ void chunk_coords(long long chunk, int KB, int nb64, int* kb, int* nb) {
  long long full = (long long)(nb64 >> 2) * 4 * KB;  // chunks in complete super-columns
  if (chunk < full) {
    int sc = (int)(chunk / (4 * KB));
    int rem = (int)(chunk % (4 * KB));
    *kb = rem >> 2;
    *nb = 4 * sc + (rem & 3);
  } else {
    int cs = nb64 & 3;
    int rem = (int)(chunk - full);
    *kb = rem / cs;
    *nb = 4 * (nb64 >> 2) + rem % cs;
  }
}

// The nibbles of a canonical word (row offset o in nibble o) in the packed order (nibble (o >> 1) + 4 * (o & 1)), and back.
__device__ __forceinline__ uint32_t even_nibbles(uint32_t w) {  // nibbles 0, 2, 4, 6 side by side in the low half
  w &= 0x0f0f0f0fu;
  w = (w | (w >> 4)) & 0x00ff00ffu;
  return (w | (w >> 8)) & 0xffffu;
}
__device__ __forceinline__ uint32_t spread_nibbles(uint32_t h) {  // its inverse
  h = (h | (h << 8)) & 0x00ff00ffu;
  return (h | (h << 4)) & 0x0f0f0f0fu;
}
__device__ __forceinline__ uint32_t to_packed_word(uint32_t w) { return even_nibbles(w) | (even_nibbles(w >> 4) << 16); }
__device__ __forceinline__ uint32_t to_canonical_word(uint32_t w) {
  return spread_nibbles(w & 0xffffu) | (spread_nibbles(w >> 16) << 4);
}

// scale at packed position x -> its canonical position
__device__ __forceinline__ long long canonical_scale(long long x, int N, int sub) {
  const int pos = (int)(x & 63);  // packed position inside the run of 64
  const int g = pos >> 3, j = (pos >> 1) & 3, b = pos & 1;
  const int c64 = 16 * j + 8 * b + g;  // column inside the run
  if (sub == 1) return (x & ~63LL) + c64;
  // packed [kb][tile][r][256]  <->  canonical row kb * sub + r, column 256 * tile + ...
  const long long rec = x >> 8;  // (kb * NT + tile) * sub + r
  const int r = (int)(rec % sub);
  const long long kt = rec / sub;
  const int NT = N / 256;
  const long long kb = kt / NT, tile = kt % NT;
  return (kb * sub + r) * (long long)N + tile * 256 + (x & 192) + c64;
}
__device__ __forceinline__ void permute_scales(const uint16_t* __restrict__ in, uint16_t* __restrict__ out, long long total,
                                               int N, int sub, bool inverse, int block, int blocks) {
  for (long long x = block * (long long)blockDim.x + threadIdx.x; x < total; x += (long long)blocks * blockDim.x) {
    const long long canon = canonical_scale(x, N, sub);
    if (inverse)
      out[canon] = in[x];
    else
      out[x] = in[canon];
  }
}

// Codes and scales of a dense layer in one launch: the first `code_blocks` blocks take the chunks, the others the scales.
// A chunk is 16 canonical word rows x 64 columns, and every packed word is one canonical word with its nibbles permuted:
// the block moves the chunk through shared memory so that both sides are read and written 16 bytes a thread in whole
// lines.  Bound: DRAM, both buffers once.  (One thread per packed word that gathered its canonical word took 25 us on
// 4096 x 11008, the scales another launch of 4 us; both together take 13 us now.)
constexpr int kPackThreads = 256;
__global__ void __launch_bounds__(kPackThreads)
repack_dense_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, const uint16_t* __restrict__ s_src,
                    uint16_t* __restrict__ s_dst, int K, int N, long long scales, int sub, int code_blocks, bool inverse) {
  if ((int)blockIdx.x >= code_blocks) {
    permute_scales(s_src, s_dst, scales, N, sub, inverse, blockIdx.x - code_blocks, gridDim.x - code_blocks);
    return;
  }
  // rows padded by four words: the 32 words a warp takes by vectors (four rows, eight columns) lie in different banks
  __shared__ __align__(16) uint32_t tile[16][kChunkN + 4];
  const int t = threadIdx.x;
  const int KB = K / kTileK, nb64 = N / kChunkN;
  const int row = t >> 4, c4 = t & 15;  // by rows: four columns of a word row
  // by vectors: vector t of the chunk holds rows 16c .. and 64 + 16c .. of column 8i + g, slot = (c + g / 2) % 4
  const int i = t >> 5, g = (t & 31) >> 2, c = ((t & 3) - (g >> 1)) & 3;
  const int col = 8 * i + g;
  for (long long chunk = blockIdx.x; chunk < (long long)KB * nb64; chunk += code_blocks) {
    int kb, nb;
    chunk_coords(chunk, KB, nb64, &kb, &nb);
    const size_t canon = (((size_t)kb * 16 + row) * N + (size_t)nb * kChunkN) / 4 + c4;
    const size_t packed = (size_t)chunk * kPackThreads + t;
    if (!inverse) {
      *reinterpret_cast<uint4*>(&tile[row][4 * c4]) = src[canon];
      __syncthreads();
      uint4 v;
      v.x = to_packed_word(tile[2 * c][col]);
      v.y = to_packed_word(tile[2 * c + 1][col]);
      v.z = to_packed_word(tile[8 + 2 * c][col]);
      v.w = to_packed_word(tile[8 + 2 * c + 1][col]);
      dst[packed] = v;
    } else {
      const uint4 v = src[packed];
      tile[2 * c][col] = to_canonical_word(v.x);
      tile[2 * c + 1][col] = to_canonical_word(v.y);
      tile[8 + 2 * c][col] = to_canonical_word(v.z);
      tile[8 + 2 * c + 1][col] = to_canonical_word(v.w);
      __syncthreads();
      dst[canon] = *reinterpret_cast<const uint4*>(&tile[row][4 * c4]);
    }
    __syncthreads();
  }
}

__global__ void permute_scales_kernel(const uint16_t* __restrict__ in, uint16_t* __restrict__ out, long long total,
                                      int N, int sub, bool inverse) {
  permute_scales(in, out, total, N, sub, inverse, blockIdx.x, gridDim.x);
}

// zero points: the same permutation, uint8 codes on the canonical side and fp16 values on the packed side
__global__ void permute_zeros_kernel(uint8_t* __restrict__ z, uint16_t* __restrict__ zq, long long total, int N, int sub,
                                     bool inverse) {
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total;
       x += (long long)gridDim.x * blockDim.x) {
    const long long canon = canonical_scale(x, N, sub);
    if (inverse)
      z[canon] = (uint8_t)__half2float(__ushort_as_half(zq[x]));
    else
      zq[x] = __half_as_ushort(__float2half_rn((float)z[canon]));
  }
}

// out[row][n], n = 16 b + r: r < 8 -> gate[row][8 b + r], else up[row][8 b + r - 8]
template <typename T>
__global__ void interleave_gate_up_kernel(const T* __restrict__ gate, const T* __restrict__ up, T* __restrict__ out,
                                          long long rows, int I) {
  const long long total = rows * 2 * I;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total; x += (long long)gridDim.x * blockDim.x) {
    const long long row = x / (2 * I);
    const int n = (int)(x % (2 * I));
    const int b = n >> 4, r = n & 15;
    out[x] = r < 8 ? gate[row * I + 8 * b + r] : up[row * I + 8 * b + r - 8];
  }
}

// 8-bit codes: one thread per 16-byte vector of the packed buffer = rows 128 kb + 16 c + 0..15 of column 256 T + n
__global__ void pack_w8_kernel(uint8_t* __restrict__ q8, uint8_t* __restrict__ wq, int K, int N, bool inverse) {
  const long long vecs = (long long)K * N / 16;
  const int KB = K / 128;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < vecs; v += (long long)gridDim.x * blockDim.x) {
    const int n = (int)(v & 255);
    const int c = (int)((v >> 8) & 7);
    const long long rec = v >> 11;  // T * KB + kb
    const int kb = (int)(rec % KB);
    const long long T = rec / KB;
    uint8_t* canon = q8 + ((size_t)kb * 128 + 16 * c) * N + T * 256 + n;
    uint8_t* packed = wq + v * 16;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      if (inverse)
        canon[(size_t)j * N] = packed[j];
      else
        packed[j] = canon[(size_t)j * N];
    }
  }
}

}  // namespace

cudaError_t launch_pack_w8(uint8_t* q8, uint8_t* wq, int K, int N, bool inverse, cudaStream_t stream) {
  const long long vecs = (long long)K * N / 16;
  const int threads = 256;
  int blocks = (int)((vecs + threads - 1) / threads);
  if (blocks > 148 * 16) blocks = 148 * 16;
  pack_w8_kernel<<<blocks, threads, 0, stream>>>(q8, wq, K, N, inverse);
  return cudaGetLastError();
}

cudaError_t launch_interleave_gate_up(const uint32_t* q_gate, const uint16_t* s_gate, const uint32_t* q_up, const uint16_t* s_up,
                                      uint32_t* q_out, uint16_t* s_out, int K, int I, int G, cudaStream_t stream) {
  const int threads = 256;
  const long long qrows = K / 8, srows = K / G;
  int blocks = (int)((qrows * 2 * I + threads - 1) / threads);
  if (blocks > 148 * 16) blocks = 148 * 16;
  interleave_gate_up_kernel<uint32_t><<<blocks, threads, 0, stream>>>(q_gate, q_up, q_out, qrows, I);
  blocks = (int)((srows * 2 * I + threads - 1) / threads);
  if (blocks > 148 * 16) blocks = 148 * 16;
  interleave_gate_up_kernel<uint16_t><<<blocks, threads, 0, stream>>>(s_gate, s_up, s_out, srows, I);
  return cudaGetLastError();
}

cudaError_t launch_permute_zeros(uint8_t* z, uint16_t* zq, int K, int N, int G, bool inverse, cudaStream_t stream) {
  const long long ns = (long long)(K / G) * N;
  const int sub = G >= kTileK ? 1 : kTileK / G;
  const int threads = 256;
  int blocks = (int)((ns + threads - 1) / threads);
  if (blocks > 148 * 16) blocks = 148 * 16;
  permute_zeros_kernel<<<blocks, threads, 0, stream>>>(z, zq, ns, N, sub, inverse);
  return cudaGetLastError();
}

cudaError_t launch_pack_dense(uint32_t* q, uint16_t* s, uint32_t* wq, uint16_t* sq, int K, int N, int G, bool inverse,
                              cudaStream_t stream) {
  const long long chunks = (long long)(K / kTileK) * (N / kChunkN), ns = (long long)(K / G) * N;
  const int code_blocks = (int)(chunks < 148 * 16 ? chunks : 148 * 16);
  const long long sb = (ns + kPackThreads - 1) / kPackThreads;
  const int scale_blocks = (int)(sb < 148 * 2 ? sb : 148 * 2);
  const int sub = G < kTileK ? kTileK / G : 1;
  repack_dense_kernel<<<code_blocks + scale_blocks, kPackThreads, 0, stream>>>(
      reinterpret_cast<const uint4*>(inverse ? wq : q), reinterpret_cast<uint4*>(inverse ? q : wq), inverse ? sq : s,
      inverse ? s : sq, K, N, ns, sub, code_blocks, inverse);
  return cudaGetLastError();
}

cudaError_t launch_permute_scales(uint16_t* s, uint16_t* sq, int K, int N, int G, bool inverse, cudaStream_t stream) {
  const int threads = 256;
  const long long ns = (long long)(K / G) * N;
  const int sub = G < kTileK ? kTileK / G : 1;
  int sblocks = (int)((ns + threads - 1) / threads);
  if (sblocks > 148 * 16) sblocks = 148 * 16;
  if (!inverse)
    permute_scales_kernel<<<sblocks, threads, 0, stream>>>(s, sq, ns, N, sub, false);
  else
    permute_scales_kernel<<<sblocks, threads, 0, stream>>>(sq, s, ns, N, sub, true);
  return cudaGetLastError();
}

}  // namespace marlin_b200
