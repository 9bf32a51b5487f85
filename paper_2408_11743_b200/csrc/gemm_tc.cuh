// W4A16 layer for sm_100a on the tcgen05 tensor cores, with the WEIGHTS as the A operand in tensor memory: batches from 17
// rows, and at every batch size the 2:4 layers, the 8-bit layers and those with scale groups of 64 or 32 rows.
//
// The warp-level MMA (mma.sync) of the small-batch kernel runs at about a tenth of the tcgen05 rate on this
// architecture.  Here the product is computed transposed, as the paper does for its sparse kernel (Section 4:
// C = (B^T A^T)^T): per column tile of W and 128-row k-block
//     D_t[128 channels x MPAD batch rows] += W_t^T[128 x 128] . A^T[128 x MPAD],   t = 0 .. NT - 1
// with UMMA shape M = 128 (output channels on the TMEM lanes), N = the rows of a slab (at most MPAD), K = 16.
//
// One CTA per SM, 640 threads:
//   warps 0..11   converters, three warpgroups (two with deferred scales) that take the k-blocks in turn: one converts while
//                 another waits for codes, for an operand slot or for its tensor-memory stores.  Thread = one output
//                 channel (TMEM lane): it reads its 128 codes (four 16-byte shared loads), converts them to fp16
//                 (Section 3.4 "Dequantization and Tensor Cores") and writes them into an operand slot with tcgen05.st
//                 (64 columns, two k per column).
//   warps 12..15  drain (8..15 with deferred scales): accumulators out of tensor memory, fix-up across CTAs, C.  They have
//                 no part in the conversion, so the next column segment is converted meanwhile.  The last tile of a CTA is read
//                 out by the converters as well (not with deferred scales, whose sums are in the drain's registers).
//   warp 16       weight producer: one bulk copy of packed weights per k-block (evict-first) into a ring that the converters
//                 free.
//   warp 17       activation producer: per k-block one TMA box (two 64-wide halves, 128-byte swizzle = the canonical K-major
//                 UMMA layout, rows >= M zero-filled), into a ring of its own that the MMAs free.
//   warps 18, 19  MMA issuers, one per tile.  Warp 18 owns the TMEM allocation.
// Copies and MMAs are issued by one thread of their warp in a loop of its own (no warp-wide step per k-block: with those an
// issuer took 650-800 cycles a k-block and bounded the loop up to 64 rows).
//
// Scales (template parameter SCALE):
//   kPerColumn  one scale per column, applied to the fp32 sums when the tile is finished.
//   kInLoop     group scales multiplied into the weights in the loop (Section 3.4 "Groups and Instruction Ordering"): one
//               rounding of 2^-11 per weight, as in the paper's kernel.  kInLoopSub: the same with two or four groups in a
//               k-block (groups of 64 or 32 rows).
//   kDeferred   the weights enter as exact integers; every k-block has an accumulator of its own (a ring of them in tensor
//               memory) which the drain warps multiply by the group's scale and add up in registers, in fp32.
//               Layers whose N is not a multiple of 256 (groups of 128 rows and more).
//
// What bounds it: up to 64 rows the weights (8192 x 8192, 4-bit: 34 MB, 5.0 us at 6.8 TB/s), behind them the conversion (about
// 240 cycles per 128 x 128 k-block and scheduler) and one hand-over between the warps per k-block (about 100 cycles each); at 128 rows
// also the MMAs (64 cycles per 128 x 128 x 16); prefill from some hundreds of rows: the conversion again, and the power limit.
// Measured on B200, cold weights, launches one behind the other: 8192 x 8192 at 32 / 64 / 128 rows 12.8 / 14.6 / 17.7 us (the kernel
// with one role for conversion and drain before it: 15.2 / 17.0 / 21.5); 2:4 at 16 / 64 / 128 rows 9.8 / 11.7 / 13.8
// (11.6 / 14.0 / 17.2); 8-bit at one row 14.2 (15.3), at 100 rows 19.0.
//
// Partition: every column tile is cut into S k-ranges, one per CTA, where that keeps most SMs busy (one
// epilogue per CTA, all CTAs alike); else even stripes over all units.  Fix-up of a shared tile: the CTAs of a
// tile form thread-block clusters; every CTA leaves what belongs to the others in a workspace slot, and behind one cluster barrier
// adds the others' parts to its own share of the tile.  What several clusters (or stripes) hold of a tile goes through further slots,
// and the last arriver adds them in worker order.  The order of the fp32 sum is always the same: the same inputs give
// the same bits.  Bounded waits and programmatic dependent launch are those of the small-batch kernel (gemm_dense.cu).
#pragma once
#include <stdlib.h>

#include "device_utils.cuh"
#include "marlin_internal.cuh"
#include "tc_plan.h"
#include "tc_utils.cuh"

namespace marlin_b200 {
namespace tc {

constexpr int kAuxWarp0 = 16;  // the converting and draining warps before it, the copying and issuing ones from it on
constexpr int kWeightWarp = kAuxWarp0, kActWarp = kAuxWarp0 + 1, kMmaWarp0 = kAuxWarp0 + 2, kMmaWarps = 2;
constexpr int kThreads = (kAuxWarp0 + 4) * 32;
// 640 threads start with 96 registers each; the copying and issuing warps give most of theirs to the drain
constexpr int kLaunchRegs = 96, kAuxRegs = 40;
constexpr int kTmemCols = 512;
constexpr int kMaxWStages = 12, kMaxAStages = 8, kMaxSlots = 4;

constexpr int kFmtDense4 = 0, kFmtSparse4 = 1, kFmtDense8 = 2;
constexpr int kPerColumn = 0, kInLoop = 1, kDeferred = 2, kInLoopSub = 3;

constexpr int imin(int a, int b) { return a < b ? a : b; }

// NT: 128-channel UMMA tiles per CTA (the column tile has 128 NT columns).
// FMT: 0 = dense 4-bit codes; 1 = the 2:4 variant: a stage holds the 64 kept codes per column and the metadata words of the
// tensor-memory lanes, an operand slot 32 columns of kept values and 4 of metadata per tile; 2 = 8-bit codes
// (W = (q - 128) * s): [8 vectors][256 columns][16 bytes] per stage.
template <int NT, int MPAD, int SCALE, int FMT>
struct Geometry {
  static constexpr bool SP = FMT == kFmtSparse4, W8 = FMT == kFmtDense8, DEF = SCALE == kDeferred;
  static constexpr bool LOOP = SCALE == kInLoop || SCALE == kInLoopSub, SUB = SCALE == kInLoopSub;
  // Warpgroups that convert and that drain.  With deferred scales the drain reads an accumulator per k-block, half of the
  // batch rows each.
  static constexpr int CONV_GROUPS = DEF ? 2 : 3, DRAIN_GROUPS = 4 - CONV_GROUPS;
  static constexpr int CONV_WARPS = 4 * CONV_GROUPS, DRAIN_WARPS = 4 * DRAIN_GROUPS;
  static constexpr int CONV_REGS = DRAIN_GROUPS == 1 ? kLaunchRegs : MPAD == 128 ? 80 : 88;
  static constexpr int DRAIN_REGS = DRAIN_GROUPS == 1 ? 152 : MPAD == 128 ? 136 : 128;
  static_assert(CONV_WARPS * 32 * CONV_REGS + DRAIN_WARPS * 32 * DRAIN_REGS + 128 * kAuxRegs <= kThreads * kLaunchRegs,
                "setmaxnreg draws on the registers of the launch");
  static constexpr int TN = 128 * NT;
  static constexpr int A_BYTES = MPAD * 256;
  static constexpr int CODE_BYTES = SP ? TN * 32 : (W8 ? TN * 128 : TN * 64);
  static constexpr int META_BYTES = SP ? TN * 16 : 0;
  static constexpr int W_BYTES = CODE_BYTES + META_BYTES;
  static constexpr int BAR_BYTES = 1024;
  static constexpr int OUT_WARP = 1024;                     // two buffers of 8 rows x 32 columns of fp16 per warp
  static constexpr int OUT_BYTES = kAuxWarp0 * OUT_WARP;
  // activations: three stages are the least (see the waits below); more where they are small
  static constexpr int A_STAGES = NT == 1 ? (MPAD == 128 ? 4 : W8 ? 4 : 6) : (MPAD == 128 ? 3 : (W8 || MPAD == 64 ? 4 : 6));
  static constexpr int AVAIL = kSmemBudget - BAR_BYTES - OUT_BYTES - 1024 - 1024 - A_STAGES * A_BYTES;
  // A parity wait on an mbarrier tells "the phase before the current one" from the current one and no more, so whoever waits
  // for a filling of a stage must know that the filling before it has landed.  The weight ring's length is a multiple of
  // the converting warpgroups, so that each waits for consecutive fillings of its stages in its own program order;
  // where that would cost too many stages (8-bit codes), the converters first wait for the release of the filling
  // before (which the producer, in order, had issued before a k-block that this warpgroup has already seen).
  static constexpr int W_FIT = imin(kMaxWStages, AVAIL / W_BYTES);
  static constexpr int W_STAGES = (W8 && W_FIT >= 4) ? W_FIT : W_FIT / CONV_GROUPS * CONV_GROUPS;
  static constexpr bool W_GUARD = W_STAGES % CONV_GROUPS != 0;
  static constexpr int FIXED_BYTES = ((BAR_BYTES + OUT_BYTES + 1023) / 1024) * 1024;
  static constexpr int RING_BYTES = A_STAGES * A_BYTES + W_STAGES * W_BYTES;
  static constexpr int SMEM_BYTES = FIXED_BYTES + 1024 + RING_BYTES;  // 1024: alignment
  // One issuing warp per tile; with one tile the two warps take half of a k-block each, into accumulators of their own that
  // the drain adds (deferred: whole k-blocks, in turn or all of them by one warp).
  static constexpr int KH = (DEF || NT == 2) ? 1 : 2;
  static constexpr int STAGE_WARPS = DEF ? 1 : kMmaWarps;     // issuing warps whose commits complete a stage
  // Accumulators with a barrier pair of their own.  Deferred, 128 rows: three of them leave room for two operand slots, which is
  // the faster split (two and four: the MMAs wait for the read-out; 777 x 4096 x 5504 47.2 us so, 45.0 with three).
  static constexpr int ND = DEF ? (MPAD <= 32 ? 6 : MPAD <= 64 ? 4 : 3) : NT;
  static constexpr int ISSUERS = DEF && MPAD == 128 ? 1 : kMmaWarps;  // (an odd ring has one issuer, see the waits)
  static constexpr int D_COLS = DEF ? ND * MPAD : NT * KH * MPAD;
  static constexpr int TILE_A_COLS = SP ? 32 : 64;
  // 2:4: metadata behind the kept values, on even columns (the instruction names a pair of them and which of the two)
  static constexpr int SLOT_COLS = SP ? NT * 32 + 8 : NT * 64;
  static constexpr int META_COL = NT * 32;
  static constexpr int SLOTS = imin(imin((kTmemCols - D_COLS) / SLOT_COLS, kMaxSlots), A_STAGES);
  static constexpr int A_COL0 = kTmemCols - SLOTS * SLOT_COLS;
  static constexpr int RB = MPAD / 8;                      // blocks of eight batch rows
  static constexpr bool FIXED_ROWS = tc_fixed_rows(DEF, MPAD, NT);  // slabs of MPAD rows, always
  static_assert(W_STAGES >= 3 && A_STAGES >= 3 && SLOTS >= 2 && SLOTS <= A_STAGES, "pipeline");
  static_assert(A_STAGES <= kMaxAStages && W_STAGES <= kMaxWStages, "barrier area");
  static_assert(A_COL0 >= D_COLS && A_COL0 % 2 == 0 && SLOT_COLS % 2 == 0, "tensor memory");
  static_assert(W_BYTES % 1024 == 0 && A_BYTES % 1024 == 0, "swizzled tiles need 1024-byte alignment");
  static_assert(SMEM_BYTES <= kSmemBudget, "shared memory");
  static_assert(!DEF || (NT == 1 && FMT == kFmtDense4), "deferred scales: dense, one tile");
  // deferred: each issuer sees its own stages, slots and accumulators
  static_assert(!DEF || ISSUERS == 1 || (A_STAGES % 2 == 0 && SLOTS % 2 == 0 && ND % 2 == 0), "the two issuers take the k-blocks in turn");
  // who waits for the MMAs of k-block it - SLOTS knows that those of it - SLOTS - CONV_GROUPS are done (the unit before of the
  // same warpgroup and tile), which has to be past the completion before on the same barrier
  static_assert(A_STAGES >= CONV_GROUPS, "parity of the completion barriers");
};

// ---- small device helpers ---------------------------------------------------------------------------------------
// one lane of the warp, the same one every time
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "elect.sync _|p, 0xffffffff;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(p));
  return p != 0;
}
// 16 lanes x 16 columns in the MMA's fragment order: registers 4b + e hold columns 8b ..; e = 0, 1: row lane / 4, columns
// 2 (lane % 4) and the next; e = 2, 3: row lane / 4 + 8
__device__ __forceinline__ void tc_ld_frag(uint32_t taddr, float* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
               : "r"(taddr)
               : "memory");
}
// the same, 8 columns: registers e
__device__ __forceinline__ void tc_ld_frag8(uint32_t taddr, float* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3])
               : "r"(taddr)
               : "memory");
}
// 8 x 8 fragments of 16-bit values, transposed: lanes 8i .. 8i + 7 give the row addresses of matrix i
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t saddr, const uint32_t (&r)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(saddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void stmatrix_x2_trans(uint32_t saddr, uint32_t a, uint32_t b) {
  asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1, %2};" ::"r"(saddr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// The codes of a word as s * (q - 8), rounded once, where s * 2^20 is finite (|s| <= kFastScaleBits as fp16 bits, 0.0624):
// three of the four pairs of nibbles are moved to bits 4..7, where an AND alone leaves the fp16 subnormal q * 2^-20, and one
// fma with s * 2^20 and -8 s (both exact) is the scaled weight; the fourth goes through the exponent trick.  Eleven
// instructions for eight weights, five of them on the fp16 pipe, instead of thirteen with eight: that pipe, which issues a
// packed operation every two cycles, bounds the conversion (236 against 299 cycles per 128-channel k-block and scheduler,
// measured alone with three warps on it).
constexpr uint32_t kFastScaleBits = 0x2bffu;
__device__ __forceinline__ void dequant8_scaled(uint32_t w, uint32_t* a, uint32_t s2, uint32_t s2_up, uint32_t minus8s) {
  constexpr uint32_t LO = 0x000f000fu, HI = 0x00f000f0u, EX = 0x64006400u;
  a[0] = hmul2_u32(hsub2_u32(lop3<0xea>(w, LO, EX), 0x64086408u), s2);
  a[1] = hfma2_u32(w & HI, s2_up, minus8s);
  a[2] = hfma2_u32((w >> 4) & HI, s2_up, minus8s);
  a[3] = hfma2_u32((w >> 8) & HI, s2_up, minus8s);
}

template <bool V>
struct BoolC {
  static constexpr bool value = V;
};
template <int V>
struct IntC {
  static constexpr int value = V;
};
struct Int {
  int value;
};

// ---- the kernel ---------------------------------------------------------------------------------------------------
template <int NT, int MPAD, int SCALE, int FMT>
__global__ void __launch_bounds__(kThreads, 1)
gemm_tc_kernel(const GemmParams p, const __grid_constant__ CUtensorMap tmap_a) {
  using G = Geometry<NT, MPAD, SCALE, FMT>;
  constexpr bool SP = G::SP, W8 = G::W8, DEF = G::DEF, LOOP = G::LOOP, SUB = G::SUB;
  constexpr int WS = G::W_STAGES, AS = G::A_STAGES, NSLOTS = G::SLOTS, KH = G::KH, RB = G::RB;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* wfull = reinterpret_cast<uint64_t*>(smem);          // [12]   weights of a stage have landed
  uint64_t* wempty = reinterpret_cast<uint64_t*>(smem + 128);   // [12]   the codes of a stage have been converted
  uint64_t* xfull = reinterpret_cast<uint64_t*>(smem + 256);    // [8]    activation tile of a stage has landed
  uint64_t* mdone = reinterpret_cast<uint64_t*>(smem + 384);    // [8]    the MMAs of an activation stage have completed
  uint64_t* afull = reinterpret_cast<uint64_t*>(smem + 576);    // [4]    operand slot written
  uint64_t* dfull = reinterpret_cast<uint64_t*>(smem + 704);    // [8]    accumulator complete
  uint64_t* dempty = reinterpret_cast<uint64_t*>(smem + 768);   // [8]    accumulator read out
  uint32_t* tmem_base_slot = reinterpret_cast<uint32_t*>(smem + 832);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 836);
  volatile int* last_flag = reinterpret_cast<volatile int*>(smem + 840);
  volatile int* others_flag = reinterpret_cast<volatile int*>(smem + 844);  // the others have left their parts of the last tile
  uint8_t* a_ring = smem + G::FIXED_BYTES;
  uint8_t* w_ring = a_ring + AS * G::A_BYTES;

  // the warp index, broadcast from lane 0 so that the compiler knows it is the same in all lanes (every role branch
  // and loop bound below depends on it: otherwise each warp-wide instruction gets a divergence check)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const uint32_t buf_s = smem_u32(smem) + G::BAR_BYTES + (uint32_t)(warp * G::OUT_WARP);  // this warp's output buffers
  const uint32_t worker = blockIdx.x;
  const uint32_t U = p.units, P = p.workers, KB = p.kb;
  // split > 0: one k-range of one column tile per CTA (the last range of a tile ends where the next tile begins)
  // whole: the stripes are cut at tile boundaries (many more tiles than workers: nothing is shared, no fix-up)
  const uint32_t u0 = p.split   ? split_begin32(worker, KB, p.split)
                      : p.whole ? stripe_begin32(worker, (uint32_t)p.ncols, P) * KB
                                : stripe_begin32(worker, U, P);
  const uint32_t u1 = p.split   ? split_begin32(worker + 1, KB, p.split)
                      : p.whole ? stripe_begin32(worker + 1, (uint32_t)p.ncols, P) * KB
                                : stripe_begin32(worker + 1, U, P);
  const uint32_t total = u1 - u0;  // k-blocks of this CTA
  // rows of a slab: a multiple of 16, at most MPAD (see tc_slab_rows)
  const uint32_t slab_rows = G::FIXED_ROWS ? (uint32_t)MPAD : p.slab_rows;
  const bool zp = SCALE != kPerColumn && p.zq != nullptr;  // zero points: rows of the same shape and order as the scales

  pdl_launch_dependents();
  if (warp == kWeightWarp) {
    // This warp sets up all barriers that it needs itself and does not wait for the others: its copies go out first
    // (issuing one takes a few hundred cycles; behind the block barrier the first weights landed 1 us later).
    if (lane < WS) {
      mbar_init(&wfull[lane], 1);
      mbar_init(&wempty[lane], 4);  // the warps of the warpgroup that converts it
    }
    if (lane == 0) *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    // (a barrier of its own: with few k-blocks this warp is done while another still allocates tensor memory, and its arrival
    // at the block's last barrier must not count for this one)
    asm volatile("bar.arrive 2, %0;" ::"n"(kThreads) : "memory");
  } else {
    if (warp == kActWarp) {
      if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_a) : "memory");
      if (lane < AS) {
        mbar_init(&xfull[lane], 1);
        mbar_init(&mdone[lane], G::STAGE_WARPS);
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (warp == kMmaWarp0) {
      tmem_alloc(tmem_base_slot, kTmemCols);
      tmem_relinquish();
    } else if (warp == kMmaWarp0 + 1) {
      if (lane < NSLOTS) mbar_init(&afull[lane], 4);
      if (lane < G::ND) {
        mbar_init(&dfull[lane], KH);
        mbar_init(&dempty[lane], G::DRAIN_WARPS);
      }
      if (lane == 0) *last_flag = 0;
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before_sync();
    asm volatile("bar.sync 2, %0;" ::"n"(kThreads) : "memory");
    tc_fence_after_sync();
  }
  const uint32_t tmem_base = warp == kWeightWarp ? 0u : *tmem_base_slot;

  // ---- finished sums to C, and the last steps of the fix-up: used by the drain and, behind clusters, by the converters ----
  // A block of eight batch rows x 32 channels in fragment order (r[2h + x]: channels 16h + 8x + lane / 4, rows
  // 2 (lane % 4) and the next, fp16); with the fused activation every 16 channels are eight gate channels and the same
  // eight up channels, and activate() leaves r[h]: products 8h + lane / 4.
  auto activate = [&](uint32_t (&r)[4]) {
    if (p.swiglu) {
      r[0] = swiglu2(r[0], r[1]);
      r[1] = swiglu2(r[2], r[3]);
    }
  };
  const int ldc = p.swiglu ? p.N / 2 : p.N;
  // ... to C: through a buffer of the warp, so that C is written in runs of 64 bytes (32 with the fused activation)
  auto emit = [&](const uint32_t (&r)[4], uint32_t buf, int m0, int m_lim, size_t row0, uint32_t n0) {
    const int i = lane >> 3, rr = lane & 7;
    if (!p.swiglu) {
      stmatrix_x4_trans(buf + (uint32_t)(rr * 64 + ((i ^ ((rr >> 1) & 3)) * 16)), r);
      __syncwarp();
      const int row = lane >> 2, ch = lane & 3;
      const uint4 v = lds128(buf + (uint32_t)(row * 64 + ((ch ^ ((row >> 1) & 3)) * 16)));
      if (m0 + row < m_lim) *reinterpret_cast<uint4*>(p.C + (row0 + m0 + row) * ldc + n0 + ch * 8) = v;
    } else {
      stmatrix_x2_trans(buf + (uint32_t)(rr * 32 + (((i & 1) ^ ((rr >> 2) & 1)) * 16)), r[0], r[1]);
      __syncwarp();
      const int row = (lane & 15) >> 1, ch = lane & 1;
      const uint4 v = lds128(buf + (uint32_t)(row * 32 + ((ch ^ ((row >> 2) & 1)) * 16)));
      if (lane < 16 && m0 + row < m_lim) *reinterpret_cast<uint4*>(p.C + (row0 + m0 + row) * ldc + n0 / 2 + ch * 8) = v;
    }
  };
  auto pack8 = [&](const float* f, uint32_t (&r)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) r[e] = pack_half2(f[2 * e], f[2 * e + 1]);
  };
  // float4 index of half h of block (32 channels c32, eight rows b) in a partial tile
  auto frag_index = [&](int c32, int b, int h) { return (uint32_t)(((c32 * RB + b) * 2 + h) * 32 + lane); };
  // workspace slots: with clusters one per worker and then one per cluster, else two per worker (a worker shares at most its
  // first and last tile)
  auto slot_ptr = [&](uint32_t index) { return reinterpret_cast<float4*>(p.partials + (size_t)index * (G::TN * MPAD)); };
  // Blocks x of a tile (x = c32 * nb + b, every `step`-th from x0 on) summed over the slots slot(0) .. slot(n - 1), in order;
  // done(c32, b, f) takes the sums.  Two blocks and two slots at a time, or one block and four slots where that is all a warp
  // has (deferred scales, 32 rows: 20 x 11008 x 1088 8.4 us, 7.8 so): eight 16-byte loads of a lane are in flight together.  What a slot
  // held is cleared behind its last read, so that a workspace comes back from most calls as it was given (not with deferred scales, and
  // not past the last column); nothing relies on it: slots are written before they are read.
  auto sum_some = [&](auto ib_c, int x0, int step, int items, int nb, uint32_t col, int n, auto slot, auto done) {
    constexpr int IB = decltype(ib_c)::value, QN = 4 / IB;
    for (int x = x0; x < items; x += IB * step) {
      int c32[IB], b[IB];
      bool ok[IB];
#pragma unroll
      for (int i = 0; i < IB; ++i) {
        const int xi = x + i * step;
        c32[i] = xi / nb;
        b[i] = xi - c32[i] * nb;
        ok[i] = xi < items && col * G::TN + (uint32_t)c32[i] * 32 < (uint32_t)p.N;
      }
      float f[IB][8];
#pragma unroll
      for (int i = 0; i < IB; ++i)
#pragma unroll
        for (int e = 0; e < 8; ++e) f[i][e] = 0.f;
      for (int src = 0; src < n; src += QN) {
        float4 v[QN][IB][2];
#pragma unroll
        for (int q = 0; q < QN; ++q)
          if (src + q < n) {
            const float4* from = slot(src + q);
#pragma unroll
            for (int i = 0; i < IB; ++i)
#pragma unroll
              for (int h = 0; h < 2; ++h)
                if (ok[i]) v[q][i][h] = ld_cg_f4(from + frag_index(c32[i], b[i], h));
          }
#pragma unroll
        for (int q = 0; q < QN; ++q)
          if (src + q < n) {
#pragma unroll
            for (int i = 0; i < IB; ++i)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                f[i][4 * h] = __fadd_rn(f[i][4 * h], v[q][i][h].x); f[i][4 * h + 1] = __fadd_rn(f[i][4 * h + 1], v[q][i][h].y);
                f[i][4 * h + 2] = __fadd_rn(f[i][4 * h + 2], v[q][i][h].z); f[i][4 * h + 3] = __fadd_rn(f[i][4 * h + 3], v[q][i][h].w);
              }
          }
        if constexpr (!DEF) {
#pragma unroll
          for (int q = 0; q < QN; ++q)
            if (src + q < n) {
              float4* to = slot(src + q);
#pragma unroll
              for (int i = 0; i < IB; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                  if (ok[i]) to[frag_index(c32[i], b[i], h)] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
      }
#pragma unroll
      for (int i = 0; i < IB; ++i)
        if (ok[i]) done(c32[i], b[i], f[i], i);
    }
  };
  auto sum_blocks = [&](int x0, int step, int items, int nb, uint32_t col, int n, auto slot, auto done) {
    if (DEF && MPAD == 32 && x0 + step >= items)
      sum_some(IntC<1>{}, x0, step, items, nb, col, n, slot, done);
    else
      sum_some(IntC<2>{}, x0, step, items, nb, col, n, slot, done);
  };
  // sums to C
  auto store_block = [&](int c32, int b, const float (&f)[8], int i, uint32_t col, int m_lim, size_t row0) {
    uint32_t r[4];
    pack8(f, r);
    activate(r);
    emit(r, buf_s + (uint32_t)i * 512, b * 8, m_lim, row0, col * G::TN + (uint32_t)c32 * 32);
  };
  // stripes: the slot of worker w for virtual column tile vcol
  auto stripe_slot = [&](int w, uint32_t vcol) {
    return slot_ptr((uint32_t)(2 * w + ((!p.split && vcol != stripe_begin32((uint32_t)w, U, P) / KB) ? 1 : 0)));
  };

  // Split tile, CTAs in clusters (deferred scales; the others: drain_last): every CTA has left its partial tile in its slot.  Behind the cluster barrier a CTA adds up
  // its share of the (32 channels, eight rows) blocks over the cluster, in rank order, and stores that part of C; where a
  // tile has several clusters the share goes to the cluster's slot and the last of them adds the shares in order.
  // (Through the L2 and not through distributed shared memory, which moves about 12 bytes per clock and SM here against
  // 60 and more, and would need a second barrier before a CTA may exit.)  `w16`: the warp among the converting and draining ones.
  auto finish_cluster = [&](int w16) {
    const int cs = (int)p.cluster, C = (int)p.split / cs, r = (int)cluster_ctarank();
    const uint32_t vcol = u0 / KB, col = vcol / p.slabs, slab = vcol - col * p.slabs;
    const size_t row0 = (size_t)slab * slab_rows;
    const int m_lim = min(p.M - (int)row0, (int)slab_rows);
    const int nb = (m_lim + 7) >> 3, items = nb * (G::TN / 32);
    cluster_sync_all();  // every CTA's partial tile is in its slot
    if (w16 < G::CONV_WARPS) pdl_wait_prior_grids();
    const uint32_t first = worker - (uint32_t)r, shares = P + vcol * (uint32_t)C;
    auto to_c = [&](int c32, int b, const float (&f)[8], int i) { store_block(c32, b, f, i, col, m_lim, row0); };
    auto exchanged = [&](int q) { return slot_ptr(first + (uint32_t)q); };
    const int x0 = r + cs * w16, step = cs * kAuxWarp0;
    if (C == 1) {
      sum_blocks(x0, step, items, nb, col, cs, exchanged, to_c);
      return;
    }
    float4* mine = slot_ptr(shares + (worker / (uint32_t)cs) % (uint32_t)C);
    sum_blocks(x0, step, items, nb, col, cs, exchanged, [&](int c32, int b, const float (&f)[8], int) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        mine[frag_index(c32, b, h)] = make_float4(f[4 * h], f[4 * h + 1], f[4 * h + 2], f[4 * h + 3]);
    });
    // the CTAs of rank r of the tile's clusters hold the same share: whoever of them comes last adds it up
    named_bar_sync(1, kAuxWarp0 * 32);
    if (w16 == 0 && lane == 0) {
      int* counter = &p.counters[vcol * (uint32_t)cs + r];
      const int is_last = atom_add_acq_rel_gpu(counter, 1) == C - 1 ? 1 : 0;
      if (is_last) *counter = 0;
      *last_flag = is_last;
    }
    named_bar_sync(1, kAuxWarp0 * 32);
    if (*last_flag != 0)
      sum_blocks(x0, step, items, nb, col, C, [&](int q) { return slot_ptr(shares + (uint32_t)q); }, to_c);
  };

  // Stripes, the last segment of a CTA (deferred scales, likewise): its partial tile is in its slot; the last arriver at the tile adds all of them up, all
  // converting and draining warps together (they are done, and nothing else is left to hide the loads behind).
  // One counter per virtual column tile; where there are more of those than workers, per tile that can be shared, numbered by
  // the first worker on it (at most one tile runs over the end of a worker's stripe).
  auto finish_stripe = [&](int w16) {
    // nothing is shared: out, in front of the divisions (32 x 1024 x 14400 with deferred scales 5.92 us behind them, 5.67 so)
    if (p.whole || p.split == 1) return;
    const uint32_t vcol = (u1 - 1) / KB, col = vcol / p.slabs, slab = vcol - col * p.slabs;
    const int first_w = p.split ? (int)(vcol * p.split) : (int)stripe_owner32(vcol * KB, U, P);
    const int last_w = p.split ? (int)(vcol * p.split + p.split - 1) : (int)stripe_owner32((vcol + 1) * KB - 1, U, P);
    if (last_w == first_w) return;
    if (w16 < G::CONV_WARPS) pdl_wait_prior_grids();
    const size_t row0 = (size_t)slab * slab_rows;
    const int m_lim = min(p.M - (int)row0, (int)slab_rows);
    const int nb = (m_lim + 7) >> 3, items = nb * (G::TN / 32);
    named_bar_sync(1, kAuxWarp0 * 32);
    if (w16 == 0 && lane == 0) {
      int* counter = &p.counters[(uint32_t)p.ncols <= P ? vcol : (uint32_t)first_w];
      const int is_last = atom_add_acq_rel_gpu(counter, 1) == last_w - first_w ? 1 : 0;
      if (is_last) *counter = 0;
      *last_flag = is_last;
    }
    named_bar_sync(1, kAuxWarp0 * 32);
    if (*last_flag != 0) {
      sum_blocks(w16, kAuxWarp0, items, nb, col, last_w - first_w + 1, [&](int q) { return stripe_slot(first_w + q, vcol); },
                 [&](int c32, int b, const float (&f)[8], int i) { store_block(c32, b, f, i, col, m_lim, row0); });
    }
  };

  // ---- read-out of accumulators: used by the drain and, for a CTA's last tile, by the converters too ----
  const uint32_t quad = (uint32_t)(warp & 3);  // 32 TMEM lanes = channels of a tile
  // the scales of channels lane / 4, +8, +16, +24 of the warp's 32 are four halves in a row
  const uint32_t spos2 = ((quad >> 1) * 64 + 8 * (uint32_t)(lane >> 2) + 4 * (quad & 1)) * 2;
  auto column_scales = [&](uint32_t col, int t, float (&sc)[4]) {
    sc[0] = sc[1] = sc[2] = sc[3] = 1.f;
    if constexpr (SCALE == kPerColumn) {
      uint2 sv = make_uint2(0, 0);
      if (col * G::TN + (uint32_t)t * 128 + quad * 32 < (uint32_t)p.N)
        sv = __ldg(reinterpret_cast<const uint2*>(p.sq + ((size_t)col * G::TN + (size_t)t * 128) * 2 + spos2));
      const float2 s01 = __half22float2(*reinterpret_cast<const __half2*>(&sv.x));
      const float2 s23 = __half22float2(*reinterpret_cast<const __half2*>(&sv.y));
      sc[0] = s01.x; sc[1] = s01.y; sc[2] = s23.x; sc[3] = s23.y;
    }
  };
  // 8 NBK rows from row m on out of tensor memory, the halves of the k-blocks added, scaled: f[8b + 4h + e].  Every product and sum
  // of the fix-up is rounded by itself (no fma): whether a CTA's part goes into the sum from registers or through a slot depends on
  // who comes first and must not show.
  auto load_rows = [&](auto nbk_c, int t, int m, const float (&sc)[4], float* f) {
    constexpr int NBK = decltype(nbk_c)::value;
    float a[2][4 * NBK], a2[2][4 * NBK];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t at = tmem_base + ((quad * 32u + (uint32_t)(16 * h)) << 16) + (uint32_t)(t * KH * MPAD + m);
      if constexpr (NBK == 2) {
        tc_ld_frag(at, a[h]);
        if constexpr (KH == 2) tc_ld_frag(at + MPAD, a2[h]);
      } else {
        tc_ld_frag8(at, a[h]);
        if constexpr (KH == 2) tc_ld_frag8(at + MPAD, a2[h]);
      }
    }
    tc_wait_ld();
#pragma unroll
    for (int x = 0; x < 8 * NBK; ++x) {
      const int h = (x >> 2) & 1, i = 4 * (x >> 3) + (x & 3);
      f[x] = a[h][i];
      if constexpr (KH == 2) f[x] = __fadd_rn(f[x], a2[h][i]);
      if constexpr (SCALE == kPerColumn) f[x] = __fmul_rn(f[x], sc[2 * h + ((x >> 1) & 1)]);
    }
  };
  // The CTA's last tile (not with deferred scales): the converters have nothing else left to do, so all 16 warps read it out, in pieces
  // of 16 rows x 32 channels; piece c: tile c % NT, rows 16 (c / NT).  With the four draining warps alone this took 0.55 us (32 rows,
  // two tiles) to 2.1 us (128 rows) at the end of every launch.
  auto drain_last = [&](int w16) {
    const uint32_t vcol = (u1 - 1) / KB, col = vcol / p.slabs, slab = vcol - col * p.slabs;
    const uint32_t phase = (vcol - u0 / KB) & 1u;
    const size_t row0 = (size_t)slab * slab_rows;
    const int m_lim = min(p.M - (int)row0, (int)slab_rows);
    const int pieces = NT * ((m_lim + 15) >> 4), units = NT * ((m_lim + 7) >> 3), g = w16 >> 2;
    const int first_w = p.split ? (int)(vcol * p.split) : (int)stripe_owner32(vcol * KB, U, P);
    const int last_w = p.split ? (int)(vcol * p.split + p.split - 1) : (int)stripe_owner32((vcol + 1) * KB - 1, U, P);
    const bool shared_tile = !p.whole && last_w > first_w, clustered = p.cluster > 1;
    int* stripe_counter = &p.counters[(uint32_t)p.ncols <= P ? vcol : (uint32_t)first_w];
    constexpr IntC<1> one{};
    constexpr IntC<2> two{};
    // NBK blocks of eight rows from block b on (of tile t) out of tensor memory
    auto own_sums = [&](auto nbk_c, int t, int b, float* f) {
      float sc[4];
      column_scales(col, t, sc);
      mbar_wait(&dfull[t], phase, abort_flag, p.status);
      tc_fence_after_sync();
      load_rows(nbk_c, t, 8 * b, sc, f);
    };
    // half y % 2 (channels) of block b + y / 2 in a slot
    auto index_of = [&](int t, int b, int y) { return frag_index(t * 4 + (int)quad, b + (y >> 1), y & 1); };
    auto has = [&](int b, int y) { return 8 * (b + (y >> 1)) < m_lim; };  // (its rows exist)
    auto to_slot = [&](auto nbk_c, int t, int b, const float* f, float4* slot) {
#pragma unroll
      for (int y = 0; y < 2 * decltype(nbk_c)::value; ++y)
        if (has(b, y)) slot[index_of(t, b, y)] = make_float4(f[4 * y], f[4 * y + 1], f[4 * y + 2], f[4 * y + 3]);
    };
    auto to_c = [&](auto nbk_c, int t, int b, const float* f) {
      const int c32 = t * 4 + (int)quad;
      if (col * G::TN + (uint32_t)c32 * 32 >= (uint32_t)p.N) return;
#pragma unroll
      for (int i = 0; i < decltype(nbk_c)::value; ++i) {
        float fb[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) fb[x] = f[8 * i + x];
        store_block(c32, b + i, fb, i, col, m_lim, row0);
      }
    };
    // Block b of n partial tiles in their order: tile `own` (n: none) from tensor memory, the others from their slots, three of them
    // on their way at a time (a cluster of four: one latency of the L2), and cleared behind the read (a workspace comes back as it was
    // given; behind the stores of C, in a loop of its own, it takes 0.1 to 0.3 us longer).  The sums go to `to` or, without one, to C.
    auto gather = [&](int t, int b, int n, int own, auto slot, float4* to) {
      float f[8], sum[8];
      if (own < n) own_sums(one, t, b, f);
#pragma unroll
      for (int x = 0; x < 8; ++x) sum[x] = 0.f;
      const int others = own < n ? n - 1 : n;
      constexpr int UN = 3;
      for (int o = 0; o < others; o += UN) {
        float4 v[UN][2];
        float4* from[UN];
#pragma unroll
        for (int i = 0; i < UN; ++i)
          if (o + i < others) {
            from[i] = slot(o + i + (o + i >= own ? 1 : 0));
#pragma unroll
            for (int y = 0; y < 2; ++y)
              if (has(b, y)) v[i][y] = ld_cg_f4(from[i] + index_of(t, b, y));
          }
#pragma unroll
        for (int i = 0; i < UN; ++i)
          if (o + i < others) {
            if (o + i == own) {
#pragma unroll
              for (int x = 0; x < 8; ++x) sum[x] = __fadd_rn(sum[x], f[x]);
            }
#pragma unroll
            for (int y = 0; y < 2; ++y)
              if (has(b, y)) {  // (always so here; without the condition the loop is compiled to 1 to 4 % longer launches)
                sum[4 * y] = __fadd_rn(sum[4 * y], v[i][y].x); sum[4 * y + 1] = __fadd_rn(sum[4 * y + 1], v[i][y].y);
                sum[4 * y + 2] = __fadd_rn(sum[4 * y + 2], v[i][y].z); sum[4 * y + 3] = __fadd_rn(sum[4 * y + 3], v[i][y].w);
                from[i][index_of(t, b, y)] = make_float4(0.f, 0.f, 0.f, 0.f);
              }
          }
      }
      if (own == n - 1) {
#pragma unroll
        for (int x = 0; x < 8; ++x) sum[x] = __fadd_rn(sum[x], f[x]);
      }
      if (to)
        to_slot(one, t, b, sum, to);
      else
        to_c(one, t, b, sum);
    };
    pdl_wait_prior_grids();
    float f[16];
    if (clustered) {
      // CTAs of a split tile in clusters: the tile is dealt out to them in units of 32 channels x 8 rows; unit c: tile c % NT, block
      // c / NT, to rank c % cluster and warpgroup c / cluster % 4 of it.  A CTA leaves the units of the others in its slot and, behind the
      // cluster barrier, adds the others' parts of its own units to what it has in tensor memory, in rank order.  (In whole pieces
      // four CTAs with two tiles of 32 rows had four warps each at work, twice as long, and up to 16 rows two of them nothing to do:
      // 8192 x 8192 at 24 / 32 / 64 rows 13.2 / 13.3 / 14.7 us so, 12.6 / 12.8 / 14.5 in units; 4096 x 4096 at 64 rows 8.7 / 7.9; 8-bit, four
      // rows of 8192 x 8192 14.6 / 14.2; 2:4, 64 rows 11.9 / 11.7.  One body for all steps and partitions, its numbers in variables: half the
      // code, and 1 to 10 % longer.  Through the L2 and not
      // through distributed shared memory: bulk copies from one shared memory into another, which exchange 32 KB among four CTAs in 2630
      // cycles instead of 4170, need a handshake before them and a barrier before a CTA may exit, and took 1 to 1.5 us longer in all.)
      const int cs = (int)p.cluster, C = (int)p.split / cs, r = (int)cluster_ctarank();
      float4* mine = slot_ptr(worker);
      for (int c = g; c < pieces; c += 4) {
        const int t = c % NT, b = c / NT * 2;
        const bool lo = (t + NT * b) % cs != r, hi = (t + NT * (b + 1)) % cs != r && has(b, 2);
        if (!lo && !hi) continue;
        own_sums(two, t, b, f);
        if (lo) to_slot(one, t, b, f, mine);
        if (hi) to_slot(one, t, b + 1, f + 8, mine);
      }
      cluster_sync_all();
      const uint32_t first = worker - (uint32_t)r, shares = P + vcol * (uint32_t)C;
      float4* share = C == 1 ? nullptr : slot_ptr(shares + (worker / (uint32_t)cs) % (uint32_t)C);
      for (int c = r + cs * g; c < units; c += 4 * cs)
        gather(c % NT, c / NT, cs, r, [&](int q) { return slot_ptr(first + (uint32_t)q); }, share);
      if (C == 1) return;
      // the CTAs of rank r of the tile's clusters hold the same units: whoever of them comes last adds them up
      named_bar_sync(1, kAuxWarp0 * 32);
      if (w16 == 0 && lane == 0) {
        int* counter = &p.counters[vcol * (uint32_t)cs + r];
        const int is_last = atom_add_acq_rel_gpu(counter, 1) == C - 1 ? 1 : 0;
        if (is_last) *counter = 0;
        *last_flag = is_last;
      }
      named_bar_sync(1, kAuxWarp0 * 32);
      if (*last_flag != 0)
        for (int c = r + cs * g; c < units; c += 4 * cs)
          gather(c % NT, c / NT, C, C, [&](int q) { return slot_ptr(shares + (uint32_t)q); }, nullptr);
      return;
    }
    // Stripes.  Where the other CTAs of the tile have left their parts already (it was their first tile), this one adds them to what it
    // has and writes C; otherwise it leaves its own, and the last arriver adds up all of them.  All that needs a division is worked out in
    // front, while the last MMAs run, and the parts of three CTAs come in one latency of the L2 (24 x 8192 x 22016, 2:4, 86 tiles on 148 CTAs:
    // 21.2 us with the general code of finish_stripe at the end, 19.9 so; in pieces of 16 rows 20.3).
    const uint32_t slot0 = 2u * (uint32_t)first_w + ((!p.split && shared_tile && vcol != stripe_begin32((uint32_t)first_w, U, P) / KB) ? 1u : 0u);
    auto part_slot = [&](int q) { return slot_ptr(q == 0 ? slot0 : 2u * (uint32_t)(first_w + q)); };  // (see stripe_slot)
    if (w16 == 0 && lane == 0) *others_flag = shared_tile && ld_acquire_gpu(stripe_counter) == last_w - first_w ? 1 : 0;
    named_bar_sync(1, kAuxWarp0 * 32);  // (also: the drain is done with the tile before, which went through all output buffers)
#ifdef MARLIN_TEST_HOOKS
    const bool onto = *others_flag != 0 && p.status[7] != kTestLeaveMagic;
#else
    const bool onto = *others_flag != 0;
#endif
    if (shared_tile && !onto) {
      float4* mine = part_slot((int)worker - first_w);
      for (int c = g; c < pieces; c += 4) {
        own_sums(two, c % NT, c / NT * 2, f);
        to_slot(two, c % NT, c / NT * 2, f, mine);
      }
      named_bar_sync(1, kAuxWarp0 * 32);
      if (w16 == 0 && lane == 0) *last_flag = atom_add_acq_rel_gpu(stripe_counter, 1) == last_w - first_w ? 1 : 0;
      named_bar_sync(1, kAuxWarp0 * 32);
      if (*last_flag == 0) return;
    }
    if (shared_tile) {
      const int parts = last_w - first_w + 1, own = onto ? (int)worker - first_w : parts;
      for (int c = g; c < units; c += 4) gather(c % NT, c / NT, parts, own, part_slot, nullptr);
      if (w16 == 0 && lane == 0) *stripe_counter = 0;
    } else {
      for (int c = g; c < pieces; c += 4) {
        own_sums(two, c % NT, c / NT * 2, f);
        to_c(two, c % NT, c / NT * 2, f);
      }
    }
  };

  if (warp >= kAuxWarp0) {
    setmaxnreg_dec<kAuxRegs>();
    if (warp == kWeightWarp) {
      if (elect_one()) {
#ifdef MARLIN_TEST_HOOKS
        const bool withhold = worker == 0 && p.status[7] == kTestWithholdMagic;
#else
        constexpr bool withhold = false;
#endif
        const uint32_t vcol = u0 / KB;
        uint32_t kb = u0 - vcol * KB, col = vcol / p.slabs, slab = vcol - col * p.slabs;
        // one slab: every weight byte is read once; several slabs read the layer once each, from the L2 after the first
        // (normal priority: marked to stay, the weights of the layers before would crowd the L2)
        const uint64_t pol_w = p.slabs > 1 ? policy_evict_normal() : policy_evict_first();
        for (uint32_t it = 0; it < total; ++it) {
          const uint32_t ws = it % WS;
          if (it >= (uint32_t)WS) mbar_wait<20>(&wempty[ws], (it / WS - 1) & 1u, abort_flag, p.status);
          if (!(withhold && it == 1)) {
            // The last column tile of a layer may be narrower: its chunks are fewer, what the stage held before stays in
            // the rest, and the channels that come of it are not stored.
            uint8_t* st = w_ring + (size_t)ws * G::W_BYTES;
            const uint32_t cols = (SP || W8) ? (uint32_t)G::TN : min((uint32_t)G::TN, (uint32_t)p.N - col * G::TN);
            const uint32_t code_bytes = (SP || W8) ? (uint32_t)G::CODE_BYTES : cols * 64u;
            mbar_expect_tx(&wfull[ws], code_bytes + G::META_BYTES);
            if constexpr (SP || W8) {
              // one record per (256 columns, k-block), of vectors of 16 bytes per column; 128 columns are half of each vector
              constexpr int VECS = G::CODE_BYTES / (G::TN * 16);
              const size_t rec = (size_t)(col * NT / 2) * KB + kb;
              const uint8_t* codes = p.wq + rec * (size_t)(VECS * 4096);
              if constexpr (NT == 2) {
                bulk_g2s(st, codes, G::CODE_BYTES, &wfull[ws], pol_w);
              } else {
#pragma unroll
                for (int v = 0; v < VECS; ++v) bulk_g2s(st + v * 2048, codes + v * 4096 + (col & 1u) * 2048u, 2048, &wfull[ws], pol_w);
              }
              if constexpr (SP)
                bulk_g2s(st + G::CODE_BYTES, p.meta + rec * 4096 + (NT == 1 ? (col & 1u) * 2048u : 0u), G::META_BYTES, &wfull[ws], pol_w);
            } else {
              // super-columns of four chunks (fewer in the last), k-blocks contiguous inside a super-column
              const uint32_t nb = col * (2 * NT), sc = nb >> 2, cs = min(4u, (uint32_t)p.N / kChunkN - 4u * sc);
              bulk_g2s(st, p.wq + ((size_t)sc * 4u * KB + (size_t)kb * cs + (nb & 3u)) * kChunkBytes, code_bytes, &wfull[ws],
                       pol_w);
            }
          }
          if (++kb == KB) {
            kb = 0;
            if (++slab == p.slabs) { slab = 0; ++col; }
          }
        }
        if (*abort_flag) {
          // give copies that may still be in flight time to land before the CTA's shared memory goes away
          for (int x = 0; x < 1000; ++x) __nanosleep(1000);
        }
      }
    } else if (warp == kActWarp) {
      if (elect_one()) {
        const uint64_t pol_a = policy_evict_last();
        uint32_t vcol = u0 / KB, kb = u0 - vcol * KB, slab = vcol % p.slabs;
        pdl_wait_prior_grids();
        for (uint32_t it = 0; it < total; ++it) {
          const uint32_t s = it % AS;
          if (it >= (uint32_t)AS) mbar_wait<20>(&mdone[s], (it / AS - 1) & 1u, abort_flag, p.status);
          mbar_expect_tx(&xfull[s], slab_rows * 256u);
          tma_load_3d(a_ring + (size_t)s * G::A_BYTES, &tmap_a, 0, (int)(slab * slab_rows), (int)(2 * kb), &xfull[s], pol_a);
          if (++kb == KB) {
            kb = 0;
            if (++slab == p.slabs) slab = 0;
          }
        }
        if (*abort_flag) {
          for (int x = 0; x < 1000; ++x) __nanosleep(1000);
        }
      }
    } else if (elect_one()) {
      // ------------------------------- MMA issuers (one thread each) -------------------------------------------------
      constexpr int KS = 8 / KH;  // K = 16 steps per warp and k-block
      const int mw = warp - kMmaWarp0;
      const int t = NT == 2 ? mw : 0;
      const int h = KH == 2 ? mw : 0;  // half of the k-block
      // the MMAs of the k-block in stage s and operand slot `slot` into d_tmem; `fresh`: overwrite what is there.  N: the rows of
      // a slab (`rows.value`); the halves of an activation tile lie that many rows apart.
      auto issue = [&](auto rows, uint32_t s, uint32_t slot, uint32_t d_tmem, bool fresh) {
        const uint32_t idesc = instr_desc_f16(128, (int)rows.value), half_step = (uint32_t)rows.value * 8u;
        // descriptor of the first K = 16 step of the stage; the others differ in the address field only
        const uint64_t desc0 = smem_desc_k_sw128(smem_u32(a_ring) + s * (uint32_t)G::A_BYTES);
        const uint32_t slot_col = tmem_base + (uint32_t)G::A_COL0 + slot * (uint32_t)G::SLOT_COLS;
        const uint32_t a_tmem = slot_col + (uint32_t)(t * G::TILE_A_COLS);
        if constexpr (!SP) {
#pragma unroll
          for (int k2 = 0; k2 < KS; ++k2) {
            const int ks = h * KS + k2;
            const uint64_t bdesc = desc0 + (uint64_t)((ks >> 2) * half_step + (ks & 3) * 2);
            tc_mma_ts(d_tmem, a_tmem + ks * 8, bdesc, idesc, (fresh && k2 == 0) ? 0u : 1u);
          }
        } else {
          // 2:4 (Section 4): one instruction takes 32 rows of k (16 kept values per channel = 8 columns of
          // the slot) and the metadata column of that step; four steps per k-block
          const uint32_t e_tmem = slot_col + (uint32_t)(G::META_COL + t * 4);
#pragma unroll
          for (int k2 = 0; k2 < KS / 2; ++k2) {
            const int i = h * (KS / 2) + k2;
            const uint64_t bdesc = desc0 + (uint64_t)((i >> 1) * half_step + (i & 1) * 4);
            tc_mma_sp_ts(d_tmem, a_tmem + i * 8, bdesc, e_tmem + (uint32_t)(i & ~1), idesc | kIdescSparse | (uint32_t)(i & 1),
                         (fresh && k2 == 0) ? 0u : 1u);
          }
        }
      };
      if constexpr (DEF && G::ISSUERS == 1) {
        // Every k-block into the next accumulator of the ring.  The accumulators' round trip (wait, MMAs, completion, read-out,
        // release) bounds the loop, so the barriers of the next k-block are asked for behind the MMAs of this one, all in one go: one after
        // the other in front of the MMAs they took 250 cycles.
        if (mw == 0) {
          uint32_t s = 0, x_par = 0, slot = 0, a_par = 0, d = 0, d_par = 1;  // (the first filling of an accumulator waits for nothing)
          bool ready = false;
          for (uint32_t it = 0; it < total; ++it) {
            if (!ready) {
              mbar_wait(&xfull[s], x_par, abort_flag, p.status);
              mbar_wait(&afull[slot], a_par, abort_flag, p.status);
              mbar_wait(&dempty[d], d_par, abort_flag, p.status);
            }
            tc_fence_after_sync();
            issue(IntC<MPAD>{}, s, slot, tmem_base + d * (uint32_t)MPAD, true);
            const uint32_t d_now = d, s_now = s;
            if (++s == (uint32_t)AS) {
              s = 0;
              x_par ^= 1u;
            }
            if (++slot == (uint32_t)NSLOTS) {
              slot = 0;
              a_par ^= 1u;
            }
            if (++d == (uint32_t)G::ND) {
              d = 0;
              d_par ^= 1u;
            }
            ready = mbar_test3(&xfull[s], x_par, &afull[slot], a_par, &dempty[d], d_par);
            tc_commit(&dfull[d_now]);
            tc_commit(&mdone[s_now]);
          }
        }
      } else if constexpr (DEF) {
        // whole k-blocks, the two warps in turn, each into the next accumulator of the ring
        for (uint32_t it = mw; it < total; it += kMmaWarps) {
          const int s = (int)(it % AS), slot = (int)(it % NSLOTS), d = (int)(it % G::ND);
          if (it >= (uint32_t)G::ND) mbar_wait(&dempty[d], (it / G::ND - 1) & 1u, abort_flag, p.status);
          mbar_wait(&xfull[s], (it / AS) & 1u, abort_flag, p.status);
          mbar_wait(&afull[slot], (it / NSLOTS) & 1u, abort_flag, p.status);
          tc_fence_after_sync();
          issue(IntC<MPAD>{}, (uint32_t)s, (uint32_t)slot, tmem_base + (uint32_t)(d * MPAD), true);
          tc_commit(&dfull[d]);
          tc_commit(&mdone[s]);
        }
      } else {
        const uint32_t d_tmem = tmem_base + (uint32_t)((t * KH + h) * MPAD);
        auto run = [&](auto rows) {
          uint32_t it = 0, seg = 0;
          for (uint32_t u = u0; u < u1; ++seg) {
            const uint32_t len = min(KB - u % KB, u1 - u);
            // the accumulators are overwritten by the first MMA of the segment: the previous one must be read out
            if (seg > 0) mbar_wait(&dempty[t], (seg - 1) & 1u, abort_flag, p.status);
            for (uint32_t x = 0; x < len; ++x, ++it) {
              const int s = (int)(it % AS), slot = (int)(it % NSLOTS);
              mbar_wait(&xfull[s], (it / AS) & 1u, abort_flag, p.status);
              mbar_wait(&afull[slot], (it / NSLOTS) & 1u, abort_flag, p.status);
              tc_fence_after_sync();
              issue(rows, (uint32_t)s, (uint32_t)slot, d_tmem, x == 0);
              // one arrival when these MMAs are done: the slot may be rewritten, the activation tile refilled
              tc_commit(&mdone[s]);
              if (x + 1 == len) tc_commit(&dfull[t]);
            }
            u += len;
          }
        };
        // The rows as a constant where there are one or two of them: from a register they take the issuer, which is on the critical path
        // of a short launch, 1 to 4 % longer (4096 x 4096 at 64 rows 8.87 us so, 8.70 with the constant; a loop for each of 48 and 64 rows
        // costs as much again, 8.03 / 7.84 behind the other changes of that instance).  At 128 rows, where there are four, it does not show.
        if constexpr (G::FIXED_ROWS) {
          run(IntC<MPAD>{});
        } else if constexpr (MPAD == 32) {
          if (slab_rows == 16)
            run(IntC<16>{});
          else
            run(IntC<32>{});
        } else {
          run(Int{(int)slab_rows});
        }
      }
    }
    __syncwarp();
    if (p.cluster > 1) cluster_sync_all();  // every thread of every CTA of the cluster takes part
  } else {  // converters and drain: two roles with one end
  if (warp < G::CONV_WARPS) {
    // --------------------------------- converters ------------------------------------------------------------------
    if constexpr (G::CONV_REGS < kLaunchRegs) setmaxnreg_dec<G::CONV_REGS>();
    const uint32_t wg = (uint32_t)(warp >> 2);
    const uint32_t lane_win = (uint32_t)(warp & 3) * 32u;  // this warp's TMEM lanes
    const int n128 = (int)lane_win + lane;                 // channel of the thread inside a 128-channel tile
    const int j = (n128 & 63) >> 4, b = (n128 >> 3) & 1, g = n128 & 7;
    // the column's vectors in its 4096-byte chunk; position of its scale in the tile's row
    const uint32_t vec_off = (uint32_t)(n128 >> 6) * kChunkBytes + (uint32_t)(((2 * j + b) * 32 + 4 * g) * 16);
    const uint32_t spos = (uint32_t)((n128 & 64) + 8 * g + 2 * j + b);
    const uint32_t tmem_lane = tmem_base + (lane_win << 16);
    const uint32_t w_ring_s = smem_u32(w_ring);
    uint32_t it = wg;  // the warpgroups take the k-blocks in turn
    const uint32_t v0 = u0 / KB;
    uint32_t s_kb = u0 - v0 * KB, s_col = v0 / p.slabs, s_slab = v0 - s_col * p.slabs;  // where the next scales lie
    // The scales and zero points of the next k-block are loaded while this one is converted (from global memory: one line per
    // warp and tile; a bulk copy per k-block would cost its issuing warp more than all of the codes do).  The drain has
    // asked for them to be brought into the L2 (from DRAM they are 1500 cycles away).
    constexpr int SROWS = SUB ? 4 : 1;
    uint32_t sn[NT][SROWS] = {}, zn[NT][SROWS] = {};
    auto advance_scales = [&](uint32_t n) {
      s_kb += n;
      while (s_kb >= KB) {
        s_kb -= KB;
        if (++s_slab == p.slabs) { s_slab = 0; ++s_col; }
      }
    };
    auto load_scales = [&]() {
      if constexpr (SCALE != kPerColumn) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const uint32_t n0 = s_col * G::TN + (uint32_t)t * 128;
          if (n0 + (uint32_t)(n128 & 64) >= (uint32_t)p.N) continue;  // past the last column
          if constexpr (SUB) {
            const uint32_t sub = (uint32_t)p.sub_groups;
            const size_t at = ((size_t)s_kb * (p.N / 256) + n0 / 256) * sub * 256 + n0 % 256 + spos;
#pragma unroll
            for (uint32_t qd = 0; qd < 4; ++qd) {
              const size_t row = at + ((qd * sub) >> 2) * 256;
              sn[t][qd] = __ldg(reinterpret_cast<const uint16_t*>(p.sq) + row);
              if (zp) zn[t][qd] = __ldg(reinterpret_cast<const uint16_t*>(p.zq) + row);
            }
          } else {
            const uint32_t gi = p.group_shift >= 0 ? (s_kb >> p.group_shift) : (s_kb / (uint32_t)p.kb_per_group);
            const size_t at = (size_t)gi * p.N + n0 + spos;
            if constexpr (LOOP) sn[t][0] = __ldg(reinterpret_cast<const uint16_t*>(p.sq) + at);
            if (zp) zn[t][0] = __ldg(reinterpret_cast<const uint16_t*>(p.zq) + at);
          }
        }
      }
    };
    if (it < total) {
      advance_scales(it);
      load_scales();
    }

    // One tile of a k-block.  FAST: every scale of the warp's channels is in the range of dequant8_scaled and there are no zero
    // points.
    auto convert = [&](auto fast_c, int t, uint32_t wstage, uint32_t slot_col, const uint32_t (&sq)[4], const uint32_t (&zq4)[4]) {
      constexpr bool FAST = decltype(fast_c)::value;
      const uint32_t wbase = wstage + ((SP || W8) ? (uint32_t)(t * 128 + n128) * 16u : (uint32_t)t * 2 * kChunkBytes + vec_off);
      const uint32_t a_col = slot_col + (uint32_t)(t * G::TILE_A_COLS);
      if constexpr (W8) {
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          uint4 v[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) v[c] = lds128(wbase + (uint32_t)(4 * hh + c) * (G::TN * 16));  // rows 64hh + 16c ..
          uint32_t r[32];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t w4[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              // bytes (b0, b1) and (b2, b3) of the word under the exponent of 1024: 1024 + b, minus 1152 = b - 128
              const uint32_t lo = hsub2_u32(__byte_perm(w4[e], 0x64646464u, 0x4140), 0x64806480u);
              const uint32_t hi = hsub2_u32(__byte_perm(w4[e], 0x64646464u, 0x4342), 0x64806480u);
              r[8 * c + 2 * e] = LOOP ? hmul2_u32(lo, sq[2 * hh + (c >> 1)]) : lo;
              r[8 * c + 2 * e + 1] = LOOP ? hmul2_u32(hi, sq[2 * hh + (c >> 1)]) : hi;
            }
          }
          tc_st_x32(a_col + (uint32_t)(32 * hh), r);  // column = row / 2
        }
      } else if constexpr (SP) {
        const uint4 v[2] = {lds128(wbase), lds128(wbase + G::TN * 16)};  // kept values 0..31, 32..63 of the column
        const uint4 vm = lds128(wbase + (uint32_t)G::CODE_BYTES);         // the metadata words of this lane
        // 32 columns: column G holds the two kept values of the k-block's group G of four rows
        uint32_t r[32];
#pragma unroll
        for (int qd = 0; qd < 4; ++qd) {
          const uint4 vv = v[qd >> 1];
          const uint32_t w0 = (qd & 1) ? vv.z : vv.x, w1 = (qd & 1) ? vv.w : vv.y;
          if constexpr (FAST) {
            const uint32_t up = hmul2_u32(hmul2_u32(sq[qd], 0x64006400u), 0x64006400u), m8 = hmul2_u32(sq[qd], 0xc800c800u);
            dequant8_scaled(w0, r + 8 * qd, sq[qd], up, m8);
            dequant8_scaled(w1, r + 8 * qd + 4, sq[qd], up, m8);
          } else {
            uint32_t a0[4], a1[4];
            dequant8(w0, a0);
            dequant8(w1, a1);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              r[8 * qd + e] = LOOP ? hmul2_u32(a0[e], sq[qd]) : a0[e];
              r[8 * qd + 4 + e] = LOOP ? hmul2_u32(a1[e], sq[qd]) : a1[e];
            }
          }
        }
        tc_st_x32(a_col, r);
        const uint32_t mwords[4] = {vm.x, vm.y, vm.z, vm.w};
        tc_st_x4(slot_col + (uint32_t)(G::META_COL + t * 4), mwords);
      } else {
        uint4 v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = lds128(wbase + (uint32_t)(((c + (g >> 1)) & 3) * 16));  // rows 16c.. sit in slot (c + g/2) % 4
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          // 64 rows of k = 32 columns of the slot, written with one store
          uint32_t r[32];
#pragma unroll
          for (int qh = 0; qh < 2; ++qh) {
            const uint32_t s2 = sq[2 * hh + qh];
            // s * 2^20 and -8 s, or the subtrahends of the conversion: {1024 + z, 1024 + z} and {-(64 + z), -(64 + z)}, z = 8
            // without zero points
            uint32_t k0 = 0x64086408u, k1 = 0xd480d480u;
            if constexpr (FAST) {
              k0 = hmul2_u32(hmul2_u32(s2, 0x64006400u), 0x64006400u);
              k1 = hmul2_u32(s2, 0xc800c800u);
            } else if (zp) {
              k0 = hadd2_u32(zq4[2 * hh + qh], 0x64006400u);
              k1 = hsub2_u32(0xd400d400u, zq4[2 * hh + qh]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const uint4 vc = v[2 * qh + (e >> 1)];  // rows 64hh + 16c .., c = 2 qh + e / 2
              const uint32_t w = hh == 0 ? ((e & 1) ? vc.y : vc.x) : ((e & 1) ? vc.w : vc.z);
              uint32_t* out = r + 16 * qh + 4 * e;
              if constexpr (FAST) {
                dequant8_scaled(w, out, s2, k0, k1);
              } else {
                uint32_t a[4];
                dequant8_zp(w, a, k0, k1);
#pragma unroll
                for (int x = 0; x < 4; ++x) out[x] = LOOP ? hmul2_u32(a[x], s2) : a[x];
              }
            }
          }
          tc_st_x32(a_col + (uint32_t)(32 * hh), r);  // column = row / 2
        }
      }
    };
    auto convert_all = [&](auto fast_c, const uint32_t (&sq)[NT][4], const uint32_t (&zq4)[NT][4]) {
      const int s = (int)(it % WS), slot = (int)(it % NSLOTS);
      const uint32_t jt = it - NSLOTS;  // the k-block whose MMAs last read the slot
      if (G::W_GUARD && it >= (uint32_t)WS) mbar_wait(&wempty[s], (it / WS - 1) & 1u, abort_flag, p.status);
      mbar_wait(&wfull[s], (it / WS) & 1u, abort_flag, p.status);
      if (it >= (uint32_t)NSLOTS) mbar_wait(&mdone[jt % AS], (jt / AS) & 1u, abort_flag, p.status);
      tc_fence_after_sync();
#pragma unroll
      for (int t = 0; t < NT; ++t)
        convert(fast_c, t, w_ring_s + (uint32_t)s * G::W_BYTES, tmem_lane + (uint32_t)(G::A_COL0 + slot * G::SLOT_COLS), sq[t], zq4[t]);
      // The codes have been converted, so the shared loads that fetched them have certainly delivered: only now is
      // the stage released.  (An arrival issued right behind the loads can be performed before a multi-wavefront
      // shared load has read its data: a refill that followed at once overwrote codes still being read.)
      __syncwarp();
      if (lane == 0) mbar_arrive(&wempty[s]);
      tc_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&afull[slot]);
    };

    for (; it < total; it += G::CONV_GROUPS) {
      // the scales of rows 32 qd .. of the k-block, twice in a word, and likewise the zero points
      uint32_t sq[NT][4], zq4[NT][4];
      bool small = true;
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int qd = 0; qd < 4; ++qd) {
          sq[t][qd] = sn[t][SUB ? qd : 0] * 0x10001u;
          zq4[t][qd] = zn[t][SUB ? qd : 0] * 0x10001u;
          if (SUB || qd == 0) small = small && (sq[t][qd] & 0x7fffu) <= kFastScaleBits;
        }
      if (it + G::CONV_GROUPS < total) {
        advance_scales(G::CONV_GROUPS);
        load_scales();
      }
      if constexpr (LOOP && !W8) {
        if (__all_sync(0xffffffffu, small) != 0 && !zp)
          convert_all(BoolC<true>{}, sq, zq4);
        else
          convert_all(BoolC<false>{}, sq, zq4);
      } else {
        convert_all(BoolC<false>{}, sq, zq4);
      }
    }
  } else {
    // --------------------------------- drain: accumulators, fix-up, C ----------------------------------------------
    setmaxnreg_inc<G::DRAIN_REGS>();
    constexpr int kDrainThreads = G::DRAIN_WARPS * 32;
    const int dw = (warp - G::CONV_WARPS) & 3;                   // 32 channels of a tile
    constexpr int RBG = RB / G::DRAIN_GROUPS;                    // blocks of batch rows of a warpgroup, from b_first on
    const int b_first = (warp - G::CONV_WARPS) / 4 * RBG;
    const uint32_t tmem_lane = tmem_base + ((uint32_t)dw * 32u << 16);  // this warp's TMEM lanes = channels of a tile
    const int dtid = (int)threadIdx.x - G::CONV_WARPS * 32;
    auto release = [&](int d) {
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&dempty[d]);
    };
    // A finished tile to C: its fp16 blocks (eight rows x 32 channels in fragment order) into this warp's buffers, several of them
    // (put_block), then from there to C in runs of 64 bytes (write_blocks; 32 with the fused activation, applied on the way).
    // These warps get the issue slots that the converters leave: block after block, each a store, a warp barrier, a load and a store
    // to C that wait for one another, a tile of 128 rows took 4000 to 7000 cycles, and with two tiles the MMAs of the next
    // segment waited for the accumulators of the second one meanwhile (2:4, 2300 x 1024 x 4096: 21.9 us so, 15.7 this way;
    // 2048 x 4096 x 22016 226 / 218; 4-bit, 2048 x 1024 x 8192 44.7 / 38.4; 100 x 4096 x 12288 17.0 / 16.2).
    // The buffers of the converting warps are free here: those use theirs behind the block's barriers only.
    constexpr int kBufBlocks = imin(RBG, G::OUT_BYTES / G::DRAIN_WARPS / 512);
    const uint32_t tile_buf = smem_u32(smem) + G::BAR_BYTES + (uint32_t)((warp - G::CONV_WARPS) * kBufBlocks * 512);
    const uint32_t put_at = tile_buf + (uint32_t)((lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) * 16));
    auto put_block = [&](int x, const uint32_t (&r)[4]) { stmatrix_x4_trans(put_at + (uint32_t)(x * 512), r); };
    auto write_blocks = [&](auto count_c, int b0, int m_lim, size_t row0, uint32_t n0) {
      constexpr int COUNT = decltype(count_c)::value;
      __syncwarp();
      if (!p.swiglu) {
        const int row = lane >> 2, ch = lane & 3;
        const uint32_t from = tile_buf + (uint32_t)(row * 64 + ((ch ^ ((row >> 1) & 3)) * 16));
        uint16_t* c = p.C + (row0 + (size_t)(8 * b0 + row)) * ldc + n0 + ch * 8;
#pragma unroll
        for (int x = 0; x < COUNT; x += imin(COUNT, 4)) {
          uint4 v[imin(COUNT, 4)];
#pragma unroll
          for (int y = 0; y < imin(COUNT, 4); ++y) v[y] = lds128(from + (uint32_t)((x + y) * 512));
#pragma unroll
          for (int y = 0; y < imin(COUNT, 4); ++y)
            if ((b0 + x + y) * 8 + row < m_lim) *reinterpret_cast<uint4*>(c + (size_t)(8 * (x + y)) * ldc) = v[y];
        }
      } else {
        // two blocks at a time; of every 16 channels the gate piece and the up piece of a row lie side by side
        const int row = (lane & 15) >> 1, ch = lane & 1, half = lane >> 4;
        const uint32_t at = tile_buf + (uint32_t)(half * 512 + row * 64), turn = (uint32_t)((row >> 1) & 3);
        const uint32_t gate = at + (((uint32_t)(2 * ch) ^ turn) * 16), up = at + (((uint32_t)(2 * ch + 1) ^ turn) * 16);
        uint16_t* c = p.C + (row0 + (size_t)(8 * (b0 + half) + row)) * ldc + n0 / 2 + ch * 8;
#pragma unroll
        for (int x = 0; x < COUNT; x += 2) {
          const uint4 v = swiglu8(lds128(gate + (uint32_t)(x * 512)), lds128(up + (uint32_t)(x * 512)));
          if ((b0 + x + half) * 8 + row < m_lim) *reinterpret_cast<uint4*>(c + (size_t)(8 * x) * ldc) = v;
        }
      }
      __syncwarp();  // everybody has read: the buffers may be written again
    };
    uint32_t it = 0, seg = 0;
    bool waited_for_prior_grid = false;
    for (uint32_t u = u0; u < u1; ++seg) {
      // virtual column tile = (column tile of W, slab of batch rows): batches above MPAD rows replicate the
      // layer in the unit numbering (Section 3.4, last paragraph), slab after slab of one column tile
      const uint32_t vcol = u / KB;
      const uint32_t col = vcol / p.slabs, slab = vcol - col * p.slabs;
      const size_t row0 = (size_t)slab * slab_rows;
      const int m_lim = min(p.M - (int)row0, (int)slab_rows);  // rows of this slab that exist
      const uint32_t len = min(KB - u % KB, u1 - u);
      const uint32_t ncol0 = col * G::TN + (uint32_t)dw * 32;  // first channel of this warp in tile 0
      const int first_w = p.split ? (int)(vcol * p.split) : (int)stripe_owner32(vcol * KB, U, P);
      const int last_w = p.split ? (int)(vcol * p.split + p.split - 1) : (int)stripe_owner32((vcol + 1) * KB - 1, U, P);
      const bool shared_tile = !p.whole && last_w > first_w;
      auto before_first_write = [&]() {
        // first write to C or the workspace: the previous kernel of the stream must be done with them
        if (!waited_for_prior_grid) pdl_wait_prior_grids();
        waited_for_prior_grid = true;
      };
      if constexpr (SCALE != kPerColumn) {
        // the segment's scale rows (and zero points) into the L2, a line per lane: the converters and, with deferred scales, the
        // loop below will read them
        constexpr uint32_t LINES = G::TN * 2 / 128;
        const uint32_t rows = len * (SUB ? (uint32_t)p.sub_groups : 1u), kb0 = u % KB;
        for (uint32_t x = (uint32_t)dtid; x < rows * LINES; x += kDrainThreads) {
          const uint32_t row = x / LINES, line = x % LINES;
          const uint32_t c0 = col * G::TN + line * 64;
          if (c0 >= (uint32_t)p.N) continue;
          size_t at;
          if constexpr (SUB) {
            const uint32_t sub = (uint32_t)p.sub_groups;
            at = (((size_t)(kb0 + row / sub) * (p.N / 256) + c0 / 256) * sub + row % sub) * 256 + c0 % 256;
          } else {
            const uint32_t kb = kb0 + row;
            const uint32_t gi = p.group_shift >= 0 ? (kb >> p.group_shift) : (kb / (uint32_t)p.kb_per_group);
            at = (size_t)gi * p.N + c0;
          }
          asm volatile("prefetch.global.L2 [%0];" ::"l"(p.sq + at * 2));
          if (zp) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.zq + at * 2));
        }
      }
      if (!DEF && u + len == u1) break;  // the last tile: drain_last
      // where the partial tile goes, if this is one
      float4* part = p.cluster > 1 ? slot_ptr(worker) : (shared_tile ? stripe_slot((int)worker, vcol) : nullptr);

      if constexpr (DEF) {
        // sums of two neighbouring batch rows in a register pair: two rows to an instruction (fma.rn.f32x2)
        f32x2 acc2[RBG * 4];
#pragma unroll
        for (int e = 0; e < RBG * 4; ++e) acc2[e] = pack2(0.f, 0.f);
        // the scales of a k-block, loaded (from the L2, see above) while the one before is added
        auto load_scale = [&](uint32_t x) {
          uint2 v = make_uint2(0, 0);
          if (x < len && ncol0 < (uint32_t)p.N) {
            const uint32_t kb = u % KB + x;
            const uint32_t gi = p.group_shift >= 0 ? (kb >> p.group_shift) : (kb / (uint32_t)p.kb_per_group);
            v = __ldg(reinterpret_cast<const uint2*>(p.sq + ((size_t)gi * p.N + (size_t)col * G::TN) * 2 + spos2));
          }
          return v;
        };
        uint2 sv = load_scale(0);
        for (uint32_t x = 0; x < len; ++x, ++it) {
          const int d = (int)(it % G::ND);
          const float2 s01 = __half22float2(*reinterpret_cast<const __half2*>(&sv.x));
          const float2 s23 = __half22float2(*reinterpret_cast<const __half2*>(&sv.y));
          const f32x2 sc2[4] = {pack2(s01.x, s01.x), pack2(s01.y, s01.y), pack2(s23.x, s23.x), pack2(s23.y, s23.y)};
          sv = load_scale(x + 1);
          mbar_wait(&dfull[d], (it / G::ND) & 1u, abort_flag, p.status);
          tc_fence_after_sync();
          // (64 rows of a warpgroup: 32 at a time, to spare registers)
          constexpr int MG = RBG * 8, MC = imin(MG, 32);
#pragma unroll
          for (int m0 = 0; m0 < MG; m0 += MC) {
            float dd[MC / 16][2][8];
#pragma unroll
            for (int m = 0; m < MC / 16; ++m)
#pragma unroll
              for (int h = 0; h < 2; ++h)
                tc_ld_frag(tmem_lane + ((uint32_t)(16 * h) << 16) + (uint32_t)(d * MPAD + b_first * 8 + m0 + 16 * m), dd[m][h]);
            tc_wait_ld();
            if (m0 + MC == MG) release(d);
#pragma unroll
            for (int b = 0; b < MC / 8; ++b)
#pragma unroll
              for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                  const float* v = &dd[b >> 1][h][4 * (b & 1) + 2 * e];
                  f32x2& a = acc2[(m0 / 8 + b) * 4 + 2 * h + e];
                  a = fma2(sc2[2 * h + e], pack2(v[0], v[1]), a);
                }
          }
        }
        float acc[RBG * 8];
#pragma unroll
        for (int e = 0; e < RBG * 4; ++e) unpack2(acc2[e], acc[2 * e], acc[2 * e + 1]);
        before_first_write();
        if (part) {
#pragma unroll
          for (int b = 0; b < RBG; ++b)
            if ((b_first + b) * 8 < m_lim)
#pragma unroll
              for (int h = 0; h < 2; ++h)
                part[frag_index(dw, b_first + b, h)] =
                    make_float4(acc[8 * b + 4 * h], acc[8 * b + 4 * h + 1], acc[8 * b + 4 * h + 2], acc[8 * b + 4 * h + 3]);
        } else if (ncol0 < (uint32_t)p.N) {
#pragma unroll
          for (int b = 0; b < RBG; b += kBufBlocks)
            if ((b_first + b) * 8 < m_lim) {
#pragma unroll
              for (int x = 0; x < kBufBlocks; ++x) {
                uint32_t r[4];
                pack8(acc + 8 * (b + x), r);
                put_block(x, r);
              }
              write_blocks(IntC<kBufBlocks>{}, b_first + b, m_lim, row0, ncol0);
            }
        }
      } else {
#pragma unroll 1
        for (int t = 0; t < NT; ++t) {
          float sc[4];
          const uint32_t n0 = ncol0 + (uint32_t)t * 128;
          column_scales(col, t, sc);
          before_first_write();
          mbar_wait(&dfull[t], seg & 1u, abort_flag, p.status);
          tc_fence_after_sync();
          if (part) {
#pragma unroll 1  // (by two: 184 bytes of spills in the instance of 64 rows with one scale per column)
            for (int m = 0; m < (int)slab_rows; m += 16) {
              float f[16];
              load_rows(IntC<2>{}, t, m, sc, f);
              if (m + 16 >= (int)slab_rows) release(t);
#pragma unroll
              for (int b = 0; b < 2; ++b)
                if (m + 8 * b < m_lim)
#pragma unroll
                  for (int h = 0; h < 2; ++h)
                    part[frag_index(t * 4 + dw, m / 8 + b, h)] =
                        make_float4(f[8 * b + 4 * h], f[8 * b + 4 * h + 1], f[8 * b + 4 * h + 2], f[8 * b + 4 * h + 3]);
            }
          } else {
            // All of it out of tensor memory as fp16 first, as much as fits into the buffers and the rest into registers: the
            // MMAs of the next segment may start while C is written.
            constexpr int REST = RB - kBufBlocks;
            uint32_t rest[REST > 0 ? REST : 1][4];
#pragma unroll
            for (int m = 0; m < MPAD; m += 16) {
              if (MPAD == 128 && m >= (int)slab_rows) break;  // (what no MMA has written; what is put away of it is not stored)
              float f[16];
              load_rows(IntC<2>{}, t, m, sc, f);
#pragma unroll
              for (int b = 0; b < 2; ++b) {
                const int x = m / 8 + b;
                uint32_t r[4];
                pack8(f + 8 * b, r);
                if (x < kBufBlocks) {
                  put_block(x, r);
                } else {
#pragma unroll
                  for (int e = 0; e < 4; ++e) rest[x - kBufBlocks][e] = r[e];
                }
              }
            }
            release(t);
            if (n0 < (uint32_t)p.N) {
              write_blocks(IntC<kBufBlocks>{}, 0, m_lim, row0, n0);
              if constexpr (REST > 0) {
                if (kBufBlocks * 8 < m_lim) {
#pragma unroll
                  for (int x = 0; x < REST; ++x) put_block(x, rest[x]);
                  write_blocks(IntC<REST>{}, kBufBlocks, m_lim, row0, n0);
                }
              }
            }
          }
        }
      }

      if (p.cluster <= 1 && shared_tile && u + len < u1) {
        // not the CTA's last segment: the drain counts, and if it comes last it adds the partial tiles up alone
        const uint32_t fix = (uint32_t)p.ncols <= P ? vcol : (uint32_t)first_w;
        named_bar_sync(3, kDrainThreads);
        if (dtid == 0) {
          const int old = atom_add_acq_rel_gpu(&p.counters[fix], 1);
          const int is_last = (old == last_w - first_w) ? 1 : 0;
          if (is_last) p.counters[fix] = 0;
          *last_flag = is_last;
        }
        named_bar_sync(3, kDrainThreads);
        if (*last_flag != 0) {
          const int nb = (m_lim + 7) >> 3;
          sum_blocks(warp - G::CONV_WARPS, G::DRAIN_WARPS, nb * (G::TN / 32), nb, col, last_w - first_w + 1,
                     [&](int q) { return stripe_slot(first_w + q, vcol); },
                     [&](int c32, int b, const float (&f)[8], int i) { store_block(c32, b, f, i, col, m_lim, row0); });
        }
        named_bar_sync(3, kDrainThreads);  // last_flag may be rewritten by the next segment
      }
      u += len;
    }
    setmaxnreg_dec<G::CONV_REGS>();  // what follows is the converters' code as well
  }

  // --------------------------------- the end of the CTA's last tile ----------------------------------------------
  if constexpr (!DEF)
    drain_last(warp);
  else if (p.cluster > 1)
    finish_cluster(warp);
  else
    finish_stripe(warp);
  if (*abort_flag) {
    // a wait gave up: copies may still be in flight towards this CTA's shared memory
    for (int x = 0; x < 1000; ++x) __nanosleep(1000);
  }
  }

  // ---- the TMEM owner waits for everybody who touches tensor memory, then frees it ----
  tc_fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp0) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

template <int NT, int MPAD, int SCALE, int FMT>
cudaError_t launch(const GemmParams& p, cudaStream_t stream) {
  using G = Geometry<NT, MPAD, SCALE, FMT>;
  auto kernel = gemm_tc_kernel<NT, MPAD, SCALE, FMT>;
  const int workers = (int)p.workers;
  static bool attr_set[64] = {};
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (dev < 0 || dev >= 64 || !attr_set[dev]) {
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM_BYTES);
    if (err != cudaSuccess) return err;
    // the register split above counts on what the kernel is launched with
    cudaFuncAttributes fa;
    if ((err = cudaFuncGetAttributes(&fa, kernel)) != cudaSuccess) return err;
    if (fa.numRegs != kLaunchRegs) return cudaErrorInvalidConfiguration;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  alignas(64) CUtensorMap tmap;
  if (!make_a_tensor_map_3d(&tmap, p.A, p.M, p.K, (int)p.slab_rows)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(workers);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = G::SMEM_BYTES;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  GemmParams q = p;
  // Clusters of a split tile, if this device can co-schedule them (all of them at once: a GPC holds only so many
  // clusters of a size, and a second wave would cost far more than a smaller cluster); else the next smaller divisor.
  static int max_clusters[64][9] = {};  // per device and cluster size: clusters resident at once (0 unknown, -1 none)
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  for (; q.cluster > 1; --q.cluster) {
    if (q.split % q.cluster) continue;
    const int cs = (int)q.cluster;
    int nmax = (dev >= 0 && dev < 64) ? max_clusters[dev][cs] : 0;
    attr[1].val.clusterDim.x = (unsigned)cs;
    cfg.numAttrs = 2;
    if (nmax == 0) {
      int n = 0;
      nmax = (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0) ? n : -1;
      (void)cudaGetLastError();
      if (dev >= 0 && dev < 64) max_clusters[dev][cs] = nmax;
    }
    if (nmax > 0 && (long long)nmax * cs >= workers) break;
  }
  cfg.numAttrs = q.cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, q, tmap);
}

template <int NT, int SCALE, int FMT>
cudaError_t launch_mpad(int mpad, const GemmParams& p, cudaStream_t stream) {
  if (mpad == 32) return launch<NT, 32, SCALE, FMT>(p, stream);
  if (mpad == 64) return launch<NT, 64, SCALE, FMT>(p, stream);
  return launch<NT, 128, SCALE, FMT>(p, stream);
}
template <int NT, int FMT>
cudaError_t launch_scale(int mpad, int scale, const GemmParams& p, cudaStream_t stream) {
  if (scale == kInLoop) return launch_mpad<NT, kInLoop, FMT>(mpad, p, stream);
  if (scale == kPerColumn) return launch_mpad<NT, kPerColumn, FMT>(mpad, p, stream);
  if (scale == kInLoopSub) return launch_mpad<NT, kInLoopSub, FMT>(mpad, p, stream);
  return cudaErrorInvalidValue;
}

// one translation unit per format
cudaError_t launch_dense(int nt, int mpad, int scale, const GemmParams& p, cudaStream_t stream);
cudaError_t launch_sparse(int nt, int mpad, int scale, const GemmParams& p, cudaStream_t stream);
cudaError_t launch_w8(int nt, int mpad, int scale, const GemmParams& p, cudaStream_t stream);

}  // namespace tc
}  // namespace marlin_b200
