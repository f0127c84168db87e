// Persistent, SM-budgeted bf16 GEMM on the 5th-generation tensor cores (tcgen05) with the step's
// element-wise work fused into its epilogues.
//
//   tile        pair kernel (more than 128 tokens): 256 x 256 per PAIR of blocks (a cluster of two SMs,
//               tcgen05.mma.cta_group::2): each block stages its 128 token rows of A and ONE 128-row half
//               of B per 64-wide K block (32 KB, 6-stage ring), the leader block issues M256 N256 K16 MMAs
//               that read both blocks' shared memory, and each block owns the accumulator rows of its
//               SM's tensor memory.  Halving the B bytes per SM is what lifts the operand-feed limit of the
//               single-block kernel (128 x 256 tile, 48 KB per K block, 4-stage ring), which remains for
//               small token counts, for sm_budget 1 and for the K-split path; both produce the same bits.
//   operands    TMA (128-byte swizzle) -> shared-memory ring -> tcgen05.mma, fp32 accumulators in tensor
//               memory, two accumulator buffers so the epilogue of tile i overlaps the main loop of i+1
//   roles       warp 0: TMA producer, warp 1: MMA issuer (one thread, leader block only), warps 2..9:
//               epilogue, two per 32 rows of the accumulator.  Cross-block signalling in a pair: both blocks'
//               TMA bytes are counted on the leader's "full" barrier; the leader's tcgen05.commit arrives on the
//               "empty" and "accumulator full" barriers of both blocks; epilogue warps of both blocks arrive on the
//               leader's "accumulator empty" barrier.
//   schedule    unit = worker + i * workers, workers <= sm_budget (pairs: sm_budget / 2), one block per
//               SM.  Each output tile is produced by one block (pair) with a fixed K order, so results do
//               not depend on the budget.
//
// Epilogues: residual add (the fp32 tile is ADDED into the residual stream by a TMA reduction, so the
// stream is never read by the SM), QKV (rotate-half RoPE; a row's 64 contiguous bytes of q, k or v from the
// registers, k and v into the paged cache), gate/up (silu(gate) * up -> bf16 by TMA store).  Output blocks are staged in shared memory
// in the 128-byte-swizzled layout the tensor maps expect (conflict-free for one-row-per-thread writes).
#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "ptx.cuh"

namespace hs {
namespace {

static_assert(kGuMinWidth + 16 * kGuNarrow == 128, "a step of 16 columns from one width to the next");

constexpr int BM = 128, BN = 256, BK = 64;
constexpr int A_BYTES = BM * BK * 2;            // 16 KB
constexpr int BH_BYTES = 128 * BK * 2;          // one 128-row half of the B tile, 16 KB
// One block per tile: a stage holds A and both halves of B, 4 stages.  Block pair per 256 x 256 tile: every
// block stages A and ONE half of B (the MMA reads the other half from the other block), 6 stages.
template <bool PAIR> struct Ring {
  static constexpr int STAGE_BYTES = PAIR ? A_BYTES + BH_BYTES : A_BYTES + 2 * BH_BYTES;
  static constexpr int STAGES = PAIR ? 6 : 4;
};
constexpr int RING_BYTES = 4 * (A_BYTES + 2 * BH_BYTES);
static_assert(Ring<true>::STAGES * Ring<true>::STAGE_BYTES == RING_BYTES, "both rings fill the same space");
constexpr int kMaxStages = 12;                  // barrier slots; the ring holds fewer when stages are large
constexpr int EPI_WARPS = 8, GEMM_THREADS = 64 + EPI_WARPS * 32;
constexpr int TMEM_COLS = 512;                  // two 128 x 256 fp32 accumulators
constexpr int EPI_BUF_BYTES = 4096;             // 32 rows x 128 B: a 32 x 32 fp32 or 32 x 64 bf16 output block
constexpr int EPI_BYTES = EPI_WARPS * EPI_BUF_BYTES;   // one block per epilogue warp
constexpr int GEMM_SMEM = 1024 + RING_BYTES + EPI_BYTES + 384;
static_assert(GEMM_SMEM <= 227 * 1024, "fits one SM");
static_assert(GEMM_SMEM >= kMinSmemBytes, "one block per SM");

// Qkv mode, single blocks: tiles of 128 virtual columns (one B box) when p.bn says so -- a step asks for
// them, since the tile count decides how many SMs stream weights; 256 otherwise.  A 128-column
// tile never straddles q | k | v (their widths are multiples of 128) and holds whole heads.
// Pairs: 256, or 192 where p.bn says so (gemm_pick_pair_qkv_width).  Such a tile is three units of two 32-column pieces that rotate
// with each other, 32 p .. of the two halves of a head; each piece is a B box of its own, so that a tile may begin and end inside a
// head or a projection.  Single blocks also have tiles of one such unit (gemm_pick_qkv_width).
constexpr int QKV_NARROW = 192, QKV_UNIT = 64;
__host__ __device__ __forceinline__ int gemm_qkv_width(const GemmParams& p) {
  return p.pair ? (p.bn == QKV_NARROW ? QKV_NARROW : BN) : p.bn == 128 || p.bn == QKV_UNIT ? p.bn : BN;
}
// First column of unit u of [q | k | v]; its partners are half a head further.
__device__ __forceinline__ int qkv_unit_col(const GemmParams& p, int u) {
  return p.head_dim == 128 ? (u >> 1) * 128 + (u & 1) * 32 : u * 64;
}

// GateUp mode: activation columns of a tile, 128 or p.gu_width.
__host__ __device__ __forceinline__ int gemm_gu_width(const GemmParams& p) { return p.gu_width > 0 ? p.gu_width : 128; }

// Output-tile width: 256 virtual columns, except in Resid mode where the launcher picks p.bn (a multiple
// of 32 in [128, 256]) from the problem shape so that the tile count fills whole waves of SMs, and in GateUp mode.
__host__ __device__ __forceinline__ int gemm_n_tiles(const GemmParams& p) {
  if (p.mode == kGemmGateUp) return (p.N + gemm_gu_width(p) - 1) / gemm_gu_width(p);
  const int bn = p.mode == kGemmResid ? p.bn : gemm_qkv_width(p);
  return (p.N + bn - 1) / bn;
}

struct BSource { int map, row; };
__device__ __forceinline__ BSource qkv_source(const GemmParams& p, int v) {
  if (v < p.q_dim) return {0, v};
  v -= p.q_dim;
  if (v < p.kv_dim) return {1, v};
  return {2, v - p.kv_dim};
}
__device__ __forceinline__ BSource b_source(const GemmParams& p, int n_tile, int half, int qkv_width) {
  if (p.mode == kGemmResid) return {0, n_tile * p.bn + half * 128};
  if (p.mode == kGemmGateUp) return {half, n_tile * gemm_gu_width(p)};
  return qkv_source(p, n_tile * qkv_width + half * 128);
}
// Piece `piece` of a tile of `units` units (past the end of v the boxes lie outside the matrix and read zeros)
__device__ __forceinline__ BSource qkv_piece(const GemmParams& p, int n_tile, int units, int piece) {
  return qkv_source(p, qkv_unit_col(p, n_tile * units + (piece >> 1)) + (piece & 1) * (p.head_dim >> 1));
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

__device__ __forceinline__ void st_global_32b(void* dst, const uint32_t (&w)[8]) {      // a lane's whole sector
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
               "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
// n_valid (a multiple of 8) of 32 values of one row -> 16-bit values at dst: 32-byte stores where dst is aligned to that.
__device__ __forceinline__ void store_act32(__nv_bfloat16* dst, const float (&v)[32], bool f16, int n_valid) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = pack_act(v[i * 16 + 2 * e], v[i * 16 + 2 * e + 1], f16);
    if (16 * i + 16 <= n_valid && (reinterpret_cast<uintptr_t>(dst) & 31) == 0) {
      st_global_32b(dst + 16 * i, w);
    } else {
      if (16 * i + 8 <= n_valid) *reinterpret_cast<uint4*>(dst + 16 * i) = make_uint4(w[0], w[1], w[2], w[3]);
      if (16 * i + 16 <= n_valid) *reinterpret_cast<uint4*>(dst + 16 * i + 8) = make_uint4(w[4], w[5], w[6], w[7]);
    }
  }
}
// 32 fp32 values (raw bits) of one row -> 64 contiguous bytes of bf16, 32-byte aligned.
__device__ __forceinline__ void store_bf16x32(__nv_bfloat16* dst, const uint32_t (&r)[32]) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = pack_bf16(__uint_as_float(r[i * 16 + 2 * e]), __uint_as_float(r[i * 16 + 2 * e + 1]));
    st_global_32b(dst + 16 * i, w);
  }
}

// Staging layout of an output block: row r (one thread of the warp) is 128 bytes = 8 units of 16 B,
// unit u stored at r * 128 + ((u ^ (r & 7)) << 4): the 128-byte swizzle of the output tensor maps.
__device__ __forceinline__ void stage_f32x32(uint8_t* buf, int lane, const uint32_t (&r)[32]) {
#pragma unroll
  for (int u = 0; u < 8; ++u)
    *reinterpret_cast<uint4*>(buf + lane * 128 + ((u ^ (lane & 7)) << 4)) =
        make_uint4(r[4 * u], r[4 * u + 1], r[4 * u + 2], r[4 * u + 3]);
}
// 32 values -> bf16 into units u0 .. u0+3 of the thread's row (u0 = 0 or 4: which 32 of the 64 columns).
__device__ __forceinline__ void stage_bf16x32(uint8_t* buf, int lane, int u0, const float (&v)[32], bool f16 = false) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint4 w;
    w.x = pack_act(v[i * 8 + 0], v[i * 8 + 1], f16);
    w.y = pack_act(v[i * 8 + 2], v[i * 8 + 3], f16);
    w.z = pack_act(v[i * 8 + 4], v[i * 8 + 5], f16);
    w.w = pack_act(v[i * 8 + 6], v[i * 8 + 7], f16);
    *reinterpret_cast<uint4*>(buf + lane * 128 + (((u0 + i) ^ (lane & 7)) << 4)) = w;
  }
}

__device__ __forceinline__ void ldg_f32x8(float (&t)[8], const float2* src) {      // 32 bytes, 32-byte aligned, read-only data
  asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(t[0]), "=f"(t[1]), "=f"(t[2]), "=f"(t[3]), "=f"(t[4]), "=f"(t[5]), "=f"(t[6]), "=f"(t[7])
               : "l"(src));
}

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Bounded spin on a global word written by another block (same limits as the mbarrier waits).
__device__ __forceinline__ bool spin_until_equal(const int* word, int value, volatile int* abort_flag, int* status) {
  const unsigned long long t0 = globaltimer_ns();
  for (uint32_t spins = 0;; ++spins) {
    if (ld_acquire(word) == value) return true;
    if ((spins & 0x3f) == 0x3f) {
      if (*abort_flag) return false;
      if (globaltimer_ns() - t0 > kWaitLimitNs) {
        *abort_flag = 1;
        atomicExch(status, kErrTimeout);
        return false;
      }
      __nanosleep(100);
    }
  }
}

// r[0..31] += b[0..31]: fp32 values held as raw bits, bias in bf16 (64-byte aligned; the same for every row,
// so the loads of a warp are broadcasts out of the L1).
__device__ __forceinline__ void add_bias32(uint32_t (&r)[32], const __nv_bfloat16* b) {
  const uint4* src = reinterpret_cast<const uint4*>(b);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const uint4 w = __ldg(src + u);
    const uint32_t pk[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      r[u * 8 + 2 * e] = __float_as_uint(__uint_as_float(r[u * 8 + 2 * e]) + __uint_as_float(pk[e] << 16));
      r[u * 8 + 2 * e + 1] = __float_as_uint(__uint_as_float(r[u * 8 + 2 * e + 1]) + __uint_as_float(pk[e] & 0xffff0000u));
    }
  }
}

// r[0..31] *= s (fp32 values held as raw bits)
__device__ __forceinline__ void scale32(uint32_t (&r)[32], float s) {
#pragma unroll
  for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * s);
}

// Folded RMSNorm, producing side: a thread leaves the sum of x^2 of its row over one tile column; the warp that
// delivers the last tile column of its 32 rows (counted per row group) adds each row's partials in tile-column order --
// the same sum whoever comes last -- and writes r = rsqrt(mean(x^2) + eps) for the GEMM that follows.
__device__ __forceinline__ void finish_row_norm(const GemmParams& p, int row, bool row_ok, int row_group, int n,
                                                int n_n_tiles, float ss, int lane) {
  if (row_ok) p.row_ss[size_t(row) * p.ss_stride + n] = ss;
  __syncwarp();
  // (One lane's count releases the warp's partials and acquires the others'.  A fence of every lane on both sides: out and down of a
  // small backbone, 5776 rows, 61.6 and 99.7 us instead of 60.6 and 98.7.)
  int last = 0;
  if (lane == 0) {
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(last) : "l"(p.row_group_done + row_group) : "memory");
    last = last == n_n_tiles - 1;
  }
  last = __shfl_sync(0xffffffffu, last, 0);
  if (!last) return;
  __syncwarp();
  if (row_ok) {
    float sum = 0.f;
    for (int i = 0; i < n_n_tiles; ++i) sum += __ldcg(p.row_ss + size_t(row) * p.ss_stride + i);
    p.row_rs[row] = rsqrtf(sum / float(p.N) + p.norm_eps);
  }
  if (lane == 0) p.row_group_done[row_group] = 0;      // ready for the next launch
}

// Address of element e of (slot, kv head) in one layer's K or V pages.
__device__ __forceinline__ __nv_bfloat16* cache_ptr(__nv_bfloat16* base, int slot, int hk, int n_kv_heads, int Dh,
                                                    int e) {
  const size_t row = (size_t(slot >> 4) * n_kv_heads + hk) * 16 + (slot & 15);
  return base + row * Dh + e;
}

// One work unit of a block (pair): the K blocks [kb_begin, kb_end) of an output tile.  `seg` counts the earlier K
// segments of the same tile (their sums are added into the output before this one's), `last` marks the tile's final
// segment.
struct Unit { int tile, kb_begin, kb_end, seg, last, half; };

// Hands a worker its units, in the same order for the producer, the MMA issuer and the epilogue warps.
//   plain / split-K   unit u = worker + i * workers over tiles x splits, split-major (a split's predecessors have
//                     smaller unit numbers).
//   stream-K          (Resid mode on pairs, chosen by shape) the tiles' K blocks, laid end to end tile after tile, are
//                     cut into `n_slots` equal runs -- one per pair of the whole device, whatever the budget -- so that
//                     no pair idles through a ragged last wave.  A run is a tail segment of one tile, whole tiles, and
//                     a head segment of another; slot s is worked by worker s mod workers.  Within a slot the head
//                     segment comes first and the tail segment last: the tail's predecessor is the head segment of
//                     the previous slot, which that slot has done first, so the ordered add never waits long.
//                     With sm_budget 1 there is no pair: the single block then works the same slots on the same
//                     256-row tiles, each unit twice -- once per 128-row half (`half`) -- so that every output
//                     element still receives the same partial sums in the same order.
struct UnitWalk {
  int stream_k, parts, n_tiles, k_blocks, ksplit, n_workers, n_slots;
  int halves, n_m_tiles, M;  // halves = 2: a single block standing in for a pair
  int cur;                 // unit (plain) or slot (stream-K) being handed out
  int idx, n_seg, first_tile;
  long long lo, hi;
  __device__ __forceinline__ void init(const GemmParams& p, bool pair, bool emulate_pair, int n_m_tiles_, int n_tiles_,
                                       int k_blocks_, int worker, int n_workers_) {
    stream_k = (pair || emulate_pair) && p.mode == kGemmResid && p.stream_k_slots > 0;
    parts = p.mode == kGemmResid && p.part_rows > 0;
    halves = emulate_pair ? 2 : 1;
    n_m_tiles = n_m_tiles_;
    M = p.M;
    n_tiles = n_tiles_; k_blocks = k_blocks_; n_workers = n_workers_;
    ksplit = (!pair || parts) && p.mode == kGemmResid && p.ksplit > 1 ? p.ksplit : 1;
    n_slots = stream_k ? p.stream_k_slots : n_tiles * ksplit;
    cur = worker - n_workers;
    idx = n_seg = 0; first_tile = 0; lo = hi = 0;
  }
  __device__ __forceinline__ bool next(Unit& u) {
    if (halves == 2 && idx > 0 && u.half == 0) {   // the second half of the unit handed out last, if it has rows
      if ((2 * (u.tile % n_m_tiles) + 1) * BM < M) {
        u.half = 1;
        return true;
      }
    }
    u.half = 0;
    if (!stream_k) {
      cur += n_workers;
      if (cur >= n_slots) return false;
      const int ks = cur / n_tiles;
      u.tile = cur - ks * n_tiles;
      u.kb_begin = parts ? k_blocks * ks / ksplit : gemm_split_begin(k_blocks, ksplit, ks);
      u.kb_end = parts ? k_blocks * (ks + 1) / ksplit : gemm_split_begin(k_blocks, ksplit, ks + 1);
      u.seg = ks;
      u.last = ks == ksplit - 1;
      return true;
    }
    const long long total = (long long)n_tiles * k_blocks;
    while (idx == n_seg) {                         // next slot of this worker (empty slots are skipped)
      cur += n_workers;
      if (cur >= n_slots) return false;
      lo = total * cur / n_slots;
      hi = total * (cur + 1) / n_slots;
      idx = 0;
      n_seg = 0;
      if (hi > lo) {
        first_tile = int(lo / k_blocks);
        n_seg = int((hi - 1) / k_blocks) - first_tile + 1;
      }
    }
    const int nat = n_seg == 1 ? 0 : (idx == 0 ? n_seg - 1 : (idx == n_seg - 1 ? 0 : idx));
    const int t = first_tile + nat;
    const long long t0 = (long long)t * k_blocks;
    const long long b = lo > t0 ? lo : t0, e = hi < t0 + k_blocks ? hi : t0 + k_blocks;
    u.tile = t;
    u.kb_begin = int(b - t0);
    u.kb_end = int(e - t0);
    // earlier segments of the tile = slot boundaries inside the tile before this segment; the slot that holds the
    // tile's first K block is ceil((t0 + 1) n_slots / total) - 1
    u.seg = u.kb_begin == 0 ? 0 : cur - (int(((t0 + 1) * n_slots + total - 1) / total) - 1);
    u.last = u.kb_end == k_blocks;
    ++idx;
    return true;
  }
};

// (One instantiation per mode: an epilogue does not pay with registers for the others.  UNIT: Qkv tiles of 64 columns on single blocks.  In
// one instantiation with the others, and with a tile width that the pairs' read from the parameters alike, those cost every launch:
// denoising step, 1024 rows on pairs 892.2 -> 884.5 us.)
template <bool PAIR, int MODE, bool UNIT = false>
__device__ __forceinline__ void gemm_body(const GemmParams& p) {
  const int qkv_width = PAIR ? (p.bn == QKV_NARROW ? QKV_NARROW : BN) : UNIT ? QKV_UNIT : p.bn == 128 ? 128 : BN;      // (Qkv mode)
  // Ring geometry.  Pairs: 6 stages of 32 KB.  Single blocks: a stage holds the A box (128 rows, or only 64 / 32
  // when the step is that small) and one or two 128-row B boxes, and the ring holds as many stages as fit (at
  // most kMaxStages): a block's streaming rate is stages in flight / memory latency, so the small stages of a
  // small step buy depth -- 8 or 9 stages instead of 4.
  const bool b_two = MODE == kGemmGateUp || (MODE == kGemmResid ? p.bn > 128 : UNIT || qkv_width > 128);   // (64 columns: two pieces of 32)
  const int a_bytes = (p.a_box_rows > 0 && !PAIR ? p.a_box_rows : BM) * BK * 2;
  // (a narrow GateUp tile: its gate rows, and right behind them -- in a pair, in the other block -- its up rows, one operand of
  // 2 gu_w rows)
  const int gu_w = MODE == kGemmGateUp ? gemm_gu_width(p) : 128;
  const int bh_bytes = (MODE != kGemmQkv ? gu_w : PAIR ? qkv_width / 2 : UNIT ? 32 : 128) * BK * 2;
  constexpr int narrow_units = PAIR ? 3 : 1, pieces = PAIR ? 3 : 2;      // of a narrow tile, and of those a block's
  const bool qkv_narrow = UNIT || (PAIR && MODE == kGemmQkv && qkv_width == narrow_units * QKV_UNIT);
  const int STAGE_BYTES = PAIR ? Ring<true>::STAGE_BYTES : a_bytes + (b_two ? 2 : 1) * bh_bytes;
  // (a pair kernel that folds the following RMSNorm into its epilogue runs its ring one stage short and uses the last
  // stage's 32 KB as landing blocks for the residual stream: see the epilogue)
  const bool fold_pair = PAIR && MODE == kGemmResid && p.norm_gain != nullptr;
  const int STAGES = PAIR ? Ring<true>::STAGES - (fold_pair ? 1 : 0)
                          : (RING_BYTES / STAGE_BYTES < kMaxStages ? RING_BYTES / STAGE_BYTES : kMaxStages);
  const int b_off = PAIR ? A_BYTES : a_bytes;     // B boxes follow the A box inside a stage
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* epi_smem = smem + RING_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(epi_smem + EPI_BYTES);
  uint64_t* empty = full + kMaxStages;
  uint64_t* tfull = empty + kMaxStages;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint64_t* xbar = reinterpret_cast<uint64_t*>(epi_smem + EPI_BYTES + 256);   // [4 warps][4] landing-block barriers (three used)

  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (uniform)
  // Residual GEMMs on pairs, and those that fold the norm, leave the second warps of the quarters idle: their epilogue is bound by
  // the residual stream's way through shared memory, and the idle warps' staging blocks serve the first (both at work with a
  // block each: out and down at 7B dimensions, 2112 rows, 224 -> 230 us on average, partial sums of 401 rows 49.0 -> 49.8).
  const bool solo = MODE == kGemmResid && (PAIR || p.norm_gain != nullptr);
  log_smid(p.smid_log);
  // In pair mode the two blocks of a cluster share every work unit: a unit's tile is 256 rows tall and
  // block `rank` owns rows 128 * rank .. 128 * rank + 127 of it.
  const uint32_t rank = PAIR ? blockIdx.x & 1 : 0;              // (clusters of two along x)
  const int worker = PAIR ? int(blockIdx.x >> 1) : int(blockIdx.x);
  const int n_workers = PAIR ? int(gridDim.x >> 1) : int(gridDim.x);
  // a single block that stands in for a pair (stream-K form at sm_budget 1) walks the pair's 256-row tiles
  const bool emulate_pair = !PAIR && p.pair && MODE == kGemmResid && p.stream_k_slots > 0;
  const int n_m_tiles = PAIR || emulate_pair ? (p.M + 2 * BM - 1) / (2 * BM) : (p.M + BM - 1) / BM;
  const int n_n_tiles = MODE == kGemmQkv ? (p.N + qkv_width - 1) / qkv_width : gemm_n_tiles(p);
  const int n_tiles = n_m_tiles * n_n_tiles;
  const int k_blocks = (p.K + BK - 1) / BK;
  // Work unit = (output tile, run of K blocks): see UnitWalk.  Runs shorter than the whole K range exist only in
  // Resid mode, whose epilogue adds partial sums into the output in a fixed order.
  UnitWalk walk;
  walk.init(p, PAIR, emulate_pair, n_m_tiles, n_tiles, k_blocks, worker, n_workers);
  const bool ordered = !walk.parts && (walk.stream_k || walk.ksplit > 1);
  Unit un;

  // (a lane per barrier: a block that starts when its predecessor's leaves has its set-up, 2 us of it, on the critical path)
  if (warp == 0) {
    if (lane < STAGES) {
      mbar_init(&full[lane], 1);
      mbar_init(&empty[lane], 1);
    } else if (lane >= 16 && lane < 18) {
      mbar_init(&tfull[lane - 16], 1);
      mbar_init(&tempty[lane - 16], (PAIR ? 2 : 1) * (solo ? EPI_WARPS / 2 : EPI_WARPS));   // one arrival per epilogue warp (of both blocks)
    } else if (lane == 18) {
      *abort_flag = 0;
    }
    if (lane >= 16) mbar_init(&xbar[lane - 16], 1);
    fence_barrier_init();
  } else if (warp == 2) {
    if (lane == 0) tma_prefetch_desc(&p.tm_a);
    if (lane == 1) tma_prefetch_desc(&p.tm_b[0]);
    if (lane == 2 && MODE != kGemmQkv) tma_prefetch_desc(MODE == kGemmResid ? &p.tm_out : &p.tm_act);
  }
  if (warp == 1) {
    if (PAIR) {
      tmem_alloc_pair(tmem_slot, TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, TMEM_COLS);
      tmem_relinquish();
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (PAIR) cluster_sync_all();               // the other block's barriers exist before anything targets them
  tc_fence_after_sync();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  // A small step's A box holds only the rows that exist (32 or 64 instead of 128): the MMA still reads 128
  // rows starting at the stage's base -- beyond the A box that is the B data of the stage, finite values
  // that only reach accumulator rows no epilogue stores
  const bool two_halves = b_two;
  // One stage's requests of the producer thread: the weight boxes (which also arm the barrier) and the A box.  In a
  // pair both blocks' bytes are counted on the leader's barrier, which the leader arms for both.
  auto load_b = [&](int s, int kb, const BSource& b0, const BSource& b1, const BSource& b2) {
    uint8_t* st = smem + s * STAGE_BYTES;
    if (PAIR) {
      if (rank == 0) mbar_expect_tx(&full[s], 2 * (A_BYTES + bh_bytes));
      const uint32_t bar = mapa_u32(smem_u32(&full[s]), 0);
      tma_load_2d_pair(st + b_off, &p.tm_b[b0.map], bar, kb * BK, b0.row);
      if (qkv_narrow) {
        tma_load_2d_pair(st + b_off + 32 * BK * 2, &p.tm_b[b1.map], bar, kb * BK, b1.row);
        tma_load_2d_pair(st + b_off + 64 * BK * 2, &p.tm_b[b2.map], bar, kb * BK, b2.row);
      }
    } else {
      mbar_expect_tx(&full[s], a_bytes + (two_halves ? 2 * bh_bytes : bh_bytes));
      tma_load_2d(st + b_off, &p.tm_b[b0.map], &full[s], kb * BK, b0.row);
      if (two_halves) tma_load_2d(st + b_off + bh_bytes, &p.tm_b[b1.map], &full[s], kb * BK, b1.row);
    }
  };
  auto load_a = [&](int s, int kb, int m, int half) {
    uint8_t* st = smem + s * STAGE_BYTES;
    if (PAIR) tma_load_2d_pair(st, &p.tm_a, mapa_u32(smem_u32(&full[s]), 0), kb * BK, (2 * m + int(rank)) * BM);
    else tma_load_2d(st, &p.tm_a, &full[s], kb * BK, (emulate_pair ? 2 * m + half : m) * BM);
  };
  // The weights never change: the producer asks for the weight boxes of its first unit's first stages before the wait
  // for the previous kernel, and for the A boxes of those stages after it.
  bool have_unit = false;
  int b_ahead = 0;
  if (warp == 0) {
    have_unit = walk.next(un);
    if (have_unit) {
      const int n = un.tile / n_m_tiles;
      const BSource b0 = qkv_narrow ? qkv_piece(p, n, narrow_units, pieces * int(rank)) : b_source(p, n, PAIR ? int(rank) : 0, qkv_width);
      const BSource b1 = qkv_narrow ? qkv_piece(p, n, narrow_units, pieces * int(rank) + 1) : b_source(p, n, 1, qkv_width);
      const BSource b2 = PAIR && qkv_narrow ? qkv_piece(p, n, narrow_units, pieces * int(rank) + 2) : b1;
      b_ahead = un.kb_end - un.kb_begin < STAGES ? un.kb_end - un.kb_begin : STAGES;
      if (elect_one())
        for (int i = 0; i < b_ahead; ++i) load_b(i, un.kb_begin + i, b0, b1, b2);
    }
  }
  griddep_wait();                 // everything above is set-up; the operands belong to the previous kernel until here
  griddep_launch_dependents(p.overlap);

  // The producer and the MMA issuer are whole warps in uniform control flow, one elected lane issuing: the descriptors,
  // coordinates and barrier addresses then live in uniform registers.  With a loop inside `if (lane == 0)` every
  // instruction fetched its operands through a move of its own, about 60 cycles per MMA, and the issuing thread was
  // what bounded the main loop (it never waited for data): 565 cycles per 64-wide K block for 128 columns and for pairs
  // alike; now 405 and 520 (a pair's tensor time is 512).
  if (warp == 0) {
    // ------------------------------------------------------- TMA producer --
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    while (ok && have_unit) {
      const int tile = un.tile;
      const int m = tile % n_m_tiles, n = tile / n_m_tiles;
      const BSource b0 = qkv_narrow ? qkv_piece(p, n, narrow_units, pieces * int(rank)) : b_source(p, n, PAIR ? int(rank) : 0, qkv_width);
      const BSource b1 = qkv_narrow ? qkv_piece(p, n, narrow_units, pieces * int(rank) + 1) : b_source(p, n, 1, qkv_width);
      const BSource b2 = PAIR && qkv_narrow ? qkv_piece(p, n, narrow_units, pieces * int(rank) + 2) : b1;
      const int kb_end = un.kb_end;
      for (int kb = un.kb_begin; kb < kb_end; ++kb) {
        ok = mbar_wait(&empty[s], ph ^ 1, abort_flag, p.status);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        if (elect_one()) {
          if (b_ahead == 0) load_b(s, kb, b0, b1, b2);
          load_a(s, kb, m, un.half);
        }
        if (b_ahead > 0) --b_ahead;
        if (++s == STAGES) { s = 0; ph ^= 1; }
      }
      have_unit = walk.next(un);
    }
  } else if (warp == 1) {
    // --------------------------------------------------------- MMA issuer --
    if (rank == 0) {
      // both operands are fp16 or both bf16 (one MMA cannot mix the two): the format fields of A (bits 7..9)
      // and B (bits 10..12) are 0 for fp16 and 1 for bf16
      const uint32_t idesc = umma_idesc_bf16_f32(PAIR ? 2 * BM : BM,
                                                 MODE == kGemmGateUp ? 2 * gu_w : MODE == kGemmQkv ? qkv_width : PAIR ? BN : p.bn) &
                             (p.ab_f16 ? ~(63u << 7) : ~0u);
      int s = 0, acc = 0;
      uint32_t ph = 0, acc_ph = 0;
      bool ok = true;
      const uint64_t a_desc0 = umma_desc_kmajor_sw128(smem_u32(smem));
      while (ok && walk.next(un)) {
        ok = mbar_wait(&tempty[acc], acc_ph ^ 1, abort_flag, p.status);
        if (!__all_sync(0xffffffffu, ok)) break;
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + acc * BN;
        const int kb_begin = un.kb_begin, kb_end = un.kb_end;
        for (int kb = kb_begin; kb < kb_end; ++kb) {
          ok = mbar_wait(&full[s], ph, abort_flag, p.status);
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
          tc_fence_after_sync();
          // descriptors of stage s: those of stage 0 plus the stage's offset in the address field (units of 16 bytes;
          // shared memory is below 256 KB, so nothing carries out of the field)
          const uint64_t a_desc = a_desc0 + uint64_t(s * (STAGE_BYTES >> 4));
          const uint64_t b_desc = a_desc + uint64_t(b_off >> 4);
          const uint32_t acc0 = kb != kb_begin ? 1u : 0u;
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {  // 16 bf16 = 32 B along K: +2 in the (address / 16) field
              if (PAIR) umma_bf16_pair(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, k != 0 ? 1u : acc0);
              else umma_bf16(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, k != 0 ? 1u : acc0);
            }
            // frees the stage (in both blocks) once these MMAs have read it
            if (PAIR) umma_commit_pair_both(&empty[s]);
            else umma_commit(&empty[s]);
          }
          if (++s == STAGES) { s = 0; ph ^= 1; }
        }
        if (ok && elect_one()) {
          if (PAIR) umma_commit_pair_both(&tfull[acc]);
          else umma_commit(&tfull[acc]);
        }
        acc ^= 1;
        if (acc == 0) acc_ph ^= 1;
      }
    }
  } else {
    // ----------------------------------------------------------- epilogue --
    // Two warps per quarter, each with half of the tile's columns: an epilogue is a chain of latencies (tensor memory,
    // shared memory, stores) of one warp per scheduler otherwise, and where a GEMM has a tile or two per SM it is exposed.
    // Measured on B200, 1024 conditioned rows of d = 1024, per launch: QKV 18.7 -> 15.5 us, with 32-byte loads of the rotation
    // and 32-byte stores (a lane's whole sector: its row is its own), out-projection 11.9 -> 10.7; step 984 -> 933 us.
    const int quarter = warp & 3;             // the TMEM lane quarter this warp may read
    const int cg = (warp - 2) >> 2;           // its half of the columns
    int acc = 0;
    uint32_t acc_ph = 0;
    const int Dh = p.head_dim;
    uint8_t* epi_buf = epi_smem + (quarter + 4 * cg) * EPI_BUF_BYTES;
    int epi_sel = 0;                          // staging block to fill next, of the two that a lone warp has
    uint32_t xph = 0;                         // phase bits of this warp's landing-block barriers
    while (!(solo && cg == 1) && walk.next(un)) {
      const int tile = un.tile, ks = un.seg;
      const int m = PAIR ? 2 * (tile % n_m_tiles) + int(rank)
                         : emulate_pair ? 2 * (tile % n_m_tiles) + un.half : tile % n_m_tiles,
                n = tile / n_m_tiles;
      const int row = m * BM + quarter * 32 + lane;
      const bool row_ok = row < p.M;
      const int row_base = m * BM + quarter * 32;          // first row of this warp's 32
      // folded RMSNorm, consuming side: r of this thread's row, requested before the wait for the accumulator
      float rs = 1.f;
      if (p.in_row_rs != nullptr && MODE != kGemmResid && row_ok) rs = __ldcg(p.in_row_rs + row);
      // QKV: the row's position and cache slot, and its rotation's cosines and sines on their way into the L1
      int pos = 0, slot = 0;
      if (MODE == kGemmQkv) {
        if (row_ok) {
          pos = p.tok_pos[row];
          slot = p.tok_slot[row];
        }
        const float2* cs = p.rope + size_t(pos) * (Dh >> 1) + (Dh == 128 ? 32 * ((n * (qkv_width / 64) + cg) & 1) : 0);
        asm volatile("prefetch.global.L1 [%0];\n\tprefetch.global.L1 [%0 + 128];" ::"l"(cs));
      }
      // folded RMSNorm, producing side: the first two blocks of this warp's rows of y are on their way before the
      // tile's products are complete
      const bool fold_now = fold_pair && un.last;
      // three landing blocks per warp that folds: two in the ring's unused last stage, the third is its idle neighbour's
      // staging block
      uint8_t* xb_stage = smem + (Ring<true>::STAGES - 1) * Ring<true>::STAGE_BYTES + quarter * 2 * EPI_BUF_BYTES;
      auto landing = [&](int i) -> uint8_t* { return i < 2 ? xb_stage + i * EPI_BUF_BYTES : epi_buf + 4 * EPI_BUF_BYTES; };
      uint64_t* xb_bar = xbar + quarter * 4;
      // this warp's 32-column chunks of the tile: c_lo .. c_hi - 1
      const int n_chunks = min(p.bn / 32, (p.N - n * p.bn + 31) / 32), c_mid = solo ? n_chunks : min((p.bn / 32 + 1) / 2, n_chunks);
      const int c_lo = cg ? c_mid : 0, c_hi = cg ? n_chunks : c_mid;
      if (fold_now) {
        if (ordered && ks > 0) {              // every earlier segment of the tile must be in y before y is read
          int* turn = p.tile_turn + (tile * 2 + int(rank)) * EPI_WARPS + quarter + 4 * cg;
          bool go = true;
          if (lane == 0) go = spin_until_equal(turn, ks, abort_flag, p.status);
          if (!__shfl_sync(0xffffffffu, go, 0)) break;
        }
        if (lane == 0) {
          bulk_wait_read<0>();                // nothing of an earlier unit still reads the staging blocks
          for (int c = 0; c < 3 && c < n_chunks; ++c) {
            mbar_expect_tx(&xb_bar[c], EPI_BUF_BYTES);
            tma_load_2d(landing(c), &p.tm_out, &xb_bar[c], n * p.bn + c * 32, row_base);
          }
        }
      }
      const bool ok = mbar_wait(&tfull[acc], acc_ph, abort_flag, p.status);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after_sync();
      const uint32_t taddr = tmem_base + acc * BN + (uint32_t(quarter * 32) << 16);
      uint32_t r0[32], r1[32];
      float v0[32];

      if (MODE == kGemmResid) {
        // Ordered split-K: the partial sums of a tile are added into the output in split order, so the
        // result is the same fixed sum whatever block computed which split.  This warp owns 32 rows of half the
        // tile's columns; it waits until the previous split's add of those has been performed.
        int* turn = p.tile_turn + (PAIR ? tile * 2 + int(rank) : emulate_pair ? tile * 2 + un.half : tile) * EPI_WARPS + quarter + 4 * cg;
        if (ordered && ks > 0 && !fold_now) {
          bool go = true;
          if (lane == 0) go = spin_until_equal(turn, ks, abort_flag, p.status);
          if (!__shfl_sync(0xffffffffu, go, 0)) break;
        }
        const bool add = !walk.parts && (p.accumulate || ks > 0);
        const int out_row = walk.parts ? ks * p.part_rows + row_base : row_base;
        const bool store_ok = !walk.parts || row_base < p.M;      // (a box past the rows would reach into the next split)
        // conditioned block: the product is scaled by the gate vector of the row's sequence before it is added
        const float* gate = p.gate_mod && row_ok ? p.gate_mod + (size_t(p.tok_seq[row]) * 6 + p.gate_which) * p.N : nullptr;
        if (gate) {   // pull this tile's part of the gate vector into the L1 before the chunk loop needs it
          const int chunk = lane % (p.bn / 32), col = n * p.bn + chunk * 32;
          if (col < p.N) asm volatile("prefetch.global.L1 [%0];" ::"l"(gate + col));
        }
        if (fold_now) {
          // Final segment of the tile with the following RMSNorm folded in: x = y + acc is formed here (every
          // earlier segment has been added into y), written back, and reused for h = 16-bit(x o g) and sum x^2.
          // The 32 x 32 blocks of y come in by TMA, one chunk ahead, into two landing blocks per warp (the ring's
          // unused last stage), are updated in place and leave by TMA stores; the 16-bit block of a pair of chunks
          // is staged beside them.
          const bool h16 = p.norm_h_f16 != 0;
          float ss = 0.f;
          uint8_t* buf_h = epi_buf;
          bool okx = true;
          for (int c = 0; c < n_chunks; ++c) {
            const int col0 = n * p.bn + c * 32;
            const int xi = c % 3;
            uint8_t* bx = landing(xi);
            tmem_ld32(taddr + c * 32, r0);
            uint4 gw[4];                               // 32 gains (bf16), the same for every row
            const int nv = p.N - col0 >= 32 ? 8 : (p.N - col0) >> 2;
#pragma unroll
            for (int e = 0; e < 4; ++e)
              gw[e] = 2 * e < nv ? __ldg(reinterpret_cast<const uint4*>(p.norm_gain + col0) + e) : make_uint4(0, 0, 0, 0);
            okx = mbar_wait(&xb_bar[xi], (xph >> xi) & 1, abort_flag, p.status);
            if (!__all_sync(0xffffffffu, okx)) { okx = false; break; }
            xph ^= 1u << xi;
            tmem_ld_wait();
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              float4* slot = reinterpret_cast<float4*>(bx + lane * 128 + ((u ^ (lane & 7)) << 4));
              const float4 y4 = *slot;
              const float x0 = __uint_as_float(r0[4 * u]) + y4.x, x1 = __uint_as_float(r0[4 * u + 1]) + y4.y;
              const float x2 = __uint_as_float(r0[4 * u + 2]) + y4.z, x3 = __uint_as_float(r0[4 * u + 3]) + y4.w;
              if (u < nv) ss += (x0 * x0 + x1 * x1) + (x2 * x2 + x3 * x3);
              *slot = make_float4(x0, x1, x2, x3);
              r0[4 * u] = __float_as_uint(x0); r0[4 * u + 1] = __float_as_uint(x1);
              r0[4 * u + 2] = __float_as_uint(x2); r0[4 * u + 3] = __float_as_uint(x3);
            }
            // (here and not at the chunk's start, where that wait was 600 cycles of every chunk's 2300)
            if (lane == 0 && c > 0) {
              bulk_wait_read<0>();                         // the stores of the previous chunk have read their blocks
              if (c + 2 < n_chunks) {                      // ... so its landing block can take the chunk two further on
                const int xn = (c + 2) % 3;
                mbar_expect_tx(&xb_bar[xn], EPI_BUF_BYTES);
                tma_load_2d(landing(xn), &p.tm_out, &xb_bar[xn], col0 + 64, row_base);
              }
            }
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const uint32_t pk[4] = {gw[e].x, gw[e].y, gw[e].z, gw[e].w};
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                v0[8 * e + 2 * q] = __uint_as_float(r0[8 * e + 2 * q]) * __uint_as_float(pk[q] << 16);
                v0[8 * e + 2 * q + 1] = __uint_as_float(r0[8 * e + 2 * q + 1]) * __uint_as_float(pk[q] & 0xffff0000u);
              }
            }
            if (h16 && row_ok) note_f16_saturation(v0, p.status);
            stage_bf16x32(buf_h, lane, (c & 1) * 4, v0, h16);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&p.tm_out, bx, col0, row_base);
              if ((c & 1) || c + 1 == n_chunks) tma_store_2d(&p.tm_norm_h, buf_h, n * p.bn + (c >> 1) * 64, row_base);
              bulk_commit();
            }
          }
          if (!okx) break;
          finish_row_norm(p, row, row_ok, m * 4 + quarter, n, n_n_tiles, ss, lane);
          if (lane == 0) bulk_wait_read<0>();         // the staging blocks go back to the alternating use below
          __syncwarp();
          epi_sel = 0;
        } else if (p.norm_gain != nullptr && un.last) {
          // The same fold in the single-block kernel (reached by a folded step only at sm_budget 1): y is read with
          // plain loads; the arithmetic, and so every bit of x, h and the sums, is that of the pair form.
          const float* yrow = p.y_in + size_t(row_ok ? row : 0) * p.N;
          const bool h16 = p.norm_h_f16 != 0;
          float ss = 0.f;
          uint8_t* buf_x = epi_buf;                       // fp32 block of this chunk
          uint8_t* buf_h = epi_buf + 4 * EPI_BUF_BYTES;       // 16-bit block of a pair of chunks
          for (int c = 0; c < p.bn / 32; ++c) {
            const int col0 = n * p.bn + c * 32;
            if (col0 >= p.N) break;
            tmem_ld32(taddr + c * 32, r0);
            const int nv = p.N - col0 >= 32 ? 8 : (p.N - col0) >> 2;        // float4s of the chunk inside the row
            float4 yv[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
              yv[e] = row_ok && e < nv ? __ldcg(reinterpret_cast<const float4*>(yrow + col0) + e) : make_float4(0.f, 0.f, 0.f, 0.f);
            uint4 gw[4];                                   // 32 gains (bf16), the same for every row
#pragma unroll
            for (int e = 0; e < 4; ++e)
              gw[e] = 2 * e < nv ? __ldg(reinterpret_cast<const uint4*>(p.norm_gain + col0) + e) : make_uint4(0, 0, 0, 0);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float x0 = __uint_as_float(r0[4 * e]) + yv[e].x, x1 = __uint_as_float(r0[4 * e + 1]) + yv[e].y;
              const float x2 = __uint_as_float(r0[4 * e + 2]) + yv[e].z, x3 = __uint_as_float(r0[4 * e + 3]) + yv[e].w;
              if (e < nv) ss += (x0 * x0 + x1 * x1) + (x2 * x2 + x3 * x3);
              r0[4 * e] = __float_as_uint(x0); r0[4 * e + 1] = __float_as_uint(x1);
              r0[4 * e + 2] = __float_as_uint(x2); r0[4 * e + 3] = __float_as_uint(x3);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const uint32_t pk[4] = {gw[e].x, gw[e].y, gw[e].z, gw[e].w};
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                v0[8 * e + 2 * q] = __uint_as_float(r0[8 * e + 2 * q]) * __uint_as_float(pk[q] << 16);
                v0[8 * e + 2 * q + 1] = __uint_as_float(r0[8 * e + 2 * q + 1]) * __uint_as_float(pk[q] & 0xffff0000u);
              }
            }
            if (h16 && row_ok) note_f16_saturation(v0, p.status);
            if (lane == 0) bulk_wait_read<0>();       // both staging blocks have been read by their last stores
            __syncwarp();
            stage_f32x32(buf_x, lane, r0);
            stage_bf16x32(buf_h, lane, (c & 1) * 4, v0, h16);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&p.tm_out, buf_x, col0, row_base);
              if ((c & 1) || col0 + 32 >= p.N) tma_store_2d(&p.tm_norm_h, buf_h, n * p.bn + (c >> 1) * 64, row_base);
              bulk_commit();
            }
          }
          finish_row_norm(p, row, row_ok, m * 4 + quarter, n, n_n_tiles, ss, lane);
          if (lane == 0) bulk_wait_read<0>();         // the staging blocks go back to the alternating use below
          __syncwarp();
          epi_sel = 0;
        } else {
          float best_v = -INFINITY;              // greedy sampling: this thread's row over the tile
          int best_c = 0x7fffffff;
          for (int c = c_lo; c < c_hi; ++c) {
            const int col0 = n * p.bn + c * 32;
            tmem_ld32(taddr + c * 32, r0);
            float4 gv[8];
            const int nv = p.N - col0 >= 32 ? 8 : (p.N - col0) >> 2;          // float4s of the chunk inside the row
            if (gate) {                              // requested while the accumulator chunk is on its way
#pragma unroll
              for (int e = 0; e < 8; ++e)
                gv[e] = e < nv ? __ldg(reinterpret_cast<const float4*>(gate + col0) + e) : make_float4(1.f, 1.f, 1.f, 1.f);
            }
            tmem_ld_wait();
            if (gate) {
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                r0[4 * e] = __float_as_uint(__uint_as_float(r0[4 * e]) * gv[e].x);
                r0[4 * e + 1] = __float_as_uint(__uint_as_float(r0[4 * e + 1]) * gv[e].y);
                r0[4 * e + 2] = __float_as_uint(__uint_as_float(r0[4 * e + 2]) * gv[e].z);
                r0[4 * e + 3] = __float_as_uint(__uint_as_float(r0[4 * e + 3]) * gv[e].w);
              }
            }
            if (!PAIR && p.argmax_key != nullptr) {
              // (N is a multiple of 8; a NaN is never the maximum; columns ascend, so the first maximum stays)
              float mx = -INFINITY;
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (col0 + (e & ~7) < p.N) mx = fmaxf(mx, __uint_as_float(r0[e]));
              if (mx > best_v || best_c == 0x7fffffff) {
#pragma unroll
                for (int e = 31; e >= 0; --e)
                  if (col0 + (e & ~7) < p.N && __uint_as_float(r0[e]) == mx) best_c = col0 + e;
                best_v = mx;
              }
            }
            if (lane == 0) {                        // the staging block has been read by its last store
              if (solo) bulk_wait_read<1>();
              else bulk_wait_read<0>();
            }
            __syncwarp();
            uint8_t* buf = epi_buf + epi_sel * 4 * EPI_BUF_BYTES;
            stage_f32x32(buf, lane, r0);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              if (add) tma_reduce_add_2d(&p.tm_out, buf, col0, row_base);
              else if (store_ok) tma_store_2d(&p.tm_out, buf, col0, out_row);
              bulk_commit();
            }
            if (solo) epi_sel ^= 1;
          }
          if (!PAIR && p.argmax_key != nullptr && row_ok) {
            const uint32_t u = __float_as_uint(best_v + 0.f);                       // (-0 and +0 are the same value)
            const uint32_t ord = u & 0x80000000u ? ~u : u | 0x80000000u;
            atomicMax(p.argmax_key + row, (static_cast<unsigned long long>(ord) << 32) | (0xffffffffu - uint32_t(best_c)));
            __threadfence();
          }
        }
        if (ordered && !(ks == 0 && un.last) && lane == 0) {    // a tile with a single segment needs no turn
          bulk_wait<0>();                     // this segment's adds have been performed
          __threadfence();
          st_release(turn, un.last ? 0 : ks + 1);   // the last segment leaves the word at zero
        }
      } else if (MODE == kGemmGateUp) {
        for (int c = 2 * cg; c < 2 * cg + 2; ++c) {        // (this warp's 64 columns are one block of the output map)
          const int col0 = n * gu_w + c * 32;
          if (col0 >= p.N || c * 32 >= gu_w) break;
          tmem_ld32(taddr + c * 32, r0);          // gate
          tmem_ld32(taddr + gu_w + c * 32, r1);   // up
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const float g = __uint_as_float(r0[e]) * rs, u = __uint_as_float(r1[e]) * rs;
            v0[e] = __fdividef(g * u, 1.f + __expf(-g));   // silu(g) * u
          }
          if (gu_w < 128) {                       // a narrow tile: straight from the registers
            const int nv = min(min(32, gu_w - c * 32), p.N - col0);
            if (nv < 32)
#pragma unroll
              for (int e = 0; e < 32; ++e) v0[e] = e < nv ? v0[e] : 0.f;        // (what follows the tile's columns is not act)
            if (row_ok) {
              if (p.act_f16) note_f16_saturation(v0, p.status);
              store_act32(p.act + size_t(row) * p.N + col0, v0, p.act_f16 != 0, nv);
            }
            continue;
          }
          if (p.act_f16) note_f16_saturation(v0, p.status);
          if ((c & 1) == 0) {
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
          }
          stage_bf16x32(epi_buf, lane, (c & 1) * 4, v0, p.act_f16 != 0);
          if ((c & 1) || col0 + 32 >= p.N) {      // 64 columns staged (or the ragged end of the row)
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&p.tm_act, epi_buf, n * 128 + cg * 64, row_base);
              bulk_commit();
            }
          }
        }
      } else {
        // units of two 32-column pieces that rotate with each other, every other one this warp's
        const int half_dh = Dh >> 1, n_units = qkv_width / 64;
        const bool apart = Dh == 128 && !qkv_narrow;           // (whole heads of 128: the partners are 64 columns apart)
        for (int i = cg; i < n_units; i += 2) {
          const int unit = n * n_units + i, vcol = qkv_unit_col(p, unit), part = Dh == 128 ? unit & 1 : 0;   // column of [q | k | v]
          if (vcol >= p.N) break;
          int region = 0, col = vcol;
          if (col >= p.q_dim) { region = 1; col -= p.q_dim; }
          if (region == 1 && col >= p.kv_dim) { region = 2; col -= p.kv_dim; }
          const __nv_bfloat16* bias = p.qkv_bias[region];      // of this region's projection, or null
          const int at = apart ? (i >> 1) * 128 + (i & 1) * 32 : i * 64;
          tmem_ld32(taddr + at, r0);
          tmem_ld32(taddr + at + (apart ? 64 : 32), r1);
          tmem_ld_wait();
          if (p.in_row_rs) {
            scale32(r0, rs);
            scale32(r1, rs);
          }
          if (bias) {                                          // the bias comes before the rotation
            add_bias32(r0, bias + col);
            add_bias32(r1, bias + col + half_dh);
          }
          if (region != 2) {
            const float2* cs = p.rope + size_t(pos) * half_dh + 32 * part;
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              float t[8];                                      // cos, sin of pairs e .. e + 3
              ldg_f32x8(t, cs + e);
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                float a = __uint_as_float(r0[e + u]), b = __uint_as_float(r1[e + u]);
                rotate_pair(a, b, t[2 * u], t[2 * u + 1]);
                r0[e + u] = __float_as_uint(a);
                r1[e + u] = __float_as_uint(b);
              }
            }
          }
          if (row_ok) {
            __nv_bfloat16* to = region == 0 ? p.q_out + size_t(row) * p.q_dim + col
                                            : cache_ptr(region == 1 ? p.k_cache : p.v_cache, slot, col / Dh, p.n_kv_heads, Dh, col % Dh);
            store_bf16x32(to, r0);
            store_bf16x32(to + half_dh, r1);
          }
        }
      }
      // this warp has drained its rows of the accumulator: tell the MMA issuer (in the leader block)
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_cluster(mapa_u32(smem_u32(&tempty[acc]), 0));
        else mbar_arrive(&tempty[acc]);
      }
      acc ^= 1;
      if (acc == 0) acc_ph ^= 1;
    }
    if (lane == 0) bulk_wait<0>();            // every output block has been written
  }

  // ------------------------------------------------------------- teardown --
  __syncwarp();
  if (*abort_flag) drain_after_abort();
  tc_fence_before_sync();
  __syncthreads();
  if (!PAIR && MODE == kGemmResid && p.argmax_key != nullptr && warp == 2) {   // the last block to leave turns the keys into tokens
    int last = 0;
    if (lane == 0) {
      __threadfence();
      last = atomicAdd(p.argmax_done, 1) == int(gridDim.x) - 1;
    }
    if (__shfl_sync(0xffffffffu, last, 0)) {
      __threadfence();
      for (int r = lane; r < p.M; r += 32) {
        p.argmax_token[r] = int32_t(0xffffffffu - uint32_t(atomicExch(p.argmax_key + r, 0ull)));
      }
      if (lane == 0) *p.argmax_done = 0;
    }
  }
  if (PAIR) cluster_sync_all();               // neither block leaves while the other may still reach into it
  if (warp == 1) {
    tc_fence_after_sync();
    if (PAIR) tmem_dealloc_pair(tmem_base, TMEM_COLS);
    else tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

template <int MODE>
__global__ void __launch_bounds__(GEMM_THREADS, 1) gemm_kernel(const __grid_constant__ GemmParams p) {
  gemm_body<false, MODE>(p);
}
__global__ void __launch_bounds__(GEMM_THREADS, 1) gemm_qkv_unit_kernel(const __grid_constant__ GemmParams p) {
  gemm_body<false, kGemmQkv, true>(p);
}
// Two blocks per cluster, one 256 x 256 tile per pair.
template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM_THREADS, 1)
    gemm_pair_kernel(const __grid_constant__ GemmParams p) {
  gemm_body<true, MODE>(p);
}

template <typename F>
auto by_mode(int mode, F f) {
  return mode == kGemmResid ? f(std::integral_constant<int, kGemmResid>()) : mode == kGemmQkv ? f(std::integral_constant<int, kGemmQkv>())
                                                                                             : f(std::integral_constant<int, kGemmGateUp>());
}

}  // namespace

cudaError_t gemm_set_attributes() {
  for (const int mode : {kGemmResid, kGemmQkv, kGemmGateUp}) {
    const cudaError_t e = by_mode(mode, [](auto m) {
      const cudaError_t e1 = set_kernel_smem(gemm_pair_kernel<decltype(m)::value>, GEMM_SMEM);
      return e1 != cudaSuccess ? e1 : set_kernel_smem(gemm_kernel<decltype(m)::value>, GEMM_SMEM);
    });
    if (e != cudaSuccess) return e;
  }
  return set_kernel_smem(gemm_qkv_unit_kernel, GEMM_SMEM);
}

int gemm_pick_bn(int M, int N, int sm_count) {
  // Time of a launch ~ waves x time of one tile.  A tile's MMA work is proportional to its width, but the
  // operand feed is not (the 128-row A tile is fetched whatever the width, and narrow tiles leave less
  // time to hide the fetch): measured on B200, a 224-wide tile takes 0.95 and a 128-wide tile 0.80 of a
  // 256-wide one, i.e. about 0.6 + 0.4 * bn / 256.  The choice depends on the shape and on the device's
  // SM count only -- never on the SM budget -- so that the same tiles are computed at every budget.
  const int m_tiles = (M + BM - 1) / BM;
  int best = BN;
  double best_cost = 1e30;
  for (int bn = 256; bn >= 128; bn -= 32) {
    const int tiles = m_tiles * ((N + bn - 1) / bn);
    const int waves = (tiles + sm_count - 1) / sm_count;
    const double cost = double(waves) * (0.6 + 0.4 * bn / 256.0);
    if (cost < best_cost - 1e-9) {
      best_cost = cost;
      best = bn;
    }
  }
  return best;
}

int gemm_pick_ksplit(int M, int N, int K, int bn, int sm_count) {
  // Few tiles (small M): split K so that more SMs stream a share of the weights.  The splits of a tile add
  // their partial sums in split order, one after the other.  Measured on B200 at 64 rows (bn = 128): a block streams
  // a 64-wide K block in about 0.36 us, a link of the chain costs about 3.5 us -- the time of ten K blocks, which is
  // how much longer each split is than the one before it (gemm_split_begin), so that only the last link is exposed.
  // The split count minimises gemm_ksplit_cost_us over ks = 1 .. 8.  Depends on the shape and the device only, never
  // on the SM budget.
  const int tiles = ((M + BM - 1) / BM) * ((N + bn - 1) / bn);
  const int k_blocks = (K + BK - 1) / BK;
  int best = 1;
  double best_cost = 1e30;
  for (int ks = 1; ks <= 8 && ks <= k_blocks; ++ks) {
    if (gemm_split_begin(k_blocks, ks, ks - 1) >= k_blocks) continue;      // an empty last split
    const int waves = (tiles * ks + sm_count - 1) / sm_count;
    const double cost = gemm_ksplit_cost_us(k_blocks, ks, waves);
    if (cost < best_cost - 1e-9) {
      best_cost = cost;
      best = ks;
    }
  }
  return best;
}

namespace {
// Time (us) of a residual GEMM's launch on `sms` SMs, its longest unit `kb` K blocks of 64.  A block (pair) works a K block
// at the slowest of five rates, measured on B200: issue and tensor core (0.20 us per K block 128 columns wide, 0.27 for
// 256 and for pairs), what one SM takes in (120 KB/us) and what of it can be weights from the HBM (68 KB/us: latency
// against the ring's bytes in flight), what the L2 hands out to all SMs (14.5 MB/us) and what the HBM delivers (6.2 MB/us
// of weights, which the row tiles of a column share).  Rounds of one unit per worker, 2.5 us of start and end, 1.2 us per
// further round.
double resid_launch_us(int M, int N, bool pair, int bn, int ks, int kb, int sms) {
  const int W = pair ? sms / 2 : sms;
  if (W < 1) return 0.0;
  const int m_tiles = pair ? (M + 2 * BM - 1) / (2 * BM) : (M + BM - 1) / BM, units = m_tiles * ((N + bn - 1) / bn) * ks;
  const double a_bytes = (!pair && M <= 32 ? 32 : !pair && M <= 64 ? 64 : 128) * BK * 2;
  const double b_bytes = (pair || bn <= 128 ? 128 : 256) * BK * 2;
  auto round_us = [&](int n) {
    const double sm = pair ? 2.0 * n : n;
    double t = pair || bn > 128 ? 0.27 : 0.20;
    t = std::max(t, (a_bytes + b_bytes) / 120e3);
    t = std::max(t, b_bytes / m_tiles / 68e3);
    t = std::max(t, sm * (a_bytes + b_bytes) / 14.5e6);
    t = std::max(t, sm * b_bytes / m_tiles / 6.2e6);
    return kb * t;
  };
  const int full = units / W, rest = units - full * W;
  return full * round_us(W) + (rest ? round_us(rest) : 0.0) + 2.5 + 1.2 * (full + (rest ? 1 : 0) - 1);
}
// Time on the whole device and, with a weight of 0.15 each, on 13/16, 3/4, 13/20 and 1/2 of it (120, 111, 96 and 74 of 148
// SMs, budgets a stage with a neighbour is given), so that such a stage is not left with a short last round.
template <typename F>
double over_budgets(int sm_count, F us) {
  double sum = us(sm_count);
  for (const int eightieths : {65, 60, 52, 40}) sum += 0.15 * us(std::max(1, sm_count * eightieths / 80));
  return sum / 1.6;
}
}  // namespace

ResidPlan gemm_plan_parts(int M, int N, int K, int sm_count, int part_cap_rows, bool skinny) {
  // The best form with partial sums, read back at 12 MB/us, against the one the GEMM has without them (weight-streaming
  // kernel, or single blocks whose splits add in order), both by the times above.  Against that one the partial sums
  // count 3 MB/us where the norm kernel's threads hold eight groups each or its rows need a second round (pair of norms,
  // 1024 x 1024 with 21 MB +4 us, 1280 x 1024 with 26 MB +10, 600 x 2048 with 25 MB +11), and 3 us that no rate explains
  // (17 rows of d = 1024: out-projection +2.1 us, norm +1.7, whatever K).  Measured on B200, kernel by kernel, at 17 ..
  // 4096 rows of d = 1024 / 2048 / 3584 with K = d and 2.75 .. 5.3 d, on 148 and 74 SMs.  In steps, without -> with partial
  // sums: 128 rows of d = 1024 713 -> 574 us, 401 rows at 7B dimensions (2 layers) 501 -> 464; but 17 rows of d = 1024
  // 369 -> 426, 1280 rows 1114 -> 1209, which is why the two are compared.
  // Splits x width at 7B dimensions, down-projection (us per launch): 64 rows on 148 SMs 3 x 128 36.6, 5 x 128 33.7, 10 x
  // 128 34.2, 10 x 256 34.9; 29 rows on 96 SMs 36.5 / 42.3 / 36.9 / 39.1.
  const int k_blocks = (K + BK - 1) / BK, part_rows = (M + 31) / 32 * 32;
  const double part_bytes = double(part_rows) * N * 4.0;
  ResidPlan best{0, 0, 0};
  double best_us = 1e30;
  for (int form = 0; form < 3; ++form) {                     // single blocks 128 and 256 columns wide, pairs
    const bool pair = form == 2;
    if (pair && M <= BM) continue;
    const int bn = form == 0 ? 128 : 256;
    for (int ks = 2; ks <= 10 && ks <= k_blocks && ks * part_rows <= part_cap_rows; ++ks) {
      const double us = over_budgets(sm_count, [&](int sms) {
        return resid_launch_us(M, N, pair, bn, ks, (k_blocks + ks - 1) / ks, sms);
      }) + ks * part_bytes / 12e6;
      if (us < best_us - 1e-9) { best_us = us; best = ResidPlan{pair ? 1 : 0, bn, ks}; }
    }
  }
  const int tpr = norm_row_threads(M, N, sm_count), rows_per_block = kNormRowThreads / tpr;
  const bool wide = ((N >> 2) + tpr - 1) / tpr > 4 || (M + rows_per_block - 1) / rows_per_block > sm_count;
  if (wide) best_us += best.ks * part_bytes * (1 / 3e6 - 1 / 12e6);
  const int bn = gemm_pick_bn(M, N, sm_count), ks = gemm_pick_ksplit(M, N, K, bn, sm_count);
  const int longest = k_blocks - gemm_split_begin(k_blocks, ks, ks - 1);
  const double without = over_budgets(sm_count, [&](int sms) {
    // (units of 32 weight rows, though a launch may take others; rows past the step are not copied; from 33 rows on the MMAs of
    // 64 rows take as long as 64 rows' copies)
    if (skinny) return (((N >> 5) + sms - 1) / sms) * (1.5 + double(32 + (M <= 32 ? M : 64)) * K * 2 / 70e3);
    return resid_launch_us(M, N, false, bn, ks, longest, sms) + gemm_chain_us(k_blocks, ks);
  });
  // (A weight-streaming kernel with more units than half of the device loses in the second round under a partial budget what
  // it wins on the whole device -- 29 rows at 7B dimensions, out-projection, partial sums -> that kernel: on 148 SMs (2
  // layers) 284 -> 277 us, on 48 478 -> 487, on 96 (4 layers) 678 -> 688 -- so there it does not get the 3 us.)
  const double extra = skinny && (N >> 5) > sm_count / 2 ? 0.0 : 3.0;
  return best_us + extra < without ? best : ResidPlan{0, 0, 0};
}

int gemm_pick_stream_k(int M, int N, int K, int sm_count) {
  // Whole 256 x 256 tiles on W pairs take ceil(tiles / W) rounds; cutting the K blocks of all tiles into W equal
  // runs takes tiles / W rounds' worth, at the price of a second (ordered) add for the tiles that a cut falls into.
  // Worth it when the last round would be under about 90 % full and K is long: a run that ends inside a tile costs
  // that tile a second epilogue (the 256 x 256 fp32 block leaves by TMA add-reductions, about a third of the main
  // loop's time at K = 3584), and a short head or tail segment cannot hide its epilogue behind the next main loop.
  // Measured on B200 (per launch, whole tiles -> equal runs): 126 tiles of K = 18944 on 74 pairs (1.70 rounds run
  // as 2) 254 -> 233 us at equal clocks; 184 tiles of K = 5632 (2.49 run as 3) 114 -> 104 us; but 126 tiles of
  // K = 3584 62 -> 64 us and 184 tiles of K = 2048 53 -> 52 us: no gain below about 64 K blocks.
  const int W = sm_count / 2;
  const int tiles = ((M + 2 * BM - 1) / (2 * BM)) * ((N + BN - 1) / BN);
  const int k_blocks = (K + BK - 1) / BK;
  if (W < 1 || tiles * 2 * EPI_WARPS > kGemmTurnWords || k_blocks < 64) return 0;
  if (tiles * 2 < W) return 0;                       // few tiles: single blocks with a K split serve better
  const int rounds = (tiles + W - 1) / W;
  return double(tiles) / W < 0.92 * rounds ? W : 0;
}

// Activation columns of a GateUp tile of at most 128 rows, from the SMs the launch gets: an output element's sum is the same
// whatever the tile's width, so this choice may look at the budget.  Tiles of 128 columns at 7B dimensions, 148 of them, are
// one round on the whole device but two on 96 to 147 SMs.  Time per K block: the larger of issue, shared memory, an SM's intake
// -- 80 KB/us of the weights and 4.5 KB more, which is what narrow boxes pay -- and its share of the HBM; 1.1 us per further
// round.  Measured on B200, us per launch at 7B dimensions, 128 columns -> the width taken: 29 rows on 96 SMs 53.8 -> 50.7 (112
// columns); steps of 2 layers, 5 rows on 64 SMs 297 -> 283 (112), on 112 245 -> 233 (96), on 120 249 -> 232 (80), on 28 475 (128; 80
// columns, which the bytes alone would have, 509).
int gemm_pick_gu_width(int M, int N, int K, int sms) {
  if (M > BM) return 128;
  const double a_bytes = (M <= 32 ? 32 : M <= 64 ? 64 : 128) * BK * 2, k_blocks = (K + BK - 1) / BK;
  int best = 128;
  double best_us = 1e30;
  for (int w = 128; w >= kGuMinWidth; w -= 16) {
    const int tiles = (N + w - 1) / w, rounds = (tiles + sms - 1) / sms;
    const double b_bytes = 2.0 * w * BK * 2;
    auto k_block_us = [&](int n) {
      return std::max(std::max(0.27 * (0.4 + 0.6 * w / 128), (a_bytes + b_bytes) / 120e3), std::max((b_bytes + 4608) / 80e3, n * b_bytes / 6.2e6));
    };
    const int rest = tiles - (rounds - 1) * sms;
    const double us = k_blocks * ((rounds - 1) * k_block_us(sms) + k_block_us(rest)) + (rounds - 1) * 1.1;
    if (us < best_us * 0.97) { best_us = us; best = w; }
  }
  return best;
}

// The same for more than 128 rows: rounds, times the longer of the tensor core's time and of an SM's intake per K block (127 KB/us out of
// the L2; a block has its rows and, of a pair, half of the weight rows).  Tiles of 128 columns left the last round of 1024 rows and d_ffn
// 2816 nearly empty -- 88 tiles on 74 pairs.  Measured on B200, us per launch there (K = 1024), 128 / 112 / 96 / 80 / 64 / 48 columns: 17.4 /
// 16.4 / 15.5 / 15.3 (taken) / 17.8 / 20.8.  Steps, 128 columns -> the width taken: that one 925 -> 908; 400 rows on 148 / 120 / 112 / 74 / 37
// SMs 730 -> 708 (80), 745 -> 728 (96), 746 -> 739 (112), 942 -> 910 (80), 1189 -> 1167 (112); 504 rows of a small backbone (d_ffn 5632) on
// 148 SMs 395 -> 378 (80).  On single blocks, 256 rows, 148 / 120 / 96 / 74 SMs: 679 -> 657 (48), 758 -> 731 (48), 759 -> 732 (64), 759 -> 738
// (80).  5776 rows of the backbone keep 128 (16 rounds of 112 columns for 14 are 2.5 us slower).
int gemm_pick_tall_gu_width(int M, int N, int sms, bool pair) {
  const int units = pair ? sms / 2 : sms, m_tiles = (M + (pair ? 2 : 1) * BM - 1) / ((pair ? 2 : 1) * BM);
  if (units < 1) return 128;
  int best = 128;
  double best_us = 1e30;
  for (int w = 128; w >= kGuMinWidth; w -= 16) {
    const int rounds = (m_tiles * ((N + w - 1) / w) + units - 1) / units;
    const double us = rounds * std::max(0.275 * w / 128, (A_BYTES + (pair ? 1 : 2) * w * BK * 2) / 127e3);
    if (us < best_us * 0.97) { best_us = us; best = w; }
  }
  return best;
}

// Columns of a single block's Qkv tile, 128 or 64, by rounds and an SM's intake per K block -- 64 where that is one round still.  Steps on
// B200, 128 -> 64 columns: denoising, one image, 70 rows 538 -> 524 us, 256 on 148 / 120 / 96 SMs 670 -> 655, 743 -> 728, 745 -> 730; 128 decode
// rows of the talker 709 -> 689, at 7B dimensions (2 layers) 320 -> 315; a small backbone, 84 rows 266 -> 260.  In two rounds 64 columns
// lose: 256 rows of the denoising stage on 74 SMs 751 -> 778, 400 on 148 740 -> 759.  Not for at most 64 rows, whose A boxes of 64 or
// 32 rows would leave a stage (12 KB) shorter than the 128 rows that an MMA reads.
int gemm_pick_qkv_width(int M, int N, int sms) {
  if (M <= 64) return 128;
  const int m_tiles = (M + BM - 1) / BM;
  auto cost = [&](int w) { return (m_tiles * ((N + w - 1) / w) + sms - 1) / sms * double(A_BYTES + w * BK * 2); };
  return cost(QKV_UNIT) < 0.97 * cost(128) ? QKV_UNIT : 128;
}

// Columns of a pair's Qkv tile, 256 or 192, by the same rounds and times: 48 tiles of 256 columns (1024 rows, 3072 columns) leave a third of
// the 74 pairs idle, 64 of 192 do not and are shorter (15.6 -> 13.8 us a launch); 162 tiles (2112 rows, 4608 columns) are 2.19 rounds run
// as three, 216 are 2.92 (75 -> 68 us).  Steps on B200, 256 -> 192 columns: denoising, 1024 rows, 909 -> 887 us; a small backbone (K = 2048,
// 3072 columns), 1004 and 2104 rows 537 -> 526, 834 -> 816; 7B dimensions, 4 layers, 604, 1104, 1504, 2052 rows 1353 -> 1337, 2053 ->
// 2035, 2519 -> 2463, 3657 -> 3617; 2 layers on 96 SMs, 904 and 1504 rows 1112 -> 1086, 1601 -> 1583.  Not where the last round of 256
// columns is nearly empty, which is then a fast one: 1254 rows of the small backbone on 112 SMs (60 tiles on 56 pairs) 779 -> 797, 3204 rows
// on 148 (156 on 74) 1198 -> 1207; nor for more rounds (5404 rows, five for four, 1892 -> 1935).
int gemm_pick_pair_qkv_width(int M, int N, int sms) {
  const int pairs = sms / 2, m_tiles = (M + 2 * BM - 1) / (2 * BM);
  if (pairs < 1) return BN;
  auto tiles = [&](int w) { return m_tiles * ((N + w - 1) / w); };
  auto cost = [&](int w) { return (tiles(w) + pairs - 1) / pairs * std::max(0.275 * w / BN, (A_BYTES + w * BK) / 127e3); };
  const int rest = tiles(BN) % pairs;
  if (tiles(BN) > pairs && rest > 0 && rest * 8 < pairs) return BN;
  return cost(QKV_NARROW) < 0.97 * cost(BN) ? QKV_NARROW : BN;
}

cudaError_t launch_gemm(const GemmParams& p, int sm_budget, cudaStream_t stream) {
  const int n_m_tiles = (p.M + BM - 1) / BM;
  const int n_n_tiles = gemm_n_tiles(p);
  const int n_tiles = n_m_tiles * n_n_tiles * (p.mode == kGemmResid && p.ksplit > 1 ? p.ksplit : 1);
  if (n_tiles <= 0) return cudaSuccess;
  if (p.pair && sm_budget >= 2) {
    // pairs of blocks (clusters of two SMs) on 256 x 256 tiles; an odd budget leaves one SM unused
    const int pair_tiles = ((p.M + 2 * BM - 1) / (2 * BM)) * n_n_tiles;
    const int pairs = p.mode == kGemmResid && p.stream_k_slots > 0 ? p.stream_k_slots
                      : p.mode == kGemmResid && p.part_rows > 0 && p.ksplit > 1 ? pair_tiles * p.ksplit : pair_tiles;
    const int grid = 2 * (pairs < sm_budget / 2 ? pairs : sm_budget / 2);
    return by_mode(p.mode, [&](auto m) {
      return launch_step_kernel(gemm_pair_kernel<decltype(m)::value>, grid, GEMM_THREADS, GEMM_SMEM, stream, p.overlap != 0, p);
    });
  }
  const int grid = n_tiles < sm_budget ? n_tiles : sm_budget;
  if (p.mode == kGemmQkv && gemm_qkv_width(p) == QKV_UNIT)
    return launch_step_kernel(gemm_qkv_unit_kernel, grid, GEMM_THREADS, GEMM_SMEM, stream, p.overlap != 0, p);
  return by_mode(p.mode, [&](auto m) {
    return launch_step_kernel(gemm_kernel<decltype(m)::value>, grid, GEMM_THREADS, GEMM_SMEM, stream, p.overlap != 0, p);
  });
}

}  // namespace hs
