// A decode-only step of at most 16 rows in one cooperative launch: the phases of a layer -- QKV, attention, out-projection,
// gate/up, down -- follow each other inside the kernel.  As separate launches such a step (the talker: 12 layers) is a chain of 61
// kernels of 3.6 us each, 5 to 6 under a partial budget, of which 1.2 are work; what bounds it is the way from one phase's last
// store to the next one's first MMA.  So:
//   * No barrier between phases and no flag beside the data.  A phase writes its 16-bit results (and the rows' sums of squares)
//     into an exchange buffer every word of which reads 0xffffffff until it is written: two NaNs of a kind that no conversion
//     returns.  A consumer's lanes ask for just the fragments that they feed their MMAs with, and again while some are not there
//     yet: one store and one load instead of store, fence, flag, poll, load.  What is left of the way is the L2's: a load of a
//     line that another SM has just written takes about 800 cycles (280 of one that has been there), and more while the whole
//     device asks for the same few lines.  Hence fewer blocks than SMs for one launch (see launch_small_step).
//   * Three exchange buffers, layer l uses number l mod 3.  A thread that writes X of layer l then wipes what it wrote into X of
//     layer l - 1: its block has seen inputs that were formed from all of that.  One fence of every thread per layer lies between
//     the wiping and the thread's store of X of layer l + 1, and on the other side between seeing that store and asking for X of
//     layer l + 2, which is the wiped buffer.  The step's first act is to wipe all three (a step that was given up leaves them as
//     they are), followed by the one barrier over all blocks.
//   * Weights and the cache's pages do not wait for anything: one warp copies them, in the order of their use and across phases
//     and layers, into a ring of 32 KB slots, as the slots are emptied.  Bulk copies: a fence also waits for a thread's cp.async,
//     which took 1 to 6 us when those brought the weights.
// A piece is what a unit of 16 weight rows is in gemm_skinny.cu, its K range dealt to eight warps in the same way and added in the
// same order; the attention is the group mode of attention_decode.cuh, slice by slice.  So the bits are those of the separate
// launches, whatever the grid.  The new token's key and value come from the exchange buffer too: its page is fetched as it
// stands and the row put in place in shared memory.
// Measured on B200, talker step, rows of 128 .. 1024 cached tokens (eleven: .. 1500), separate launches behind a copy of the metadata -> this
// behind the kernel that fetches it, on 148 / 96 / 52 / 28 SMs: one row 223 -> 174, 270 -> 174, 316 -> 210, 461 -> 288 us; eight 258 -> 206,
// 309 -> 208, 350 -> 260, 536 -> 374; eleven 297 -> 280, 344 -> 281, 384 -> 371, 595 -> 575; sixteen 281 -> 260, 326 -> 266, 411 -> 399,
// 609 -> 590.
#include "attention_decode.cuh"
#include "hs_internal.h"
#include "weight_stream.cuh"

namespace hs {
namespace {

constexpr int DH = 64, PAGE2 = 2 * Geom<DH>::PAGE_BYTES;      // a page's keys and values of one KV head
constexpr int kStepWidth = SK_WARPS * 32, kSteps = kSmallMaxWidth / kStepWidth;      // columns of a K step of all warps
constexpr int kChunk = 4;                                     // K steps (of every warp) of a copy
constexpr int kTile = kChunk * SK_WARPS * 512, kSlot = 2 * kTile;    // bytes of eight weight rows in it, and of sixteen
static_assert(kSlot == SK_WARPS * PAGE2, "a slot holds a piece's chunk, or a page for every warp");
constexpr int kRing = 5;                                      // slots
constexpr int kTileRows = 64, kPartRow = 20;                  // rows of all the partial tiles reduced at a time; floats between two
constexpr int kGroupRows = 8, kSlicePitch = kGroupRows * kPartPitch<DH> * 4 + kGroupRows * 8;     // most heads of a group; a warp's part of a slice
constexpr int kPartBytes = SK_WARPS * kTileRows * kPartRow * 4, kPartAt = kRing * kSlot, kTailAt = kPartAt + kPartBytes;
constexpr int kBarriers = 2 * kRing + 2, kSmallSmem = 1024 + kTailAt + kBarriers * 8 + 256;
static_assert(SK_WARPS * kSlicePitch <= kPartBytes, "the parts of a slice lie where the partial tiles do");
static_assert(kSmallSmem <= 227 * 1024, "one SM's shared memory");
// Two warp groups that compute, and one of which a warp copies and one watches the time.  A thread that computes keeps up to 96
// registers of row fragments, and a spilled register comes back from the L2, the fences having emptied the L1 (one row 195 -> 311
// us).  So the registers are shared out unevenly, 256 x 232 + 128 x 40 = 384 x 168.
constexpr int kSmallThreads = SK_THREADS + 128, kComputeRegs = 232, kServiceRegs = 40;
constexpr uint32_t kEmpty = 0xffffffffu;

// (v stays as it is where i is not below n)
__device__ __forceinline__ void load_below(uint4& v, const void* at, int i, int n) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %5, %6;\n\t@p ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}\n"
               : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "l"(at), "r"(i), "r"(n) : "memory");
}
__device__ __forceinline__ void load_below(uint2& v, const void* at, int i, int n) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %3, %4;\n\t@p ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];\n\t}\n"
               : "+r"(v.x), "+r"(v.y) : "l"(at), "r"(i), "r"(n) : "memory");
}
__device__ __forceinline__ void load_below(uint32_t& v, const void* at, int i, int n) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %2, %3;\n\t@p ld.relaxed.gpu.global.u32 %0, [%1];\n\t}\n"
               : "+r"(v) : "l"(at), "r"(i), "r"(n) : "memory");
}
__device__ __forceinline__ uint32_t load_word(const void* at) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(at) : "memory");
  return v;
}
// (kEmpty is the largest word)
__device__ __forceinline__ uint32_t largest(uint32_t m, const uint2& v) { return max(max(m, v.x), v.y); }
__device__ __forceinline__ uint32_t largest(uint32_t m, const uint4& v) { return max(max(max(m, v.x), max(v.y, v.z)), v.w); }
// (a word that would read as "not there" is a NaN, whatever its bits: it becomes the one that conversions return)
__device__ __forceinline__ uint32_t there(uint32_t v) { return v == kEmpty ? 0x7fff7fffu : v; }
__device__ __forceinline__ void put1(void* at, uint32_t v) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(at), "r"(v) : "memory"); }
__device__ __forceinline__ void put2(void* at, uint32_t a, uint32_t b) {
  asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1, %2};" ::"l"(at), "r"(a), "r"(b) : "memory");
}
// A result for layer l's buffer, and the wiping of the same place in layer l - 1's.
__device__ __forceinline__ void hand_over(uint8_t* now, uint8_t* before, uint32_t v) {
  put1(now, there(v));
  put1(before, kEmpty);
}

// Every wait of the block ends when the block gives up, which a warp of its own sees to (`watch`): the waits themselves have no clock.
// Whatever a wait ended without is not stored: between a phase's waits and its stores lies a barrier, behind which every thread looks
// at the flag once more; and once a layer the warps leave together.  (Together in every phase: one row 184 -> 187 us, eleven on 52
// SMs 364 -> 367.)
// (a whole warp: true = some lane still misses something)
__device__ __forceinline__ bool again(bool more, volatile int* gave_up) { return __any_sync(0xffffffffu, more && *gave_up == 0); }
__device__ __forceinline__ bool copied(uint64_t* bar, uint32_t parity, volatile int* gave_up) {       // a whole warp; false = given up
  bool ok;
  while (!(ok = mbar_try_wait(bar, parity)))
    if (*gave_up != 0) break;
  return __all_sync(0xffffffffu, ok);
}
// Until the block is done: gives up when it has made no progress for limit_ns, or when
// another block has.
__device__ __forceinline__ void watch(uint64_t* done, volatile int* progress, volatile int* gave_up, int* all_gave_up, int* status, unsigned long long limit_ns) {
  unsigned long long t0 = globaltimer_ns();
  int seen = -1;
  for (uint32_t turn = 1; !mbar_try_wait(done, 0); ++turn) {
    if ((turn & 31u) != 0) continue;
    const int at = *progress;
    const unsigned long long now = globaltimer_ns();
    if (at != seen) { seen = at; t0 = now; }
    const bool late = now - t0 > limit_ns;
    if (late || load_word(all_gave_up) != 0) {
      if (late) {
        atomicExch(status, kErrTimeout);
        put1(all_gave_up, 1u);
      }
      *gave_up = 1;
      return;
    }
  }
}

// Barriers of the eight warps that compute.
__device__ __forceinline__ void block_sync() { named_barrier_sync(1, SK_THREADS); }
__device__ __forceinline__ bool block_any(bool mine) {
  int any;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.b32 %0, 1, 0, q;\n\t}\n"
               : "=r"(any) : "r"(int(mine)), "n"(SK_THREADS) : "memory");
  return any != 0;
}

enum Phase : int { kQkv = 0, kOut = 1, kGateUp = 2, kDown = 3 };

// Its code is run once per layer, a few thousand instructions in a row: beyond 8 KB an instruction comes at 2.4 cycles, beyond 32 KB
// at 6.  So there is one projection for all phases, its rare cases cost few instructions, and rows beyond eight are an instantiation
// of their own.  F16: format of h, o and act; NT: tiles of eight rows.
template <bool F16, int NT>
__global__ void __launch_bounds__(kSmallThreads, 1) small_step_kernel(const __grid_constant__ SmallStepParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *full = reinterpret_cast<uint64_t*>(smem + kTailAt), *free_ = full + kRing, *all_done = free_ + kRing;
  volatile int* gave_up = reinterpret_cast<volatile int*>(full + kBarriers);
  float* row_r = reinterpret_cast<float*>(full + kBarriers) + 4;      // [16]
  float* red = row_r + 16;                                                // [16]
  volatile int* progress = gave_up + 1;                                   // counts what thread 0 has done
  int* runs = reinterpret_cast<int*>(red + 16);                           // [4][2]: this block's pieces of every phase
  float* tiles = reinterpret_cast<float*>(smem + kPartAt);
  const int block = int(blockIdx.x), n_blocks = int(gridDim.x), tid = int(threadIdx.x);
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int T = p.T, L = p.n_layers, G = p.n_q_heads / p.n_kv_heads;
  constexpr bool f16 = F16;
  constexpr int kRound = kTileRows / (8 * NT);                  // pieces reduced at a time: at most a task per thread

  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&free_[i], SK_WARPS);
    }
    mbar_init(all_done, SK_WARPS);
    *gave_up = 0;
    *progress = 0;
    fence_barrier_init();
    tma_prefetch_desc(&p.tm_kv_page);
  }

  const int n_qkv = (p.q_dim + 2 * p.kv_dim) >> 4, n_d = p.d >> 4, n_gu = p.F >> 3;
  auto pieces = [&](int ph) { return ph == kQkv ? n_qkv : ph == kGateUp ? n_gu : n_d; };
  // (fewer pieces than blocks: on the last blocks, the slices of the attention being on the first)
  auto run_begin = [&](int ph, int b) {
    const int n = pieces(ph);
    return n >= n_blocks ? b * n / n_blocks : max(0, b - (n_blocks - n));
  };
  auto width = [&](int ph) { return ph == kOut ? p.q_dim : ph == kDown ? p.F : p.d; };
  if (tid < 8) runs[tid] = run_begin(tid >> 1, block + (tid & 1));
  __syncthreads();

  // ---- what comes from memory whatever the step computes, in the order in which the block will use it: the weights of its pieces,
  // kChunk K steps at a time, and behind those of QKV the pages of its slices, one for every warp at a time.  By a warp of its own.
  if (warp >= SK_WARPS) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kServiceRegs));
    if (tid == SK_THREADS + 32) watch(all_done, progress, gave_up, p.sync + 1, p.status, p.wait_limit_ns != 0 ? p.wait_limit_ns : kWaitLimitNs);
    if (warp != SK_WARPS) return;
    // (the maps lie in the stage's workspace, where another stage's may have been before)
    for (int i = lane; i < L * 7; i += 32) tma_acquire_desc(p.maps + i);
    __syncwarp();
    int slot = 0;
    uint32_t parity = 1;                                        // (a fresh barrier's phase before the first counts as done)
    bool ok = true;
    auto turn = [&]() {
      if (++slot == kRing) { slot = 0; parity ^= 1; }
    };
    for (int l = 0; l < L && ok; ++l) {
      const CUtensorMap* m = p.maps + l * 7;                    // w_q, w_k, w_v, w_o, w_gate, w_up, w_down
      for (int ph = kQkv; ph <= kDown && ok; ++ph) {
        const int n = width(ph) >> 8, last = runs[2 * ph + 1];
        for (int piece = runs[2 * ph]; piece < last && ok; ++piece) {
          const CUtensorMap *map0, *map1;
          int row0, row1;
          if (ph == kQkv) {                                     // eight rotation pairs of a head
            int col = (piece >> 2) * DH + (piece & 3) * 8, which = 0;
            if (col >= p.q_dim) {
              col -= p.q_dim;
              which = 1;
              if (col >= p.kv_dim) { col -= p.kv_dim; which = 2; }
            }
            map0 = map1 = m + which;
            row0 = col;
            row1 = col + DH / 2;
          } else if (ph == kGateUp) {                           // eight gate rows and the same of up
            map0 = m + 4;
            map1 = m + 5;
            row0 = row1 = piece * 8;
          } else {
            map0 = map1 = m + (ph == kOut ? 3 : 6);
            row0 = piece * 16;
            row1 = row0 + 8;
          }
          for (int k = 0; k < n && ok; k += kChunk) {
            ok = copied(&free_[slot], parity, gave_up);
            if (ok && lane == 0) {
              mbar_expect_tx(&full[slot], kSlot);
              tma_load_4d(smem + slot * kSlot, map0, &full[slot], 0, row0, 0, k);
              tma_load_4d(smem + slot * kSlot + kTile, map1, &full[slot], 0, row1, 0, k);
            }
            turn();
          }
        }
        if (ph == kQkv) {
          for (int i = block; i < p.n_slices && ok; i += n_blocks) {      // lane w: warp w's eighth of the slice
            int4 it = make_int4(0, 0, 0, 0);
            const int32_t* table = p.block_tables;
            if (lane < SK_WARPS) {
              it = __ldg(reinterpret_cast<const int4*>(p.decode_items) + 2 * (i * SK_WARPS + lane));
              table += size_t(__ldg(p.decode_items + 8 * (i * SK_WARPS + lane) + 4)) * p.max_pages_per_seq + (it.z >> 4);
            }
            const int n_pages = (it.w - it.z + 15) >> 4, columns = __shfl_sync(0xffffffffu, n_pages, 0);
            for (int c = 0; c < columns && ok; ++c) {
              const int page = c < n_pages ? __ldg(table + c) : 0;
              ok = copied(&free_[slot], parity, gave_up);
              if (!ok) break;
              const uint32_t with = __ballot_sync(0xffffffffu, c < n_pages);
              if (lane == 0) mbar_expect_tx(&full[slot], __popc(with) * PAGE2);
              __syncwarp();
              if (c < n_pages)
                tma_load_4d(smem + slot * kSlot + lane * PAGE2, &p.tm_kv_page, &full[slot], 0, (page * p.n_kv_heads + it.y) * 16, 0, l * 2);
              turn();
            }
          }
        }
      }
    }
    if (*gave_up) drain_after_abort();
    return;
  }
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kComputeRegs));
  const uint32_t k_off = uint32_t(warp * 32 + t * 8) * 2;       // of this lane's fragment of a K step, which is 256 columns
  int slot = 0;                                                 // the next one to use
  uint32_t parity = 0;
  bool dead = false;                                            // this warp has given up on a copy
  auto release = [&]() {                                        // the slot may be filled again
    __syncwarp();
    if (lane == 0) mbar_arrive(&free_[slot]);
    if (++slot == kRing) { slot = 0; parity ^= 1; }
  };

  // ---- wiped exchange buffers, then the one barrier over all blocks; the first RMSNorm meanwhile
  {
    const uint4 e = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    const uint32_t off[11] = {p.at.h_attn, p.at.h_mlp, p.at.q, p.at.k, p.at.v, p.at.o, p.at.act, p.at.ss_attn, p.at.ss_mlp, p.at.slice_o, p.at.slice_ml};
    const int bytes[11] = {T * p.d * 2, T * p.d * 2, T * p.q_dim * 2, T * p.kv_dim * 2, T * p.kv_dim * 2, T * p.q_dim * 2, T * p.F * 2,
                           T * (p.d >> 4) * 4, T * (p.d >> 4) * 4, p.n_slices * G * DH * 4, p.n_slices * G * 8};
#pragma unroll
    for (int r = 0; r < 11; ++r)
#pragma unroll 1
      for (int b = 0; b < 3; ++b) {
        uint4* at = reinterpret_cast<uint4*>(p.exchange + b * p.at.bytes + off[r]);
#pragma unroll 1
        for (int i = block * SK_THREADS + tid; i < (bytes[r] + 15) >> 4; i += n_blocks * SK_THREADS) at[i] = e;
      }
  }
  __threadfence();
  block_sync();
  if (tid == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.sync) : "memory");

  // Row r is normalised by block r mod n_blocks: as rmsnorm_row_kernel with 512 threads on a row, each thread here two of those.
  auto arrived = [&]() {                                        // false: given up, as below
    if (tid < 32) {
      int n;
      do asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(n) : "l"(p.sync) : "memory");
      while (again(n < n_blocks, gave_up));
    }
    if (block_any(*gave_up != 0)) return false;
    if (tid == 0) *progress = 1;
    return true;
  };
  const int d4 = p.d >> 2;
  bool first_row = true, on = true;                             // (on: the same in every warp that computes)
  for (int row = block; row < T; row += n_blocks) {
    constexpr int V = (kSmallMaxWidth / 4 + 511) / 512;
    float4 a[2][V];
    uint2 gw[2][V];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float ss = 0.f;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int i = tid + 256 * j + 512 * v;
        a[j][v] = make_float4(0.f, 0.f, 0.f, 0.f);
        gw[j][v] = make_uint2(0u, 0u);
        if (i < d4) {
          const uint2 w = reinterpret_cast<const uint2*>(p.x_in + size_t(row) * p.d)[i];
          gw[j][v] = __ldg(reinterpret_cast<const uint2*>(p.layers[0].g_attn) + i);
          a[j][v] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                                __uint_as_float(w.y & 0xffff0000u));
        }
        ss += square_sum(a[j][v]);
      }
      ss = warp_sum(ss);
      if (lane == 0) red[warp + 8 * j] = ss;
    }
    block_sync();
    float ss = 0.f;
    for (int w = 0; w < 16; ++w) ss += red[w];
    const float r = rsqrtf(ss / float(p.d) + p.eps);
    if (first_row) on = arrived();
    else block_sync();
    first_row = false;
    if (!on) break;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int i = tid + 256 * j + 512 * v;
        if (i < d4) {
          const float v4[4] = {a[j][v].x * r * __uint_as_float(gw[j][v].x << 16), a[j][v].y * r * __uint_as_float(gw[j][v].x & 0xffff0000u),
                               a[j][v].z * r * __uint_as_float(gw[j][v].y << 16), a[j][v].w * r * __uint_as_float(gw[j][v].y & 0xffff0000u)};
          if (f16) note_f16_saturation(v4, p.status);
          put2(p.exchange + p.at.h_attn + (size_t(row) * p.d + 4 * i) * 2, there(pack_act(v4[0], v4[1], f16)), there(pack_act(v4[2], v4[3], f16)));
        }
      }
  }
  if (first_row) on = arrived();

  // ---- a projection: this block's pieces of it
  uint8_t *now = p.exchange, *past = p.exchange + 2 * p.at.bytes, *next = p.exchange + p.at.bytes;     // buffers of layers l, l - 1, l + 1
  const int t_i = tid / (4 * T), t_row = (tid - t_i * 4 * T) >> 2, t_q = tid & 3;       // this thread's part of an epilogue: piece, row, quarter
  const int n_ss = p.d >> 4;
  uint4 a[kSteps][NT];                                          // the rows' fragments; zeros for rows past the step
#pragma unroll
  for (int s = 0; s < kSteps; ++s)
#pragma unroll
    for (int h = 0; h < NT; ++h) a[s][h] = make_uint4(0u, 0u, 0u, 0u);
  auto project = [&](int ph, int l) {
    const int begin = runs[2 * ph], end = runs[2 * ph + 1];
    if (begin >= end) return;
    const bool resid = (ph & 1) != 0, last = l + 1 == L;
    const bool emits = resid && !(ph == kDown && last);           // h of the norm behind it
    const bool scaled = ph == kGateUp || (ph == kQkv && l > 0);   // by the folded norm's factor (the first norm is a plain one)
    const int K = width(ph), n = K >> 8;
    const uint8_t* src = now + (ph == kQkv ? p.at.h_attn : ph == kOut ? p.at.o : ph == kGateUp ? p.at.h_mlp : p.at.act);
    uint8_t *to = ph == kDown ? next : now, *wiped = ph == kDown ? now : past;

#pragma unroll 1
    for (int p0 = begin; p0 < end; p0 += kRound) {
      const int np = min(kRound, end - p0), piece = p0 + t_i;
      const bool mine = t_i < np;                               // (a round has at most a task per thread)
      // what the epilogue reads from memory
      float pre[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t gain[2] = {0u, 0u};
      int kv_slot = 0;
      const int col = resid ? piece * 16 + t_q * 4 : piece * 8 + t_q * 2;        // (gate/up; in QKV's terms below)
      const int head = piece >> 2, i0 = (piece & 3) * 8 + t_q * 2;
      if (mine) {
        if (resid) {
          if (ph == kOut && l == 0) {
            const uint2 x = *reinterpret_cast<const uint2*>(p.x_in + size_t(t_row) * p.d + col);
            pre[0] = __uint_as_float(x.x << 16); pre[1] = __uint_as_float(x.x & 0xffff0000u);
            pre[2] = __uint_as_float(x.y << 16); pre[3] = __uint_as_float(x.y & 0xffff0000u);
          } else {
            ldcg_f32<4>(pre, p.y + size_t(t_row) * p.d + col);
          }
          if (emits) ldg_u32<2>(gain, (ph == kOut ? p.layers[l].g_mlp : p.layers[l + 1].g_attn) + col);
        } else if (ph == kQkv) {
          kv_slot = __ldg(p.tok_slot + t_row);
          if (head < p.n_q_heads + p.n_kv_heads)
            ldg_f32<4>(pre, reinterpret_cast<const float*>(p.rope + size_t(__ldg(p.tok_pos + t_row)) * (DH / 2) + i0));
        }
      }
#pragma unroll 1
      for (int i = 0; i < np; ++i) {
        // the piece's weights: there, or on their way whatever comes, so no part of what follows the rows
        const int chunks = (n + kChunk - 1) / kChunk, slot0 = slot;
#pragma unroll 1
        for (int c = 0; c < chunks; ++c) {
          if (!dead) dead = !copied(&full[slot], parity, gave_up);
          if (++slot == kRing) { slot = 0; parity ^= 1; }
        }
        if (p0 == begin && i == 0) {
          // The rows' fragments, and the partial sums of squares of row tid / 16: first one fragment of the first row until it is
          // there, then all of them, usually once or twice.  Asking for all of them all the time loads the lines on their way: one
          // row on 148 SMs 220 -> 258 us, eight 233 -> 310; with few rows on few SMs it is the shorter way (one row on 64 / 52 SMs
          // 227 -> 218, 245 -> 237; four 237 -> 232, 268 -> 259; eight on 52 273 -> 280).
          const uint8_t* rows = src + uint32_t(g * K * 2) + k_off;
          const uint8_t* sums = now + (ph == kQkv ? p.at.ss_attn : p.at.ss_mlp) + uint32_t((tid >> 4) * n_ss + (tid & 15)) * 4;
          const int n_lo = g < T ? n : 0, n_hi = g + 8 < T ? n : 0, n_sums = scaled && (tid >> 4) < T ? (n_ss - (tid & 15) + 15) >> 4 : 0;
          uint4 first = make_uint4(0u, 0u, 0u, 0u);
          if (T > 4 || n_blocks > 64) {
            do load_below(first, rows, g, 1);
            while (again(largest(0u, first) == kEmpty, gave_up));
          }
          uint32_t most;
          float sum;
          do {
#pragma unroll
            for (int c = 0; c < kSteps; c += kChunk)
              if (c < n) {
#pragma unroll
                for (int s = c; s < c + kChunk; ++s) {
                  load_below(a[s][0], rows + s * 512, s, n_lo);
                  if (NT == 2) load_below(a[s][NT - 1], rows + 16 * K + s * 512, s, n_hi);
                }
              }
            most = 0u;
            sum = 0.f;
#pragma unroll 1
            for (int u0 = 0; scaled && 16 * u0 < n_ss; u0 += 4) {
              uint32_t ss[4] = {0u, 0u, 0u, 0u};
#pragma unroll
              for (int u = 0; u < 4; ++u) load_below(ss[u], sums + 64 * (u0 + u), u0 + u, n_sums);
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                most = max(most, ss[u]);
                sum += __uint_as_float(ss[u]);
              }
            }
#pragma unroll
            for (int s = 0; s < kSteps; ++s)
#pragma unroll
              for (int h = 0; h < NT; ++h) most = largest(most, a[s][h]);
          } while (again(most == kEmpty, gave_up));
          if (scaled) {                                           // sixteen threads per row, as row_norm_factor
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if ((tid & 15) == 0) row_r[tid >> 4] = rsqrtf(sum / float(p.d) + p.eps);
          }
        }

        // Sixteen weight rows times the rows of a tile; even and odd steps apart and halves of a step in gemm_skinny.cu's order, so
        // that a sum is the same.
        float acc[2][NT][4];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
          for (int h = 0; h < NT; ++h)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[x][h][e] = 0.f;
#pragma unroll
        for (int c = 0; c < kSteps / kChunk; ++c)
          if (c < chunks) {
            const uint8_t* at = smem + (slot0 + c < kRing ? slot0 + c : slot0 + c - kRing) * kSlot + warp * 512 + lane * 16;
#pragma unroll
            for (int s = c * kChunk; s < (c + 1) * kChunk; ++s)
              if (s < n) {
                const uint4 b0 = *reinterpret_cast<const uint4*>(at + (s - c * kChunk) * SK_WARPS * 512);
                const uint4 b1 = *reinterpret_cast<const uint4*>(at + (s - c * kChunk) * SK_WARPS * 512 + kTile);
#pragma unroll
                for (int h = 0; h < NT; ++h) mma_16816<F16>(acc[s & 1][h], b0.x, b1.x, b0.y, b1.y, a[s][h].x, a[s][h].y);
#pragma unroll
                for (int h = 0; h < NT; ++h) mma_16816<F16>(acc[s & 1][h], b0.z, b1.z, b0.w, b1.w, a[s][h].z, a[s][h].w);
              }
          }
        __syncwarp();                                           // the slots may be filled again
        if (lane < chunks) mbar_arrive(&free_[slot0 + lane < kRing ? slot0 + lane : slot0 + lane - kRing]);
        if (i == 0) block_sync();                               // what the tiles' area held before has been read
        float* at = tiles + ((warp * kRound + i) * 8 * NT + 2 * t) * kPartRow + g;
#pragma unroll
        for (int h = 0; h < NT; ++h)
#pragma unroll
          for (int e = 0; e < 4; ++e) at[(8 * h + (e & 1)) * kPartRow + 8 * (e >> 1)] = acc[0][h][e] + acc[1][h][e];
      }
      block_sync();
      if (!mine) continue;
      const bool all_there = *gave_up == 0;

      constexpr int PITCH = kTileRows * kPartRow;
      const float* at = tiles + (t_i * 8 * NT + t_row) * kPartRow + (resid ? 4 * t_q : 2 * t_q);
      const int to_hi = resid ? 2 : 8;
      float v[4];
      lds_f32<2>(v, at);
      lds_f32<2>(v + 2, at + to_hi);
#pragma unroll
      for (int x = 1; x < SK_WARPS; ++x) {
        float u[4];
        lds_f32<2>(u, at + x * PITCH);
        lds_f32<2>(u + 2, at + x * PITCH + to_hi);
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] += u[e];
      }
      if (scaled) {
        const float rs = row_r[t_row];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] *= rs;
      }
      // what goes to the others, in one or two words, and where; what may have been clamped; where the stage's own buffers or the
      // cache take it
      uint32_t w0 = 0u, w1 = 0u, at0 = 0u, step = 0u;           // (step: bytes to the second word, 0 = none)
      float clamped[4] = {0.f, 0.f, 0.f, 0.f};
      uint8_t* copy = nullptr;
      if (resid) {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] += pre[e];
        if (emits) {
          clamped[0] = v[0] * __uint_as_float(gain[0] << 16);
          clamped[1] = v[1] * __uint_as_float(gain[0] & 0xffff0000u);
          clamped[2] = v[2] * __uint_as_float(gain[1] << 16);
          clamped[3] = v[3] * __uint_as_float(gain[1] & 0xffff0000u);
          w0 = pack_act(clamped[0], clamped[1], f16);
          w1 = pack_act(clamped[2], clamped[3], f16);
          at0 = uint32_t(t_row * p.d + col) * 2;
          if (last) copy = reinterpret_cast<uint8_t*>(p.h) + at0;
          at0 += ph == kOut ? p.at.h_mlp : p.at.h_attn;
          step = 4;
        }
      } else if (ph == kGateUp) {
#pragma unroll
        for (int e = 0; e < 2; ++e) clamped[e] = __fdividef(v[e] * v[2 + e], 1.f + __expf(-v[e]));   // silu(gate) * up
        w0 = pack_act(clamped[0], clamped[1], f16);
        at0 = uint32_t(t_row * p.F + col) * 2;
        if (last) copy = reinterpret_cast<uint8_t*>(p.act) + at0;
        at0 += p.at.act;
      } else {
        const int region = head < p.n_q_heads ? 0 : head < p.n_q_heads + p.n_kv_heads ? 1 : 2;
        const int hk = head - (region == 0 ? 0 : region == 1 ? p.n_q_heads : p.n_q_heads + p.n_kv_heads);   // head of its region
        const __nv_bfloat16* bias = p.layers[l].bias[region];
        if (bias) {                                             // the bias comes before the rotation
          uint32_t wl[1], wh[1];
          ldg_u32<1>(wl, bias + hk * DH + i0);
          ldg_u32<1>(wh, bias + hk * DH + i0 + DH / 2);
          v[0] += __uint_as_float(wl[0] << 16);
          v[1] += __uint_as_float(wl[0] & 0xffff0000u);
          v[2] += __uint_as_float(wh[0] << 16);
          v[3] += __uint_as_float(wh[0] & 0xffff0000u);
        }
        if (region != 2) {                                      // q and k heads are rotated
          rotate_pair(v[0], v[2], pre[0], pre[1]);
          rotate_pair(v[1], v[3], pre[2], pre[3]);
        }
        w0 = pack_bf16(v[0], v[1]);
        w1 = pack_bf16(v[2], v[3]);
        at0 = uint32_t(t_row * (region == 0 ? p.q_dim : p.kv_dim) + hk * DH + i0) * 2;
        step = DH;
        if (region != 0)
          copy = reinterpret_cast<uint8_t*>(cache_row(p.kv_pool + (size_t(l) * 2 + (region - 1)) * p.layer_kv_elems, kv_slot, hk, p.n_kv_heads, DH) + i0);
        else if (last)
          copy = reinterpret_cast<uint8_t*>(p.q) + at0;
        at0 += region == 0 ? p.at.q : region == 1 ? p.at.k : p.at.v;
      }
      if (!all_there) continue;
      if (!resid || emits) {
        put1(to + at0, there(w0));
        if (step != 0) put1(to + at0 + step, there(w1));
        if (resid) {
          float sq = 0.f;
#pragma unroll
          for (int e = 0; e < 4; ++e) sq += v[e] * v[e];
          const uint32_t mask = 0xfu << (lane & ~3);
          sq += __shfl_xor_sync(mask, sq, 1);
          sq += __shfl_xor_sync(mask, sq, 2);
          const uint32_t at_ss = (ph == kOut ? p.at.ss_mlp : p.at.ss_attn) + uint32_t(t_row * n_ss + piece) * 4;
          if (t_q == 0) hand_over(to + at_ss, wiped + at_ss, __float_as_uint(sq));
        }
        put1(wiped + at0, kEmpty);
        if (step != 0) put1(wiped + at0 + step, kEmpty);
        if (copy != nullptr) {
          *reinterpret_cast<uint32_t*>(copy) = w0;
          if (step != 0) *reinterpret_cast<uint32_t*>(copy + step) = w1;
        }
        if (f16 && ph != kQkv) note_f16_saturation(clamped, p.status);
      }
      if (resid) stg_f32<4>(p.y + size_t(t_row) * p.d + col, v);    // (read again by this thread only)
    }
  };

  // ---- the attention: slices block, block + n_blocks, ... of the groups; then the merge of the groups whose first slice it had
  const float scale_log2 = kLog2e / sqrtf(float(DH));
  struct Slice { int4 it, dr; int columns; };                   // this warp's eighth: its record; pages of the longest eighth
  auto slice_of = [&](int i) {
    const int4* r = reinterpret_cast<const int4*>(p.decode_items) + 2 * i * SK_WARPS;
    Slice s;
    s.it = __ldg(r + 2 * warp);
    s.dr = __ldg(r + 2 * warp + 1);
    s.columns = (__ldg(&r->w) - __ldg(&r->z) + 15) >> 4;
    return s;
  };
  Slice mine;
  if (block < p.n_slices) mine = slice_of(block);
  auto attend = [&](int l) {                                    // false: given up
    if (block_any(*gave_up != 0)) return false;                 // (and what the tiles' area held before has been read)
    if (block >= p.n_slices) return true;
    auto store = [&](const Slice& s, int gh, int col, float o0, float o1, float ll) {
      const float inv = 1.f / ll;
      const uint32_t o2 = pack_act(o0 * inv, o1 * inv, f16);
      const uint32_t at = uint32_t(s.dr.y * p.q_dim + (s.it.y * G + gh) * DH + col), at_o = p.at.o + at * 2;
      hand_over(now + at_o, past + at_o, o2);
      if (f16) {
        const float v2[2] = {o0, o1};
        note_f16_saturation(v2, p.status, inv);
      }
      if (l + 1 == L) *reinterpret_cast<uint32_t*>(p.o + at) = o2;
    };
#pragma unroll 1
    for (int i = block; i < p.n_slices; i += n_blocks) {
      const Slice s = i == block ? mine : slice_of(i);
      const int hk = s.it.y, k0 = s.it.z, k1 = s.it.w, tok = s.dr.y, splits = s.dr.w & 0xffff, n_pages = (k1 - k0 + 15) >> 4;
      // q of the group's heads, and for the warp with the last key the new token's key and value (16 bytes a lane)
      HeadsAsColumns<DH> at;
      at.clear();
      uint4 kv = make_uint4(0u, 0u, 0u, 0u);
      const bool has_new = n_pages > 0 && k1 == __ldg(p.seq_ctx + s.dr.x) + 1;
      const int need_q = n_pages > 0 && g < G ? 1 : 0, need_kv = has_new ? 16 : 0;
#pragma unroll
      for (int ks = 0; ks < DH / 16; ++ks) at.qf[ks][0] = at.qf[ks][1] = 0u;
      const uint8_t* q_src = now + p.at.q + uint32_t(tok * p.q_dim + (hk * G + g) * DH + 2 * t) * 2;
      const uint8_t* kv_src = now + (lane < 8 ? p.at.k : p.at.v) + uint32_t(tok * p.kv_dim + hk * DH + (lane & 7) * 8) * 2;
      uint32_t most;
      do {
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) {
          load_below(at.qf[ks][0], q_src + ks * 32, 0, need_q);
          load_below(at.qf[ks][1], q_src + ks * 32 + 16, 0, need_q);
        }
        load_below(kv, kv_src, lane, need_kv);
        most = largest(0u, kv);
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) most = max(most, max(at.qf[ks][0], at.qf[ks][1]));
      } while (again(most == kEmpty, gave_up));
      bool ok = true;
#pragma unroll 1
      for (int c = 0; c < s.columns; ++c) {
        ok = copied(&full[slot], parity, gave_up);
        if (!ok) break;
        if (c < n_pages) {
          uint8_t* page = smem + slot * kSlot + warp * PAGE2;
          const int n_valid = k1 - (k0 + c * 16);
          if (has_new && c == n_pages - 1) {
            if (lane < 16) *reinterpret_cast<uint4*>(page + (lane >> 3) * Geom<DH>::PAGE_BYTES + kv_off(n_valid - 1, lane & 7)) = kv;
            fence_proxy_async();                                // (the slot goes back to the copy engine)
            __syncwarp();
          }
          const uint32_t k_base = smem_u32(page);
          at.page(k_base, k_base + Geom<DH>::PAGE_BYTES, n_valid, lane, scale_log2);
        }
        release();
      }
      uint8_t* part = smem + kPartAt + warp * kSlicePitch;
      at.put(reinterpret_cast<float*>(part), kPartPitch<DH>, reinterpret_cast<float2*>(part + kGroupRows * kPartPitch<DH> * 4), G, lane);
      if (block_any(!ok || *gave_up != 0)) return false;
#pragma unroll 1
      for (int e = tid; e < G * (DH / 2); e += SK_THREADS) {
        const int gh = e / (DH / 2), col = 2 * (e - gh * (DH / 2));
        float mm, ll, o0, o1;
        merge_eight<DH, kGroupRows, kSlicePitch, 2>(smem + kPartAt, gh, col, mm, ll, o0, o1);
        if (splits == 1) {
          store(s, gh, col, o0, o1, ll);
        } else {
          const uint32_t at_o = p.at.slice_o + uint32_t((i * G + gh) * DH + col) * 4, at_ml = p.at.slice_ml + uint32_t(i * G + gh) * 8;
          hand_over(now + at_o, past + at_o, __float_as_uint(o0));
          hand_over(now + at_o + 4, past + at_o + 4, __float_as_uint(o1));
          if (col == 0) {
            hand_over(now + at_ml, past + at_ml, __float_as_uint(mm));
            hand_over(now + at_ml + 4, past + at_ml + 4, __float_as_uint(ll));
          }
        }
      }
      if (i + n_blocks < p.n_slices) block_sync();              // (before the next one's parts)
    }
#pragma unroll 1
    for (int i = block; i < p.n_slices; i += n_blocks) {
      const Slice s = i == block ? mine : slice_of(i);
      const int splits = s.dr.w & 0xffff;
      if (splits == 1 || (s.dr.w >> 16) != 0) continue;         // (the same for every warp of the block)
      const int rounds = (G * (DH / 2) + SK_THREADS - 1) / SK_THREADS;
#pragma unroll 1
      for (int rd = 0; rd < rounds; ++rd) {
        const int e = tid + rd * SK_THREADS, gh = e / (DH / 2), col = 2 * (e - gh * (DH / 2));
        const bool active = e < G * (DH / 2);
        const uint8_t* o_src = now + p.at.slice_o + uint32_t((i * G + gh) * DH + col) * 4;
        const uint8_t* ml_src = now + p.at.slice_ml + uint32_t(i * G + gh) * 8;
        float mm = -INFINITY, ll = 0.f, o0 = 0.f, o1 = 0.f;
#pragma unroll 1
        for (int j0 = 0; j0 < splits; j0 += 8) {
          uint2 ml[8], ov[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) ml[u] = ov[u] = make_uint2(0u, 0u);
          const int left = active ? splits - j0 : 0;
          uint32_t most;
          do {
            most = 0u;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              load_below(ml[u], ml_src + uint32_t((j0 + u) * G * 8), u, left);
              load_below(ov[u], o_src + uint32_t((j0 + u) * G * DH * 4), u, left);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) most = largest(largest(most, ml[u]), ov[u]);
          } while (again(most == kEmpty, gave_up));
          float2 mlf[8], ovf[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            mlf[u] = make_float2(__uint_as_float(ml[u].x), __uint_as_float(ml[u].y));
            ovf[u] = make_float2(__uint_as_float(ov[u].x), __uint_as_float(ov[u].y));
          }
          merge_slices(mlf, ovf, splits - j0, mm, ll, o0, o1);
        }
        if (active && *gave_up == 0) store(s, gh, col, o0, o1, ll);
      }
    }
    return true;
  };

#pragma unroll 1
  for (int l = 0; l < L && on; ++l) {
#pragma unroll 1
    for (int ph = kQkv; ph <= kDown && on; ++ph) {
      project(ph, l);
      if (ph == kQkv) {
        on = attend(l);
        __threadfence();                                        // the layer's (see above), where most blocks wait longest
      }
      if (tid == 0) *progress = 4 * l + ph + 2;
    }
    uint8_t* const oldest = past;
    past = now;
    now = next;
    next = oldest;
  }
  if (*gave_up) drain_after_abort();
  __syncwarp();
  if (lane == 0) mbar_arrive(all_done);
}

}  // namespace

SmallExchange small_exchange(int d, int q_dim, int kv_dim, int F, int heads_per_group, int slices) {
  SmallExchange x{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += align_up(bytes, 128);
    return uint32_t(o);
  };
  const size_t R = kSmallMaxRows;
  x.h_attn = take(R * d * 2);
  x.h_mlp = take(R * d * 2);
  x.q = take(R * q_dim * 2);
  x.k = take(R * kv_dim * 2);
  x.v = take(R * kv_dim * 2);
  x.o = take(R * q_dim * 2);
  x.act = take(R * F * 2);
  x.ss_attn = take(R * (d / 16) * 4);
  x.ss_mlp = take(R * (d / 16) * 4);
  x.slice_o = take(size_t(slices) * heads_per_group * DH * 4);
  x.slice_ml = take(size_t(slices) * heads_per_group * 8);
  x.bytes = uint32_t(align_up(off, 1024));
  return x;
}

bool small_step_supports(int T, int d, int q_dim, int kv_dim, int F, int head_dim, int n_layers) {
  auto fits = [](int K, int most) { return K >= kStepWidth && K <= most && K % kStepWidth == 0; };
  return T >= 1 && T <= kSmallMaxRows && head_dim == DH && n_layers <= kSmallMaxLayers && kv_dim > 0 && kv_dim % DH == 0 && q_dim <= kGroupRows * kv_dim &&
         fits(d, kSmallMaxModel) && fits(q_dim, kSmallMaxModel) && fits(F, kSmallMaxWidth);
}

bool small_step_wins(int T, int d, int q_dim, int sm_budget) {
  return T <= 8 || (d <= 1024 && q_dim <= 1024 && sm_budget >= 32);
}

cudaError_t small_step_set_attributes() {
  cudaError_t e = cudaSuccess;
  for (const auto k : {small_step_kernel<true, 1>, small_step_kernel<true, 2>, small_step_kernel<false, 1>, small_step_kernel<false, 2>})
    if (e == cudaSuccess) e = set_kernel_smem(k, kSmallSmem);
  return e;
}

cudaError_t launch_small_step(const SmallStepParams& p, int sm_budget, cudaStream_t stream) {
  // At most 96 blocks, 120 for more than eight rows: they take in what the HBM gives, and every further one asks for the same
  // lines (148 -> 96: one row 220 -> 211 us, eight 233 -> 224; eleven and sixteen 148 -> 120: 282 -> 273, 275 -> 267, 96: 288 and 285).
  const int most = std::max(std::max(p.F / 8, p.n_slices), std::max((p.q_dim + 2 * p.kv_dim) / 16, p.d / 16));
  const bool two = p.T > 8;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(std::min(std::min(sm_budget, most), two ? 120 : 96)), 1, 1);
  cfg.blockDim = dim3(kSmallThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmallSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;                  // its blocks wait for one another
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const auto kernel = two ? (p.f16 ? small_step_kernel<true, 2> : small_step_kernel<false, 2>) : (p.f16 ? small_step_kernel<true, 1> : small_step_kernel<false, 1>);
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

}  // namespace hs
