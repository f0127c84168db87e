// The projections of a small step (at most 64 token rows).  With so few rows every GEMM of the layer is a
// weight-streaming problem, and what counts is how many SMs pull weights and how directly.  The tcgen05 kernel
// of gemm.cu feeds 128-row tiles through TMA boxes of 128-byte pieces and needs a K split with an ordered
// chain of adds to occupy the GPU; this kernel does the opposite:
//   * one block per unit of 16 .. 112 weight rows and the WHOLE K range: no K split across blocks, no chain;
//   * inside the block the K range is dealt over 8 warps; every warp streams its K steps of the unit's
//     weight rows with 16-byte cp.async copies into a private ring of shared memory (every lane reads back exactly the
//     16 bytes it copied, so the ring needs no barrier at all), the matching slice of the activations the same
//     way, and feeds mma.sync m16n8k16 fragments from the ring -- no TMA, no TMEM, no mbarrier;
//   * the 8 partial accumulators meet in shared memory and are summed in warp order, then the epilogue of the
//     mode runs: residual add, RoPE + cache write + q store, or SwiGLU.
// Units are listed independently of the SM budget and a unit's arithmetic is one fixed sequence, so the results
// do not depend on the budget -- nor on the width of a unit: an output element's sum is its own, and a folded norm's
// partial sums of squares are kept per 16 columns.  So the width may be chosen by the budget (pick_width).  A unit's
// columns are chosen per mode so that the epilogue finds its partner columns in the same thread: with P pairs of
// 8-column tiles, Qkv units take columns c .. c + 8 P - 1 and the same of the head's other half (the rotation pairs),
// GateUp units 8 P gate columns and the same 8 P up columns.
//
// Fragment trick: a lane loads 8 consecutive K elements (16 bytes) of its weight row and of its two
// activation rows; the two MMAs of a 32-wide K step use elements 0..3 and 4..7 of those.  That is a
// permutation of the K index inside the step, applied to both operands alike, so the dot products are
// unchanged and every load is a full 16 bytes.
#include <algorithm>

#include "weight_stream.cuh"

namespace hs {
namespace {

// Weight row that feeds column g (0..7) of tile j (0 .. 2 P - 1) of unit `unit`.  The last unit of a width that P does not
// divide reads the last row again; its columns past the end are not stored.
template <int P>
__device__ __forceinline__ const uint8_t* unit_row(const SkinnyParams& p, int unit, int j, int g) {
  const size_t row_bytes = size_t(p.K) * 2;
  if (p.mode == kGemmResid) return static_cast<const uint8_t*>(p.w[0]) + size_t(min(unit * 16 * P + j * 8 + g, p.N - 1)) * row_bytes;
  const int hi = j >= P ? 1 : 0, jj = j - hi * P;                    // tiles 0 .. P - 1 and their partners
  if (p.mode == kGemmGateUp) return static_cast<const uint8_t*>(p.w[hi]) + size_t(min(unit * 8 * P + jj * 8 + g, p.N - 1)) * row_bytes;
  const int upr = p.head_dim / (16 * P);                             // units per head
  const int head = unit / upr, sub = unit - head * upr;
  int col = head * p.head_dim + sub * 8 * P + jj * 8 + g + hi * (p.head_dim >> 1);
  int which = 0;
  if (col >= p.q_dim) { col -= p.q_dim; which = 1; }
  if (which == 1 && col >= p.kv_dim) { col -= p.kv_dim; which = 2; }
  return static_cast<const uint8_t*>(p.w[which]) + size_t(col) * row_bytes;
}
__host__ __device__ __forceinline__ int skinny_units(int N, int mode, int P) {
  const int w = mode == kGemmGateUp ? 8 * P : 16 * P;
  return (N + w - 1) / w;
}

// Shared memory of an instantiation: the warps' rings, the partial tiles of the reduction -- of their own where all fits, else
// in the rings -- and a tail: r of a folded norm's 16 rows and its last-unit flag.
template <int MT, int P, int DB>
struct SkinnySmem {
  static constexpr int STAGE_BYTES = (2 * P + 2 * MT) * 512;        // per warp and K step: 2 P weight tiles, 2 MT row groups
  static constexpr int RING_BYTES = DB * STAGE_BYTES;               // per warp
  static constexpr int PART_STRIDE = 16 * P + 8;                    // floats between rows of a warp's partial tile
  static constexpr int PART_FLOATS = MT * 16 * PART_STRIDE;         // per warp
  static constexpr int TAIL_BYTES = 16 * 4 + 16, MAX_BYTES = 227 * 1024;
  static constexpr bool ALIAS = SK_WARPS * (RING_BYTES + PART_FLOATS * 4) + TAIL_BYTES > MAX_BYTES;
  static constexpr int TAIL_AT = SK_WARPS * (RING_BYTES + (ALIAS ? 0 : PART_FLOATS * 4));
  static constexpr int BYTES = TAIL_AT + TAIL_BYTES < kMinSmemBytes ? kMinSmemBytes : TAIL_AT + TAIL_BYTES;
  static_assert(!ALIAS || PART_FLOATS * 4 <= RING_BYTES, "a warp's partial tile must fit its own ring");
  static_assert(BYTES <= MAX_BYTES, "rings and partial tiles must fit one SM");
};

// What a launch takes once the kernel in front is done, in timestamps at the talker's dimensions (K = 1024): 1.1 us until the
// activations are there, 0.4 in the K loop, 0.45 until the last warp's partial tile is, 0.6 in the epilogue.  So with a K range
// that fits the rings there is one wait and no refills, the chains of MMAs are halved, an epilogue thread has four columns
// instead of eight, and the divisions of the unit's geometry and the first look at the arguments stand in front of the wait:
// talker step of one row 232 -> 225 us, of 16 rows 288 -> 276, all of it together.
// MT: 16-row tiles of activations (T <= 16 MT); P: pairs of 8-column tiles per unit; DB: depth of a warp's ring of K steps.
// FOLD: the instantiation that knows the folded RMSNorm (producing side in Resid mode, consuming side in the others; steps
// of at most 16 rows); the plain one carries none of its code.
template <int MT, int P, int DB, bool F16, bool FOLD>
__global__ void __launch_bounds__(SK_THREADS, 1) gemm_skinny_kernel(const SkinnyParams p) {
  extern __shared__ __align__(16) uint8_t sk_smem[];
  log_smid(p.smid_log);
  const int block = int(blockIdx.x), n_blocks = int(gridDim.x);
  static_assert(!FOLD || MT == 1, "the folded norm's rows are those of one row tile");
  constexpr int NT = 2 * P;                                 // n8 tiles of a unit
  using Smem = SkinnySmem<MT, P, DB>;
  constexpr int PART_STRIDE = Smem::PART_STRIDE, STAGE_BYTES = Smem::STAGE_BYTES, RING_BYTES = Smem::RING_BYTES, PART_FLOATS = Smem::PART_FLOATS;
  constexpr bool ALIAS = Smem::ALIAS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const uint8_t* ring_at = sk_smem + warp * RING_BYTES + lane * 16;
  const uint32_t ring = smem_u32(ring_at);
  float* part_all = reinterpret_cast<float*>(sk_smem + (ALIAS ? 0 : SK_WARPS * RING_BYTES));
  constexpr int PART_PITCH = ALIAS ? RING_BYTES / 4 : PART_FLOATS;   // floats between two warps' partial tiles
  float* part = part_all + warp * PART_PITCH;

  const int units = skinny_units(p.N, p.mode, P);
  // 32-wide K steps, dealt to the warps in turn: warp w takes steps w, w + 8, ...  The eight warps move through
  // the K range together, so at any moment the block reads 512 contiguous bytes of each weight row -- a run long
  // enough for the DRAM pages it opens.  (Contiguous per-warp K slices would make 8 x 32 separate 64-byte streams.)
  const int steps = p.K >> 5;
  const int n = (steps - warp + SK_WARPS - 1) / SK_WARPS;
  const size_t k_off = (size_t(warp) * 32 + t * 8) * 2;     // byte offset of this lane's first 16 bytes in a row
  constexpr int STEP_BYTES = SK_WARPS * 64;                 // from one of the warp's steps to its next
  // A K range that fits the rings is copied whole: one wait, no refills.  Otherwise DB - 1 steps are kept in flight.  (Not with
  // four row tiles, whose MMAs take long enough to start on the first step that is there: 64 rows of the talker on 112 / 37 SMs
  // 594 -> 556, 1023 -> 967 us with that and a step's weights and activations in one group, as below, for every unit but the
  // first, whose weights go ahead of the wait; 16 .. 32 rows, several units a block, 370 for 404 on 112 SMs.)
  const bool whole = MT < 4 && steps <= SK_WARPS * DB;
  const int n_first = whole ? n : min(n, DB - 1);

  const uint8_t* wrow[NT];
  auto set_rows = [&](int unit) {
#pragma unroll
    for (int j = 0; j < NT; ++j) wrow[j] = unit_row<P>(p, unit, j, g) + k_off;
  };
  // Activation rows of this lane: rows 16 i + g and 16 i + g + 8.  Rows past the step are not copied: whatever their
  // ring bytes hold reaches only accumulator rows that no epilogue stores.  (Copying the last row in their place made
  // every lane of every block ask the L2 for the same lines: talker step of one row 334 -> 236 us.)
  const uint8_t* arow[MT][2];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) arow[i][h] = static_cast<const uint8_t*>(p.a) + size_t(16 * i + 8 * h + g) * p.K * 2 + k_off;
  auto issue_b = [&](int s, int slot) {                     // weights of step s of this warp's slice
#pragma unroll
    for (int j = 0; j < NT; ++j) cp_async16(ring + slot * STAGE_BYTES + j * 512, wrow[j] + size_t(s) * STEP_BYTES);
  };
  auto issue_a = [&](int s, int slot) {                     // activations of the same step
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (16 * i + 8 * h + g < p.T) cp_async16(ring + slot * STAGE_BYTES + (NT + 2 * i + h) * 512, arow[i][h] + size_t(s) * STEP_BYTES);
  };
  // (groups: one per step, or with a whole range a single one, the others empty)
  auto first_b = [&]() {
#pragma unroll
    for (int s = 0; s < DB; ++s)
      if (s < n_first) issue_b(s, s);
  };
  auto first_a = [&]() {
#pragma unroll
    for (int s = 0; s < DB; ++s) {
      if (s < n_first) issue_a(s, s);
      if (s < DB - 1) cp_async_commit();
    }
    if (whole) cp_async_commit();
  };
  auto first_both = [&]() {                                 // both, a step's weights and activations in its own group
#pragma unroll
    for (int s = 0; s < DB; ++s) {
      if (s < n_first) {
        issue_b(s, s);
        issue_a(s, s);
      }
      if (s < DB - 1) cp_async_commit();
    }
    if (whole) cp_async_commit();
  };
  // Unit geometry of the Qkv mode: head, and first rotation pair inside it (the divisions stay in front of the wait)
  int u_head = 0, u_pair = 0;
  auto set_unit = [&](int unit) {
    set_rows(unit);
    if (p.mode == kGemmQkv) {
      const int upr = p.head_dim / (16 * P);
      u_head = unit / upr;
      u_pair = (unit - u_head * upr) * 8 * P;
    }
  };

  int unit = block;
  if (unit < units) {                                       // weights never change: fetch them before the wait
    set_unit(unit);
    first_b();
  }
  // This thread's part of the epilogue -- its row, and in Resid mode 2 Q consecutive columns, else Q columns of the first
  // half and their partners -- and what it needs from the step's metadata (there since two launches at least, see launch_fetch_metadata).
  constexpr int Q = MT == 1 && P <= 4 ? 2 : 4, TPR = 16 * P / (2 * Q);  // threads of a row
  static_assert(MT * 16 * TPR <= SK_THREADS, "one epilogue task per thread");
  const int e_row = threadIdx.x / TPR, e_q = threadIdx.x - e_row * TPR;
  const bool e_ok = e_row < MT * 16 && e_row < p.T;
  int e_pos = 0, e_slot = 0;
  if (p.mode == kGemmQkv && e_ok) {
    e_pos = p.tok_pos[e_row];
    e_slot = p.tok_slot[e_row];
  }
  const int n_q_heads = p.mode == kGemmQkv ? p.q_dim / p.head_dim : 0;
  // (the arguments the epilogue will read: their first use brings their lines of the constant bank)
  asm volatile("" ::"l"(p.y), "l"(p.q_out), "l"(p.act), "l"(p.norm_gain), "l"(p.row_ss), "l"(p.in_row_ss), "l"(p.rope), "l"(p.qkv_bias[0]),
               "l"(p.k_cache), "l"(p.status), "l"(p.gate_mod));
  griddep_wait();
  griddep_launch_dependents(p.overlap);
  // folded RMSNorm, consuming side: r of this thread's epilogue row, or the partial sums it is made of, which travel with the
  // activations of the first unit
  float rs_in = 1.f;
  const bool sums_in = FOLD && p.in_row_ss != nullptr;
  float* row_r = reinterpret_cast<float*>(sk_smem + Smem::TAIL_AT);         // FOLD: r of 16 rows, and one word
  int* last_unit = reinterpret_cast<int*>(row_r + 16);
  float ss_pre[kSsPre];
  if (unit < units) first_a();
  if (sums_in) row_norm_request(ss_pre, p.in_row_ss, p.K >> 4, p.K >> 4, p.T);
  if (FOLD && p.in_row_rs != nullptr && e_ok) rs_in = __ldcg(p.in_row_rs + e_row);
  bool first = true;

  for (; unit < units; unit += n_blocks) {
    // What the epilogue will read from memory is requested now, so that it has arrived when the K loop ends: the
    // output block to add to, the gains of a folded norm, the rotation of the row's position.
    float y_pre[2 * Q], cs[2 * Q];                            // (cs: cosine and sine of Q pairs)
    uint32_t ng[Q];                                           // 2 Q gains
    const int r_col = unit * 16 * P + e_q * 2 * Q;            // Resid: this thread's first column
    const bool r_ok = e_ok && r_col < p.N;
    const int head = u_head, i0 = u_pair + e_q * Q;           // Qkv: head and first rotation pair
    if (p.mode == kGemmResid) {
      if (r_ok) {
        if (p.accumulate) ldcg_f32<2 * Q>(y_pre, p.y + size_t(e_row) * p.N + r_col);
        if (FOLD && p.norm_gain != nullptr) ldg_u32<Q>(ng, p.norm_gain + r_col);
      }
    } else if (p.mode == kGemmQkv) {
      if (e_ok && head < n_q_heads + p.n_kv_heads) ldg_f32<2 * Q>(cs, reinterpret_cast<const float*>(p.rope + size_t(e_pos) * (p.head_dim >> 1) + i0));
    }
    // even and odd K steps of the warp in accumulators of their own (MT = 1: their chains of MMAs are what a short K range
    // takes), added at the end
    constexpr int NA = MT == 1 ? 2 : 1;
    float acc[NA][MT][NT][4];
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[a][i][j][e] = 0.f;
    auto step = [&](float (&d)[MT][NT][4], int slot) {
      const uint8_t* at = ring_at + slot * STAGE_BYTES;
      uint4 b[NT];
#pragma unroll
      for (int j = 0; j < NT; ++j) b[j] = *reinterpret_cast<const uint4*>(at + j * 512);
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        const uint4 lo = *reinterpret_cast<const uint4*>(at + (NT + 2 * i) * 512), hi = *reinterpret_cast<const uint4*>(at + (NT + 2 * i + 1) * 512);
        // the two MMAs on one accumulator are kept apart: independent ones run between them
#pragma unroll
        for (int j = 0; j < NT; ++j) mma_16816<F16>(d[i][j], lo.x, hi.x, lo.y, hi.y, b[j].x, b[j].y);
#pragma unroll
        for (int j = 0; j < NT; ++j) mma_16816<F16>(d[i][j], lo.z, hi.z, lo.w, hi.w, b[j].z, b[j].w);
      }
    };
    if (whole) {
      cp_async_wait<0>();
#pragma unroll 2
      for (int s = 0; s + NA <= n; s += NA) {
#pragma unroll
        for (int a = 0; a < NA; ++a) step(acc[a], s + a);
      }
      if (NA == 2 && (n & 1)) step(acc[0], n - 1);
    } else {
      int slot = 0, fill = DB - 1;                          // ring slot of step s / of step s + DB - 1
      auto turn = [&](float (&d)[MT][NT][4], int s) {
        if (s + DB - 1 < n) {
          issue_b(s + DB - 1, fill);
          issue_a(s + DB - 1, fill);
        }
        cp_async_commit();
        cp_async_wait<DB - 1>();
        step(d, slot);
        slot = slot + 1 == DB ? 0 : slot + 1;
        fill = fill + 1 == DB ? 0 : fill + 1;
      };
      for (int s = 0; s < n; s += NA) {
        turn(acc[0], s);
        if (NA == 2 && s + 1 < n) turn(acc[NA - 1], s + 1);
      }
      cp_async_wait<0>();
    }
    if (NA == 2)
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[0][0][j][e] += acc[NA - 1][0][j][e];

    // the next unit's first steps travel while this one is reduced and written (when the rings stay free)
    const int next = unit + n_blocks;
    if (!ALIAS && next < units) {
      set_unit(next);
      first_both();
    }

    // partial tiles -> shared memory (rows past the step are not read)
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        float* at = part + (16 * i + g) * PART_STRIDE + 8 * j + 2 * t;
        *reinterpret_cast<float2*>(at) = make_float2(acc[0][i][j][0], acc[0][i][j][1]);
        if (MT > 1 || p.T > 8) *reinterpret_cast<float2*>(at + 8 * PART_STRIDE) = make_float2(acc[0][i][j][2], acc[0][i][j][3]);
      }
    if (sums_in && first) {
      const float r = row_norm_factor(ss_pre, p.in_row_ss, p.K >> 4, p.K >> 4, p.T, p.K, p.norm_eps);
      if ((threadIdx.x & 15) == 0) row_r[threadIdx.x >> 4] = r;
    }
    __syncthreads();

    // sum of the 8 warps' partials in warp order, then the epilogue of the mode
    if (sums_in && first && e_ok) rs_in = row_r[e_row];
    first = false;
    const int row = e_row;
    if (p.mode == kGemmResid ? r_ok : e_ok) {
      const float* src = part_all + row * PART_STRIDE + (p.mode == kGemmResid ? e_q * 2 * Q : e_q * Q);
      const int to_hi = p.mode == kGemmResid ? Q : 8 * P;
      float v[2 * Q];                                       // the Q first columns, then the Q others
      lds_f32<Q>(v, src);
      lds_f32<Q>(v + Q, src + to_hi);
#pragma unroll
      for (int w = 1; w < SK_WARPS; ++w) {
        float u[2 * Q];
        lds_f32<Q>(u, src + w * PART_PITCH);
        lds_f32<Q>(u + Q, src + w * PART_PITCH + to_hi);
#pragma unroll
        for (int e = 0; e < 2 * Q; ++e) v[e] += u[e];
      }
      if (FOLD && (p.in_row_rs != nullptr || sums_in)) {
#pragma unroll
        for (int e = 0; e < 2 * Q; ++e) v[e] *= rs_in;
      }
      if (p.mode == kGemmResid) {
        if (p.gate_mod) {                                    // conditioned block: gate vector of the row's sequence
          float gt[2 * Q];
          ldg_f32<2 * Q>(gt, p.gate_mod + (size_t(p.tok_seq[row]) * 6 + p.gate_which) * p.N + r_col);
#pragma unroll
          for (int e = 0; e < 2 * Q; ++e) v[e] *= gt[e];
        }
        if (p.accumulate) {
#pragma unroll
          for (int e = 0; e < 2 * Q; ++e) v[e] += y_pre[e];
        }
        stg_f32<2 * Q>(p.y + size_t(row) * p.N + r_col, v);
        if (FOLD && p.norm_gain != nullptr) {
          // folded RMSNorm, producing side: the next GEMM's operand and the share of the row's sum of squares of these 16
          // columns (neighbouring threads)
          float h[2 * Q];
#pragma unroll
          for (int e = 0; e < Q; ++e) {
            h[2 * e] = v[2 * e] * __uint_as_float(ng[e] << 16);
            h[2 * e + 1] = v[2 * e + 1] * __uint_as_float(ng[e] & 0xffff0000u);
          }
          if (p.norm_h_f16 && p.status) note_f16_saturation(h, p.status);
          stg_act<2 * Q>(p.norm_h + size_t(row) * p.N + r_col, h, p.norm_h_f16 != 0);
          float ss = 0.f;
#pragma unroll
          for (int e = 0; e < 2 * Q; ++e) ss += v[e] * v[e];
          constexpr int L = 8 / Q;                           // threads of 16 columns
          const uint32_t mask = ((1u << L) - 1) << (lane & ~(L - 1));
#pragma unroll
          for (int o = 1; o < L; o <<= 1) ss += __shfl_xor_sync(mask, ss, o);
          if ((e_q & (L - 1)) == 0) p.row_ss[size_t(row) * p.ss_stride + (r_col >> 4)] = ss;
        }
      } else if (p.mode == kGemmGateUp) {
        const int col = unit * 8 * P + e_q * Q;
        float o[Q];
#pragma unroll
        for (int e = 0; e < Q; ++e) o[e] = __fdividef(v[e] * v[Q + e], 1.f + __expf(-v[e]));   // silu(gate) * up
        if (col < p.N) {
          if (p.act_f16 && p.status) note_f16_saturation(o, p.status);
          stg_act<Q>(p.act + size_t(row) * p.N + col, o, p.act_f16 != 0);
        }
      } else {
        const int Dh = p.head_dim, half = Dh >> 1;
        const int region = head < n_q_heads ? 0 : head < n_q_heads + p.n_kv_heads ? 1 : 2;
        if (p.qkv_bias[region]) {                            // the bias comes before the rotation
          const __nv_bfloat16* bias = p.qkv_bias[region] + (head - (region == 0 ? 0 : region == 1 ? n_q_heads : n_q_heads + p.n_kv_heads)) * Dh + i0;
          uint32_t wl[Q / 2], wh[Q / 2];
          ldg_u32<Q / 2>(wl, bias);
          ldg_u32<Q / 2>(wh, bias + half);
#pragma unroll
          for (int e = 0; e < Q / 2; ++e) {
            v[2 * e] += __uint_as_float(wl[e] << 16);
            v[2 * e + 1] += __uint_as_float(wl[e] & 0xffff0000u);
            v[Q + 2 * e] += __uint_as_float(wh[e] << 16);
            v[Q + 2 * e + 1] += __uint_as_float(wh[e] & 0xffff0000u);
          }
        }
        if (region != 2) {                                   // q and k heads are rotated
#pragma unroll
          for (int e = 0; e < Q; ++e) rotate_pair(v[e], v[Q + e], cs[2 * e], cs[2 * e + 1]);
        }
        __nv_bfloat16* dst = region == 0 ? p.q_out + size_t(row) * p.q_dim + head * Dh + i0
                                         : cache_row(region == 1 ? p.k_cache : p.v_cache, e_slot,
                                                     head - n_q_heads - (region == 1 ? 0 : p.n_kv_heads), p.n_kv_heads, Dh) + i0;
        stg_act<Q>(dst, v, false);
        stg_act<Q>(dst + half, v + Q, false);
      }
    }
    __syncthreads();                                         // the partial tiles are free again
    if (FOLD && p.mode == kGemmResid && p.norm_gain != nullptr && p.units_done != nullptr) {
      // the block that delivers the last unit turns the partial sums into every row's r (for a tiled GEMM behind the
      // norm).  (The barrier above orders the block's stores before thread 0's fence.)
      if (threadIdx.x == 0) {
        __threadfence();
        *last_unit = atomicAdd(p.units_done, 1) == units - 1;
      }
      __syncthreads();
      if (*last_unit) {
        __threadfence();
        float v[kSsPre];
        row_norm_request(v, p.row_ss, p.ss_stride, p.N >> 4, p.T);
        const float r = row_norm_factor(v, p.row_ss, p.ss_stride, p.N >> 4, p.T, p.N, p.norm_eps);
        if ((threadIdx.x & 15) == 0 && int(threadIdx.x >> 4) < p.T) p.row_rs[threadIdx.x >> 4] = r;
        if (threadIdx.x == 0) *p.units_done = 0;             // ready for the next launch
      }
    }
    if (ALIAS && next < units) {
      set_unit(next);
      first_both();
    }
  }
}

// Ring depth: what fits one SM beside the activations.  Weights in the rings of a block: 96 .. 192 KB with one row tile, 64
// (P = 1) and 96 KB with two, 32 P KB with four; of a K range that does not fit them, one step of each warp less is in flight.
constexpr int ring_depth(int MT, int P) {
  return MT == 1 ? (P == 1 ? 12 : P == 2 ? 8 : P == 3 ? 6 : P <= 6 ? 4 : 3) : MT == 2 ? (P == 1 ? 8 : P == 2 ? 6 : P == 3 ? 4 : 3) : 4;
}

template <int MT, int P>
cudaError_t launch_one(const SkinnyParams& p, int grid, cudaStream_t stream) {
  constexpr int DB = ring_depth(MT, P), smem = SkinnySmem<MT, P, DB>::BYTES;
  const bool early = p.overlap != 0;
  if constexpr (MT == 1) {
    if (p.norm_gain != nullptr || p.in_row_rs != nullptr || p.in_row_ss != nullptr) {
      if (p.ab_f16) return launch_step_kernel(gemm_skinny_kernel<MT, P, DB, true, true>, grid, SK_THREADS, smem, stream, early, p);
      return launch_step_kernel(gemm_skinny_kernel<MT, P, DB, false, true>, grid, SK_THREADS, smem, stream, early, p);
    }
  }
  if (p.ab_f16) return launch_step_kernel(gemm_skinny_kernel<MT, P, DB, true, false>, grid, SK_THREADS, smem, stream, early, p);
  return launch_step_kernel(gemm_skinny_kernel<MT, P, DB, false, false>, grid, SK_THREADS, smem, stream, early, p);
}
template <int MT, int P>
cudaError_t set_one() {
  constexpr int DB = ring_depth(MT, P), smem = SkinnySmem<MT, P, DB>::BYTES;
  cudaError_t e = set_kernel_smem(gemm_skinny_kernel<MT, P, DB, true, false>, smem);
  if (e == cudaSuccess) e = set_kernel_smem(gemm_skinny_kernel<MT, P, DB, false, false>, smem);
  if constexpr (MT == 1) {
    if (e == cudaSuccess) e = set_kernel_smem(gemm_skinny_kernel<MT, P, DB, true, true>, smem);
    if (e == cudaSuccess) e = set_kernel_smem(gemm_skinny_kernel<MT, P, DB, false, true>, smem);
  }
  return e;
}

// Width of a launch's units.  A block takes in about 70 KB/us, weights and activations alike -- 56 with units of 16 weight
// rows beside at most 16 of activations -- with about 1.5 us per unit beside that, and units run in rounds of one per SM.  The results do not depend on the width, so the rule may look at the
// budget.  Units wider than 64 weight rows, for a gate/up projection on few SMs, keep eight columns per epilogue thread and
// their partial tiles in the rings: steps of a small backbone (4 layers, d_ffn 5632), next best width -> this one, 80 rows: one
// row on 74 SMs 210 -> 201 us, 96: nine rows on 120 188 -> 183, 112: nine rows on 112 192 -> 184.  Measured on B200 against 32 rows throughout: talker step of 16 rows at 112 / 96 / 28 SMs
// 352 -> 333, 351 -> 333, 683 -> 632 us, of 11 rows at 52 (51 units of 112 rows instead of 176 of 32) 395 -> 382; at 7B
// dimensions 9 rows, 4 layers, at 96 / 74 / 37 SMs 606 -> 546, 594 -> 562, 963 -> 897; one row, 2 layers, at 52 SMs 344 -> 331 (two
// rounds of 48 rows; five rounds of 16, which 70 KB/us would have, 370).
int pick_width(int T, int K, int N, int mode, int head_dim, int sms) {
  const int max_p = T <= 16 && mode == kGemmGateUp ? 7 : T <= 32 ? 4 : 2;
  int best = 2;
  double best_us = 1e30;
  for (int P = 1; P <= max_p; ++P) {
    if (mode == kGemmQkv && (head_dim >> 4) % P != 0) continue;
    const int units = skinny_units(N, mode, P), rounds = (units + sms - 1) / sms;
    const double us = rounds * (1.5 + double(16 * P + (T <= 32 ? T : 64)) * K * 2 / (P == 1 && T <= 16 ? 56e3 : 70e3));
    if (us < best_us - 1e-9) { best_us = us; best = P; }
  }
  return best;
}

}  // namespace

bool gemm_skinny_supports(int T, int K, int N, int mode, int head_dim) {
  if (T < 1 || T > 64 || K < 32 || K % 32 != 0) return false;
  if (mode == kGemmResid) return N % 32 == 0;
  if (mode == kGemmGateUp) return N % 16 == 0;
  return head_dim % 32 == 0 && N % head_dim == 0;
}

// Which kernel is faster for this shape, from measurements on B200 (config-3 and talker dimensions, 8 .. 64 rows).
// The rule counts this kernel as it was when they were taken: units of 32 weight rows in rounds of one per SM, 70 KB/us of
// those and of 16 MT activation rows of width K, 1.5 us per unit for set-up, reduction and epilogue.  A launch today takes
// 16 .. 112 weight rows (pick_width) and copies the step's rows alone, so where units of 32 rows are several rounds -- gate/up
// of a wide FFN above all -- the rule holds this kernel for slower than it is.
// The tiled kernel streams a 64-wide K block in about 0.36 us (0.8 us with two weight boxes per stage, gate/up)
// and pays 3.5 us per link of a K-split chain.  So this kernel wins where the tiled one has too few tiles to
// occupy the device or needs a long chain (QKV, out-projection, down at few rows), and loses where there are
// tiles enough (gate/up of a wide FFN), because here every unit re-reads the activations.
// Depends on the shape and the device only, never on the SM budget: the two kernels round differently, and a
// step's result must not depend on its budget.  Rounds and waves are counted for the whole device.  Measured
// against the alternatives over budgets 148 / 111 / 74 at config-3 dimensions (ms per 28-layer decode-only step,
// all projections tiled -> this rule): 16 rows 4.39 -> 3.49, 5.42 -> 5.14, 5.74 -> 5.27; 32 rows 4.91 -> 4.36,
// 5.99 -> 5.80, 6.34 -> 6.15; 64 rows 5.72 -> 5.38, 7.21 -> 7.43, 8.06 -> 8.32 (with its unit count just below
// the SM count this kernel needs a second round as soon as the budget drops, which at 64 rows costs 3 %).
bool gemm_skinny_wins(int T, int K, int N, int mode, int head_dim, int sm_count) {
  if (!gemm_skinny_supports(T, K, N, mode, head_dim)) return false;
  const int mt = T <= 16 ? 1 : T <= 32 ? 2 : 4;
  const int units = mode == kGemmGateUp ? N / 16 : N / 32;
  const int rounds = (units + sm_count - 1) / sm_count;
  const double mine = rounds * (1.5 + double(32 + 16 * mt) * K * 2 / 70e3);
  const int k_blocks = (K + 63) / 64;
  double tiled;
  if (mode == kGemmResid) {
    const int bn = gemm_pick_bn(T, N, sm_count), ks = gemm_pick_ksplit(T, N, K, bn, sm_count);
    const int tiles = (N + bn - 1) / bn, waves = (tiles * ks + sm_count - 1) / sm_count;
    tiled = gemm_ksplit_cost_us(k_blocks, ks, waves);
  } else {
    const int tiles = (N + 127) / 128, waves = (tiles + sm_count - 1) / sm_count;
    tiled = double(waves) * k_blocks * (mode == kGemmGateUp ? 0.8 : 0.36);
  }
  return mine < tiled;
}

cudaError_t gemm_skinny_set_attributes() {
  cudaError_t e = cudaSuccess;
  for (const auto set : {set_one<1, 1>, set_one<1, 2>, set_one<1, 3>, set_one<1, 4>, set_one<1, 5>, set_one<1, 6>, set_one<1, 7>, set_one<2, 1>, set_one<2, 2>, set_one<2, 3>,
                         set_one<2, 4>, set_one<4, 1>, set_one<4, 2>})
    if (e == cudaSuccess) e = set();
  return e;
}

int gemm_skinny_rows(int T, int K, int N, int mode, int head_dim, int sms) { return 16 * pick_width(T, K, N, mode, head_dim, sms); }

cudaError_t launch_gemm_skinny(const SkinnyParams& p, int sm_budget, cudaStream_t stream) {
  if (p.T <= 0) return cudaSuccess;
  const int P = pick_width(p.T, p.K, p.N, p.mode, p.head_dim, sm_budget), units = skinny_units(p.N, p.mode, P);
  const int grid = units < sm_budget ? units : sm_budget;
  if (p.T <= 16) {
    switch (P) {
      case 1: return launch_one<1, 1>(p, grid, stream);
      case 2: return launch_one<1, 2>(p, grid, stream);
      case 3: return launch_one<1, 3>(p, grid, stream);
      case 4: return launch_one<1, 4>(p, grid, stream);
      case 5: return launch_one<1, 5>(p, grid, stream);
      case 6: return launch_one<1, 6>(p, grid, stream);
      default: return launch_one<1, 7>(p, grid, stream);
    }
  }
  if (p.T <= 32) {
    switch (P) {
      case 1: return launch_one<2, 1>(p, grid, stream);
      case 2: return launch_one<2, 2>(p, grid, stream);
      case 3: return launch_one<2, 3>(p, grid, stream);
      default: return launch_one<2, 4>(p, grid, stream);
    }
  }
  return P == 1 ? launch_one<4, 1>(p, grid, stream) : launch_one<4, 2>(p, grid, stream);
}

}  // namespace hs
