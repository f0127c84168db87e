// Launcher interfaces of the step's kernels.  Every launcher enqueues one persistent kernel of at most
// `sm_budget` thread blocks (one per SM: each block asks for more than half of an SM's shared memory)
// on `stream` and returns the launch status.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace hs {

// Dynamic shared memory every kernel requests at least, so that two blocks (of this or of a co-running
// stage's kernel) never share an SM: more than half of the 227 KB an SM offers.
constexpr int kMinSmemBytes = 117 * 1024;
// Warps per block of the decode attention kernel (each works through one item at a time); the planner sizes its
// work items for sm_count x this many warps.
constexpr int kDecodeKernelWarps = 8;

// ------------------------------------------------------------------ GEMM --
// out = A[M,K] * W^T with W given as up to three row blocks [rows, K] (bf16, K contiguous).  The output
// tile is 128 x 256 "virtual" columns; each 128-column half of a tile is fetched from one weight matrix.
enum GemmMode : int {
  kGemmResid = 0,   // out[M,N] fp32 (+)= A W^T: TMA store, or TMA add-reduction into out (out-proj, down)
  kGemmQkv = 1,     // virtual columns [q | k | v]; RoPE on q,k; q -> bf16 buffer, k,v -> paged cache
  kGemmGateUp = 2   // tile = 128 gate columns + the same 128 up columns; act = silu(gate) * up -> bf16
};

struct GemmParams {
  CUtensorMap tm_a;          // activations [rows >= M, K], box 64 x 128
  CUtensorMap tm_b[3];       // weights, box 64 x 128: Resid {W}, Qkv {Wq, Wk, Wv}, GateUp {Wgate, Wup}
  int M, N, K;               // N: Resid output width; Qkv (Hq + 2 Hkv) * Dh; GateUp F (activation width)
  int mode;
  int ab_f16;                // 1: both operands hold fp16 values; 0: both bf16
  int a_box_rows;            // rows of tm_a's box: 128, or 64 / 32 when M is that small (0 means 128); single blocks only
  int overlap;               // OverlapMode: how the launch overlaps the previous kernel's drain
  int pair;                  // 1: run on pairs of SMs (256 x 256 tiles, bn = 256, no K split) when the budget allows
  // Resid
  CUtensorMap tm_out;        // fp32 [M, N], box 32 x 32, 128-byte swizzle (rows past M are clipped)
  int accumulate;            // 1: out += A W^T (the residual add), 0: out = A W^T
  int bn;                    // tile width of this launch (gemm_pick_bn); 256 when unused
  int ksplit;                // K splits per output tile, added in split order (gemm_pick_ksplit); 0/1 = none
  int stream_k_slots;        // pairs only: > 0 = cut the tiles' K blocks into this many equal runs (gemm_pick_stream_k)
  // Resid in store mode on single blocks, optional: greedy sampling of every row (argmax_key non-null).  The tile's
  // epilogue, which holds the values in registers, maximises the row's key -- order-preserving bits of the value above
  // the complement of the column, so that the first maximum wins whatever the order -- and the block that leaves last
  // turns the keys into tokens.
  unsigned long long* argmax_key;   // [M], zero at entry and at exit
  int* argmax_done;          // one counter, zero at entry and at exit
  int32_t* argmax_token;     // [M]: lowest column of the row's maximum
  int part_rows;             // > 0: partial sums -- K split ks of the tile goes, unadded, to rows ks * part_rows ... of
                             // tm_out (a scratch [ksplit * part_rows, N] fp32 matrix; part_rows a multiple of 32, at
                             // least M), in equal splits; the RMSNorm behind the GEMM adds them (NormParams::part)
  int* tile_turn;            // [tiles * 8] ([tiles * 16] on pairs) whose-turn words for the ordered adds; zero at entry and at exit
  // Qkv
  int q_dim, kv_dim, head_dim, n_kv_heads;
  __nv_bfloat16* q_out;      // bf16 q [M, q_dim]
  __nv_bfloat16* k_cache;    // this layer's K pages: [page][kv_head][16][Dh]
  __nv_bfloat16* v_cache;
  const int32_t* tok_pos;    // [M]
  const int32_t* tok_slot;   // [M]
  const float2* rope;        // [max_position][Dh/2] (cos, sin)
  const __nv_bfloat16* qkv_bias[3];   // optional biases of the q, k, v projections ([q_dim], [kv_dim], [kv_dim]); null = none
  // Resid, optional: out += gate * (A W^T) with the gate vector of the row's sequence: gate_mod is this layer's
  // fp32 [max_seqs][6][N], gate_which the row of the gate vector (2 or 5), tok_seq the sequence of every row
  const float* gate_mod;
  const int32_t* tok_seq;
  int gate_which;
  // GateUp
  CUtensorMap tm_act;        // bf16 act [M, N], box 64 x 32, 128-byte swizzle
  int gu_width;              // activation columns per tile when not 128 (gemm_pick_gu_width); then tm_b has
  __nv_bfloat16* act;        // boxes of as many rows, and act [M, N] is written with plain stores
  int* status;               // device status word; with act_f16 the word after it counts saturated act values
  int act_f16;               // GateUp: 1 = write act as fp16, 0 = bf16
  int* smid_log;             // nullable: SM census slots of this launch (see log_smid)
  // RMSNorm folded into the GEMMs around it: rmsnorm(x) W^T = diag(r) ((x o g) W^T), r = rsqrt(mean(x^2) + eps).
  //   Resid, producing side (norm_gain non-null): the tile's final segment does not add-reduce its block into the
  //   output but reads it, adds, writes x back and, from the same registers, emits the next GEMM's A operand
  //   h = 16-bit(x o g) (not yet normalised) and the sum of x^2 over the tile's columns, one partial per (row, tile
  //   column), into row_ss[row * ss_stride + tile column]; the warp that delivers a row group's last tile column sums
  //   the partials in tile-column order and writes r into row_rs[row] (row_group_done: one counter per 32 rows,
  //   zero at entry and at exit).
  const __nv_bfloat16* norm_gain;   // [N] gains of the norm that follows, or null
  CUtensorMap tm_norm_h;     // h [M, N] 16-bit, box 64 x 32, 128-byte swizzle
  float* row_ss;             // [M][ss_stride]
  int ss_stride;
  float* row_rs;             // [M] r of every row, for the consuming GEMM
  int* row_group_done;       // [ceil(M / 32)]
  const float* y_in;         // the output as plain memory (the residual stream to read)
  int norm_h_f16;            // 1 = h in fp16, 0 = bf16
  //   Qkv / GateUp, consuming side (in_row_rs non-null): every accumulator row is scaled by r of its token before
  //   bias / RoPE / SiLU.
  const float* in_row_rs;    // [M]
  float norm_eps;            // producing side: eps of the norm that follows
};
cudaError_t launch_gemm(const GemmParams& p, int sm_budget, cudaStream_t stream);
cudaError_t gemm_set_attributes();
// Tile width for a Resid-mode GEMM of this shape on a device with sm_count SMs (budget independent).
int gemm_pick_bn(int M, int N, int sm_count);
int gemm_pick_ksplit(int M, int N, int K, int bn, int sm_count);
// Activation columns per tile of a GateUp GEMM with `sms` SMs: 128, or kGuMinWidth + 16 i, i < kGuNarrow.  Of at most 128 rows (128 for
// more), and of more, on pairs or on single blocks.
constexpr int kGuMinWidth = 48, kGuNarrow = 5;
int gemm_pick_gu_width(int M, int N, int K, int sms);
int gemm_pick_tall_gu_width(int M, int N, int sms, bool pair);
// Columns per tile of a Qkv GEMM with `sms` SMs, on pairs 256 or 192, on single blocks 128 or 64 (192 and 64: tm_b has boxes of 32 rows).
int gemm_pick_pair_qkv_width(int M, int N, int sms);
int gemm_pick_qkv_width(int M, int N, int sms);
// Where split i (0 .. ks) of a tile's k_blocks begins.  The splits add their sums one after the other, a link of that
// chain costing about as long as kSplitSkew K blocks take to stream; so each split is that much longer than the one
// before it and finishes just when its turn comes, instead of all finishing together and then queueing.  Equal
// lengths when K is too short for that.  A function of the shape only.
constexpr int kSplitSkew = 10;
__host__ __device__ inline int gemm_split_begin(int k_blocks, int ks, int i) {
  if (i >= ks) return k_blocks;
  const int tri = kSplitSkew * ks * (ks - 1) / 2;
  if (ks < 2 || k_blocks < tri + ks * kSplitSkew) {
    const int per = (k_blocks + ks - 1) / ks;
    return i * per < k_blocks ? i * per : k_blocks;
  }
  return i * ((k_blocks - tri) / ks) + kSplitSkew * i * (i - 1) / 2;
}
// What of the chain of adds is not hidden behind the longest split's stream (us).
inline double gemm_chain_us(int k_blocks, int ks) {
  const bool skewed = gemm_split_begin(k_blocks, ks, 1) != (k_blocks + ks - 1) / ks || ks == 1;
  return ks > 1 ? (skewed ? 3.5 : (ks - 1) * 3.5) : 0.0;
}
// Modelled time (us) of a K-split residual GEMM of `waves` rounds on single blocks: the longest split's stream and
// what of the chain of adds is not hidden behind it.
inline double gemm_ksplit_cost_us(int k_blocks, int ks, int waves) {
  const int last = k_blocks - gemm_split_begin(k_blocks, ks, ks - 1);
  return double(waves) * last * 0.36 + gemm_chain_us(k_blocks, ks);
}
// Runs for the stream-K form of a Resid-mode GEMM on pairs (one per pair of the device), or 0 when whole tiles
// already fill their waves well enough (budget independent).
int gemm_pick_stream_k(int M, int N, int K, int sm_count);
// Form of a residual GEMM whose K splits leave partial sums for the RMSNorm behind it (GemmParams::part_rows): tile width,
// pairs or single blocks, and the number of splits, or ks = 0 where no such form fits `part_cap_rows` rows of scratch or
// is expected to be faster, with the reading of the partial sums, than the form on single blocks -- on the weight-streaming
// kernel with `skinny` -- that it replaces.  A function of the shape and the device's SM count only.
struct ResidPlan { int pair, bn, ks; };
ResidPlan gemm_plan_parts(int M, int N, int K, int sm_count, int part_cap_rows, bool skinny);
// The same three GEMMs for steps of at most 64 rows (gemm_skinny.cu): weight streaming on plain loads and
// warp-level MMAs, one block per 16 .. 112 weight rows and the whole K range, no K split across blocks.
struct SkinnyParams {
  const void* a;             // activations [rows >= T, K], 16-bit (fp16 or bf16 as ab_f16 says), row-major
  const void* w[3];          // Resid {W}, Qkv {Wq, Wk, Wv}, GateUp {Wgate, Wup}; 16-bit [out, K] row-major
  int T, K, N;               // N: Resid output width; Qkv (Hq + 2 Hkv) * Dh; GateUp F
  int mode, ab_f16, overlap;
  float* y;                  // Resid: fp32 [T, N]
  int accumulate;            // Resid: 1: y += A W^T, 0: y = A W^T
  int q_dim, kv_dim, head_dim, n_kv_heads;      // Qkv
  __nv_bfloat16* q_out;      // bf16 [T, q_dim]
  __nv_bfloat16* k_cache;
  __nv_bfloat16* v_cache;
  const int32_t* tok_pos;
  const int32_t* tok_slot;
  const float2* rope;
  const __nv_bfloat16* qkv_bias[3];   // optional, as in GemmParams
  const float* gate_mod;     // Resid, optional, as in GemmParams
  const int32_t* tok_seq;
  int gate_which;
  __nv_bfloat16* act;        // GateUp: 16-bit [T, N]
  int act_f16;
  int* status;               // nullable: the stage's device status words (the second one counts fp16 saturations)
  int* smid_log;
  // RMSNorm folded into the GEMMs around it, as in GemmParams (rmsnorm(x) W^T = diag(r) ((x o g) W^T)).
  //   Resid, producing side (norm_gain non-null): the epilogue also emits h = 16-bit(y o g) for the next GEMM and the
  //   sum of y^2 over every 16 columns into row_ss[row * ss_stride + column / 16].  When the GEMM behind the norm is the
  //   tiled kernel (units_done non-null), the block that delivers the last unit (units_done: one counter, zero at entry
  //   and at exit) sums every row's partials and writes r = rsqrt(mean(y^2) + norm_eps) into row_rs[row]; when it is
  //   this kernel, that GEMM sums the partials itself (in_row_ss) and the producer's tail stays short.
  const __nv_bfloat16* norm_gain;   // [N]
  __nv_bfloat16* norm_h;     // 16-bit [T, N]
  int norm_h_f16;
  float* row_ss;             // [T][ss_stride], ss_stride >= N / 16
  int ss_stride;
  float* row_rs;             // [T]
  int* units_done;
  float norm_eps;            // both sides
  //   Qkv / GateUp, consuming side: every output row is scaled by r of its token before bias / RoPE / SiLU; r comes
  //   from in_row_rs[row], or (in_row_ss non-null) from the K / 16 partials in_row_ss[row * (K / 16) + i], which sixteen
  //   threads per row add in the order the producer's last block would have.
  const float* in_row_rs;    // [T]
  const float* in_row_ss;    // [T][K / 16]
};
// True when the skinny kernel covers this shape (few rows, K a multiple of 32, widths it can tile).
bool gemm_skinny_supports(int T, int K, int N, int mode, int head_dim);
// True when it is also expected to be faster than the tiled kernel for this shape (budget independent).
bool gemm_skinny_wins(int T, int K, int N, int mode, int head_dim, int sm_count);
// Weight rows of a block's unit on `sms` SMs (the results do not depend on it).
int gemm_skinny_rows(int T, int K, int N, int mode, int head_dim, int sms);
cudaError_t launch_gemm_skinny(const SkinnyParams& p, int sm_budget, cudaStream_t stream);
cudaError_t gemm_skinny_set_attributes();
constexpr int kGemmTurnWords = 8192;   // capacity of the whose-turn array: splits are used only when tiles * 8 fits

// The step's metadata from pinned host memory (a multiple of four words, 16-byte aligned), as the step's first launch.
// The kernels of a step may read work lists, positions and slots in front of their own wait for the kernel before them, which this
// launch allows to all but the kernel directly behind it: that one may be running while the block is written.  So (1) the kernel
// behind it, the first RMSNorm or the one-launch step, touches no metadata before it has waited, and (2) like every kernel of a step it
// lets its successor go behind that wait only, when the block is complete.
cudaError_t launch_fetch_metadata(const void* host, void* dev, int words, int overlap, int sm_budget, cudaStream_t stream);
cudaError_t metadata_set_attributes();

// ------------------------------------------------- a small step in one launch --
// Decode-only step of at most 16 rows whose projections all stream weights past the rows, head_dim 64, at most eight query heads
// per KV head, d_model and q_dim up to kSmallMaxModel, d_ffn up to kSmallMaxWidth, all three multiples of 256, as ONE cooperative
// launch: every block goes through the phases of every layer, and what one phase leaves for the next travels through buffers in
// which a value that is not there yet reads as a pattern that no value has (small_step.cu).  The same units, slices and orders as
// the kernels of their own: the same bits.
constexpr int kSmallMaxRows = 16, kSmallMaxModel = 2048, kSmallMaxWidth = 3072, kSmallMaxLayers = 32;
struct SmallLayer {
  const __nv_bfloat16 *g_attn, *g_mlp;
  const __nv_bfloat16* bias[3];                                    // of q, k, v, or null
};
// Byte offsets inside one of the three exchange buffers of a stage: 16 rows of h in front of the attention and of the MLP, q, k,
// v, o and act, the sums of squares that belong to the two h, and the partial results of `slices` slices of the attention.
struct SmallExchange {
  uint32_t h_attn, h_mlp, q, k, v, o, act, ss_attn, ss_mlp, slice_o, slice_ml, bytes;
};
SmallExchange small_exchange(int d, int q_dim, int kv_dim, int F, int heads_per_group, int slices);
struct SmallStepParams {
  CUtensorMap tm_kv_page;          // as in AttnParams
  const CUtensorMap* maps;         // device, [n_layers][7]: w_q, w_k, w_v, w_o, w_gate, w_up, w_down (encode_small_weight)
  SmallLayer layers[kSmallMaxLayers];
  SmallExchange at;
  uint8_t* exchange;               // three buffers of at.bytes
  int n_layers, T, d, F, q_dim, kv_dim, n_q_heads, n_kv_heads, max_pages_per_seq;
  int n_slices;                    // of the decode attention in group mode
  int f16;                         // format of h, o and act
  float eps;
  const __nv_bfloat16* x_in;       // [T, d]
  float* y;                        // [T, d]
  __nv_bfloat16 *h, *q, *o, *act;  // the stage's own buffers, which hold the last layer's values after a step
  __nv_bfloat16* kv_pool;
  size_t layer_kv_elems;           // elements of one layer's K (or V) pages
  const int32_t *tok_pos, *tok_slot, *decode_items, *seq_ctx, *block_tables;
  const float2* rope;
  int* sync;                       // two words, zero at entry: blocks that have arrived, and a flag of blocks that gave up
  int* status;
  unsigned long long wait_limit_ns;    // without progress, before a block gives up; 0: kWaitLimitNs
};
// Tensor map of a 16-bit weight matrix [rows, K], K a multiple of 256, from which one copy brings eight rows of four consecutive
// 256-column blocks as [block][eighth of it: one warp's 32 columns][row][64 bytes].
template <typename Encode>
inline bool encode_small_weight(Encode encode, CUtensorMap* m, const void* w, int rows, int K) {
  cuuint64_t dims[4] = {32, cuuint64_t(rows), 8, cuuint64_t(K) / 256}, strides[3] = {cuuint64_t(K) * 2, 64, 512};
  cuuint32_t box[4] = {32, 8, 8, 4}, estr[4] = {1, 1, 1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(w), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// The sizes of a stage and the rows of a step that the kernel takes.  Wider stages would fit, but their weights are long enough to
// hide the launches: d_model = q_dim = 3072, 4 layers, one / eight rows on 148 SMs 146 -> 158, 146 -> 163 us (2048, 8 layers: 235 ->
// 214, 228 -> 224, on 74 SMs 317 -> 233, 311 -> 238).
bool small_step_supports(int T, int d, int q_dim, int kv_dim, int F, int head_dim, int n_layers);
// Where it is the faster form.  Up to eight rows at every budget tried (2 .. 148 SMs).  With more, a block's load of the rows is
// what a phase waits for, which wide rows and few blocks lengthen: 13 rows, d_model 2048, on 148 SMs 229 -> 255 us; the talker's 13 on
// 28 / 8 / 2 540 -> 507, 1325 -> 1379, 4524 -> 5031; d_model 768 on 148 / 52 / 28 162 -> 161, 204 -> 187, 297 -> 273; 512 on 28 201 -> 209.
// 75 steps drawn over the sizes that it takes (d_model 256 .. 2048, q_dim 256 .. 2048, d_ffn 256 .. 3072, 4 .. 12 layers, 1 .. 16 rows of up to 4000
// keys, 2 .. 148 SMs; the chain where this says so): 1.00 to 1.7 times as fast as the chain with a copied block of metadata, 1.29 on average.
// The results are the same bits, so the choice may look at the budget.
bool small_step_wins(int T, int d, int q_dim, int sm_budget);
cudaError_t launch_small_step(const SmallStepParams& p, int sm_budget, cudaStream_t stream);
cudaError_t small_step_set_attributes();

// ---------------------------------------------------------------- RMSNorm --
// h[t,:] = bf16(x[t,:] * rsqrt(mean(x[t,:]^2) + eps) * g).  x comes either as bf16 (x_bf16, first layer;
// x_f32_out then receives the widened copy that starts the fp32 residual stream) or as fp32 (x_f32).
struct NormParams {
  const __nv_bfloat16* x_bf16;
  const float* x_f32;
  float* x_f32_out;
  const __nv_bfloat16* gain;
  __nv_bfloat16* h;
  int T, d;
  float eps;
  const int* row_index;      // nullable: input row of output row t is row_index[t] (device int32 [T]); else t
  // optional modulation of a conditioned block: h = rmsnorm(x) g (1 + scale) + shift with the vectors of the
  // row's sequence; mod is this layer's fp32 [max_seqs][6][d], mod_which the row of the shift vector (0 or 3,
  // the scale follows it), tok_seq the sequence of every row.  mod null = none.
  const float* mod;
  const int32_t* tok_seq;
  int mod_which;
  // optional partial sums of the residual GEMM in front (GemmParams::part_rows): x += gate * (part[0] + part[1] + ...),
  // added in split order, written to x_f32_out; gate_which > 0 takes the gate vector from `mod_gate` (the layer's vectors
  // the branch belongs to), else the gate is 1.  h null: only this sum is formed.
  const float* part;         // [n_parts][part_stride] floats, rows of d
  int n_parts;
  size_t part_stride;
  const float* mod_gate;
  int gate_which;
  int sm_count;              // > 0: SMs of the device, for the choice of the kernel (never the budget)
  int h_f16;                 // 1 = write h as fp16, 0 = bf16
  int overlap;               // OverlapMode: how the launch overlaps the previous kernel's drain
  int* status;               // device status word (bounded waits report HS_ERR_TIMEOUT here)
  int* smid_log;             // nullable: SM census slots of this launch
};
cudaError_t launch_rmsnorm(const NormParams& p, int sm_budget, cudaStream_t stream);
constexpr int kNormRowThreads = 512;
constexpr int kNormRowMaxD = kNormRowThreads * 8 * 4;    // widest row of the kernel that adds partial sums
// Threads per row of that kernel: as many as leave one round of rows on the device, with at most eight groups of four
// columns each.
inline int norm_row_threads(int T, int d, int sms) {
  int tpr = kNormRowThreads;
  while (tpr > 32 && (T + kNormRowThreads / tpr - 1) / (kNormRowThreads / tpr) > sms && ((d >> 2) + tpr / 2 - 1) / (tpr / 2) <= 8)
    tpr >>= 1;
  return tpr;
}

// Embedding lookup (head.cu).
struct EmbedParams {
  const int32_t* tokens;           // device [n]
  const __nv_bfloat16* table;      // [vocab, d]
  __nv_bfloat16* x_out;            // [n, d]
  int n, vocab, d;
  int* status;                     // receives HS_ERR_INVALID_ARG for an id outside the table
};
cudaError_t head_set_attributes();
cudaError_t launch_embed(const EmbedParams& p, int sm_budget, cudaStream_t stream);
// dst[i] = fp16(src[i]) for n bf16 values (n a multiple of 8, both 16-byte aligned); used once per weight
// matrix when a stage is created
cudaError_t launch_bf16_to_f16(const void* src, void* dst, size_t n, cudaStream_t stream);
cudaError_t norm_set_attributes();

// -------------------------------------------------------------- attention --
// Tensor map of a whole KV pool from which ONE copy brings the K and the V block of a (page, KV head): dimensions
// {64 elements, rows of one layer's K or V, Dh / 64 halves of a row, K | V blocks of all layers}, box {64, 16, Dh / 64, 2},
// so that it lands as [K | V][half][16 keys][128 bytes] with the 128-byte swizzle.  Lane 0 of a warp issues it between two
// pages, so one request instead of 2 * Dh / 64 shortens every page: step of 29 decode rows at config-3 dimensions, 4
// layers, 96 SMs 810 -> 795 us; talker steps 0.3-0.5 %.  `encode` is cuTensorMapEncodeTiled.
template <typename Encode>
inline bool encode_kv_pages(Encode encode, CUtensorMap* m, const void* pool, int n_layers, int num_pages, int n_kv_heads,
                            int head_dim) {
  const cuuint64_t rows = cuuint64_t(num_pages) * n_kv_heads * 16, halves = cuuint64_t(head_dim) / 64;
  cuuint64_t dims[4] = {64, rows, halves, cuuint64_t(n_layers) * 2};
  cuuint64_t strides[3] = {cuuint64_t(head_dim) * 2, 128, rows * head_dim * 2};
  cuuint32_t box[4] = {64, 16, static_cast<cuuint32_t>(halves), 2};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(pool), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
struct AttnParams {
  CUtensorMap tm_kv;               // prefill kernel: whole pool as rows of Dh bf16: box 64 x 16, 128-byte swizzle
  CUtensorMap tm_kv_page;          // decode kernel: one box = the K and the V block of a (page, KV head) (encode_kv_pages)
  CUtensorMap tm_q;                // q [max_tokens, q_dim]: box 64 x prefill_tokens, 128-byte swizzle
  int prefill_tokens;              // tokens per prefill work item
  int o_f16;                       // 1 = write o as fp16, 0 = bf16 (q, K, V are always bf16)
  int overlap;               // OverlapMode: how the launch overlaps the previous kernel's drain
  const __nv_bfloat16* q;          // [T, q_dim] (after RoPE)
  __nv_bfloat16* o;                // [T, q_dim]
  int n_q_heads, n_kv_heads, head_dim, num_pages, max_pages_per_seq, layer;
  const int32_t* seq_tok0;
  const int32_t* seq_ctx;
  const int32_t* seq_qlen;   // new tokens per sequence (prefill kernel, bidirectional only)
  int bidirectional;         // prefill kernel: 1 = no causal mask, a row sees every key of its sequence
  const int32_t* block_tables;
  const int32_t* prefill_items;    // two int4 per item: {seq, kv head, first token, tokens} {cached tokens, first token
                                   //                    row and new tokens of the sequence, 0}
  int n_prefill_items;
  const int32_t* decode_items;     // two int4 per item: {decode row, kv head, first key, end key}
                                   //                    {seq, token row, first item of its group, splits}
  int n_decode_items;
  int decode_group;                // 1: the items come in eights: a block's eight warps share a slice of a (sequence, KV
                                   //    head)'s pages and meet in shared memory (small batches); first item and splits of
                                   //    the record then count slices
  int decode_sliced;               // 1: group mode, and a group has more than one slice
  const int32_t* decode_rows;      // int4 per decode sequence
  int n_decode_rows;
  float* part_o;                   // [max_decode_items][16][Dh] unnormalised partial outputs
  float* part_ml;                  // [max_decode_items][16][2]  running max (log2 domain) and sum
  int* counters;                   // two work-queue heads of this layer (prefill, decode), zero at entry
  int* group_done;                 // [n_decode_rows * n_kv_heads] finished splits per group, zero at entry
                                   // and left at zero by the kernel
  int* status;
  int* smid_log;                   // nullable: SM census slots; prefill uses [0, 160), decode [160, 320)
};
cudaError_t launch_attention_prefill(const AttnParams& p, int sm_budget, cudaStream_t stream);
cudaError_t launch_attention_decode(const AttnParams& p, int sm_budget, cudaStream_t stream);
cudaError_t attention_set_attributes();
cudaError_t attention_prefill_set_attributes();

}  // namespace hs
