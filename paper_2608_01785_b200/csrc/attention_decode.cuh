// Decode-side causal GQA attention over the paged bf16 KV cache: TMA-staged K/V pages, warp-level
// tensor-core tiles (mma.sync m16n8k16) and an fp32 online softmax in the log2 domain.  (The prefill
// kernel lives in attention_prefill.cu.)
//
//   decode kernel    work item = (sequence, KV head, run of at most 512 keys); rows = the G query heads of the
//                    single new token.  Eight autonomous warps per block, each streaming its own item's
//                    pages through a private TMA ring and writing one partial (max, sum, output) per
//                    item.  HBM-bound: 8 warps x 2 (K page, V page) pairs x 8 KB in flight per SM.
//                    The warp that finishes the last split of a (sequence, KV head) merges that group's
//                    partials in split order (a group with a single split writes its output directly).
// Work items are listed on the host independently of the SM budget and handed out through an atomic
// queue head; an item's result does not depend on which block ran it, and every reduction has a fixed
// order, so outputs are bit-identical across budgets.
//
// A page block [16 keys][Dh] arrives as Dh/64 tiles of [16][64] with the 128-byte swizzle, which makes
// every ldmatrix below bank-conflict free.  Keys past the end of a sequence (the unused tail of its last
// page, or pages of a ragged last block that were never fetched) may hold arbitrary bytes: scores are
// masked by selection and the matching V fragments are zeroed, so they cannot reach the output.
#pragma once
#include <math.h>

#include <type_traits>

#include "kernels.h"
#include "ptx.cuh"

namespace hs {
namespace {

constexpr float kLog2e = 1.4426950408889634f;

template <int DH>
struct Geom {
  static constexpr int HALVES = DH / 64;
  static constexpr int PAGE_BYTES = HALVES * 2048;   // [HALVES][16 keys][128 B]
  static constexpr int CHUNKS = DH / 8;              // 16-byte chunks per row
};

// Byte offset of (key kk, 16-byte chunk cc) inside a page block.
__device__ __forceinline__ int kv_off(int kk, int cc) {
  return (cc >> 3) * 2048 + kk * 128 + (((cc & 7) ^ (kk & 7)) << 4);
}
// Requests the K and the V block of (layer, page, KV head) with one copy: [K | V][half][16 keys][128 B].
template <int DH>
__device__ __forceinline__ void load_page(const AttnParams& p, uint8_t* dst, uint64_t* bar, int page, int hk) {
  tma_load_4d(dst, &p.tm_kv_page, bar, 0, (page * p.n_kv_heads + hk) * 16, 0, p.layer * 2);
}
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
// The same over the eight lanes that share lane % 4, and over the four of those that share lane % 8.
__device__ __forceinline__ float column_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
}
__device__ __forceinline__ float half_column_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 8);
  return v + __shfl_xor_sync(0xffffffffu, v, 16);
}
// Transposes an 8 x 8 matrix of 16-bit values of which lane l holds row l / 4, columns 2 (l % 4) and the next.
__device__ __forceinline__ uint32_t transpose_8x8(uint32_t v) {
  uint32_t t;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(t) : "r"(v));
  return t;
}
// Zeroes the halves of a V fragment register whose keys (k, k + 1) are not below n_valid.
__device__ __forceinline__ uint32_t mask_v(uint32_t r, int k, int n_valid) {
  if (k >= n_valid) return 0u;
  if (k + 1 >= n_valid) return r & 0x0000ffffu;
  return r;
}

// Running state of one warp's attention over the pages of an item: the group's queries, unnormalised outputs, maxima (log2 domain)
// and sums.  page(): one page in shared memory, n_valid keys of which belong to the item (16 or more: all).  put(): what an item
// leaves, output rows `pitch` floats apart and (max, sum) per head.  store(): the normalised output of an item that is a whole
// sequence, with the saturation report of fp16 (see note_f16_saturation).
// A page is a chain of dependent steps in one warp (two warps per scheduler): its latency, not the bytes, is what
// bounds a batch that does not saturate the HBM.  So the scores of a page are two chains of DH / 32 MMAs,
// the V fragments are fetched while the scores are on their way, and a page on which no row's maximum moves --
// most of them, after the first few -- needs a vote, but no shuffles and no rescale.  (A reference that follows the
// maximum only beyond a factor of 256 is another 1 - 2 % faster, but leaves the largest weight rounded: error against
// 64 bits up to 6 % larger.)  Against a loop with one chain of MMAs, shuffles and exp2f on every page and V fetched
// behind the softmax (1250 cycles per page at head_dim 128 with the page already in shared memory): talker step of 16
// rows 300.5 -> 289 us, of 11 rows on 52 SMs 471 -> 457; at config-3 dimensions 9 rows, 4 layers 493 -> 483 us, 29 rows
// on 96 SMs 796 -> 782, 64 rows, 28 layers (HBM-bound) 5.20 -> 5.16 ms.
//
// More than eight heads: the heads are the MMA's sixteen rows; this lane has rows lane / 4 and lane / 4 + 8.
template <int DH>
struct HeadsAsRows {
  uint32_t qf[DH / 16][4];
  float o[DH / 8][4], m_a, m_b, l_a, l_b;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < DH / 8; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
    m_a = m_b = -INFINITY;
    l_a = l_b = 0.f;
  }
  __device__ __forceinline__ void load_q(const __nv_bfloat16* q, int G, int lane) {
    const int ra = lane >> 2, rb = ra + 8;
#pragma unroll
    for (int ks = 0; ks < DH / 16; ++ks) {
      const int c = ks * 16 + 2 * (lane & 3);
      qf[ks][0] = ra < G ? __ldcg(reinterpret_cast<const uint32_t*>(q + ra * DH + c)) : 0u;
      qf[ks][1] = rb < G ? __ldcg(reinterpret_cast<const uint32_t*>(q + rb * DH + c)) : 0u;
      qf[ks][2] = ra < G ? __ldcg(reinterpret_cast<const uint32_t*>(q + ra * DH + c + 8)) : 0u;
      qf[ks][3] = rb < G ? __ldcg(reinterpret_cast<const uint32_t*>(q + rb * DH + c + 8)) : 0u;
    }
  }
  __device__ __forceinline__ void page(uint32_t k_base, uint32_t v_base, int n_valid, int lane, float scale_log2) {
    float sc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float sd[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int ks = 0; ks < DH / 16; ks += 2) {
      uint32_t kf[4], kg[4];
      const int kk = (lane & 7) + (lane >> 4) * 8, cc = 2 * ks + ((lane >> 3) & 1);
      ldmatrix_x4(kf, k_base + kv_off(kk, cc));
      ldmatrix_x4(kg, k_base + kv_off(kk, cc + 2));
      mma_bf16_16816(sc[0], qf[ks], kf[0], kf[1]);
      mma_bf16_16816(sc[1], qf[ks], kf[2], kf[3]);
      mma_bf16_16816(sd[0], qf[ks + 1], kg[0], kg[1]);
      mma_bf16_16816(sd[1], qf[ks + 1], kg[2], kg[3]);
    }
    uint32_t vf[DH / 16][4];
#pragma unroll
    for (int dp = 0; dp < DH / 16; ++dp) {
      const int kk = (lane & 7) + ((lane >> 3) & 1) * 8, cc = 2 * dp + (lane >> 4);
      ldmatrix_x4_trans(vf[dp], v_base + kv_off(kk, cc));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) sc[j][e] += sd[j][e];
    if (n_valid < 16) {
      const int k = 2 * (lane & 3);
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (8 * j + k + (e & 1) >= n_valid) sc[j][e] = -INFINITY;
#pragma unroll
      for (int dp = 0; dp < DH / 16; ++dp)
#pragma unroll
        for (int e = 0; e < 4; ++e) vf[dp][e] = mask_v(vf[dp][e], k + 8 * (e & 1), n_valid);
    }
    const float mx_a = fmaxf(fmaxf(sc[0][0], sc[0][1]), fmaxf(sc[1][0], sc[1][1])) * scale_log2;
    const float mx_b = fmaxf(fmaxf(sc[0][2], sc[0][3]), fmaxf(sc[1][2], sc[1][3])) * scale_log2;
    if (__any_sync(0xffffffffu, mx_a > m_a || mx_b > m_b)) {
      const float mn_a = fmaxf(m_a, quad_max(mx_a)), mn_b = fmaxf(m_b, quad_max(mx_b));
      const float al_a = fast_exp2(m_a - mn_a), al_b = fast_exp2(m_b - mn_b);
      m_a = mn_a;
      m_b = mn_b;
      l_a *= al_a;
      l_b *= al_b;
#pragma unroll
      for (int j = 0; j < DH / 8; ++j) {
        o[j][0] *= al_a; o[j][1] *= al_a;
        o[j][2] *= al_b; o[j][3] *= al_b;
      }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      sc[j][0] = fast_exp2(fmaf(sc[j][0], scale_log2, -m_a));
      sc[j][1] = fast_exp2(fmaf(sc[j][1], scale_log2, -m_a));
      sc[j][2] = fast_exp2(fmaf(sc[j][2], scale_log2, -m_b));
      sc[j][3] = fast_exp2(fmaf(sc[j][3], scale_log2, -m_b));
    }
    l_a += (sc[0][0] + sc[0][1]) + (sc[1][0] + sc[1][1]);
    l_b += (sc[0][2] + sc[0][3]) + (sc[1][2] + sc[1][3]);
    uint32_t pf[4];
    pf[0] = pack_bf16(sc[0][0], sc[0][1]);
    pf[1] = pack_bf16(sc[0][2], sc[0][3]);
    pf[2] = pack_bf16(sc[1][0], sc[1][1]);
    pf[3] = pack_bf16(sc[1][2], sc[1][3]);
#pragma unroll
    for (int dp = 0; dp < DH / 16; ++dp) {
      mma_bf16_16816(o[2 * dp], pf, vf[dp][0], vf[dp][1]);
      mma_bf16_16816(o[2 * dp + 1], pf, vf[dp][2], vf[dp][3]);
    }
  }
  __device__ __forceinline__ void put(float* po, int pitch, float2* pml, int G, int lane) {
    const int ra = lane >> 2, rb = ra + 8;
    l_a = quad_sum(l_a);
    l_b = quad_sum(l_b);
#pragma unroll
    for (int j = 0; j < DH / 8; ++j) {
      const int col = 8 * j + 2 * (lane & 3);
      if (ra < G) *reinterpret_cast<float2*>(po + ra * pitch + col) = make_float2(o[j][0], o[j][1]);
      if (rb < G) *reinterpret_cast<float2*>(po + rb * pitch + col) = make_float2(o[j][2], o[j][3]);
    }
    if ((lane & 3) == 0) {
      if (ra < G) pml[ra] = make_float2(m_a, l_a);
      if (rb < G) pml[rb] = make_float2(m_b, l_b);
    }
  }
  __device__ __forceinline__ void store(__nv_bfloat16* out, bool f16, int* status, int G, int lane) {
    const int ra = lane >> 2, rb = ra + 8;
    const float inv_a = 1.f / quad_sum(l_a), inv_b = 1.f / quad_sum(l_b);
#pragma unroll
    for (int j = 0; j < DH / 8; ++j) {
      const int col = 8 * j + 2 * (lane & 3);
      const float a[2] = {o[j][0], o[j][1]}, b[2] = {o[j][2], o[j][3]};
      if (ra < G) {
        if (f16) note_f16_saturation(a, status, inv_a);
        *reinterpret_cast<uint32_t*>(out + ra * DH + col) = pack_act(a[0] * inv_a, a[1] * inv_a, f16);
      }
      if (rb < G) {
        if (f16) note_f16_saturation(b, status, inv_b);
        *reinterpret_cast<uint32_t*>(out + rb * DH + col) = pack_act(b[0] * inv_b, b[1] * inv_b, f16);
      }
    }
  }
};
// At most eight: the keys are the rows of the scores' MMA and the head dimension those of the outputs', the heads their eight
// columns, so that no half of a tile is padding: half the MMAs, and as an MMA takes its scheduler ten cycles, they were most of a
// page (in shared memory, cycles at head_dim 128 / 64: 784 -> 597, 473 -> 392).  This lane has heads 2 (lane % 4) and the next one; keys, and
// dimensions, lane / 4 and lane / 4 + 8.  The scores become the second product's operand by two 8 x 8 transpositions.
// The weights of a head are added in the order of HeadsAsRows, so that a group's bits do not depend on the form: keys 2 i, 2 i + 1,
// 2 i + 8 and 2 i + 9 of a page in one lane, page after page, then the four lanes.  Lanes 8 i .. 8 i + 3 do that for their even head,
// lanes 8 i + 4 .. 8 i + 7 for the odd one; they give each other what they lack.
// Steps, us: eleven rows of the talker on 52 SMs 368 -> 364, 16 on 148 260.2 -> 259.6; at 7B dimensions 29 rows on 96 SMs 642 -> 639, 64
// rows 4801 -> 4787.  (Of that the order of the weights takes back 0 to 0.2 %: against eight lanes that add two keys each, 64 rows
// 4622.8 -> 4628.3, 29 rows on 96 SMs 633.3 -> 634.1, sixteen of the talker 260.2 -> 260.2.)
template <int DH>
struct HeadsAsColumns {
  uint32_t qf[DH / 16][2];
  float o[DH / 16][4], m[2], l;               // (l: of the even head in lanes with an even key, of the odd one in the others)
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < DH / 16; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
    m[0] = m[1] = -INFINITY;
    l = 0.f;
  }
  __device__ __forceinline__ void load_q(const __nv_bfloat16* q, int G, int lane) {
    const int h = lane >> 2;
#pragma unroll
    for (int ks = 0; ks < DH / 16; ++ks)
#pragma unroll
      for (int e = 0; e < 2; ++e) qf[ks][e] = h < G ? __ldcg(reinterpret_cast<const uint32_t*>(q + h * DH + ks * 16 + 8 * e + 2 * (lane & 3))) : 0u;
  }
  __device__ __forceinline__ void page(uint32_t k_base, uint32_t v_base, int n_valid, int lane, float scale_log2) {
    const int key = lane >> 2;
    const bool odd = (lane & 4) != 0;
    float s[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
    {
      const int kk = (lane & 7) + ((lane >> 3) & 1) * 8, cc = lane >> 4;
#pragma unroll
      for (int ks = 0; ks < DH / 16; ks += 2) {
        uint32_t kf[4], kg[4];
        ldmatrix_x4(kf, k_base + kv_off(kk, 2 * ks + cc));
        ldmatrix_x4(kg, k_base + kv_off(kk, 2 * ks + 2 + cc));
        mma_bf16_16816(s, kf, qf[ks][0], qf[ks][1]);
        mma_bf16_16816(s2, kg, qf[ks + 1][0], qf[ks + 1][1]);
      }
    }
    uint32_t vf[DH / 16][4];
    {
      const int kk = (lane & 7) + (lane >> 4) * 8, cc = (lane >> 3) & 1;
#pragma unroll
      for (int dp = 0; dp < DH / 16; ++dp) ldmatrix_x4_trans(vf[dp], v_base + kv_off(kk, 2 * dp + cc));
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e] += s2[e];
    if (n_valid < 16) {
      if (key >= n_valid) s[0] = s[1] = -INFINITY;
      if (key + 8 >= n_valid) s[2] = s[3] = -INFINITY;
#pragma unroll
      for (int dp = 0; dp < DH / 16; ++dp)
#pragma unroll
        for (int e = 0; e < 4; ++e) vf[dp][e] = mask_v(vf[dp][e], 2 * (lane & 3) + 8 * (e >> 1), n_valid);
    }
    const float mx0 = fmaxf(s[0], s[2]) * scale_log2, mx1 = fmaxf(s[1], s[3]) * scale_log2;
    if (__any_sync(0xffffffffu, mx0 > m[0] || mx1 > m[1])) {
      const float mn0 = fmaxf(m[0], column_max(mx0)), mn1 = fmaxf(m[1], column_max(mx1));
      const float al0 = fast_exp2(m[0] - mn0), al1 = fast_exp2(m[1] - mn1);
      m[0] = mn0;
      m[1] = mn1;
      l *= odd ? al1 : al0;
#pragma unroll
      for (int j = 0; j < DH / 16; ++j) {
        o[j][0] *= al0; o[j][1] *= al1;
        o[j][2] *= al0; o[j][3] *= al1;
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e] = fast_exp2(fmaf(s[e], scale_log2, -m[e & 1]));
    const float near_ = (odd ? s[1] : s[0]) + __shfl_xor_sync(0xffffffffu, odd ? s[0] : s[1], 4);
    const float far_ = (odd ? s[3] : s[2]) + __shfl_xor_sync(0xffffffffu, odd ? s[2] : s[3], 4);
    l += near_ + far_;
    const uint32_t p0 = transpose_8x8(pack_bf16(s[0], s[1])), p1 = transpose_8x8(pack_bf16(s[2], s[3]));
#pragma unroll
    for (int dp = 0; dp < DH / 16; ++dp) mma_bf16_16816(o[dp], vf[dp], p0, p1);
  }
  __device__ __forceinline__ void put(float* po, int pitch, float2* pml, int G, int lane) {
    const int d = lane >> 2, h = 2 * (lane & 3);
    l = half_column_sum(l);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (h + e < G) {
#pragma unroll
        for (int j = 0; j < DH / 16; ++j) {
          po[(h + e) * pitch + 16 * j + d] = o[j][e];
          po[(h + e) * pitch + 16 * j + d + 8] = o[j][e + 2];
        }
        if (d == e) pml[h + e] = make_float2(m[e], l);
      }
    }
  }
  __device__ __forceinline__ void store(__nv_bfloat16* out, bool f16, int* status, int G, int lane) {
    const int d = lane >> 2, h = 2 * (lane & 3);
    l = half_column_sum(l);
    const float other = __shfl_xor_sync(0xffffffffu, l, 4);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float inv = 1.f / ((d & 1) == e ? l : other);
      if (h + e < G) {
#pragma unroll
        for (int j = 0; j < DH / 16; ++j) {
          const float v[2] = {o[j][e], o[j][e + 2]};
          if (f16) note_f16_saturation(v, status, inv);
          const uint32_t w = pack_act(v[0] * inv, v[1] * inv, f16);
          uint16_t* at = reinterpret_cast<uint16_t*>(out) + (h + e) * DH + 16 * j + d;
          at[0] = uint16_t(w);
          at[8] = uint16_t(w >> 16);
        }
      }
    }
  }
};
template <int DH, bool TWO>
using Heads = std::conditional_t<TWO, HeadsAsRows<DH>, HeadsAsColumns<DH>>;

// Merges the partials of one (sequence, KV head) group -- items first .. first + splits - 1 -- in split
// order and writes the normalised output rows.  LPH lanes share one query head, each owning DH / LPH
// contiguous columns.  A lone warp does this at the tail of the kernel, so what counts is latency: the
// partial outputs travel by asynchronous copies into the warp's own (now idle) page ring, used as two
// halves of PS splits each -- while one half is folded into the running sum the other is in flight -- laid
// out [split][float4 index][lane] so that every lane reads back only what it copied itself, conflict-free.
// The running maximum is updated per half (online rescaling); the order of all operations is fixed.
template <int DH, int LPH, int RING_BYTES>
__device__ __forceinline__ void merge_group(const float* part_o, const float* part_ml, uint8_t* ring, int first,
                                            int splits, int G, int lane, __nv_bfloat16* orow, bool f16, int* status) {
  constexpr int NV = DH / 4 / LPH;                 // float4 per lane and split
  constexpr int PS = RING_BYTES / 2 / (NV * 512) < 4 ? RING_BYTES / 2 / (NV * 512) : 4;   // splits per half
  static_assert(PS >= 1, "half a ring holds one split");
  const int g = lane / LPH, part = lane % LPH;
  if (g < G) {
    const float2* ml_g = reinterpret_cast<const float2*>(part_ml) + size_t(first) * 16 + g;   // + j * 16
    const uint32_t ring_u32 = smem_u32(ring) + lane * 16;
    const float4* ring_f4 = reinterpret_cast<const float4*>(ring) + lane;
    float2 mlv[2][PS];
    auto request = [&](int j0, int half) {         // splits j0 .. j0 + PS - 1 into one half of the ring
#pragma unroll
      for (int u = 0; u < PS; ++u) {
        if (j0 + u < splits) {
          const float4* src = reinterpret_cast<const float4*>(part_o + (size_t(first + j0 + u) * 16 + g) * DH) + part * NV;
#pragma unroll
          for (int i = 0; i < NV; ++i)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring_u32 + ((half * PS + u) * NV + i) * 512),
                         "l"(src + i)
                         : "memory");
          mlv[half][u] = __ldcg(&ml_g[size_t(j0 + u) * 16]);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float mm = -INFINITY, ll = 0.f;
    float4 acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    request(0, 0);
    request(PS, 1);
    int half = 0;
    for (int j0 = 0; j0 < splits; j0 += PS, half ^= 1) {
      asm volatile("cp.async.wait_group 1;" ::: "memory");     // the older of the two halves has landed
      float pm = mm;
      if (half == 0) {
#pragma unroll
        for (int u = 0; u < PS; ++u) if (j0 + u < splits) pm = fmaxf(pm, mlv[0][u].x);
      } else {
#pragma unroll
        for (int u = 0; u < PS; ++u) if (j0 + u < splits) pm = fmaxf(pm, mlv[1][u].x);
      }
      const float sc = exp2f(mm - pm);                         // 0 on the first half (mm = -inf)
      mm = pm;
      ll *= sc;
#pragma unroll
      for (int i = 0; i < NV; ++i) { acc[i].x *= sc; acc[i].y *= sc; acc[i].z *= sc; acc[i].w *= sc; }
#pragma unroll
      for (int u = 0; u < PS; ++u) {
        if (j0 + u < splits) {
          const float2 ml = half == 0 ? mlv[0][u] : mlv[1][u];
          const float f = exp2f(ml.x - mm);
          ll += f * ml.y;
#pragma unroll
          for (int i = 0; i < NV; ++i) {
            const float4 v = ring_f4[((half * PS + u) * NV + i) * 32];
            acc[i].x += f * v.x; acc[i].y += f * v.y; acc[i].z += f * v.z; acc[i].w += f * v.w;
          }
        }
      }
      if (half == 0) request(j0 + 2 * PS, 0);                  // refill the half just read (may be empty)
      else request(j0 + 2 * PS, 1);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const float inv = 1.f / ll;
    if (f16) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float v4[4] = {acc[i].x, acc[i].y, acc[i].z, acc[i].w};
        note_f16_saturation(v4, status, inv);
      }
    }
    __nv_bfloat16* dst = orow + g * DH + part * NV * 4;
#pragma unroll
    for (int i = 0; i < NV; ++i)
      *reinterpret_cast<uint2*>(dst + 4 * i) =
          make_uint2(pack_act(acc[i].x * inv, acc[i].y * inv, f16), pack_act(acc[i].z * inv, acc[i].w * inv, f16));
  }
  // the ring goes back to the copy engine for the next item: order these generic-proxy accesses before it
  fence_proxy_async();
  __syncwarp();
}

// ==================================================================== decode ==
// Every warp is its own pipeline: it pulls a work item from the queue, streams the item's pages through
// a private ring of DC_STAGES (K page, V page) slots that its lane 0 fills by TMA a few pages ahead, and
// writes the item's partial (max, sum, output) straight from its registers.  There is no producer warp,
// no "slot free" barrier (a slot is refilled by the warp that has just finished reading it) and no
// block-level synchronisation after start-up, so an SM keeps DC_WARPS x (DC_STAGES - 1) pages in flight.
// Measured on B200 (warps x slots of 8 KB, the 192 KB an SM offers): 8 x 3 and 6 x 4 take the same time at the full
// budget (config-3 decode tick 5.17 / 5.15 ms), 8 x 3 is 5-8 % faster at 74 and 37 SMs, 4 x 6 is 9 % slower everywhere.
constexpr int DC_WARPS = kDecodeKernelWarps, DC_THREADS = DC_WARPS * 32, DC_STAGES = 3;

template <int DH>
constexpr int dc_smem_bytes() {
  int b = 1024 + DC_WARPS * DC_STAGES * 2 * Geom<DH>::PAGE_BYTES + 512;
  return b > kMinSmemBytes ? b : kMinSmemBytes;
}

// Floats between the heads of a warp's part of a slice in shared memory (conflict-free for HeadsAsColumns::put).
template <int DH>
constexpr int kPartPitch = DH + 4;
// The eight warps' parts of a slice, [ROWS][kPartPitch] output and [ROWS] (max, sum) each, PITCH bytes apart, merged in order: head g, columns col and col + 1, unnormalised, with the
// maximum and the sum.
template <int DH, int ROWS, int PITCH, int UNROLL = DC_WARPS>
__device__ __forceinline__ void merge_eight(const uint8_t* parts, int g, int col, float& mm, float& ll, float& o0, float& o1) {
  mm = -INFINITY;
#pragma unroll UNROLL
  for (int w = 0; w < DC_WARPS; ++w) mm = fmaxf(mm, reinterpret_cast<const float2*>(parts + w * PITCH + ROWS * kPartPitch<DH> * 4)[g].x);
  ll = 0.f, o0 = 0.f, o1 = 0.f;
#pragma unroll UNROLL
  for (int w = 0; w < DC_WARPS; ++w) {
    const uint8_t* base = parts + w * PITCH;
    const float2 ml = reinterpret_cast<const float2*>(base + ROWS * kPartPitch<DH> * 4)[g];
    const float f = exp2f(ml.x - mm);                 // 0 for an empty slice (max = -inf)
    const float2 v = *reinterpret_cast<const float2*>(reinterpret_cast<const float*>(base) + g * kPartPitch<DH> + col);
    ll += f * ml.y;
    o0 += f * v.x;
    o1 += f * v.y;
  }
}
// The next eight (or `left`) slices of a group: their (max, sum) and two columns of their outputs into the running ones.
__device__ __forceinline__ void merge_slices(const float2 (&ml)[8], const float2 (&ov)[8], int left, float& mm, float& ll, float& o0, float& o1) {
  float pm = mm;
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (u < left) pm = fmaxf(pm, ml[u].x);
  const float sc = exp2f(mm - pm);                 // 0 the first time (mm = -inf)
  mm = pm;
  ll *= sc; o0 *= sc; o1 *= sc;
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (u < left) {
      const float f = exp2f(ml[u].x - mm);
      ll += f * ml[u].y;
      o0 += f * ov[u].x;
      o1 += f * ov[u].y;
    }
}

// The body of the decode kernel.  `smem`: 1024-byte aligned, DC_WARPS * DC_STAGES * 2 pages; `full_all`: DC_WARPS *
// DC_STAGES mbarriers followed by two ints (the abort flag; a flag of the block's) in shared memory outside that area.
// SLICED: group mode with groups of several slices (the merge of those is no part of the other instantiation: it was 2 us of the
// talker step of 16 rows, twelve launches, that has none).  TWO: groups of more than eight heads (Heads).
template <int DH, bool SLICED, bool TWO>
__device__ __forceinline__ void attn_decode_body(const AttnParams& p, uint8_t* smem, uint64_t* full_all) {
  using G_ = Geom<DH>;
  constexpr int SLOT_BYTES = 2 * G_::PAGE_BYTES;    // K page then V page
  volatile int* abort_flag = reinterpret_cast<volatile int*>(full_all + DC_WARPS * DC_STAGES);
  volatile int* block_flag = abort_flag + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int block = int(blockIdx.x), n_blocks = int(gridDim.x);
  const int G = TWO ? p.n_q_heads / p.n_kv_heads : min(p.n_q_heads / p.n_kv_heads, 8);     // (so that the compiler knows)
  const int q_dim = p.n_q_heads * DH;
  const float scale_log2 = kLog2e / sqrtf(float(DH));
  constexpr int kRows = TWO ? 16 : 8;               // heads that a warp's part of a slice has room for
  static_assert(kRows * kPartPitch<DH> * 4 + kRows * 8 <= DC_STAGES * SLOT_BYTES, "in the warp's ring");

  if (threadIdx.x == 0) {
    for (int i = 0; i < DC_WARPS * DC_STAGES; ++i) mbar_init(&full_all[i], 1);
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&p.tm_kv_page);
  }
  __syncthreads();

  uint8_t* slots = smem + warp * DC_STAGES * SLOT_BYTES;
  uint64_t* full = full_all + warp * DC_STAGES;
  int fill = 0;                           // ring slot of the next page to request, over all items of this warp
  int cur = 0;                            // ring slot of the next page to read, and its phase
  uint32_t cur_phase = 0;
  auto issue = [&](int page, int hk) {      // lane 0: request one page of an item
    mbar_expect_tx(&full[fill], SLOT_BYTES);
    load_page<DH>(p, slots + fill * SLOT_BYTES, &full[fill], page, hk);
    if (++fill == DC_STAGES) fill = 0;
  };

  // A warp's first item is its own index in the grid (no round trip to the queue head before the first page request);
  // the queue hands out the items after those.  The first item's record, its page ids and those of its first pages
  // that lie wholly inside the cached context are fetched before the wait for the previous kernel: the step's
  // metadata is there since two launches at least (see launch_fetch_metadata), and this step writes K / V at positions >= ctx only.
  int item = block * DC_WARPS + warp;
  int4 it = make_int4(0, 0, 0, 0), dr = it;
  int my_page = 0, ahead = 0;             // ahead: pages of the current item already requested
  if (item < p.n_decode_items) {
    it = reinterpret_cast<const int4*>(p.decode_items)[2 * item];
    dr = reinterpret_cast<const int4*>(p.decode_items)[2 * item + 1];
    const int n_pages = (it.w - it.z + 15) >> 4;
    my_page = lane < n_pages ? p.block_tables[size_t(dr.x) * p.max_pages_per_seq + (it.z >> 4) + lane] : 0;
    const int ctx = p.seq_ctx[dr.x];
#pragma unroll
    for (int pi = 0; pi < DC_STAGES - 1; ++pi) {
      const int page = __shfl_sync(0xffffffffu, my_page, pi);
      const bool stable = pi < n_pages && it.z + (pi + 1) * 16 <= ctx && ahead == pi;
      if (stable) {
        if (lane == 0) issue(page, it.y);
        ++ahead;
      }
    }
  }
  griddep_wait();
  griddep_launch_dependents(p.overlap);

  // Group mode (p.decode_group, a batch small enough that one round of blocks reads all of it): a group = (sequence, KV
  // head) is cut into slices of whole pages, item 8 i + w is the w-th eighth of slice i; a block takes whole slices -- i =
  // block, block + n_blocks, ... -- and its eight warps' partial results meet in the block's shared memory.  A group of
  // several slices leaves one partial result per slice in global memory, and the block that delivers the last one merges
  // them in slice order.  Every warp of the block goes through the same barriers whatever happens to it.
  const bool group_mode = p.decode_group != 0;
  bool first_round = true;
  for (int round = 0;; ++round) {
    if (!first_round) {
      if (group_mode) {
        item = (block + round * n_blocks) * DC_WARPS + warp;
      } else {
        if (lane == 0) item = n_blocks * DC_WARPS + atomicAdd(p.counters + 1, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
      }
    }
    if (item >= p.n_decode_items || (!group_mode && *abort_flag)) break;
    // one 32-byte record: {decode row, kv head, first key, end key} {seq, token row, the group's first partial slot,
    // splits | index within the group << 16}: the queue hands the items out longest first, the partials of a group
    // stay in key order
    if (!first_round) {
      it = reinterpret_cast<const int4*>(p.decode_items)[2 * item];
      dr = reinterpret_cast<const int4*>(p.decode_items)[2 * item + 1];
      ahead = 0;
    }
    const int drow = it.x, hk = it.y, k0 = it.z, k1 = it.w;
    const int seq = dr.x, tok = dr.y, splits = dr.w & 0xffff, part = dr.z + (dr.w >> 16);
    const int n_pages = (k1 - k0 + 15) >> 4;
    // the item's page ids, one per lane, fetched with a single load: reading the block table page by page
    // would put one dependent round trip to memory in front of every request
    if (!first_round) {
      const int32_t* table = p.block_tables + size_t(seq) * p.max_pages_per_seq + (k0 >> 4);
      my_page = lane < n_pages ? table[lane] : 0;      // the planner keeps items within 32 pages
    }
    first_round = false;
#pragma unroll
    for (int pi = 0; pi < DC_STAGES - 1; ++pi) {
      const int page = __shfl_sync(0xffffffffu, my_page, pi);
      if (lane == 0 && pi >= ahead && pi < n_pages) issue(page, hk);
    }

    // Q fragments straight from global memory: rows = query heads hk*G .. hk*G + G - 1 of the new token
    const __nv_bfloat16* qrow = p.q + size_t(tok) * q_dim + size_t(hk) * G * DH;
    Heads<DH, TWO> at;
    at.load_q(qrow, G, lane);
    at.clear();
    bool ok = true;

    for (int pi = 0; pi < n_pages; ++pi) {
      // the slot read in the previous iteration is free: keep DC_STAGES - 1 pages in flight
      const int page_ahead = __shfl_sync(0xffffffffu, my_page, (pi + DC_STAGES - 1) & 31);
      if (lane == 0 && pi + DC_STAGES - 1 < n_pages) issue(page_ahead, hk);
      ok = mbar_wait(&full[cur], cur_phase, abort_flag, p.status);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      const uint32_t k_base = smem_u32(slots + cur * SLOT_BYTES);
      const uint32_t v_base = k_base + G_::PAGE_BYTES;
      if (++cur == DC_STAGES) { cur = 0; cur_phase ^= 1; }
      const int n_valid = k1 - (k0 + pi * 16);            // keys of this page that belong to the item
      at.page(k_base, v_base, n_valid, lane, scale_log2);
      __syncwarp();                         // every lane is done with this slot before lane 0 refills it
    }
    if (!ok && !group_mode) break;

    __nv_bfloat16* orow = p.o + size_t(tok) * q_dim + size_t(hk) * G * DH;
    if (group_mode) {
      // this slice's part into the warp's own (now idle) page ring
      at.put(reinterpret_cast<float*>(slots), kPartPitch<DH>, reinterpret_cast<float2*>(slots + kRows * kPartPitch<DH> * 4), G, lane);
      const bool failed = __syncthreads_or(!ok) != 0;      // the same answer in every warp of the block
      if (!failed) {
        // the eight partials are merged in order by the whole block: a thread per pair of output columns
        const bool f16 = p.o_f16 != 0;
        auto store = [&](int g, int col, float o0, float o1, float ll) {
          const float inv = 1.f / ll;
          if (f16) {
            const float v2[2] = {o0, o1};
            note_f16_saturation(v2, p.status, inv);
          }
          *reinterpret_cast<uint32_t*>(orow + g * DH + col) = pack_act(o0 * inv, o1 * inv, f16);
        };
        for (int e = threadIdx.x; e < G * (DH / 2); e += DC_THREADS) {
          const int g = e / (DH / 2), col = 2 * (e - g * (DH / 2));
          float mm, ll, o0, o1;
          merge_eight<DH, kRows, DC_STAGES * SLOT_BYTES>(smem, g, col, mm, ll, o0, o1);
          if (!SLICED || splits == 1) {
            store(g, col, o0, o1, ll);
          } else {
            __stcg(reinterpret_cast<float2*>(p.part_o + (size_t(part) * 16 + g) * DH + col), make_float2(o0, o1));
            if (col == 0) __stcg(reinterpret_cast<float2*>(p.part_ml) + size_t(part) * 16 + g, make_float2(mm, ll));
          }
        }
        if (SLICED && splits > 1) {
          // the block that delivers the group's last slice merges all of them, in slice order whoever it is
          __threadfence();
          __syncthreads();
          int* done = p.group_done + drow * p.n_kv_heads + hk;
          if (threadIdx.x == 0) *block_flag = atomicAdd(done, 1) == splits - 1;
          __syncthreads();
          if (*block_flag) {
            __threadfence();
            for (int e = threadIdx.x; e < G * (DH / 2); e += DC_THREADS) {
              const int g = e / (DH / 2), col = 2 * (e - g * (DH / 2));
              const float2* ml_g = reinterpret_cast<const float2*>(p.part_ml) + size_t(dr.z) * 16 + g;
              const float* po_g = p.part_o + (size_t(dr.z) * 16 + g) * DH + col;
              float mm = -INFINITY, ll = 0.f, o0 = 0.f, o1 = 0.f;
              for (int j0 = 0; j0 < splits; j0 += 8) {       // eight slices on their way at a time
                float2 ml[8], ov[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const int j = min(j0 + u, splits - 1);
                  ml[u] = __ldcg(ml_g + size_t(j) * 16);
                  ov[u] = __ldcg(reinterpret_cast<const float2*>(po_g + size_t(j) * 16 * DH));
                }
                merge_slices(ml, ov, splits - j0, mm, ll, o0, o1);
              }
              store(g, col, o0, o1, ll);
            }
            if (threadIdx.x == 0) *done = 0;                 // ready for the next launch
          }
        }
      }
      // the rings go back to the copy engine: order these generic-proxy accesses before its next writes
      fence_proxy_async();
      __syncthreads();
      if (failed) break;
      continue;
    }
    if (splits == 1) {
      // the whole key range was this item: normalise and write the output rows directly
      at.store(orow, p.o_f16 != 0, p.status, G, lane);
      continue;
    }
    // the item's partial: unnormalised output, running max (log2 domain) and sum, rows = query heads
    at.put(p.part_o + size_t(part) * 16 * DH, DH, reinterpret_cast<float2*>(p.part_ml) + size_t(part) * 16, G, lane);
    // The warp that completes the last split of a (sequence, KV head) merges all of its splits, always in
    // split order, so the result does not depend on which warp that is.
    __threadfence();
    __syncwarp();
    int* done = p.group_done + drow * p.n_kv_heads + hk;
    int last = 0;
    if (lane == 0) last = atomicAdd(done, 1) == splits - 1;
    last = __shfl_sync(0xffffffffu, last, 0);
    if (last) {
      __threadfence();
      const int first = dr.z;
      if (G <= 8) merge_group<DH, 4, DC_STAGES * SLOT_BYTES>(p.part_o, p.part_ml, slots, first, splits, G, lane, orow, p.o_f16 != 0, p.status);
      else merge_group<DH, 2, DC_STAGES * SLOT_BYTES>(p.part_o, p.part_ml, slots, first, splits, G, lane, orow, p.o_f16 != 0, p.status);
      if (lane == 0) *done = 0;             // ready for the next launch
    }
  }
  __syncthreads();
  if (*abort_flag) drain_after_abort();
}


}  // namespace
}  // namespace hs
