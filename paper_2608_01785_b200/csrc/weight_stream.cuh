// What the kernels that stream weights past a few activation rows share (gemm_skinny.cu, small_step.cu): warp-level MMAs,
// asynchronous copies, wide accesses of a thread's epilogue columns, the folded RMSNorm's factor.
#pragma once
#include <cuda_fp16.h>

#include "kernels.h"
#include "ptx.cuh"

namespace hs {
namespace {

constexpr int SK_WARPS = 8, SK_THREADS = SK_WARPS * 32;

template <bool F16>
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  if (F16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// cp.async.cg reads through the L2 only: right for weights that are used once and for activations that the
// kernel before this one wrote (it may still be draining when this kernel starts).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// N values with the widest accesses: N * 4 bytes (N * 2 where 16-bit values are stored), aligned to their size or to 16.
template <int N>
__device__ __forceinline__ void lds_f32(float* v, const float* src) {
  if constexpr (N == 2) {
    const float2 t = *reinterpret_cast<const float2*>(src);
    v[0] = t.x; v[1] = t.y;
  } else {
    const float4 t = *reinterpret_cast<const float4*>(src);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  }
}
template <int N>
__device__ __forceinline__ void ldcg_f32(float (&v)[N], const float* src) {      // through the L2
#pragma unroll
  for (int i = 0; i < N; i += 4) {
    const float4 t = __ldcg(reinterpret_cast<const float4*>(src + i));
    v[i] = t.x; v[i + 1] = t.y; v[i + 2] = t.z; v[i + 3] = t.w;
  }
}
template <int N>
__device__ __forceinline__ void ldg_f32(float (&v)[N], const float* src) {
#pragma unroll
  for (int i = 0; i < N; i += 4) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(src + i));
    v[i] = t.x; v[i + 1] = t.y; v[i + 2] = t.z; v[i + 3] = t.w;
  }
}
template <int N>
__device__ __forceinline__ void ldg_u32(uint32_t (&v)[N], const __nv_bfloat16* src) {
  if constexpr (N == 1) {
    v[0] = __ldg(reinterpret_cast<const uint32_t*>(src));
  } else if constexpr (N == 2) {
    const uint2 t = __ldg(reinterpret_cast<const uint2*>(src));
    v[0] = t.x; v[1] = t.y;
  } else {
    const uint4 t = __ldg(reinterpret_cast<const uint4*>(src));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  }
}
template <int N>
__device__ __forceinline__ void stg_f32(float* dst, const float (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += 4) *reinterpret_cast<float4*>(dst + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
}
template <int N>
__device__ __forceinline__ void stg_act(__nv_bfloat16* dst, const float* v, bool f16) {
  uint32_t w[N / 2];
#pragma unroll
  for (int e = 0; e < N / 2; ++e) w[e] = pack_act(v[2 * e], v[2 * e + 1], f16);
  if constexpr (N == 2) *reinterpret_cast<uint32_t*>(dst) = w[0];
  else if constexpr (N == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
  else *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}

// First element of (slot, kv head) in one layer's K or V pages: [page][kv_head][16][Dh].
__device__ __forceinline__ __nv_bfloat16* cache_row(__nv_bfloat16* base, int slot, int hk, int n_kv_heads, int Dh) {
  return base + ((size_t(slot >> 4) * n_kv_heads + hk) * 16 + (slot & 15)) * Dh;
}

// Folded RMSNorm: r = rsqrt(mean(x^2) + eps) of row threadIdx / 16 (16 rows at most) from its n partial sums of squares, one
// per 16 columns: the row's sixteen threads take every sixteenth partial each and then combine, a fixed order whoever
// calls.  In two halves, so that the K loop runs while the partials travel.  Called by all threads of the block.
constexpr int kSsPre = 16;             // partials a thread asks for ahead (all of them up to a width of 4096)
__device__ __forceinline__ void row_norm_request(float (&v)[kSsPre], const float* row_ss, int stride, int n, int T) {
  const int row = threadIdx.x >> 4, q = threadIdx.x & 15;
#pragma unroll
  for (int u = 0; u < kSsPre; ++u) v[u] = row < T && q + 16 * u < n ? __ldcg(row_ss + size_t(row) * stride + q + 16 * u) : 0.f;
}
__device__ __forceinline__ float row_norm_factor(const float (&v)[kSsPre], const float* row_ss, int stride, int n, int T, int width, float eps) {
  const int row = threadIdx.x >> 4, q = threadIdx.x & 15;
  float sum = 0.f;
#pragma unroll
  for (int u = 0; u < kSsPre; ++u) sum += v[u];
  if (row < T)
    for (int i = q + 16 * kSsPre; i < n; i += 16) sum += __ldcg(row_ss + size_t(row) * stride + i);
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return rsqrtf(sum / float(width) + eps);
}

}  // namespace
}  // namespace hs
