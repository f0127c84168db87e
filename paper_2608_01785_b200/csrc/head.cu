// The embedding lookup in front of hs_stage_step, SM-budgeted like every other kernel of the library: a persistent grid of
// at most sm_budget blocks that ask for more than half of an SM's shared memory, so one block per SM.  (Greedy sampling
// behind the step is part of the vocabulary GEMM's epilogue: GemmParams::argmax_key.)
#include "kernels.h"
#include "ptx.cuh"

namespace hs {
namespace {

constexpr int HEAD_THREADS = 512;

// x_out[t, :] = table[tokens[t], :] with 16-byte loads and stores: `tpr` threads per row, as many as leave one round of
// rows on the budget's SMs (65 rows of 3584 with a warp each took 11 us).  An id outside the table yields zeros and flags
// the status word.
__global__ void __launch_bounds__(HEAD_THREADS, 1) embed_kernel(const EmbedParams p, int tpr) {
  extern __shared__ uint8_t unused_smem[];
  griddep_wait();
  const int d8 = p.d >> 3, rows = HEAD_THREADS / tpr, group = threadIdx.x / tpr, tid = threadIdx.x - group * tpr;
  for (int t = blockIdx.x * rows + group; t < p.n; t += gridDim.x * rows) {
    const int id = p.tokens[t];
    const bool ok = id >= 0 && id < p.vocab;
    if (!ok && tid == 0) atomicExch(p.status, kErrInvalidArg);
    const uint4* src = reinterpret_cast<const uint4*>(p.table + size_t(ok ? id : 0) * p.d);
    uint4* dst = reinterpret_cast<uint4*>(p.x_out + size_t(t) * p.d);
    for (int i = tid; i < d8; i += tpr) dst[i] = ok ? src[i] : make_uint4(0, 0, 0, 0);
  }
}

}  // namespace

cudaError_t head_set_attributes() {
  return set_kernel_smem(embed_kernel, kMinSmemBytes);
}

cudaError_t launch_embed(const EmbedParams& p, int sm_budget, cudaStream_t stream) {
  if (p.n <= 0) return cudaSuccess;
  int tpr = HEAD_THREADS;
  while (tpr > 32 && (p.n + HEAD_THREADS / tpr - 1) / (HEAD_THREADS / tpr) > sm_budget) tpr >>= 1;
  const int rows = HEAD_THREADS / tpr, blocks = (p.n + rows - 1) / rows;
  // (every kernel of the library waits for its predecessor itself, so the launch may be issued ahead of its completion)
  return launch_step_kernel(embed_kernel, blocks < sm_budget ? blocks : sm_budget, HEAD_THREADS, kMinSmemBytes, stream,
                            true, p, tpr);
}

}  // namespace hs
