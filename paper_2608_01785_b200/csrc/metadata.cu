// The step's first kernel: brings the metadata block from the stage's pinned host memory into the workspace.
#include "kernels.h"
#include "ptx.cuh"

namespace hs {
namespace {

constexpr int META_THREADS = 256;

// What bounds it is the way over PCIe, once; so every thread asks for one 16-byte group, all blocks at the same time, and before
// the wait for the kernel in front: nothing on the device writes the host's block, and the workspace's is written after the wait.
// (The kernel behind is let go after the wait too: it reads weights ahead of its own, and what is in front of a step may be
// writing them.)  A copy by the copy engine costs two changes between engine and SMs: from the end of one step to the end of the
// next one's first RMSNorm 21 us (denoising) and 19 (nine decode rows at 7B dimensions), with this kernel behind the step in front
// 13.5 and 11.3, ahead of its end 7.9 and 5.7.
__global__ void __launch_bounds__(META_THREADS, 1) fetch_metadata_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, int n, int overlap) {
  extern __shared__ uint8_t unused_smem[];
  bool waited = false;
  for (int i = blockIdx.x * META_THREADS + threadIdx.x; i < n || !waited; i += gridDim.x * META_THREADS) {
    uint4 v;      // (host memory that the host has just written: never from a cache)
    if (i < n) asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(src + i) : "memory");
    if (!waited) {
      griddep_wait();
      griddep_launch_dependents(overlap);
      waited = true;
    }
    if (i < n) dst[i] = v;
  }
}

}  // namespace

cudaError_t metadata_set_attributes() { return set_kernel_smem(fetch_metadata_kernel, kMinSmemBytes); }

cudaError_t launch_fetch_metadata(const void* host, void* dev, int words, int overlap, int sm_budget, cudaStream_t stream) {
  const int n = words / 4, blocks = (n + META_THREADS - 1) / META_THREADS;
  if (n <= 0) return cudaSuccess;
  return launch_step_kernel(fetch_metadata_kernel, blocks < sm_budget ? blocks : sm_budget, META_THREADS, kMinSmemBytes, stream, launches_ahead(overlap),
                            static_cast<const uint4*>(host), static_cast<uint4*>(dev), n, overlap);
}

}  // namespace hs
