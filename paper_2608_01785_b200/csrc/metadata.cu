// The step's first kernel: brings the metadata block from the stage's pinned host memory into the workspace.
#include "kernels.h"
#include "ptx.cuh"

namespace hs {
namespace {

constexpr int META_THREADS = 256, META_AHEAD = 8;      // 16-byte groups that a thread asks for at a time

// What bounds it is the way over PCIe; so all groups are asked for at the same time, as far as the budget's threads hold them, and before
// the wait for the kernel in front: nothing on the device writes the host's block, and the workspace's is written after the wait.
// A step of one layer on 148 / 16 / 4 / 1 SMs, us, block tables of 128 KB, by the copy engine 37.7 / 42.2 / 54.6 / 113.5, with one group a
// thread 31.8 / 36.9 / 57.6 / 152.3, with eight 31.9 / 37.0 / 48.3 / 110.7; 1 MB 54.3 / 60.2 / 72.4 / 126.6, 50.8 / 61.5 / 145.8 / 498.9, 47.7 /
// 54.3 / 68.4 / 172.7.
// (The kernel behind is let go after the wait too: it reads weights ahead of its own, and what is in front of a step may be
// writing them.  It is let go before the block is written: see launch_fetch_metadata for what that asks of it.)  A copy by the copy engine costs two changes between engine and SMs: from the end of one step to the end of the
// next one's first RMSNorm 21 us (denoising) and 19 (nine decode rows at 7B dimensions), with this kernel behind the step in front
// 13.5 and 11.3, ahead of its end 7.9 and 5.7.
__global__ void __launch_bounds__(META_THREADS, 1) fetch_metadata_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, int n, int overlap) {
  extern __shared__ uint8_t unused_smem[];
  bool waited = false;
  const int stride = gridDim.x * META_THREADS;
  for (int i = blockIdx.x * META_THREADS + threadIdx.x; i < n || !waited; i += META_AHEAD * stride) {
    uint4 v[META_AHEAD];      // (host memory that the host has just written: never from a cache)
#pragma unroll
    for (int u = 0; u < META_AHEAD; ++u)
      if (i + u * stride < n)
        asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v[u].x), "=r"(v[u].y), "=r"(v[u].z), "=r"(v[u].w) : "l"(src + i + u * stride) : "memory");
    if (!waited) {
      griddep_wait();
      griddep_launch_dependents(overlap);
      waited = true;
    }
#pragma unroll
    for (int u = 0; u < META_AHEAD; ++u)
      if (i + u * stride < n) dst[i + u * stride] = v[u];
  }
}

}  // namespace

cudaError_t metadata_set_attributes() { return set_kernel_smem(fetch_metadata_kernel, kMinSmemBytes); }

cudaError_t launch_fetch_metadata(const void* host, void* dev, int words, int overlap, int sm_budget, cudaStream_t stream) {
  const int n = words / 4, blocks = (n + META_THREADS - 1) / META_THREADS;
  if (n <= 0) return cudaSuccess;
  // One SM takes in 15 GB/s, and four what the copy engine moves (50): fewer leave it large blocks (one SM, 128 / 256 / 512 KB: 111 / 120 /
  // 138 us for the engine's 114 / 115 / 120).
  if (sm_budget < 4 && n > sm_budget * (10 << 10)) return cudaMemcpyAsync(dev, host, size_t(n) * 16, cudaMemcpyHostToDevice, stream);
  return launch_step_kernel(fetch_metadata_kernel, blocks < sm_budget ? blocks : sm_budget, META_THREADS, kMinSmemBytes, stream, launches_ahead(overlap),
                            static_cast<const uint4*>(host), static_cast<uint4*>(dev), n, overlap);
}

}  // namespace hs
