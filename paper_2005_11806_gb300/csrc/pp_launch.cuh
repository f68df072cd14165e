// What a launch needs to know of a kernel, asked of the runtime once.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

namespace pp {

// Blocks of K resident at once on the current device (at least one an SM),
// with smem bytes of dynamic shared memory allowed for it: the grid of a
// persistent kernel.  One entry per kernel and device, remembered for the last
// smem asked for (three runtime calls a launch before: 1 to 2 % of a pass up
// to 256^3).
//
// Measured and dropped: programmatic stream serialization of the pass kernels
// (blocks placed early, waiting for the kernel before): 32^3 0.0567 ms a pass
// either way, 256^3 0.306 -> 0.376 ms, 512^3 2.5 -> 3.1 ms, also when only
// grids of up to 304 or 1216 blocks used it.
template <auto K>
inline cudaError_t resident_blocks(int threads, size_t smem, long long* out) {
  static std::atomic<uint64_t> known[64];  // smem << 32 | blocks
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool slot = dev >= 0 && dev < 64;
  const uint64_t seen = slot ? known[dev].load(std::memory_order_relaxed) : 0;
  if (seen != 0 && (seen >> 32) == (uint64_t)smem) {
    *out = (long long)(seen & 0xFFFFFFFFu);
    return cudaSuccess;
  }
  int per_sm = 0, nsm = 0;
  if ((e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, K, threads, smem)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  *out = (long long)nsm * (per_sm < 1 ? 1 : per_sm);
  if (slot) known[dev].store(((uint64_t)smem << 32) | (uint64_t)*out, std::memory_order_relaxed);
  return cudaSuccess;
}

}  // namespace pp
