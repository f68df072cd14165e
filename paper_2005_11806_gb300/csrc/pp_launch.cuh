// What a launch needs to know of a kernel, asked of the runtime once.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <tuple>

namespace pp {

// Kernel nodes strung one after the other in a graph under construction.
struct GraphChain {
  cudaGraph_t graph;
  cudaGraphNode_t last;
};

// Where a launch goes: to a stream, or with a chain to the chain's end.  The
// nodes are added one by one, not captured from a stream: while any stream of
// a device is being captured, another host thread may not wait for the device
// (cudaErrorStreamCaptureUnsupported), and a projection must not forbid that.
struct Queue {
  cudaStream_t stream;
  GraphChain* chain;
  Queue(cudaStream_t s, GraphChain* c = nullptr) : stream(s), chain(c) {}
};

template <class... P, class... A>
inline cudaError_t enqueue(Queue q, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, A&&... args) {
  static_assert(sizeof...(P) == sizeof...(A), "");
  std::tuple<P...> value(static_cast<P>(args)...);
  void* at[sizeof...(P)];
  std::apply([&](P&... v) {
    void* a[] = {(void*)&v...};
    for (size_t i = 0; i < sizeof...(P); ++i) at[i] = a[i];
  }, value);
  cudaError_t e;
  if (q.chain == nullptr) {
    e = cudaLaunchKernel((const void*)kernel, grid, block, at, smem, q.stream);
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
  }
  cudaKernelNodeParams kp{};
  kp.func = (void*)kernel;
  kp.gridDim = grid;
  kp.blockDim = block;
  kp.sharedMemBytes = (unsigned)smem;
  kp.kernelParams = at;
  GraphChain* c = q.chain;
  cudaGraphNode_t node = nullptr;
  e = cudaGraphAddKernelNode(&node, c->graph, c->last ? &c->last : nullptr, c->last ? 1 : 0, &kp);
  if (e == cudaSuccess) c->last = node;
  else (void)cudaGetLastError();
  return e;
}

// Lets K be launched with any dynamic shared memory that the current device
// has.  The limit belongs to the function and the process, so it is set once,
// to its largest value, and never lowered: plans of other lengths may be
// launching K from other threads.
template <auto K>
inline cudaError_t allow_smem() {
  static std::atomic<uint64_t> done;  // a bit per device
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev >= 0 && dev < 64 ? (uint64_t)1 << dev : 0;
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  cudaFuncAttributes a;
  if ((e = cudaFuncGetAttributes(&a, K)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}

// Blocks of K resident at once on the current device (at least one an SM),
// with smem bytes of dynamic shared memory: the grid of a persistent kernel.
// One entry per kernel and device, remembered for the last smem asked for
// (three runtime calls a launch before: 1 to 2 % of a pass up to 256^3).
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
  const uint64_t seen = slot ? known[dev].load(std::memory_order_acquire) : 0;
  if (seen != 0 && (seen >> 32) == (uint64_t)smem) {
    *out = (long long)(seen & 0xFFFFFFFFu);
    return cudaSuccess;
  }
  int per_sm = 0, nsm = 0;
  if ((e = allow_smem<K>()) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, K, threads, smem)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  *out = (long long)nsm * (per_sm < 1 ? 1 : per_sm);
  if (slot) known[dev].store(((uint64_t)smem << 32) | (uint64_t)*out, std::memory_order_release);
  return cudaSuccess;
}

}  // namespace pp
