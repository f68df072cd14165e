// Grouped inverse x transform and update of p of the batch (k_fftx_inv_w).
#include "pp_batch.cuh"
#include "pp_wfft_kernels.cuh"

namespace pp {

__global__ void __launch_bounds__(kBatchWThreads, 5) kb_fftx_inv_w(const GridDev* G, const int2* __restrict__ work) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int2 w = work[blockIdx.x];
  const GridDev& d = G[w.x];
  if (d.st->done) return;
  const bool fold = d.st->need_exact != 0, fresh = d.st->since_exact <= 1;
  switch (d.g.nx) {
#define PP_X(N)                                                                                                   \
  case N:                                                                                                         \
    fftx_inv_w_body<float, N>(d.g, d.twx, d.spec, d.scale, d.p, 0, true, fold, fresh, d.delta, d.sdelta, w.y, smem_raw); \
    break;
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
}

cudaError_t launch_batch_fftx_inv_w(const GridDev* G, const int2* work, int n, size_t smem, cudaStream_t s) {
  kb_fftx_inv_w<<<n, kBatchWThreads, smem, s>>>(G, work);
  return cudaGetLastError();
}

}  // namespace pp
