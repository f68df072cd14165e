// Grouped residual and forward x transform of the batch (k_resid_w).
#include "pp_batch.cuh"
#include "pp_wfft_kernels.cuh"

namespace pp {

__global__ void __launch_bounds__(kBatchWThreads, 5) kb_resid_w(const GridDev* G, const int2* __restrict__ work) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int2 w = work[blockIdx.x];
  const GridDev& d = G[w.x];
  if (d.st->done) return;
  const bool exact = d.st->need_exact != 0;
  switch (d.g.nx) {
#define PP_X(N)                                                                                               \
  case N:                                                                                                     \
    resid_w_body<float, false, N>(d.g, d.fc, d.twx, d.b, d.rho, d.p, 1, 0, 1, d.spec, d.red, exact, d.E, d.delta, \
                                  w.y, smem_raw, LoopCheck{}, 0u);                                            \
    break;
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
}

cudaError_t launch_batch_resid_w(const GridDev* G, const int2* work, int n, size_t smem, cudaStream_t s) {
  kb_resid_w<<<n, kBatchWThreads, smem, s>>>(G, work);
  return cudaGetLastError();
}

template <int N>
static void shape_x(long long nrows, BatchWShape* out) {
  using W = WPlan<N>;
  constexpr int wpb = kBatchWThreads / 32;
  const long long warps = (nrows + 2 * W::LW - 1) / (2 * W::LW);
  out->smem_x = (size_t)(N + wpb * W::LW * W::LS) * sizeof(float2);
  static_assert((N + wpb * W::LW * W::LS) * sizeof(float2) <= 48 * 1024, "fits without the opt-in attribute");
  out->nblk_x = (int)((warps + wpb - 1) / wpb);
}

void batch_wfft_x(int nx, long long nrows, BatchWShape* out) {
  switch (nx) {
#define PP_X(N) case N: shape_x<N>(nrows, out); break;
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
}

}  // namespace pp
