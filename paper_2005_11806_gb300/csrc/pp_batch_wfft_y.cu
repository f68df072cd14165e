// Grouped y transforms of the batch (k_ffty_w): a block takes as many tiles as
// its threads hold (two for the lengths with 8 threads a line).
#include "pp_batch.cuh"
#include "pp_wfft_kernels.cuh"

namespace pp {

template <int N>
struct BatchY {
  using Y = WyShape<float, N>;
  static constexpr int NS = kBatchWThreads / Y::threads;  // tiles a block
  static_assert(NS * Y::threads == kBatchWThreads, "");
  // one exchange buffer a tile, two with the pairing of the cosine transform
  static constexpr size_t smem(bool dct) { return (size_t)(N + NS * (dct ? 2 : 1) * Y::ebuf) * sizeof(float2); }
  static_assert(smem(true) <= 48 * 1024, "fits without the opt-in attribute");
};

template <int DIR, bool DCT, int N>
__device__ __forceinline__ void batch_ffty_body(const GridDev& d, int group, unsigned char* smem_raw) {
  using B = BatchY<N>;
  using Y = typename B::Y;
  float2* tw = reinterpret_cast<float2*>(smem_raw);
  const int sg = threadIdx.x / Y::threads, t = threadIdx.x - sg * Y::threads;
  float2* e0 = tw + N + (size_t)sg * (DCT ? 2 : 1) * Y::ebuf;
  float2* e1 = e0 + Y::ebuf;
  wfft_load_twiddles<WPlan<N>, float>(tw, d.twy);
  const int nxh = d.g.nxh, ntx = (nxh + kWyTx - 1) / kWyTx;
  const int x = t % kWyTx, l = t / kWyTx;
  const int tile = group * B::NS + sg, bz = tile / ntx, kx = (tile - bz * ntx) * kWyTx + x;
  const bool ok = bz < d.g.nz && kx < nxh;
  float2* col = d.spec + (ok ? (size_t)bz * N * nxh + kx : 0);
  float2 v[WPlan<N>::U1][WPlan<N>::R1];
  ffty_w_load<float, DIR, DCT, N>(v, col, nxh, l, ok, d.dcty);
  __syncthreads();  // twiddles
  ffty_w_front<float, DIR, N>(v, e0, tw, x, l);
  __syncthreads();
  ffty_w_back<float, DIR, DCT, N>(col, e0, e1, nxh, x, l, ok, d.dcty);
}

template <int DIR>
__global__ void __launch_bounds__(kBatchWThreads) kb_ffty_w(const GridDev* G, const int2* __restrict__ work) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int2 w = work[blockIdx.x];
  const GridDev& d = G[w.x];
  if (d.st->done) return;
  switch (d.g.ny) {
#define PP_X(N)                                                              \
  case N:                                                                    \
    if (d.dcty != nullptr) batch_ffty_body<DIR, true, N>(d, w.y, smem_raw);  \
    else batch_ffty_body<DIR, false, N>(d, w.y, smem_raw);                   \
    break;
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
}

cudaError_t launch_batch_ffty_w(const GridDev* G, const int2* work, int n, size_t smem, int inverse, cudaStream_t s) {
  if (inverse) kb_ffty_w<1><<<n, kBatchWThreads, smem, s>>>(G, work);
  else kb_ffty_w<-1><<<n, kBatchWThreads, smem, s>>>(G, work);
  return cudaGetLastError();
}

template <int N>
static void shape_y(int nxh, int nz, BatchWShape* out) {
  using B = BatchY<N>;
  const long long tiles = (long long)((nxh + kWyTx - 1) / kWyTx) * nz;
  out->smem_y = B::smem(true);
  out->ngroups_y = (int)((tiles + B::NS - 1) / B::NS);
}

void batch_wfft_y(int ny, int nxh, int nz, BatchWShape* out) {
  switch (ny) {
#define PP_X(N) case N: shape_y<N>(nxh, nz, out); break;
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
}

}  // namespace pp
