// One grid of a batch on the device, and the launchers of the grouped kernels
// for the lengths of PP_WFFT_LENGTHS (pp_batch_wfft_*.cu).
#pragma once
#include "pp_stages.cuh"

namespace pp {

struct GridDev {
  Geo g;
  Faces fc;
  FftDesc fx, fy;
  const float2* twx;
  const float2* twy;
  const float2* dcty;  // walls in y: exp(-i pi m / (2 ny)); null: periodic y
  const double* invd;
  const double* mtab;
  TriF32 tri;  // FP32 tables of the well-conditioned z columns
  float2* spec;
  float* E;
  float* delta;
  float* sdelta;  // increments not yet added to p (lazy update, stage_fftx_inv)
  double* b;
  double* red;
  DevStatus* st;
  // per call: this grid's fields inside the caller's packed buffers
  const double *us, *vs, *ws, *rho, *S;
  double *p, *u, *v, *w;
  double dt, inv_dt, scale;
  int rpb, nblk_x;  // x kernels: rows per block, partial-sum pairs of the residual
  int tx, ntx;      // y kernels: kx tile, tiles per plane
  int nchunk;       // elementwise chunks
  long long ncell;
};

// Grouped forms of k_resid_w, k_fftx_inv_w and k_ffty_w over a work list of
// (grid, block) or (grid, tile group), kBatchWThreads threads a block.
constexpr int kBatchWThreads = 128;
cudaError_t launch_batch_resid_w(const GridDev* G, const int2* work, int n, size_t smem, cudaStream_t s);
cudaError_t launch_batch_fftx_inv_w(const GridDev* G, const int2* work, int n, size_t smem, cudaStream_t s);
cudaError_t launch_batch_ffty_w(const GridDev* G, const int2* work, int n, size_t smem, int inverse, cudaStream_t s);
// Host: shared memory and work items of one grid's x kernels (blocks; also
// the partial-sum pairs of the residual) and y kernels (groups of tiles).
struct BatchWShape {
  size_t smem_x = 0, smem_y = 0;
  int nblk_x = 0, ngroups_y = 0;
};
void batch_wfft_x(int nx, long long nrows, BatchWShape* out);
void batch_wfft_y(int ny, int nxh, int nz, BatchWShape* out);

}  // namespace pp
