// Single-grid kernels of the eigenexpansion solve and Algorithm 1's pass;
// each is a thin wrapper around a stage of pp_stages.cuh.
#include <cmath>

#include "pp_stages.cuh"
#include "pp_wfft.cuh"

namespace pp {

// YS: stretched y between walls (row factors of Geo::ym).
template <typename T, bool YS>
__global__ void __launch_bounds__(256, 4) k_resid_fftx(Geo g, Faces fc, FftDesc fx,
                                                    const C2<T>* __restrict__ twx,
                                                    const double* __restrict__ b,
                                                    const double* __restrict__ rho,
                                                    const double* __restrict__ p, int mode, int p_zero,
                                                    int scale_rho, C2<T>* __restrict__ spec,
                                                    double* __restrict__ red, int rpb,
                                                    const DevStatus* st,
                                                    float* __restrict__ E,
                                                    const float* __restrict__ delta, LoopCheck ck) {
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const bool need_exact = (st == nullptr) || st->need_exact;
  stage_resid_fftx<T, YS>(g, fc, fx, twx, b, rho, p, mode, p_zero, scale_rho, spec, red, rpb, blockIdx.x,
                      need_exact, E, delta, smem_raw, ck, gridDim.x);
}

// DCT: the cosine transform of walls in y instead of the periodic DFT.
template <typename T, int DIR, bool DCT>
// Three blocks per SM (FP32: 52 KB of buffers each at ny = 512) measured
// faster than four; the bound also keeps the register count from deciding it.
__global__ void __launch_bounds__(256, sizeof(T) == sizeof(float) ? 3 : 2) k_ffty(Geo g, FftDesc fy, const C2<T>* __restrict__ twy,
                                              C2<T>* __restrict__ spec, int tx, long long ntiles,
                                              const DevStatus* __restrict__ st,
                                              const C2<T>* __restrict__ dct) {
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  stage_ffty_persistent<T, DIR, DCT>(g, fy, twy, spec, tx, ntiles, blockIdx.x, gridDim.x, smem_raw, dct);
}

// z solve for uniform walls in z: cosine transform along z with the
// eigenvalue divide (DIR = -1), then the inverse cosine transform (DIR = +1).
template <typename T, int DIR>
__global__ void __launch_bounds__(256, 2) k_fftz(Geo g, FftDesc fz, const C2<T>* __restrict__ twz,
                                                 C2<T>* __restrict__ spec, int tx, long long ntiles,
                                                 const DevStatus* __restrict__ st,
                                                 const C2<T>* __restrict__ dct, ZDivide zd) {
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  stage_ffty_persistent<T, DIR, true, 1>(g, fz, twz, spec, tx, ntiles, blockIdx.x, gridDim.x, smem_raw, dct, zd);
}

__global__ void __launch_bounds__(128) k_tridiag(Geo g, const double* __restrict__ invd,
                                                 double2* spec, double2* ybuf,  // ybuf may alias spec
                                                 const DevStatus* __restrict__ st) {
  if (stopped(st)) return;
  const size_t ncol = (size_t)g.ny * g.nxh;
  const size_t col = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= ncol) return;
  if (col == 0) thomas_column<true>(g, invd, spec, ybuf, col, ncol);
  else thomas_column<false>(g, invd, spec, ybuf, col, ncol);
}

// z solve of FP64 and PP_MIXED_Z64 plans: one thread per column of `spec`
// (ZForm64: complex entries; ZFormD: scalars, the components apart, which
// gives small grids twice the chains).  The warp that holds column 0 first
// takes its dzf-weighted mean and subtracts it on the way (all its lanes run
// the ZERO variant, the others with mean 0), so no warp runs two variants.
//
// Dropped: a thread taking both columns ky and ny - ky of a shared table
// column.  It halves the table traffic and leaves half the warps; one column /
// two, ms, event overhead included: mixed_z64 512^3 0.515 / 0.543, 384^3 0.235 /
// 0.270, 512 x 512 x 128 0.135 / 0.145, 256^3 0.094 / 0.150.
template <class F>
__global__ void __launch_bounds__(kZThreads) k_zsolve(Geo g, F tab, int nyt, int ysym, typename F::Val* spec,
                                                      const DevStatus* __restrict__ st) {
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int C = std::is_same<F, ZFormD>::value ? 2 : 1;  // entries per complex column
  const unsigned n = (unsigned)C * (unsigned)g.ny * (unsigned)g.nxh;  // entries of a row
  const unsigned id = blockIdx.x * kZThreads + threadIdx.x;
  const unsigned col = id / C;
  const bool first = id < 32u;  // warp-uniform
  double mx = 0.0, my = 0.0;
  if (first) {
    zero_column_mean(g, spec, n, mx, my);
    if (C == 2 && id == 1u) mx = my;  // the scalars' second entry is the imaginary part
    if (col != 0u) mx = my = 0.0;
  }
  if (id >= n) return;
  const unsigned ny = (unsigned)g.ny, nxh = (unsigned)g.nxh;
  const unsigned ky = col / nxh, kx = col - ky * nxh;
  const unsigned kyt = (ysym && 2u * ky > ny) ? ny - ky : ky;
  const size_t t = (size_t)kyt * nxh + kx, tstride = (size_t)nyt * nxh;
  if (first) zsweep<F, true>(tab, spec + id, n, t, tstride, g.nz, nullptr, smem_raw, mx, my);
  else zsweep<F, false>(tab, spec + id, n, t, tstride, g.nz, nullptr, smem_raw, 0.0, 0.0);
}

__global__ void __launch_bounds__(kZThreads, 8) k_tridiag_mixed(Geo g, const double* __restrict__ mtab,
                                                         const double* __restrict__ invd, TriF32 f,
                                                         float2* spec, const DevStatus* __restrict__ st) {
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  stage_tridiag_mixed(g, mtab, invd, f, spec, blockIdx.x, smem_raw);
}

// p += sdelta when the last residual of the loop was an updated one (the
// increments since the last exact residual are still pending).
__global__ void k_fold_pending(size_t n, double* __restrict__ p, const float* __restrict__ sdelta,
                               const DevStatus* __restrict__ st) {
  if (st->last_exact) return;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x)
    p[c] += widen_f32(sdelta[c]);
}

__global__ void k_narrow(const double* __restrict__ src, float* __restrict__ dst, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = (float)src[i];
}

template <typename T>
__global__ void __launch_bounds__(256) k_fftx_inv(Geo g, FftDesc fx, const C2<T>* __restrict__ twx,
                                                  const C2<T>* __restrict__ spec, double scale,
                                                  double* __restrict__ p, int p_zero, int rpb,
                                                  const DevStatus* __restrict__ st,
                                                  T* __restrict__ delta, float* __restrict__ sdelta) {
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const bool lazy = sdelta != nullptr && st != nullptr;
  const bool fold = lazy && st->need_exact != 0;
  const bool fresh = lazy && st->since_exact <= 1;
  stage_fftx_inv<T>(g, fx, twx, spec, scale, p, p_zero, rpb, blockIdx.x, delta, lazy ? sdelta : nullptr,
                    fold, fresh, smem_raw);
}

// ---------------------------------------------------------------------------
template <typename T>
cudaError_t launch_resid_fftx(const Geo& g, const Faces& fc, const FftDesc& fx, const C2<T>* twx,
                              const double* b, double inv_dt, const double* rho, const double* p,
                              int p_zero, int scale_rho, C2<T>* spec, double* red, const LoopCheck* ck,
                              const DevStatus* st, Queue s, float* E, const float* delta) {
  // FP32 rows of 512: the warp form for residuals; a plain solve's FP64 rows load
  // faster with the block kernel's 32 warps an SM (warp form / block kernel:
  // 512^3 0.953 / 0.855 ms, 512 x 512 x 128 0.247 / 0.222; 512 x 64 x 64 0.012 both)
  if (wfft_length(g.nx) || (g.nx == 512 && std::is_same<T, float>::value && red != nullptr))
    return launch_resid_w<T>(g, fc, twx, b, rho, p, p_zero, scale_rho, spec, red, ck, st, s, E, delta);
  const int rpb = rows_per_block(g.nx, kEpt);
  const long nrows = (long)g.nz * g.ny;
  const int nblk = (int)((nrows + rpb - 1) / rpb);
  // two transform buffers, then (FP32) the padding of the second buffer and
  // the twiddle table of the fast path
  const size_t nbuf = (size_t)(rpb / 2) * g.nx;
  const size_t smem = (sizeof(T) == sizeof(float))
                          ? (nbuf + fft_pad_elems((int)nbuf) + g.nx) * sizeof(float2)
                          : 2 * nbuf * sizeof(C2<T>);
  auto kern = (g.ym != nullptr) ? k_resid_fftx<T, true> : k_resid_fftx<T, false>;
  const cudaError_t e = (g.ym != nullptr) ? allow_smem<k_resid_fftx<T, true>>() : allow_smem<k_resid_fftx<T, false>>();
  if (e != cudaSuccess) return e;
  const int mode = (red == nullptr) ? 0 : 1;
  (void)inv_dt;
  return enqueue(s, kern, nblk, kThreads, smem, g, fc, fx, twx, b, rho, p, mode, p_zero, scale_rho, spec, red, rpb,
                 st, E, delta, ck ? *ck : LoopCheck{});
}

template <typename T>
cudaError_t launch_ffty(const Geo& g, const FftDesc& fy, const C2<T>* twy, C2<T>* spec, int inverse,
                        const DevStatus* st, Queue s, const C2<T>* dct) {
  if constexpr (std::is_same<T, float>::value) {
    if (g.ny == 512 && dct == nullptr)
      return launch_ffty512(g, reinterpret_cast<const float2*>(twy), reinterpret_cast<float2*>(spec), inverse, st, s);
  }
  if (wfft_length(g.ny)) return launch_ffty_w<T>(g, twy, spec, inverse, st, s, dct);
  const int tx = ffty_tile(g.ny, sizeof(C2<T>), kEpt);
  const int tsz = g.ny * tx;
  const size_t smem = (sizeof(T) == sizeof(float))
                          ? ((size_t)2 * tsz + fft_pad_elems(tsz) + g.ny) * sizeof(float2)
                          : (size_t)3 * tsz * sizeof(C2<T>);
  const long long ntiles = (long long)((g.nxh + tx - 1) / tx) * g.nz;
  // persistent grid: exactly the blocks that are resident at once (shared
  // memory and registers both counted), so no block waits for a second wave
  auto go = [&](auto resident, auto kern) {
    long long nblk = 0;
    const cudaError_t e = resident(&nblk);
    if (e != cudaSuccess) return e;
    return enqueue(s, kern, (unsigned)(nblk < ntiles ? nblk : ntiles), kThreads, smem, g, fy, twy, spec, tx, ntiles,
                   st, dct);
  };
#define PP_GO(...) go([&](long long* n) { return resident_blocks<__VA_ARGS__>(kThreads, smem, n); }, __VA_ARGS__)
  if (dct) return inverse ? PP_GO(k_ffty<T, 1, true>) : PP_GO(k_ffty<T, -1, true>);
  return inverse ? PP_GO(k_ffty<T, 1, false>) : PP_GO(k_ffty<T, -1, false>);
#undef PP_GO
}

template <typename T>
cudaError_t launch_zdct(const Geo& g, const FftDesc& fz, const C2<T>* twz, C2<T>* spec, int inverse,
                        const DevStatus* st, Queue s, const C2<T>* dct, const ZDivide& zd) {
  const int tx = ffty_tile(g.nz, sizeof(C2<T>), kEpt);
  const int tsz = g.nz * tx;
  const size_t smem = (sizeof(T) == sizeof(float))
                          ? ((size_t)2 * tsz + fft_pad_elems(tsz) + g.nz) * sizeof(float2)
                          : (size_t)3 * tsz * sizeof(C2<T>);
  const long long ntiles = (long long)((g.nxh + tx - 1) / tx) * g.ny;
  auto kern = inverse ? k_fftz<T, 1> : k_fftz<T, -1>;
  cudaError_t e = inverse ? allow_smem<k_fftz<T, 1>>() : allow_smem<k_fftz<T, -1>>();
  if (e != cudaSuccess) return e;
  int per_sm = 0, dev = 0, nsm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem)) != cudaSuccess) return e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  long long nblk = (long long)nsm * per_sm;
  if (nblk > ntiles) nblk = ntiles;
  return enqueue(s, kern, (int)nblk, kThreads, smem, g, fz, twz, spec, tx, ntiles, st, dct, zd);
}
template cudaError_t launch_zdct<double>(const Geo&, const FftDesc&, const double2*, double2*, int,
                                         const DevStatus*, Queue, const double2*, const ZDivide&);

int tri_mixed_blocks(size_t ncol, int nlow) {
  constexpr int kWarps = kZThreads / 32;
  return (nlow + kWarps - 1) / kWarps + (int)((ncol + kZThreads - 1) / kZThreads);
}

cudaError_t launch_tridiag(const Geo& g, const double* invd, double2* spec, double2* ybuf, const DevStatus* st,
                           Queue s) {
  const size_t ncol = (size_t)g.ny * g.nxh;
  return enqueue(s, k_tridiag, (int)((ncol + 127) / 128), 128, 0, g, invd, spec, ybuf, st);
}

cudaError_t launch_tridiag_mixed(const Geo& g, const double* invd, const double* mtab, const TriF32& f32, float2* spec,
                                 const DevStatus* st, Queue s) {
  const size_t ncol = (size_t)g.ny * g.nxh;
  return enqueue(s, k_tridiag_mixed, tri_mixed_blocks(ncol, f32.nlow), kZThreads, zsweep_smem<ZForm32>(), g, mtab,
                 invd, f32, spec, st);
}

template <typename T>
cudaError_t launch_zsolve(const Geo& g, const TriZ<T>& t, C2<T>* spec, const DevStatus* st, Queue s) {
  using F = std::conditional_t<std::is_same<T, float>::value, ZForm64, ZFormD>;
  using Val = typename F::Val;
  constexpr size_t smem = zsweep_smem<F>();
  static_assert(smem <= 48 * 1024, "fits without the opt-in attribute");
  const size_t n = (size_t)g.ny * g.nxh * (sizeof(C2<T>) / sizeof(Val));
  return enqueue(s, k_zsolve<F>, (unsigned)((n + kZThreads - 1) / kZThreads), kZThreads, smem, g, F{t.m, t.d, t.e},
                 t.nyt, t.ysym, reinterpret_cast<Val*>(spec), st);
}
template cudaError_t launch_zsolve<float>(const Geo&, const TriZ<float>&, float2*, const DevStatus*, Queue);
template cudaError_t launch_zsolve<double>(const Geo&, const TriZ<double>&, double2*, const DevStatus*, Queue);

std::vector<int> tri_low_columns(const std::vector<double>& lamx, const std::vector<double>& lamy,
                                 double thr) {
  std::vector<int> low{0};
  const int nxh = (int)lamx.size(), ny = (int)lamy.size();
  for (int j = 0; j < ny; ++j)
    for (int kx = 0; kx < nxh; ++kx)
      if ((j != 0 || kx != 0) && std::fabs(lamx[kx] + lamy[j]) < thr) low.push_back(j * nxh + kx);
  return low;
}

cudaError_t launch_fold_pending(const Geo& g, double* p, const float* sdelta, const DevStatus* st,
                                cudaStream_t s) {
  const size_t n = (size_t)g.nx * g.ny * g.nz;
  size_t nb = (n + 255) / 256;
  if (nb > (size_t)152 * 32) nb = (size_t)152 * 32;
  k_fold_pending<<<(int)(nb == 0 ? 1 : nb), 256, 0, s>>>(n, p, sdelta, st);
  return cudaGetLastError();
}

cudaError_t launch_narrow(const double* src, float* dst, size_t n, cudaStream_t s) {
  size_t nb = (n + 255) / 256;
  if (nb > (size_t)152 * 32) nb = (size_t)152 * 32;
  k_narrow<<<(int)(nb == 0 ? 1 : nb), 256, 0, s>>>(src, dst, n);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fftx_inv(const Geo& g, const FftDesc& fx, const C2<T>* twx, const C2<T>* spec,
                            double scale, double* p, int p_zero, const DevStatus* st, Queue s,
                            T* delta, float* sdelta) {
  if constexpr (std::is_same<T, float>::value) {
    if (g.nx == 512)
      return launch_fftx512_inv(g, reinterpret_cast<const float2*>(twx), reinterpret_cast<const float2*>(spec),
                                scale, p, p_zero, st, s, delta, sdelta);
  }
  if (wfft_length(g.nx)) return launch_fftx_inv_w<T>(g, twx, spec, scale, p, p_zero, st, s, delta, sdelta);
  const int rpb = rows_per_block(g.nx, kEpt);
  const long nrows = (long)g.nz * g.ny;
  const int nblk = (int)((nrows + rpb - 1) / rpb);
  // two transform buffers, then (FP32) the padding of the second buffer and
  // the twiddle table of the fast path
  const size_t nbuf = (size_t)(rpb / 2) * g.nx;
  const size_t smem = (sizeof(T) == sizeof(float))
                          ? (nbuf + fft_pad_elems((int)nbuf) + g.nx) * sizeof(float2)
                          : 2 * nbuf * sizeof(C2<T>);
  const cudaError_t e = allow_smem<k_fftx_inv<T>>();
  if (e != cudaSuccess) return e;
  return enqueue(s, k_fftx_inv<T>, nblk, kThreads, smem, g, fx, twx, spec, scale, p, p_zero, rpb, st, delta, sdelta);
}

#define PP_INST(T)                                                                                   \
  template cudaError_t launch_resid_fftx<T>(const Geo&, const Faces&, const FftDesc&, const C2<T>*,  \
                                            const double*, double, const double*, const double*,     \
                                            int, int, C2<T>*, double*, const LoopCheck*, const DevStatus*, \
                                            Queue, float*, const float*);                    \
  template cudaError_t launch_ffty<T>(const Geo&, const FftDesc&, const C2<T>*, C2<T>*, int,         \
                                      const DevStatus*, Queue, const C2<T>*);                 \
  template cudaError_t launch_fftx_inv<T>(const Geo&, const FftDesc&, const C2<T>*, const C2<T>*,    \
                                          double, double*, int, const DevStatus*, Queue,      \
                                          T*, float*);
PP_INST(double)
PP_INST(float)
#undef PP_INST

}  // namespace pp
