// k_fftx_inv_w for both spectra (pp_wfft_kernels.cuh).
#include "pp_wfft_kernels.cuh"

namespace pp {

template <typename T>
cudaError_t launch_fftx_inv_w(const Geo& g, const C2<T>* twx, const C2<T>* spec, double scale, double* p, int p_zero,
                              const DevStatus* st, Queue s, T* delta, float* sdelta) {
  switch (g.nx) {
#define PP_X(N) case N: return launch_fftx_inv_w_n<T, N>(g, twx, spec, scale, p, p_zero, st, s, delta, sdelta);
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
  return cudaErrorInvalidValue;
}
template cudaError_t launch_fftx_inv_w<float>(const Geo&, const float2*, const float2*, double, double*, int,
                                              const DevStatus*, Queue, float*, float*);
template cudaError_t launch_fftx_inv_w<double>(const Geo&, const double2*, const double2*, double, double*, int,
                                               const DevStatus*, Queue, double*, float*);

}  // namespace pp
