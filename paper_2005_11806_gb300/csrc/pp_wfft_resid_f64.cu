// k_resid_w for double spectra (pp_wfft_kernels.cuh).
#include "pp_wfft_kernels.cuh"

namespace pp {

template <>
cudaError_t launch_resid_w<double>(const Geo& g, const Faces& fc, const C2<double>* twx, const double* b, const double* rho,
                                const double* p, int p_zero, int scale_rho, C2<double>* spec, double* red,
                                const LoopCheck* ck, const DevStatus* st, Queue s, float* E, const float* delta) {
  switch (g.nx) {
#define PP_X(N) \
  case N: return launch_resid_w_n<double, N>(g, fc, twx, b, rho, p, p_zero, scale_rho, spec, red, ck, st, s, E, delta);
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
  return cudaErrorInvalidValue;
}

}  // namespace pp
