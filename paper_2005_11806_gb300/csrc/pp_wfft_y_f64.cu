// k_ffty_w for double spectra (pp_wfft_kernels.cuh).
#include "pp_wfft_kernels.cuh"

namespace pp {

template <>
cudaError_t launch_ffty_w<double>(const Geo& g, const C2<double>* twy, C2<double>* spec, int inverse, const DevStatus* st,
                               Queue s, const C2<double>* dct) {
  switch (g.ny) {
#define PP_X(N) case N: return launch_ffty_w_n<double, N>(g, twy, spec, inverse, st, s, dct);
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
  return cudaErrorInvalidValue;
}

}  // namespace pp
