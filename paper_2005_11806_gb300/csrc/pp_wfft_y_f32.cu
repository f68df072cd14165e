// k_ffty_w for float spectra (pp_wfft_kernels.cuh).
#include "pp_wfft_kernels.cuh"

namespace pp {

template <>
cudaError_t launch_ffty_w<float>(const Geo& g, const C2<float>* twy, C2<float>* spec, int inverse, const DevStatus* st,
                               Queue s, const C2<float>* dct) {
  switch (g.ny) {
#define PP_X(N) case N: return launch_ffty_w_n<float, N>(g, twy, spec, inverse, st, s, dct);
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
  }
  return cudaErrorInvalidValue;
}

}  // namespace pp
