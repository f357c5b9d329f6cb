// The Frobenius-norm kernels.
#include "fft_apply_kernel.cuh"

namespace fftgb {

template <>
fft_status launch_mode<MODE_FROB>(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    return launch_mode_impl<MODE_FROB>(g, P, st);
}
template <>
fft_status set_attr_mode<MODE_FROB>(size_t smem) {
    return set_attr_mode_impl<MODE_FROB>(smem);
}

}  // namespace fftgb
