// The support-count kernels.
#include "fft_apply_kernel.cuh"

namespace fftgb {

template <>
fft_status launch_mode<MODE_COUNT>(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    return launch_mode_impl<MODE_COUNT>(g, P, st);
}
template <>
fft_status set_attr_mode<MODE_COUNT>(size_t smem) {
    return set_attr_mode_impl<MODE_COUNT>(smem);
}

}  // namespace fftgb
