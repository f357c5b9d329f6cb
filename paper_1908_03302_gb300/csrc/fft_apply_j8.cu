// The eight-column J kernels.
#include "fft_apply_kernel.cuh"

namespace fftgb {

template <>
fft_status launch_batch<MODE_J8>(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    return launch_batch_impl<MODE_J8>(g, P, st);
}
template <>
fft_status set_attr_mode<MODE_J8>(size_t smem) {
    fft_status rc = set_attr_dt<MODE_J8, FFT_DT_STABLE, PHI_TABLE>(smem);
    if (rc != FFT_OK) return rc;
    if ((rc = set_attr_dt<MODE_J8, FFT_DT_STABLE, PHI_TRIG>(smem)) != FFT_OK) return rc;
    return set_attr_dt<MODE_J8, FFT_DT_STABLE, PHI_SEG>(smem);
}

}  // namespace fftgb
