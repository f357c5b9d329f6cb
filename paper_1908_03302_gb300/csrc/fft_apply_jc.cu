// The kernels of J with compensated sums (fft_apply_kernel.cuh).
#include "fft_apply_kernel.cuh"

namespace fftgb {

template <>
fft_status launch_mode<MODE_JC>(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    return launch_batch_impl<MODE_JC>(g, P, st);
}
template <>
fft_status set_attr_mode<MODE_JC>(size_t smem) {
    fft_status rc = set_attr_dt<MODE_JC, FFT_DT_STABLE, PHI_TABLE>(smem);
    if (rc != FFT_OK) return rc;
    if ((rc = set_attr_dt<MODE_JC, FFT_DT_STABLE, PHI_TRIG>(smem)) != FFT_OK) return rc;
    return set_attr_dt<MODE_JC, FFT_DT_STABLE, PHI_SEG>(smem);
}

}  // namespace fftgb
