// The J^T kernels.
#include "fft_apply_kernel.cuh"

namespace fftgb {

template <>
fft_status launch_mode<MODE_JT>(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    return launch_mode_impl<MODE_JT>(g, P, st);
}
template <>
fft_status set_attr_mode<MODE_JT>(size_t smem) {
    return set_attr_mode_impl<MODE_JT>(smem);
}

int apply_blocks_per_sm(bool sharp, int threads, size_t smem) {
    int b = 0;
    if (sharp)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, apply_kernel<MODE_JT, FFT_DT_STABLE, false, true, PHI_TABLE>,
                                                      threads, smem);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, apply_kernel<MODE_JT, FFT_DT_STABLE, false, false, PHI_TABLE>,
                                                      threads, smem);
    return b;
}

}  // namespace fftgb
