// lbm_step_f64.cu -- instantiation of the step, field, init and state kernels
// for the CodecF64 storage codec (see lbm_device.cuh).
#include "lbm_kernels.cuh"

AXILBM_INSTANTIATE(f64, axilbm::CodecF64)

namespace axilbm {
size_t col_tab64_size(int ncols) { return col_tab64_bytes(ncols); }
cudaError_t launch_col_tab64(double* cols, int ncols, int rate_mode, cudaStream_t st) {
    const int blocks = (ncols + 127) / 128;
    if (rate_mode == kRatesPaperRaw) col_tab64_kernel<kRatesPaperRaw><<<blocks, 128, 0, st>>>(cols, ncols);
    else col_tab64_kernel<kRatesPaper><<<blocks, 128, 0, st>>>(cols, ncols);
    return cudaGetLastError();
}
}  // namespace axilbm
