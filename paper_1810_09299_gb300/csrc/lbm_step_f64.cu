// lbm_step_f64.cu -- instantiation of the step, field, init and state kernels
// for the CodecF64 storage codec (see lbm_device.cuh).
#include "lbm_kernels.cuh"

AXILBM_INSTANTIATE(f64, axilbm::CodecF64)

namespace axilbm {
__global__ void col_tab64_kernel(double* d, int n) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const Col64 c = col64(j);
    d[j] = c.r, d[n + j] = c.inv_r;
    longlong2* s = reinterpret_cast<longlong2*>(d + 2 * n);
    const Sf v[kColSf] = {c.sr, c.s_inv_r, c.s_i6, c.s_i4, c.r03, c.r3, c.r72};
    for (int i = 0; i < kColSf; ++i) s[(int64_t)i * n + j] = longlong2{v[i].m, (long long)v[i].e};
}
size_t col_tab64_size(int ncols) { return col_tab64_bytes(ncols); }
cudaError_t launch_col_tab64(double* cols, int ncols, cudaStream_t st) {
    col_tab64_kernel<<<(ncols + 127) / 128, 128, 0, st>>>(cols, ncols);
    return cudaGetLastError();
}
}  // namespace axilbm
