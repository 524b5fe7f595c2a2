// rcp64 and sqrt64 of lbm_device.cuh over arrays on the device, for test_gpu_rcp64.py.
#include "../paper_1810_09299_gb300/csrc/lbm_device.cuh"

__global__ void rcp64_kernel(int root, int64_t n, const double* x, double* y) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = root ? axilbm::sqrt64(x[i]) : axilbm::rcp64(x[i]);
}
extern "C" int rcp64_run(int root, int64_t n, const double* x, double* y) {
    rcp64_kernel<<<(unsigned)((n + 255) / 256), 256>>>(root, n, x, y);
    return (int)cudaDeviceSynchronize();
}
