// The FP64 reciprocal and root of the phase kernels, value by value.
#include "lbm_phase.cuh"

__global__ void k(const double* x, double* r, double* s, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = lbm::rcp3(x[i]);
    s[i] = lbm::sqrt3(x[i]);
}
// x, r, s: n values on the device.
extern "C" int rcp_sqrt(const double* x, double* r, double* s, int n) {
    k<<<(n + 255) / 256, 256>>>(x, r, s, n);
    return (int)cudaDeviceSynchronize();
}
