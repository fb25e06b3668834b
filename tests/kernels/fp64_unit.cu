// The FP64 helpers of the eigenvalue kernels by themselves, for tests.
#include "../../paper_2312_16335_gb300/csrc/fp64.cuh"

__global__ void rcp_k(const double *x, int n, double *y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = lv::fast_rcp(x[i]);
}
__global__ void rsqrt_k(const double *x, int n, double *y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = lv::fast_rsqrt(x[i]);
}
__global__ void angle_k(const double *app, const double *aqq, const double *apq, int n, double *t, double *c) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) lv::jacobi_angle(app[i], aqq[i], apq[i], t[i], c[i]);
}

extern "C" int fp64_rcp(const double *x, int n, double *y) {
    rcp_k<<<(n + 255) / 256, 256>>>(x, n, y);
    return (int)cudaDeviceSynchronize();
}
extern "C" int fp64_rsqrt(const double *x, int n, double *y) {
    rsqrt_k<<<(n + 255) / 256, 256>>>(x, n, y);
    return (int)cudaDeviceSynchronize();
}
extern "C" int fp64_angle(const double *app, const double *aqq, const double *apq, int n, double *t, double *c) {
    angle_k<<<(n + 255) / 256, 256>>>(app, aqq, apq, n, t, c);
    return (int)cudaDeviceSynchronize();
}
