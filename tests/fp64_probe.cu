// Runs the double-precision refinements of eosq_fp64.cuh over arrays, for tests/test_gpu_fp64.py.
#include <cuda_runtime.h>

#include "eosq_fp64.cuh"

__global__ void rcp_kernel(const double *x, double *y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = eosq::sp_rcp(x[i]);
}

__global__ void reflector_kernel(const double *alpha, const double *ss, double *beta, double *g, double *amb, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) eosq::make_reflector(alpha[i], ss[i], beta[i], g[i], amb[i]);
}

extern "C" int probe_rcp(const double *x, double *y, int n) {
    rcp_kernel<<<(n + 255) / 256, 256>>>(x, y, n);
    return cudaDeviceSynchronize();
}

extern "C" int probe_reflector(const double *alpha, const double *ss, double *beta, double *g, double *amb, int n) {
    reflector_kernel<<<(n + 255) / 256, 256>>>(alpha, ss, beta, g, amb, n);
    return cudaDeviceSynchronize();
}
