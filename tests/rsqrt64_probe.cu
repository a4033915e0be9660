// rsqrt_fp64 of the FP64 force form over an array, for tests/test_gpu_rsqrt64.py.
#include <cuda_runtime.h>

#include "rsqrt64.cuh"

__global__ void k_probe(const double *x, double *y, long long n)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) y[i] = greem::rsqrt_fp64(x[i]);
}

extern "C" int rsqrt64_probe(const double *x, double *y, long long n)
{
    k_probe<<<(unsigned)((n + 255) / 256), 256>>>(x, y, n);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : -1;
}
