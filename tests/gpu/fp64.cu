// The operations of oca_fp64.cuh on arrays, for tests/test_gpu_fp64.py.
#include "oca_fp64.cuh"

__global__ void k_recip(const double *x, double *y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = oca::recip(x[i]);
}

extern "C" int run_recip(const double *x, double *y, int n, void *stream) {
    k_recip<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(x, y, n);
    return (int)cudaGetLastError();
}
