// The operations of oca_fp64.cuh on arrays, for tests/test_gpu_fp64.py.
#include "oca_fp64.cuh"

__global__ void k_recip(const double *x, double *y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = oca::recip(x[i]);
}

// bit 0: positive_finite, bit 1: finite
template <typename T>
__global__ void k_classes(const T *x, int *c, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) c[i] = (oca::positive_finite(x[i]) ? 1 : 0) | (oca::finite(x[i]) ? 2 : 0);
}
extern "C" int run_classes(const double *x, int *c, int n, void *stream) {
    k_classes<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(x, c, n);
    return (int)cudaGetLastError();
}
extern "C" int run_classes_f32(const float *x, int *c, int n, void *stream) {
    k_classes<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(x, c, n);
    return (int)cudaGetLastError();
}

extern "C" int run_recip(const double *x, double *y, int n, void *stream) {
    k_recip<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(x, y, n);
    return (int)cudaGetLastError();
}
