// The FP64 reciprocals of the library, element by element over host arrays.
#include "rb_fp64.cuh"

__global__ void k_probe(const double* x, int n, double* rcp, double* rsq) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    rcp[i] = rb::rcp64(x[i]);
    rsq[i] = rb::rsqrt64(x[i]);
}

extern "C" int fp64_probe(const double* x, int n, double* rcp, double* rsq) {
    double* d = nullptr;
    const size_t b = sizeof(double) * (size_t)n;
    if (cudaMalloc(&d, 3 * b) != cudaSuccess) return 1;
    cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
    k_probe<<<(n + 255) / 256, 256>>>(d, n, d + n, d + 2 * (size_t)n);
    cudaMemcpy(rcp, d + n, b, cudaMemcpyDeviceToHost);
    cudaMemcpy(rsq, d + 2 * (size_t)n, b, cudaMemcpyDeviceToHost);
    const cudaError_t e = cudaGetLastError();
    cudaFree(d);
    return e == cudaSuccess ? 0 : 2;
}
