// rsqrt_check.cu -- test helper: the library's FP64 reciprocal square root and CUDA's on an
// array.  Built by tests/test_rsqrt_gpu.py.
#include <cuda_runtime.h>

#include "../paper_1411_3487_gb300/csrc/sfp_device.cuh"

__global__ void k_rsqrt(const double* x, double* own, double* cuda, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    own[i] = sfp::rsqrt_t<double>(x[i]);
    cuda[i] = rsqrt(x[i]);
}

extern "C" int rsqrt_check(const double* x, double* own, double* cuda, int n)
{
    double* d = nullptr;
    const size_t b = (size_t)n * sizeof(double);
    if (n <= 0 || cudaMalloc(&d, 3 * b) != cudaSuccess) return -1;
    cudaError_t e = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_rsqrt<<<(n + 127) / 128, 128>>>(d, d + n, d + 2 * n, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(own, d + n, b, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(cuda, d + 2 * n, b, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : -1;
}
