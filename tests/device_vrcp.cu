// vrcp(double) of the CUDA path on an array in device memory.
#include "prc_vec.cuh"

static __global__ void k_vrcp(const double *a, double *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = prc::vrcp(a[i]);
}

extern "C" int device_vrcp(const double *a, double *y, int n)
{
    double *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 2 * sizeof(double) * (size_t)n);
    if (e != cudaSuccess) return (int)e;
    e = cudaMemcpy(d, a, sizeof(double) * (size_t)n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_vrcp<<<(n + 255) / 256, 256>>>(d, d + n, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(y, d + n, sizeof(double) * (size_t)n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
