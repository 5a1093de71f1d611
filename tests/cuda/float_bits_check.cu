// Test helper: pe_sum and to_float (csrc/float_bits.cuh) beside the plain FP64
// sum and conversion on the device, for tests/test_gpu_float_bits.py.
#include <cuda_runtime.h>

#include "../../paper_1909_07321_gb300/csrc/float_bits.cuh"

__global__ void sums_kernel(const float *v, int n, int count, double *got, double *plain)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    float x[8];
    double s = 0.0;
    for (int q = 0; q < 8; ++q) {
        x[q] = q < n ? v[(size_t)i * n + q] : 0.f;
        if (q < n) s += (double)x[q];
    }
    got[i] = rmgb::pe_sum(x, n);
    plain[i] = s;
}

__global__ void floats_kernel(const double *v, int count, float *got, float *plain)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    got[i] = rmgb::to_float(v[i]);
    plain[i] = (float)v[i];
}

// Device arrays; return a cudaError_t code.
extern "C" int sums(const float *v, int n, int count, double *got, double *plain)
{
    sums_kernel<<<(count + 255) / 256, 256>>>(v, n, count, got, plain);
    const cudaError_t e = cudaGetLastError();
    return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}

extern "C" int floats(const double *v, int count, float *got, float *plain)
{
    floats_kernel<<<(count + 255) / 256, 256>>>(v, count, got, plain);
    const cudaError_t e = cudaGetLastError();
    return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}
