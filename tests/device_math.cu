// Device functions of the step and observables kernels called one value (or one
// short sum) a thread, for tests/test_device_math_gpu.py.
#include <cuda_runtime.h>

#include "flbm_pair.cuh"

// out[k] = the FloatSum of in[k * n .. k * n + n - 1], k < count
__global__ void k_float_sum(const float *in, int n, int count, double *out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    flbm::FloatSum s;
    for (int i = 0; i < n; i++) s.add(in[(size_t)k * n + i]);
    out[k] = s.value();
}

extern "C" int float_sum(const float *in, int n, int count, double *out)
{
    float *d_in = nullptr;
    double *d_out = nullptr;
    const size_t bytes = (size_t)n * count * sizeof(float);
    cudaError_t e = cudaMalloc((void **)&d_in, bytes);
    if (e == cudaSuccess) e = cudaMalloc((void **)&d_out, (size_t)count * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpy(d_in, in, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_float_sum<<<(count + 127) / 128, 128>>>(d_in, n, count, d_out);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d_out, (size_t)count * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(d_in);
    cudaFree(d_out);
    return (int)e;
}
