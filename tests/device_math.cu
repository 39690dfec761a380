// Device functions of the step and observables kernels called one value (or one
// short sum) a thread, for tests/test_device_math_gpu.py.
#include <cuda_runtime.h>

#include "flbm_noise.cuh"
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

// every mantissa at the binary exponent e: how many values of reciprocal() and
// of rsqrt_hw() differ from __frcp_rn and rsqrtf
__global__ void k_compare(int e, unsigned *differ)
{
    const unsigned m = blockIdx.x * blockDim.x + threadIdx.x; // < 2^23
    const float x = __uint_as_float(((unsigned)(e + 127) << 23) | m);
    if (__float_as_uint(flbm::reciprocal(x)) != __float_as_uint(__frcp_rn(x))) atomicAdd(differ, 1u);
    if (__float_as_uint(flbm::rsqrt_hw(x)) != __float_as_uint(rsqrtf(x))) atomicAdd(differ + 1, 1u);
}

extern "C" int compare(int e, unsigned *differ)
{
    unsigned *d = nullptr;
    cudaError_t err = cudaMalloc((void **)&d, 2 * sizeof(unsigned));
    if (err == cudaSuccess) err = cudaMemset(d, 0, 2 * sizeof(unsigned));
    if (err == cudaSuccess) {
        k_compare<<<(1 << 23) / 256, 256>>>(e, d);
        err = cudaGetLastError();
    }
    if (err == cudaSuccess) err = cudaMemcpy(differ, d, 2 * sizeof(unsigned), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)err;
}
