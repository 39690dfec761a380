// flbm_obs.cu -- observables of the current state, off the per-step loop:
// densities, baricentric velocity (Eq. lattice-vb), FP64 conservation totals
// and the axis structure factors of Sec. VI A.  All reductions run in a fixed
// order, so repeated calls on the same state give bit-identical results.
#include "flbm_internal.h"
#include "flbm_pair.cuh"

namespace flbm {

namespace {

// fixed-order block reduction of NV doubles per thread; result valid in thread 0
template <int NV, int NT>
__device__ __forceinline__ void block_sum(double (&v)[NV], double (*sh)[NV])
{
    const int t = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
#pragma unroll
    for (int k = 0; k < NV; k++) sh[t][k] = v[k];
    __syncthreads();
    for (int stride = NT / 2; stride > 0; stride >>= 1) {
        if (t < stride)
#pragma unroll
            for (int k = 0; k < NV; k++) sh[t][k] += sh[t + stride][k];
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = sh[0][k];
}

__global__ void __launch_bounds__(256) k_sum_partials(const double *__restrict__ partials, int nblocks,
                                                      double *__restrict__ out)
{
    __shared__ double sh[256][5];
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += 256)
#pragma unroll
        for (int k = 0; k < 5; k++) v[k] += partials[(size_t)b * 5 + k];
    block_sum<5, 256>(v, sh);
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < 5; k++) out[k] = v[k];
}

// profile[c][pc] = sum of snap's plane c over the sites with coordinate pc along
// `axis`.  Along x: a block owns 8 columns (one 32-byte sector a row), 128 rows
// at a time.  128^3: 46 us from doubles with a column a block, now 27 (pairs of
// floats 22).
constexpr int kProfCols = 8, kProfRows = 128, kProfBatch = 8; // loads in flight a thread
__global__ void __launch_bounds__(kProfCols * kProfRows) k_profile_x(int nx, int rows, const float *snap, double *profile)
{
    __shared__ double sh[kProfCols * kProfRows / 32][kProfCols];
    int t = threadIdx.x;
    await_grid(t);
    const int c = blockIdx.y;
    const int x = blockIdx.x * kProfCols + t % kProfCols;
    double v = 0.0;
    if (x < nx) {
        const float *plane = snap + (size_t)c * nx * rows + x;
        FloatSum s;
        int r = t / kProfCols, left = FloatSum::kFold;
        for (; r < rows - (kProfBatch - 1) * kProfRows; r += kProfBatch * kProfRows) {
            float q[kProfBatch];
#pragma unroll
            for (int k = 0; k < kProfBatch; k++) q[k] = plane[(size_t)(r + k * kProfRows) * nx];
#pragma unroll
            for (int k = 0; k < kProfBatch; k++) s.add(q[k]);
            if ((left -= kProfBatch) < kProfBatch) {
                v += s.value();
                s = FloatSum();
                left = FloatSum::kFold;
            }
        }
        for (; r < rows; r += kProfRows) s.add(plane[(size_t)r * nx]);
        v += s.value();
    }
    for (int o = 16; o >= kProfCols; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((t & 31) < kProfCols) sh[t >> 5][t & 31] = v;
    __syncthreads();
    if (t >= 32) return;
    v = 0.0;
    for (int w = t / kProfCols; w < kProfCols * kProfRows / 32; w += 32 / kProfCols) v += sh[w][t % kProfCols];
    for (int o = 16; o >= kProfCols; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (t < kProfCols && x < nx) profile[(size_t)c * nx + x] = v;
}

// Along y or z: a block a coordinate, `rows` rows of nx sites, row r starting at
// pc * pc_stride + r * row_stride; tx threads along x (a power of two).
// kProfBatch loads in flight a thread.  us a snapshot from doubles / one load at a
// time / so: 256 x 256 x 16 along z, where 16 blocks a component read the box,
// 178 / 204 / 104; 64 x 512 x 512 1992 / 1030 / 906.
__global__ void __launch_bounds__(256) k_profile(int nx, int rows, size_t N, size_t pc_stride, size_t row_stride, int tx,
                                                 const float *snap, double *profile)
{
    __shared__ double sh[8];
    int t = threadIdx.x;
    await_grid(t);
    const int pc = blockIdx.x, c = blockIdx.y, ty = 256 / tx, x0 = t & (tx - 1);
    double v = 0.0;
    FloatSum s;
    int left = FloatSum::kFold, x = x0, r = x0 < nx ? t / tx : rows;
    const float *row = snap + (size_t)c * N + (size_t)pc * pc_stride + (size_t)r * row_stride;
    while (r < rows) {
        float q[kProfBatch];
#pragma unroll
        for (int k = 0; k < kProfBatch; k++) {
            q[k] = r < rows ? row[x] : 0.0f;
            x += tx;
            if (x >= nx) {
                x = x0;
                r += ty;
                row += (size_t)ty * row_stride;
            }
        }
#pragma unroll
        for (int k = 0; k < kProfBatch; k++) s.add(q[k]);
        if ((left -= kProfBatch) < kProfBatch) {
            v += s.value();
            s = FloatSum();
            left = FloatSum::kFold;
        }
    }
    v += s.value();
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((t & 31) == 0) sh[t >> 5] = v;
    __syncthreads();
    if (t >= 32) return;
    v = t < 8 ? sh[t] : 0.0;
    for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (t == 0) profile[(size_t)c * gridDim.x + pc] = v;
}

// One block per m, a warp a component: the Fourier coefficients of the
// profiles, accumulated |.|^2 / N.
__global__ void __launch_bounds__(160) k_dft_accumulate(int D, int n_axis, double inv_n, const double *profile,
                                                        const double2 *tw, double *acc)
{
    __shared__ double2 sh[5];
    int t = threadIdx.x;
    await_grid(t);
    const int lane = t & 31, c = t >> 5;
    const int m = blockIdx.x + 1;
    double re = 0.0, im = 0.0;
    int idx = (int)((long long)m * lane % n_axis);
    const int next = (int)((long long)m * 32 % n_axis);
    for (int pc = lane; pc < n_axis; pc += 32) {
        const double P = profile[(size_t)c * n_axis + pc];
        const double2 w = tw[idx];
        re += P * w.x;
        im -= P * w.y;
        idx += next;
        if (idx >= n_axis) idx -= n_axis;
    }
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_down_sync(0xffffffffu, re, o);
        im += __shfl_down_sync(0xffffffffu, im, o);
    }
    if (lane == 0) sh[c] = make_double2(re, im);
    __syncthreads();
    if (t >= 4) return; // thread t: S_aa, S_ab, S_bb, S_uu
    double s;
    if (t < 3) {
        const double2 a = sh[t == 2], b = sh[t > 0];
        s = a.x * b.x + a.y * b.y;
    } else {
        s = 0.0;
        for (int d = 0; d < D; d++) s += sh[2 + d].x * sh[2 + d].x + sh[2 + d].y * sh[2 + d].y;
        s /= D;
    }
    acc[(size_t)t * (n_axis / 2) + m - 1] += s * inv_n;
}

// Float densities of both species from the caller's double arrays, read
// straight from host memory (NULL: uniform rho0); the smallest index of a
// value that is not positive and finite goes to *bad (left as it is when
// there is none).
__global__ void k_densities_from_host(const double *__restrict__ ra, const double *__restrict__ rb, double r0a,
                                      double r0b, long long n, float *__restrict__ out,
                                      unsigned long long *__restrict__ bad)
{
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const double a = ra ? ra[k] : r0a, b = rb ? rb[k] : r0b;
        const bool oka = a > 0.0 && isfinite(a), okb = b > 0.0 && isfinite(b);
        if (!oka) atomicMin(bad, (unsigned long long)k);
        if (!okb) atomicMin(bad + 1, (unsigned long long)k);
        out[k] = (float)a;
        out[n + k] = (float)b;
    }
}

__global__ void k_add_u32(unsigned *p, unsigned v) { *p += v; }
__global__ void k_set_u32(unsigned *p, unsigned v) { *p = v; }

} // namespace

cudaError_t launch_add_u32(unsigned *p, unsigned v, cudaStream_t stream)
{
    k_add_u32<<<1, 1, 0, stream>>>(p, v);
    return cudaGetLastError();
}

cudaError_t launch_densities_from_host(const double *rho_a, const double *rho_b, double rho0_a, double rho0_b,
                                       int64_t n, float *out, unsigned long long *bad, cudaStream_t stream)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long long want = (n + 255) / 256, most = (long long)sms * 8;
    k_densities_from_host<<<(unsigned)(want < most ? (want > 0 ? want : 1) : most), 256, 0, stream>>>(
        rho_a, rho_b, rho0_a, rho0_b, (long long)n, out, bad);
    return cudaGetLastError();
}

cudaError_t launch_set_u32(unsigned *p, unsigned v, cudaStream_t stream)
{
    k_set_u32<<<1, 1, 0, stream>>>(p, v);
    return cudaGetLastError();
}

cudaError_t launch_sum_partials(const double *partials, int nblocks, double *out, cudaStream_t stream)
{
    k_sum_partials<<<1, 256, 0, stream>>>(partials, nblocks, out);
    return cudaGetLastError();
}

cudaError_t launch_sf_accumulate(int D, int nx, int ny, int nz, int axis, const float *snap, const double2 *tw,
                                 double *profile, double *acc, cudaStream_t stream)
{
    const int n_axis = axis == 0 ? nx : (axis == 1 ? ny : nz);
    const size_t plane = (size_t)nx * ny;
    cudaError_t e;
    if (axis == 0) {
        e = launch_chained(true, k_profile_x, dim3((nx + kProfCols - 1) / kProfCols, 2 + D), kProfCols * kProfRows, 0, stream,
                           nx, ny * nz, snap, profile);
    } else {
        int tx = 32;
        while (tx < 256 && tx < nx) tx *= 2;
        const size_t pc_stride = axis == 1 ? (size_t)nx : plane, row_stride = axis == 1 ? plane : (size_t)nx;
        e = launch_chained(true, k_profile, dim3(n_axis, 2 + D), 256, 0, stream, nx, axis == 1 ? nz : ny, plane * nz,
                           pc_stride, row_stride, tx, snap, profile);
    }
    if (e != cudaSuccess) return e;
    const double inv_n = 1.0 / ((double)nx * ny * nz);
    return launch_chained(true, k_dft_accumulate, n_axis / 2, 32 * (2 + D), 0, stream, D, n_axis, inv_n, profile, tw, acc);
}

} // namespace flbm
