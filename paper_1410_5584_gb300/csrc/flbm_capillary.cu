// flbm_capillary.cu -- capillary fluctuations of a flat interface (Sec. VI B,
// Eq. predictionspectrum): heights of the two interfaces of a stripe and the
// spectrum of their fluctuations, accumulated on the device.  D2Q9 boxes.
//
// One snapshot, in four or five launches, those after the fields each chained to the
// one before:
//   fields   rho_A - rho0_A per site in float (the fluctuation-fields kernel);
//   columns, windows (when the columns are not given) the stripe's middle column
//            x_l and the column x_g half a box away, found on the device, and
//            the means over y of that field at the two (liquid and gas bulk);
//   bulk     (when they are given) the same means at the given columns;
//   heights  per row y (one warp): the liquid fractions
//            L(y) = sum_x (rho_A - rho_g) / (rho_l - rho_g) of the windows of
//            columns [x_g, x_l) and [x_l, x_g) (periodic) place the two
//            dividing surfaces h1 = x_l - 1/2 - L1 and h2 = x_l - 1/2 + L2, in
//            the frame of x_l, column x covering [x - 1/2, x + 1/2); with
//            tracked columns each snapshot uses its own frame;
//   spectrum each interface's height in row 0 is taken off (a constant drops out of
//            every k > 0) and, for k_m = 2 pi m / n_y, |sum_y dh(y) exp(-i k_m y)|^2
//            / n_y of the two interfaces is averaged and added to an FP64 accumulator
//            (twiddles from a table indexed by m y mod n_y), a block a wavenumber;
//            the mean heights are accumulated too.
#include <cmath>
#include <vector>

#include "flbm_ctx.h"

using namespace flbm;
using namespace flbm::host;

namespace {

__device__ __forceinline__ int wrap_col(int x, int nx) { return x >= nx ? x - nx : x; }

// Columns of a stripe that may have moved: with C(x) the mean over y of
// rho_A - rho0_A, the window of nx/2 columns with the largest sum of C holds
// the A-rich stripe; its middle column is the liquid-bulk column and the one
// half a box away the gas-bulk column (ties: the lowest x).
//
// FP64 sums here are short chains on many warps: on this GPU a dependent FP64
// add takes about 80 ns and a warp's FP64 instruction about 64 cycles of its
// scheduler (measured: 512 rows summed by one thread a column take 40 us,
// whatever the number of columns a warp).  Sums of 24-bit values close to one
// another in magnitude are exact in FP64, so the order seldom matters at all.
//
// colsum[x] = sum over y.  A block owns kCols columns and cuts the rows over
// kRowLanes lanes a column.  100 x 512: columns and windows together 63 us as
// one block, 13 us now.
constexpr int kCols = 8, kRowLanes = 16;
__global__ void __launch_bounds__(kCols * kRowLanes) k_cap_columns(const float2 *z, int nx, int ny, double *colsum,
                                                                   unsigned *turn)
{
    __shared__ double sh[kCols * kRowLanes / 32][kCols];
    int t = threadIdx.x;
    await_grid(t);
    const int x = blockIdx.x * kCols + t % kCols;
    if (blockIdx.x == 0 && t == 0) *turn = 0; // for the windows
    double c = 0.0;
    if (x < nx) {
#pragma unroll 8
        for (int y = t / kCols; y < ny; y += kRowLanes) c += (double)z[(size_t)y * nx + x].x;
    }
    for (int o = 16; o >= kCols; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if ((t & 31) < kCols) sh[t >> 5][t & 31] = c;
    __syncthreads();
    if (t < kCols && x < nx) {
        for (int w = 1; w < kCols * kRowLanes / 32; w++) c += sh[w][t];
        colsum[x] = c;
    }
}

// is the window (v2, x2) ahead of (v, x)?
__device__ __forceinline__ bool ahead_of(double v2, int x2, double v, int x) { return v2 > v || (v2 == v && x2 < x); }

// The window sums, a warp a window; the last block to finish picks the window:
// cols[0] = x_l, cols[1] = x_g, bulk[0 .. 1] the columns' means.  win: nx
// doubles; *turn, zero at the start (k_cap_columns), counts the finished blocks.
constexpr int kWinWarps = 4;
__global__ void __launch_bounds__(32 * kWinWarps) k_cap_windows(const double *colsum, int nx, int ny, double *win,
                                                               unsigned *turn, int *cols, double *bulk)
{
    __shared__ unsigned last;
    __shared__ double sh_v[kWinWarps];
    __shared__ int sh_x[kWinWarps];
    int t = threadIdx.x;
    await_grid(t);
    const int lane = t & 31, warp = t >> 5;
    const int x0 = blockIdx.x * kWinWarps + warp, w = nx / 2;
    if (x0 < nx) {
        double s = 0.0;
        for (int k = lane; k < w; k += 32) s += colsum[wrap_col(x0 + k, nx)];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) __stcg(win + x0, s);
    }
    __threadfence();
    __syncthreads();
    if (t == 0) last = atomicAdd(turn, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double bv = -1e300;
    int bx = nx;
    auto take = [&](double v2, int x2) {
        if (ahead_of(v2, x2, bv, bx)) {
            bv = v2;
            bx = x2;
        }
    };
    for (int x = t; x < nx; x += 32 * kWinWarps) take(__ldcg(win + x), x);
    for (int o = 16; o > 0; o >>= 1) take(__shfl_down_sync(0xffffffffu, bv, o), __shfl_down_sync(0xffffffffu, bx, o));
    if (lane == 0) {
        sh_v[warp] = bv;
        sh_x[warp] = bx;
    }
    __syncthreads();
    if (t == 0) {
        for (int k = 1; k < kWinWarps; k++) take(sh_v[k], sh_x[k]);
        const int xl = wrap_col(bx + w / 2, nx), xg = wrap_col(xl + nx / 2, nx);
        cols[0] = xl;
        cols[1] = xg;
        bulk[0] = colsum[xl] / ny;
        bulk[1] = colsum[xg] / ny;
    }
}

// columns from the caller (fixed) or from k_cap_windows (cols)
__device__ __forceinline__ void cap_cols(int xl_in, int xg_in, const int *cols, int &xl, int &xg)
{
    if (xl_in >= 0) {
        xl = xl_in;
        xg = xg_in;
    } else {
        xl = cols[0];
        xg = cols[1];
    }
}

__global__ void __launch_bounds__(256) k_cap_bulk(const float2 *z, int nx, int ny, int xl, int xg, double *bulk)
{
    __shared__ double sh[256][2];
    double l = 0.0, g = 0.0;
    int t = threadIdx.x;
    await_grid(t);
    for (int y = t; y < ny; y += 256) {
        l += (double)z[(size_t)y * nx + xl].x;
        g += (double)z[(size_t)y * nx + xg].x;
    }
    sh[threadIdx.x][0] = l;
    sh[threadIdx.x][1] = g;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            sh[threadIdx.x][0] += sh[threadIdx.x + s][0];
            sh[threadIdx.x][1] += sh[threadIdx.x + s][1];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        bulk[0] = sh[0][0] / ny;
        bulk[1] = sh[0][1] / ny;
    }
}

// one warp per row; h[0][y] and h[1][y]
__global__ void __launch_bounds__(128) k_cap_heights(const float2 *z, int nx, int ny, int xl_in, int xg_in,
                                                     const int *cols, const double *bulk, double *h)
{
    const int lane = threadIdx.x & 31;
    int y = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    await_grid(y);
    if (y >= ny) return;
    int xl, xg;
    cap_cols(xl_in, xg_in, cols, xl, xg);
    const double rl = bulk[0], rg = bulk[1], inv = 1.0 / (rl - rg);
    const int n1 = xl - xg >= 0 ? xl - xg : xl - xg + nx; // window [x_g, x_l)
    const int n2 = nx - n1;                               // window [x_l, x_g)
    const float2 *row = z + (size_t)y * nx;
    double s1 = 0.0, s2 = 0.0;
    for (int k = lane; k < n1; k += 32) s1 += ((double)row[wrap_col(xg + k, nx)].x - rg) * inv;
    for (int k = lane; k < n2; k += 32) s2 += ((double)row[wrap_col(xl + k, nx)].x - rg) * inv;
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_down_sync(0xffffffffu, s1, o);
        s2 += __shfl_down_sync(0xffffffffu, s2, o);
    }
    if (lane == 0) {
        h[y] = xl - 0.5 - s1;
        h[ny + y] = xl - 0.5 + s2;
    }
}

constexpr int kSpecThreads = 64;
// sums of both values over the block, in a fixed order; every thread gets them
__device__ __forceinline__ double2 block_sum2(double a, double b, double2 *sh)
{
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    __syncthreads(); // sh may still be read from the last sum
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = make_double2(a, b);
    __syncthreads();
    double2 s = sh[0];
    for (int w = 1; w < kSpecThreads / 32; w++) {
        s.x += sh[w].x;
        s.y += sh[w].y;
    }
    return s;
}

// Block m - 1: wavenumber m of both interfaces, the rows over the block's
// threads; block 0 the mean heights too.  The heights are taken from that of
// row 0: a constant drops out of every m >= 1, so the mean need not be formed
// first.  One block for all m is a serial chain of n_y FP64 multiply-adds a
// thread: 100 x 512 211 us, now 11.
__global__ void __launch_bounds__(kSpecThreads) k_cap_spectrum(const double *h, int ny, const double2 *tw, double *acc,
                                                               double *hsum)
{
    __shared__ double2 sh[kSpecThreads / 32];
    int t = threadIdx.x;
    await_grid(t);
    const int m = (int)blockIdx.x + 1;
    const double ref0 = h[0], ref1 = h[ny];
    double r0 = 0.0, i0 = 0.0, r1 = 0.0, i1 = 0.0;
    int idx = (int)((long long)m * t % ny);                   // m y mod ny
    const int next = (int)((long long)m * kSpecThreads % ny); // a thread's rows are kSpecThreads apart
    for (int y = t; y < ny; y += kSpecThreads) {
        const double2 w = tw[idx]; // (cos, -sin)(2 pi idx / ny)
        const double d0 = h[y] - ref0, d1 = h[ny + y] - ref1;
        r0 += d0 * w.x;
        i0 += d0 * w.y;
        r1 += d1 * w.x;
        i1 += d1 * w.y;
        idx += next;
        if (idx >= ny) idx -= ny;
    }
    const double2 s0 = block_sum2(r0, i0, sh), s1 = block_sum2(r1, i1, sh);
    if (t == 0) acc[m - 1] += 0.5 * (s0.x * s0.x + s0.y * s0.y + s1.x * s1.x + s1.y * s1.y) / ny;
    if (m > 1) return;
    double a = 0.0, b = 0.0;
    for (int y = t; y < ny; y += kSpecThreads) {
        a += h[y];
        b += h[ny + y];
    }
    const double2 sum = block_sum2(a, b, sh);
    if (t == 0) {
        hsum[0] += sum.x / ny;
        hsum[1] += sum.y / ny;
    }
}

} // namespace

namespace flbm {
void free_cap(flbm_ctx *c)
{
    if (c->d_cap_z) cudaFree(c->d_cap_z);
    if (c->d_cap_h) cudaFree(c->d_cap_h);
    if (c->d_cap_tw) cudaFree(c->d_cap_tw);
    c->d_cap_z = nullptr;
    c->d_cap_h = nullptr;
    c->d_cap_tw = nullptr;
    c->cap_count = 0;
}
} // namespace flbm

extern "C" {

flbm_status flbm_cap_sample(flbm_ctx *c, int x_liquid, int x_gas)
{
    if (!c) return FLBM_EINVAL;
    if (is_batch(c)) return fail(c, FLBM_EINVAL, "a batch has one spectrum per replica: use flbm_batch_replica");
    if (c->lat != FLBM_D2Q9) return fail(c, FLBM_EUNSUPPORTED, "interface heights are defined for D2Q9 stripes");
    if (!c->initialised) return fail(c, FLBM_ESTATE, "flbm_cap_sample before flbm_init");
    const bool track = x_liquid < 0 && x_gas < 0;
    if (!track && (x_liquid < 0 || x_liquid >= c->nx || x_gas < 0 || x_gas >= c->nx || x_liquid == x_gas))
        return fail(c, FLBM_EINVAL, "bulk columns must be two different columns of the box, or both negative");
    if (track) x_liquid = x_gas = -1;
    if (c->cap_count > 0 && (x_liquid != c->cap_xl || x_gas != c->cap_xg))
        return fail(c, FLBM_EINVAL, "bulk columns differ from the accumulated snapshots; reset first");
    flbm_status st = ensure_obs(c); // block partials of the fields kernel
    if (st != FLBM_OK) return st;
    const int ny = c->ny, nk = ny / 2;
    const size_t words = (size_t)2 * ny + nk + 6 + 2 * c->nx;
    if (!c->d_cap_z) {
        // layout of d_cap_h: heights [2][ny], spectrum sums [nk], mean-height sums [2], bulk [2],
        // column sums [nx], tracked columns and the blocks' turn (4 ints), window sums [nx]
        if (cudaMalloc((void **)&c->d_cap_z, (size_t)c->N * sizeof(float2)) != cudaSuccess ||
            cudaMalloc((void **)&c->d_cap_h, words * sizeof(double)) != cudaSuccess ||
            cudaMalloc((void **)&c->d_cap_tw, (size_t)ny * sizeof(double2)) != cudaSuccess) {
            cudaGetLastError();
            free_cap(c);
            return fail(c, FLBM_ENOMEM, "capillary-spectrum buffers do not fit");
        }
        std::vector<double2> tw((size_t)ny);
        for (int j = 0; j < ny; j++) {
            const double a = 2.0 * M_PI * (double)j / (double)ny;
            tw[j] = make_double2(std::cos(a), -std::sin(a));
        }
        // both done on return, also when the stream is being captured: a later call
        // finds buffers that are ready, or none
        cudaError_t e = copy_in(c->d_cap_tw, tw.data(), tw.size() * sizeof(double2));
        if (e == cudaSuccess) e = cudaMemset(c->d_cap_h, 0, words * sizeof(double));
        if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
        if (e != cudaSuccess) {
            free_cap(c);
            return cuda_fail(c, e, "capillary tables");
        }
        c->cap_count = 0;
    }
    double *heights = c->d_cap_h, *spec = heights + 2 * ny, *hsum = spec + nk, *bulk = hsum + 2;
    double *colsum = bulk + 2;
    int *cols = reinterpret_cast<int *>(colsum + c->nx);
    unsigned *turn = reinterpret_cast<unsigned *>(cols + 2);
    double *win = colsum + c->nx + 2;
    const StepParams p = make_params(c);
    int nb = 0;
    FLBM_CUDA(c, launch_sfk_fields(c->lat, c->storage, layout_parity(c), p, cur_pop(c), c->d_cap_z, c->d_partials, &nb, c->stream),
              "fields kernel launch");
    cudaError_t e;
    if (track) {
        e = launch_chained(true, k_cap_columns, (c->nx + kCols - 1) / kCols, kCols * kRowLanes, 0, c->stream, c->d_cap_z,
                           c->nx, ny, colsum, turn);
        if (e == cudaSuccess)
            e = launch_chained(true, k_cap_windows, (c->nx + kWinWarps - 1) / kWinWarps, 32 * kWinWarps, 0, c->stream,
                               colsum, c->nx, ny, win, turn, cols, bulk);
    } else {
        e = launch_chained(true, k_cap_bulk, 1, 256, 0, c->stream, c->d_cap_z, c->nx, ny, x_liquid, x_gas, bulk);
    }
    if (e == cudaSuccess)
        e = launch_chained(true, k_cap_heights, (ny + 3) / 4, 128, 0, c->stream, c->d_cap_z, c->nx, ny, x_liquid, x_gas,
                           cols, bulk, heights);
    if (e == cudaSuccess && nk > 0)
        e = launch_chained(true, k_cap_spectrum, nk, kSpecThreads, 0, c->stream, heights, ny, c->d_cap_tw, spec, hsum);
    FLBM_CUDA(c, e, "capillary kernel launch");
    c->cap_xl = x_liquid;
    c->cap_xg = x_gas;
    c->cap_count++;
    return FLBM_OK;
}

flbm_status flbm_cap_spectrum(flbm_ctx *c, int nk, double *S_h, double *h_mean, int64_t *nsamples)
{
    if (!c) return FLBM_EINVAL;
    if (nsamples) *nsamples = c->cap_count;
    if (!c->d_cap_h || c->cap_count == 0) return fail(c, FLBM_ESTATE, "no capillary snapshot taken");
    const int ny = c->ny, nmax = ny / 2;
    if (nk < 1 || nk > nmax) return fail(c, FLBM_EINVAL, "nk must lie in [1, %d]", nmax);
    flbm_status st = sync_and_check(c);
    if (st != FLBM_OK) return st;
    std::vector<double> h((size_t)nmax + 2);
    FLBM_CUDA(c, cudaMemcpy(h.data(), c->d_cap_h + 2 * ny, h.size() * sizeof(double), cudaMemcpyDeviceToHost),
              "D2H spectrum");
    if (S_h)
        for (int m = 0; m < nk; m++) S_h[m] = h[m] / (double)c->cap_count;
    if (h_mean) {
        h_mean[0] = h[nmax] / (double)c->cap_count;
        h_mean[1] = h[nmax + 1] / (double)c->cap_count;
    }
    return FLBM_OK;
}

flbm_status flbm_cap_reset(flbm_ctx *c)
{
    if (!c) return FLBM_EINVAL;
    if (c->stream) cudaStreamSynchronize(c->stream);
    free_cap(c);
    return FLBM_OK;
}

} // extern "C"
