// Allocation-free row-residual check.
//
// Some callers of this library may not allocate device memory at all: a host application
// that gives every component a fixed memory budget at start-up and forbids later driver
// allocations, or a latency-critical loop that cannot afford the implicit device-wide
// synchronisation of cudaMalloc / cudaFree.  The batch API already takes its workspace from
// the caller, but a caller who only wants to audit a plan it already holds (potentials from
// an earlier solve, a warm start, another solver) would still have to size and provide
// that workspace.  This entry point needs none: the per-CTA partial sums and the arrival
// counters of the fused residual reduction live in a fixed array that is part of the
// library image, so every GPU that loads the library carries SKB_STATIC_SCRATCH_BYTES of it
// until the process exits.
//
// It is the row screen of the update kernel in its plainest form: for every lane
//     r_row = sum_i | sum_j exp((f_i + g_j - |x_i - y_j|^2) / eps) - a_i |,
// float64 arithmetic, per-CTA partial sums combined in a fixed order by the last CTA of the lane to
// arrive; up to 32 dimensions by tiles in shared memory, beyond that one thread per row.
#include <cuda_runtime.h>
#include <mutex>
#include <string>

#include "skb_pairs64.cuh"

#include "../../include/sinkhorn_batch.h"

namespace {

constexpr int NA_THREADS = 128;                       // rows per CTA
constexpr int NA_MAX_LANES = SKB_STATIC_MAX_LANES;    // 256
constexpr int NA_MAX_BLOCKS = SKB_STATIC_MAX_ROWS / NA_THREADS;   // 64 row blocks per lane
constexpr int NA_MAX_DEVICES = 64;

struct Scratch {
    double partial[NA_MAX_LANES][NA_MAX_BLOCKS];      // per-CTA L1 partial sums
    unsigned arrived[NA_MAX_LANES];                   // CTAs of the lane that have finished
};
static_assert(sizeof(Scratch) <= SKB_STATIC_SCRATCH_BYTES, "scratch larger than documented");

// The scratch itself.  In host code this name is only a handle for cudaGetSymbolAddress;
// it is not a device address and must never be handed to a kernel directly.
static __device__ __align__(256) unsigned char g_scratch[SKB_STATIC_SCRATCH_BYTES];

std::mutex g_mu;
Scratch *g_dev_scratch[NA_MAX_DEVICES] = {};
thread_local std::string g_err;       // text of the calling thread's last failure; empty after a success

__global__ void __launch_bounds__(NA_THREADS) row_residual_kernel(
    Scratch *sc, const float *x, const float *y, const float *a, const double *f, const double *g,
    const float *eps, int n, int m, int d, float *r_row)
{
    __shared__ double red[NA_THREADS / 32];
    __shared__ int is_last;
    const int lane_id = blockIdx.y, tid = threadIdx.x;
    const int i = blockIdx.x * NA_THREADS + tid;
    const double inv_eps = 1.0 / (double)eps[lane_id];
    const float *xl = x + (size_t)lane_id * n * d, *yl = y + (size_t)lane_id * m * d;
    const double *fl = f + (size_t)lane_id * n, *gl = g + (size_t)lane_id * m;
    double term = 0.0;
    if (i < n) {
        double mx = -1.0e300, s = 0.0;
        for (int j = 0; j < m; ++j) {
            double c = 0.0;
            for (int k = 0; k < d; ++k) {
                const double t = (double)xl[(size_t)i * d + k] - (double)yl[(size_t)j * d + k];
                c += t * t;
            }
            const double v = (fl[i] + gl[j] - c) * inv_eps;
            if (v > mx) { s *= exp(mx - v); mx = v; }
            s += exp(v - mx);
        }
        term = fabs(exp(mx) * s - (double)a[(size_t)lane_id * n + i]);
    }
    for (int off = 16; off > 0; off >>= 1) term += __shfl_down_sync(0xffffffffu, term, off);
    if ((tid & 31) == 0) red[tid >> 5] = term;
    __syncthreads();
    if (tid == 0) {
        double p = 0.0;
        for (int w = 0; w < NA_THREADS / 32; ++w) p += red[w];
        sc->partial[lane_id][blockIdx.x] = p;
        __threadfence();
        is_last = (atomicAdd(&sc->arrived[lane_id], 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (!is_last || tid != 0) return;
    __threadfence();
    double tot = 0.0;
    for (unsigned b = 0; b < gridDim.x; ++b) tot += reinterpret_cast<volatile double *>(sc->partial[lane_id])[b];
    sc->arrived[lane_id] = 0u;              // leave the counter ready for the next call
    r_row[lane_id] = (float)tot;
}

// The wide tiles' part of a row's sum (skb_pairs64.cuh), by differences; every NC-th of the columns.
// Out of line: its registers would come off the tiled loop's.
template <int DM, int THREADS, int NC>
__device__ __noinline__ double wide_tiles(double *tile, const double *org, const float *xi, const float *yl, const double fi, const double *gl,
                                          const int m, const int d, const double k2, const int cs, const bool row_wide)
{
    using namespace skb;
    double s = 0.0;
    for (int j0 = 0; j0 < m; j0 += P64_TJ) {
        __syncthreads();
        P64Part<DM, THREADS> part;
        p64_fetch(part, j0, m, d, [&](int j, int k) { return yl[(size_t)j * d + k]; }, [&](int j) { return gl[j]; });
        const bool wide = p64_tile<DM, THREADS>(tile, org, j0, m, d, k2, part);
        if (!__syncthreads_or(wide || row_wide)) continue;
        for (int j = j0 + cs; j < m && j < j0 + P64_TJ; j += NC)
            s += p64_entry(d, k2, fi + gl[j], [&](int k) { return xi[k]; }, [&](int k) { return yl[(size_t)j * d + k]; });
    }
    return s;
}

// The same for d <= 32: a block of WPB warps takes 16 * WPB rows, column tiles come through shared memory
// (skb_pairs64.cuh).  The entries are summed as they are; a row whose sum is not finite is redone the plain way,
// so infinite potentials give what they always gave.  32 lanes of 1024 x 1000 points, d = 15: 1040 us with one
// thread per row and the columns read from global memory, 145 us so with CUDA's exp2, 117 us with p64_exp2.
template <int DM, int WPB, int RW>
__global__ void __launch_bounds__(32 * WPB) row_residual_tiled_kernel(
    Scratch *sc, const float *x, const float *y, const float *a, const double *f, const double *g,
    const float *eps, int n, int m, int d, float *r_row)
{
    using namespace skb;
    constexpr int R = 2, NC = 32 / (RW / R);
    __shared__ double tile[P64_TILE<DM, 32 * WPB>];
    __shared__ double org[DM];
    __shared__ double red[WPB];
    __shared__ int is_last;
    const int lane_id = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cs = lane / (RW / R), i0 = blockIdx.x * (RW * WPB) + warp * RW + lane % (RW / R) * R;
    const double inv_eps = 1.0 / (double)eps[lane_id], k2 = 1.4426950408889634 * inv_eps;
    const float *xl = x + (size_t)lane_id * n * d, *yl = y + (size_t)lane_id * m * d;
    const double *fl = f + (size_t)lane_id * n, *gl = g + (size_t)lane_id * m;
    if (tid < DM) org[tid] = tid < d ? (double)xl[(size_t)blockIdx.x * (RW * WPB) * d + tid] : 0.0;
    __syncthreads();
    double xr[R][DM], ri[R], s[R];
    bool row_wide = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = i0 + r < n ? i0 + r : n - 1;
        double q = 0.0;
#pragma unroll
        for (int k = 0; k < DM; ++k) { xr[r][k] = k < d ? (double)xl[(size_t)i * d + k] - org[k] : 0.0; q = fma(xr[r][k], xr[r][k], q); }
        ri[r] = k2 * (fl[i] - q);
        row_wide = row_wide || p64_wide(k2, q);
        s[r] = 0.0;
    }
    bool any_wide = false;
    const double entry = p64_table();
    auto load = [&](int j, int k) { return yl[(size_t)j * d + k]; };
    auto pot = [&](int j) { return gl[j]; };
    P64Part<DM, 32 * WPB> part;
    if (P64_AHEAD<DM>) p64_fetch(part, 0, m, d, load, pot);
    for (int j0 = 0; j0 < m; j0 += P64_TJ) {
        if (!P64_AHEAD<DM>) p64_fetch(part, j0, m, d, load, pot);
        __syncthreads();
        const bool wide = p64_tile<DM, 32 * WPB>(tile, org, j0, m, d, k2, part);
        if (P64_AHEAD<DM>) p64_fetch(part, j0 + P64_TJ, m, d, load, pot);
        if (__syncthreads_or(wide || row_wide)) { any_wide = true; continue; }
#pragma unroll 2
        for (int jj = cs; jj < P64_TJ; jj += NC) {
            double v[R];
            const double c = tile[DM * P64_TJ + jj];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = c + ri[r];
#pragma unroll
            for (int k = 0; k < DM; ++k) {
                const double yk = tile[k * P64_TJ + jj];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = fma(xr[r][k], yk, v[r]);
            }
            p64_exp2(v, entry);
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] += v[r];
        }
    }
    if (any_wide)
        for (int r = 0; r < R; ++r) {
            const int i = i0 + r < n ? i0 + r : n - 1;
            s[r] += wide_tiles<DM, 32 * WPB, NC>(tile, org, xl + (size_t)i * d, yl, fl[i], gl, m, d, k2, cs, row_wide);
        }
    double term = 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int off = RW / R; off < 32; off *= 2) s[r] += __shfl_xor_sync(0xffffffffu, s[r], off);
        if (cs == 0 && i0 + r < n) {
            if (!isfinite(s[r])) {
                // the plain sum, with its running maximum
                double mx = -1.0e300, t = 0.0;
                for (int j = 0; j < m; ++j) {
                    double c = 0.0;
                    for (int k = 0; k < d; ++k) { const double e = (double)xl[(size_t)(i0 + r) * d + k] - (double)yl[(size_t)j * d + k]; c += e * e; }
                    const double v = (fl[i0 + r] + gl[j] - c) * inv_eps;
                    if (v > mx) { t *= exp(mx - v); mx = v; }
                    t += exp(v - mx);
                }
                s[r] = exp(mx) * t;
            }
            term += fabs(s[r] - (double)a[(size_t)lane_id * n + i0 + r]);
        }
    }
    for (int off = RW / R / 2; off > 0; off >>= 1) term += __shfl_down_sync(0xffffffffu, term, off);
    if (lane == 0) red[warp] = term;
    __syncthreads();
    if (tid == 0) {
        double p = 0.0;
        for (int w = 0; w < WPB; ++w) p += red[w];
        sc->partial[lane_id][blockIdx.x] = p;
        __threadfence();
        is_last = (atomicAdd(&sc->arrived[lane_id], 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (!is_last || tid != 0) return;
    __threadfence();
    double tot = 0.0;
    for (unsigned b = 0; b < gridDim.x; ++b) tot += reinterpret_cast<volatile double *>(sc->partial[lane_id])[b];
    sc->arrived[lane_id] = 0u;
    r_row[lane_id] = (float)tot;
}

// 32 rows to a block while the scratch has a slot for every block (n <= 2048), 64 and 128 beyond
template <int DM>
void launch_tiled(Scratch *sc, const float *x, const float *y, const float *a, const double *f, const double *g, const float *eps,
                  int W, int n, int m, int d, float *r_row, cudaStream_t st)
{
    if (n <= 32 * NA_MAX_BLOCKS) row_residual_tiled_kernel<DM, 4, 8><<<dim3((n + 31) / 32, W), 128, 0, st>>>(sc, x, y, a, f, g, eps, n, m, d, r_row);
    else if (n <= 64 * NA_MAX_BLOCKS) row_residual_tiled_kernel<DM, 4, 16><<<dim3((n + 63) / 64, W), 128, 0, st>>>(sc, x, y, a, f, g, eps, n, m, d, r_row);
    else row_residual_tiled_kernel<DM, 8, 16><<<dim3((n + 127) / 128, W), 256, 0, st>>>(sc, x, y, a, f, g, eps, n, m, d, r_row);
}

skb_status fail(skb_status st, const std::string &msg)
{
    g_err = msg;
    return st;
}

}  // namespace

extern "C" const char *sinkhorn_row_residual_static_last_error(void) { return g_err.c_str(); }

extern "C" skb_status sinkhorn_row_residual_static(const float *x, const float *y, const float *a,
                                                   const double *f, const double *g, const float *eps,
                                                   int W, int n, int m, int d, float *r_row, void *stream)
{
    std::lock_guard<std::mutex> lock(g_mu);
    if (!x || !y || !a || !f || !g || !eps || !r_row) return fail(SKB_ERR_NULL, "all data pointers are required");
    if (W < 1 || n < 1 || m < 1 || d < 1) return fail(SKB_ERR_SHAPE, "W, n, m, d must be >= 1");
    if (W > SKB_STATIC_MAX_LANES || n > SKB_STATIC_MAX_ROWS)
        return fail(SKB_ERR_SHAPE, "beyond the static scratch: at most " + std::to_string(SKB_STATIC_MAX_LANES) +
                                       " lanes and " + std::to_string(SKB_STATIC_MAX_ROWS) + " source points per lane");
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(SKB_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= NA_MAX_DEVICES) return fail(SKB_ERR_STATE, "device ordinal out of range");
    if (!g_dev_scratch[dev]) {
        // first call on this device: resolve the device address of the static array
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess) return fail(SKB_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        g_dev_scratch[dev] = reinterpret_cast<Scratch *>(p);
    }
    Scratch *sc = g_dev_scratch[dev];
    cudaStream_t st = (cudaStream_t)stream;
    // the array keeps whatever the previous call left: the arrival counters must start at zero
    e = cudaMemsetAsync(sc->arrived, 0, sizeof(sc->arrived), st);
    if (e != cudaSuccess) return fail(SKB_ERR_CUDA, std::string("cudaMemsetAsync: ") + cudaGetErrorString(e));
    if (d <= 4) launch_tiled<4>(sc, x, y, a, f, g, eps, W, n, m, d, r_row, st);
    else if (d <= 8) launch_tiled<8>(sc, x, y, a, f, g, eps, W, n, m, d, r_row, st);
    else if (d <= 16) launch_tiled<16>(sc, x, y, a, f, g, eps, W, n, m, d, r_row, st);
    else if (d <= skb::P64_MAX_D) launch_tiled<skb::P64_MAX_D>(sc, x, y, a, f, g, eps, W, n, m, d, r_row, st);
    else {
        dim3 grid((n + NA_THREADS - 1) / NA_THREADS, W);
        row_residual_kernel<<<grid, NA_THREADS, 0, st>>>(sc, x, y, a, f, g, eps, n, m, d, r_row);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(SKB_ERR_CUDA, std::string("launch: ") + cudaGetErrorString(e));
    g_err.clear();
    return SKB_OK;
}
