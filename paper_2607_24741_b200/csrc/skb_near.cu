// Large low-dimensional lanes in fp32 (d <= 4): points are kept in spatial order, a leg skips the columns that
// are too far from a group of rows to matter, and coordinates are relative to the centre of their box.
//
// At the regularisations these lanes are solved with, a plan entry is negligible beyond a few multiples of
// sqrt(eps): on the registration workload (unit sphere, eps = 0.01) an entry falls below 2^-53 of its row
// sum at a distance of 0.6, and nine tenths of all pairs are farther apart.  So
//   - at create the points of a lane are put in the order of a k-d tree (median splits along the widest
//     extent, in chunks of SORT_CHUNK points), so that 16 or 32 consecutive points are close together;
//   - every 32 consecutive points have a bounding box and the largest potential among them (`top`, kept up to
//     date by the legs' epilogues);
//   - with gam_j <= top_J, phi_i - log2 w_i <= p_G for the 32 rows of group G and d(G, J) the distance of the
//     boxes, every term of rows G and columns J relative to the sum that row i would have if its potential
//     did not move (Eq. 3 read backwards, 2^m0_i) is at most 2^(top_J + p_G - d(G, J)^2 / 2), and box J is
//     skipped for G where that is below 2^-(32 + log2 m).
// After the pass, a row whose sum has come out below 2^-6 of that estimate (its potential is about to rise by
// more than six bits: the first cycles of a cold start) is done again over all columns.  What is skipped is
// therefore below 2^-26 of any row sum - 2^-32 where the potentials have settled - against the 2^-24 of every
// fp32 term.  Whether a box is skipped depends on the group alone, and so does the order of a row's partial
// sums: its bits do not depend on the block, or the launch shape, that holds it.
//
// Arguments.  With o the centre of a point's box of 32, r = o_G + r', c = o_J + c' and D = o_G - o_J,
//     arg_ij = gam_j - |r - c|^2 / 2 + |r'|^2 / 2 = (gam_j - |c'|^2 / 2 + D.c') + r'.c' - (D.r' + |D|^2 / 2):
// three more multiply-adds per column (shared by the rows of a thread) and a shift per row and box.  All
// terms are of the size of the distance itself, where the expanded form |x|^2 + |y|^2 - 2 x.y has terms of the
// size of the cloud: the argument's rounding error falls from about 1e-5 (ulp of 150 .. 430 on the
// registration workload) to below 1e-6 for the terms that weigh.
//
// What bounds it: instruction issue and the latency of a box's chain (load, offset, multiply-adds, ex2, sums); the
// special-function unit is about half busy.  Registration workload at 32 lanes of 8192 points: a fifth of the
// pairs is kept (an eighth would be with exact distances), f-leg 610 -> 213 us, g-leg 610 -> 230 us, solve
// 376 -> 140 ms; one lane of 4096 points 22.7 -> 15 ms.  Steps on the way, f / g: Hilbert curve instead of the k-d
// tree, tiles shared by the block, expanded form 280 / 300; a warp's own 16 rows, columns through L1 216 / 290 (groups
// with outliers keep one warp of a block busy); all warps on every group 258 / 258; 32 rows to a group, four to a
// thread, columns by cp.async 213 / 230.  Two loads ahead in registers, 16 rows at four to a thread: slower (307, 268).
//
// That is the way of each leg by itself (update_near_kernel), which column checks, and g-legs whose columns' potentials rise by many
// bits, still go.  Where there is room for lists of the pairs that matter, near_rows_kernel takes both legs of a
// cycle in one pass: one exponential a pair and cycle instead of two, over 0.11 of the pairs instead of 0.22.
#include <type_traits>
#include "skb_update.cuh"
#include "skb_host.h"
#include "skb_tmem.cuh"

namespace skb {

constexpr int SORT_CHUNK = 8192;                    // points ordered together (by one block, in shared memory)
constexpr int SORT_LEAF = 16;
constexpr float NEAR_BITS = 32.f, NEAR_SLACK = 0.5f;
constexpr double NEAR_FLOOR = 0x1p-6;
// Points of the larger cloud from which the order pays: at 1024 points (16 lanes, eps 0.01) a leg is 13.7 -> 10.3 us and
// a solve of 60 cycles 2.5 -> 2.3 ms, ordering included; the boxes of smaller clouds are too wide to skip much.
constexpr int NEAR_MIN = 1024;
// ... and with lists of single points (both legs in one pass) for clouds that are too large for the on-chip kernels, beside one another:
// registration lanes, eps 0.01, a solve plain -> one pass: 32 of 520 points 17.9 -> 12.6 ms, 4 of 700 9.4 -> 8.3, 8 of 900 14.1 -> 9.6,
// 32 of 900 21.6 -> 14.9; one lane of 600 (a cycle 17.2 <- 20.8 us) has too few groups and is better off
// with its columns split over more blocks.  (Counted are the lanes a batch can take in: a queue through one slot
// has the arithmetic, and so the bits, of one batch.)
constexpr int NEAR_MIN_LISTS = 513;
constexpr int NEAR_BLOCKS = 4;                      // blocks per SM (127 registers); five and six spill: 225 and 224 us a leg

bool near_shape(int f64, int DP, int CS, int n, int m, int lanes)
{
    const int mx = n > m ? n : m;
    return !f64 && DP > 0 && DP <= 4 && CS == 4 && (mx >= NEAR_MIN || (lanes >= 2 && mx >= NEAR_MIN_LISTS));
}

// ---------------------------------------------------------------- is the order worth it
// Counts, over 4096 sampled pairs of every lane, those whose boxes a settled leg would not skip.  Edge of a box of 32
// points: that of a uniform cloud with the same variances (dimensions next to none of it left out).  A pair counts
// if its distance less one box diagonal, measured between the clouds moved onto one centre (the potentials take up
// the translation), is within the reach of 36 bits: the cut of the legs less what the largest potentials add.  The
// potentials of clouds that lie apart vary inside a box by 2 s |shift| times its size, and a quarter of that is added.
// Against the share really kept (float64 restatement of the rule, 2048 to 4096 points, d = 1 .. 4; sphere with
// outliers, normal, uniform, uniform and shifted; eps 0.001 to 0.5): 0 to 0.15 above it, 0.1 to 0.15 below it only on
// normal clouds of d = 3, 4 that keep nearly everything.
constexpr int EST_POINTS = 256;
__global__ void __launch_bounds__(EST_POINTS) near_estimate_kernel(const Dev P, const void *xin, const void *yin)
{
    __shared__ double pt[2][4][EST_POINTS], red[8][8], mean[2][4];
    __shared__ int kept_s;
    const int q = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, d = P.d;
    double v[2][4];
    auto block_sums = [&]() {                            // v -> red[0 .. 7][side * 4 + k], one partial sum per warp
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            double s = v[e >> 2][e & 3];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (lane == 0) red[warp][e] = s;
        }
        __syncthreads();
    };
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int npts = side ? P.m : P.n;
        const size_t i = (size_t)q * npts + (size_t)((2ll * tid + 1) * npts / (2 * EST_POINTS));
#pragma unroll
        for (int k = 0; k < 4; ++k) v[side][k] = pt[side][k][tid] = k < d ? (double)load_raw(P, side ? yin : xin, i * d + k) : 0.0;
    }
    if (tid == 0) kept_s = 0;
    block_sums();
    if (tid < 8) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += red[w][tid];
        mean[tid >> 2][tid & 3] = s / EST_POINTS;
    }
    __syncthreads();
    double shift = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double sh = mean[0][k] - mean[1][k];
        shift = fma(sh, sh, shift);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const double c = pt[side][k][tid] - mean[side][k];
            pt[side][k][tid] = c;
            v[side][k] = c * c;
        }
    }
    block_sums();
    double edge[4], widest = 0.0, vol = 1.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += red[w][k] + red[w][4 + k];
        edge[k] = sqrt(12.0 * s / (2 * EST_POINTS));
        widest = fmax(widest, edge[k]);
    }
    int dims = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) if (edge[k] > 0.02 * widest) { vol *= edge[k]; ++dims; }
    const double diag = dims ? pow(vol * 32.0 / (P.n > P.m ? P.n : P.m), 1.0 / dims) * sqrt((double)dims) : 0.0;
    const double s = P.scale[q], reach = 36.0 + 0.5 * s * sqrt(shift) * diag;
    int kept = 0;
    for (int r = 0; r < NEAR_PAIRS / EST_POINTS; ++r) {
        const int j = (tid + 17 * r) & (EST_POINTS - 1);
        double d2 = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) { const double t = pt[0][k][tid] - pt[1][k][j]; d2 = fma(t, t, d2); }
        const double gap = fmax(sqrt(d2) - diag, 0.0);
        kept += !(s * gap * gap > reach);                // NaN: keep
    }
    kept = __reduce_add_sync(0xffffffffu, kept);
    if (lane == 0) atomicAdd(&kept_s, kept);
    __syncthreads();
    if (tid == 0) atomicAdd(&P.ctl->near_kept, kept_s);
}
void launch_near_estimate(const Dev &P, const void *x, const void *y, int lanes, cudaStream_t st)
{
    near_estimate_kernel<<<lanes, EST_POINTS, 0, st>>>(P, x, y);
}

// ---------------------------------------------------------------- spatial order
// fp32 value -> unsigned integer of the same order
__device__ __forceinline__ unsigned ordered_bits(const float v)
{
    const unsigned u = __float_as_uint(v);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}

// One block per chunk of a cloud.  Level by level, from the whole chunk (padded to a power of two) down to
// segments of two leaves, every segment is sorted along its widest extent (bitonic, all segments at once), so
// that its halves are the two sides of a median split.
__global__ void __launch_bounds__(1024) spatial_sort_kernel(const Dev P, const void *xin, const void *yin, const int slot0)
{
    extern __shared__ unsigned long long item[];          // [size] key << 32 | index in the chunk, then [DP][SORT_CHUNK] coordinates
    float *crd = reinterpret_cast<float *>(item + SORT_CHUNK);
    __shared__ unsigned ext[2][4][SORT_CHUNK / (2 * SORT_LEAF)];       // [min, max][dimension][segment], as ordered integers
    const int q = blockIdx.y, slot = slot0 + q, side = blockIdx.z, tid = threadIdx.x;
    const int npts = side ? P.m : P.n, pp = side ? P.mp : P.np, base = (int)blockIdx.x * SORT_CHUNK;
    const int cnt = min(SORT_CHUNK, npts - base);
    if (cnt <= 0) return;
    int size = 2 * SORT_LEAF;
    while (size < cnt) size <<= 1;
    const void *in = side ? yin : xin;
    for (int e = tid; e < size; e += 1024) {
        item[e] = e < cnt ? (unsigned long long)e : ~0ull;
        if (e < cnt) for (int k = 0; k < P.d; ++k) crd[k * SORT_CHUNK + e] = load_raw(P, in, ((size_t)q * npts + base + e) * P.d + k);
    }
    for (int seg = size; seg >= 2 * SORT_LEAF; seg >>= 1) {
        const int nseg = size / seg;
        __syncthreads();
        for (int e = tid; e < nseg; e += 1024)
            for (int k = 0; k < P.d; ++k) { ext[0][k][e] = 0xffffffffu; ext[1][k][e] = 0u; }
        __syncthreads();
        for (int e = tid; e < size; e += 1024) {           // whole warps of one segment (segments hold at least 32)
            const unsigned idx = (unsigned)item[e];
            for (int k = 0; k < P.d; ++k) {
                const unsigned u = idx != 0xffffffffu ? ordered_bits(crd[k * SORT_CHUNK + idx]) : 0u;
                const unsigned lo = __reduce_min_sync(0xffffffffu, idx != 0xffffffffu ? u : 0xffffffffu), hi = __reduce_max_sync(0xffffffffu, u);
                if ((tid & 31) == 0) { atomicMin(&ext[0][k][e / seg], lo); atomicMax(&ext[1][k][e / seg], hi); }
            }
        }
        __syncthreads();
        for (int e = tid; e < size; e += 1024) {
            const unsigned idx = (unsigned)item[e];
            if (idx == 0xffffffffu) continue;
            int dim = 0;
            float widest = -1.f;
            for (int k = 0; k < P.d; ++k) {
                const unsigned lo = ext[0][k][e / seg], hi = ext[1][k][e / seg];
                const float w = __uint_as_float(hi & 0x80000000u ? hi & 0x7fffffffu : ~hi) - __uint_as_float(lo & 0x80000000u ? lo & 0x7fffffffu : ~lo);
                if (w > widest) { widest = w; dim = k; }
            }
            item[e] = ((unsigned long long)ordered_bits(crd[dim * SORT_CHUNK + idx]) << 32) | idx;
        }
        for (int k = 2; k <= seg; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                __syncthreads();
                for (int e = tid; e < size / 2; e += 1024) {
                    const int lo = 2 * (e & ~(j - 1)) | (e & (j - 1)), hi = lo | j;
                    const unsigned long long a = item[lo], b = item[hi];
                    if ((a > b) == (k == seg || (lo & k) == 0)) { item[lo] = b; item[hi] = a; }
                }
            }
        }
    }
    __syncthreads();
    int *perm = (side ? P.permy : P.permx) + (size_t)P.lane_id[slot] * pp + base;
    for (int e = tid; e < cnt; e += 1024) perm[e] = base + (int)(unsigned)item[e];
}

void launch_spatial_sort(const Dev &P, const void *x, const void *y, int slot0, int count, cudaStream_t st)
{
    const int mx = P.n > P.m ? P.n : P.m;
    const int smem = SORT_CHUNK * (8 + 4 * P.DP);
    // (the limit for any dimension: another host thread may set it between this and the launch)
    cudaFuncSetAttribute(spatial_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SORT_CHUNK * (8 + 4 * 4));
    spatial_sort_kernel<<<dim3((mx + SORT_CHUNK - 1) / SORT_CHUNK, count, 2), 1024, smem, st>>>(P, x, y, slot0);
}

// The largest potential of a box of the source (with lists: of its halves; one without points keeps this minus infinity, for
// near_rows_kernel writes the others only).
__device__ __forceinline__ void top_x(const Dev &P, const int parity, const int slot, const int box, const float top)
{
    const size_t o = (size_t)slot * P.nbx + box;
    if (P.lists) reinterpret_cast<float2 *>(P.topx[parity])[o] = make_float2(top, BOX_COLS * box + GROUP_ROWS < P.n ? top : -3.0e38f);
    else P.topx[parity][o] = top;
}
__device__ __forceinline__ GroupRecord &group_record(const Dev &P, const int home, const int group)
{
    return P.groups[(size_t)home * 2 * P.nbx + group];
}
// What near_rows_kernel starts row i from: its reference (the log-sum-exp that Eq. 3 read backwards gives, rounded up; none where
// the estimate is out of range) and weight, and the tops of its group.  Whole groups of GROUP_ROWS consecutive threads.
__device__ __forceinline__ void row_record(const Dev &P, const int home, const int i, const bool in, const double pot, const double lw,
                                           const double sq, const float w)
{
    const double est = lw + sq - pot;
    const bool has = in && fabs(est) < 1.0e7;
    float prow = has ? __double2float_ru(pot - lw) : -3.0e38f, pcol = has ? __double2float_ru(pot) : -3.0e38f;
    GroupRecord &g = group_record(P, home, i / GROUP_ROWS);
    g.row[i % GROUP_ROWS] = make_float2(has ? -ceilf((float)est) : NEG_BIG, in ? w : 0.f);
#pragma unroll
    for (int off = GROUP_ROWS / 2; off > 0; off >>= 1) {
        prow = fmaxf(prow, __shfl_xor_sync(0xffffffffu, prow, off));
        pcol = fmaxf(pcol, __shfl_xor_sync(0xffffffffu, pcol, off));
    }
    if (i % GROUP_ROWS == 0) { g.prow = prow; g.pcol = pcol; }
}
// The target's potentials as near_rows_kernel reads them, in two parts.
__device__ __forceinline__ void home_potential(const Dev &P, const int home, const int j, const double pot)
{
    const size_t o = (size_t)home * (P.mp + 1) + j;
    const float hi = (float)pot;
    (P.DP < 4 ? P.crdy + 4 * o + 3 : P.gamy + o)[0] = hi;
    P.unit_low[o].y = (float)(pot - (double)hi);
}

// Layout of lanes in spatial order: boxes, coordinates relative to their box's centre, squared norms of those,
// weights, cold potentials and their maxima, and the raw copies for the guard band in the slot's order.
__global__ void __launch_bounds__(128) prep_near_kernel(const Dev P, const void *xin, const void *yin, const float *a, const float *b, const int slot0)
{
    const int q = blockIdx.y, slot = slot0 + q, side = blockIdx.z;
    const int npts = side ? P.m : P.n, pp = side ? P.mp : P.np, nb = side ? P.nby : P.nbx;
    const int i = blockIdx.x * 128 + threadIdx.x, lane = threadIdx.x & 31, b32 = i >> 5;
    if (i >= pp) return;                                   // whole warps: pp is a multiple of 32
    float *box = (side ? P.boxy : P.boxx) + (size_t)slot * 2 * P.DP * nb;
    float *crd = reinterpret_cast<float *>(side ? P.ys : P.xs) + (size_t)slot * P.DP * pp;
    const bool in = i < npts;
    const size_t src = (size_t)q * npts + (in ? (side ? P.permy : P.permx)[(size_t)P.lane_id[slot] * pp + i] : 0);
    const double sc = sqrt(2.0 * P.scale[slot]);
    // (the first lanes find their home here, later ones take what the slot has)
    const int home = !P.lists ? 0 : (P.lane_id[slot] < P.W ? slot : P.home[slot]);
    float *box16 = P.lists && !side ? P.boxx16 + (size_t)home * 2 * P.DP * 2 * nb : nullptr;
    char *rawdst = P.guard > 0.0 ? (char *)(side ? P.yraw : P.xraw) + (size_t)slot * (side ? P.yraw_stride : P.xraw_stride) : nullptr;
    double nrm = 0.0;
    bool ok = true;
    for (int k = 0; k < P.DP; ++k) {
        double v = 0.0;
        if (in && k < P.d) {
            const float raw = load_raw(P, side ? yin : xin, src * P.d + k);
            ok = ok && isfinite(raw);
            v = sc * ((double)raw - P.center[(size_t)slot * P.DP + k]);
            if (rawdst) {
                if (P.xy_bf16) reinterpret_cast<unsigned short *>(rawdst)[(size_t)i * P.d + k] = (unsigned short)(__float_as_uint(raw) >> 16);
                else reinterpret_cast<float *>(rawdst)[(size_t)i * P.d + k] = raw;
            }
        }
        float lo = in ? __double2float_rd(v) : 3.0e38f, hi = in ? __double2float_ru(v) : -3.0e38f;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            if (off == GROUP_ROWS && box16 && lane % GROUP_ROWS == 0) {
                box16[k * 2 * nb + i / GROUP_ROWS] = lo; box16[(P.DP + k) * 2 * nb + i / GROUP_ROWS] = hi;
            }
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
        }
        if (lane == 0) { box[k * nb + b32] = lo; box[(P.DP + k) * nb + b32] = hi; }
        const float rel = in ? (float)(v - (double)(0.5f * (lo + hi))) : 0.f;
        crd[(size_t)k * pp + i] = rel;
        if (P.lists && side) {
            P.crdy[((size_t)home * (pp + 1) + i) * 4 + k] = rel;
            if (lane == 0) P.ceny[((size_t)home * (nb + 1) + b32) * 4 + k] = 0.5f * (lo + hi);
        }
        if (P.lists && !side) {
            GroupRecord &g = group_record(P, home, i / GROUP_ROWS);
            g.crd[k][i % GROUP_ROWS] = -rel;
            if (lane % GROUP_ROWS == 0) g.centre[k] = 0.5f * (lo + hi);
        }
        nrm += (double)rel * (double)rel;
    }
    const size_t o = (size_t)slot * pp + i;
    float hi0 = NEG_BIG;
    double sq = 0.0, lw = 0.0, w = 0.0;
    if (in) {
        const float wt = (side ? b : a)[src];
        ok = ok && (wt > 0.0f) && isfinite(wt);
        if (!ok) atomicOr(&P.ctl->error, ERR_VALUE);
        sq = 0.5 * nrm;
        lw = ok ? log2((double)wt) : 0.0;
        w = ok ? (double)wt : 0.0;
        hi0 = (float)(-sq);                                // cold start: phi = gam = 0
    }
    (side ? P.sqy : P.sqx)[o] = sq; (side ? P.lb2 : P.la2)[o] = lw; (side ? P.wb : P.wa)[o] = w;
    if (side) {
        reinterpret_cast<float *>(P.gt)[o] = hi0; reinterpret_cast<float *>(P.gl)[o] = 0.f; P.gam[o] = 0.0;
        if (lane == 0) P.topy[(size_t)slot * nb + b32] = 0.f;
        if (P.lists) {
            float least = in ? __double2float_rd(lw) : 3.0e38f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) least = fminf(least, __shfl_xor_sync(0xffffffffu, least, off));
            if (lane == 0) P.lby[(size_t)home * nb + b32] = least;
            const size_t ho = (size_t)home * (pp + 1) + i;
            P.unit_low[ho].x = in && ok ? ldexpf(1.f, max(-100, min(114, 44 - ilogb(w)))) : 0.f;
            home_potential(P, home, i, in ? 0.0 : (double)NEG_BIG);
            P.colacc[0][(size_t)home * pp + i] = 0ull; P.colacc[1][(size_t)home * pp + i] = 0ull;
            if (i == 0) {                                    // the point of weight zero
                for (int k = 0; k < 4; ++k) { P.crdy[((size_t)home * (pp + 1) + pp) * 4 + k] = 0.f; P.ceny[((size_t)home * (nb + 1) + pp / BOX_COLS) * 4 + k] = 0.f; }
                P.unit_low[(size_t)home * (pp + 1) + pp].x = 0.f;
                home_potential(P, home, pp, (double)NEG_BIG);
            }
            if (i == 0) { P.home[slot] = home; P.risen[home] = 0ull; P.based_at[home] = 0; P.overrun[home] = P.overrun[P.W + home] = 0u; }
        }
    } else {
        for (int e = 0; e < 2; ++e) {
            reinterpret_cast<float *>(P.ft[e])[o] = hi0; reinterpret_cast<float *>(P.fl[e])[o] = 0.f; P.phi[e][o] = 0.0;
            if (lane == 0) top_x(P, e, slot, b32, 0.f);
        }
        if (P.lists) {
            row_record(P, home, i, in, 0.0, lw, sq, (float)w);
            if (lane % GROUP_ROWS == 0) group_record(P, home, i / GROUP_ROWS).made_from = 0;       // no lists yet
        }
    }
}
void launch_prep_near(const Dev &P, const void *x, const void *y, const float *a, const float *b, int slot0, int count, cudaStream_t st)
{
    const int pp = P.np > P.mp ? P.np : P.mp;
    prep_near_kernel<<<dim3((pp + 127) / 128, count, 2), 128, 0, st>>>(P, x, y, a, b, slot0);
}

// Largest potential of every box, from the potentials (after a warm proposal; the legs keep it up to date).
__global__ void __launch_bounds__(128) near_tops_kernel(const Dev P)
{
    const int slot = blockIdx.y, side = blockIdx.z, i = blockIdx.x * 128 + threadIdx.x, lane = threadIdx.x & 31;
    const int npts = side ? P.m : P.n, nb = side ? P.nby : P.nbx;
    if (i >= (side ? P.mp : P.np)) return;
    float top = -3.0e38f;
    if (i < npts) top = __double2float_ru((side ? P.gam + (size_t)slot * P.mp : P.phi[0] + (size_t)slot * P.np)[i]);
    for (int off = 16; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
    if (P.lists && !side) {
        const size_t o = (size_t)slot * P.np + i;
        row_record(P, P.home[slot], i, i < npts, P.phi[0][o], P.la2[o], P.sqx[o], (float)P.wa[o]);
    }
    if (P.lists && side && i < npts) home_potential(P, P.home[slot], i, P.gam[(size_t)slot * P.mp + i]);
    if (lane) return;
    if (side) P.topy[(size_t)slot * nb + (i >> 5)] = top;
    else { top_x(P, 0, slot, i >> 5, top); top_x(P, 1, slot, i >> 5, top); }
}
void launch_near_tops(const Dev &P, cudaStream_t st)
{
    const int mx = P.np > P.mp ? P.np : P.mp;
    near_tops_kernel<<<dim3((mx + 127) / 128, P.W, 2), 128, 0, st>>>(P);
}

// ---------------------------------------------------------------- the legs
// What a block keeps of its rows while it walks the columns.
template <int DP, int RB>
struct NearRows {
    float crd[DP][RB];                                   // relative to the centre of the row's box
    float ref[RB];                                       // reference point: log-sum-exp if the potential did not move
    float lo[DP][RB / BOX_COLS], hi[DP][RB / BOX_COLS], top[RB / BOX_COLS];     // per group: its box, largest phi - log2 w
};

// One group's 32 rows (four per thread, eight threads across, a box's columns dealt to the four quarters of the
// warp) against every fourth box, from box `first` on; `all` takes every one of those.  A box's columns come by
// cp.async through a ring of the warp's own, three boxes ahead, so no warp waits for another.
template <int DP, int RB>
__device__ __forceinline__ void stream_near(const float *colc, const float *colt, const int cp, const int nbox, const float *box, const float *top,
                                            const bool halves, const int nb, const NearRows<DP, RB> &rows, const int g, const float cut, const bool all,
                                            const int first, const int lane, float *ring, unsigned char *list, float (&mx)[4], double (&sd)[4])
{
    constexpr int R = 4, NP = 4;                         // rows and column pairs per thread and box
    constexpr int BOX = (DP + 1) * BOX_COLS;             // floats of a box in the ring: coordinate rows, then the terms
    const int cs = lane >> 3, r0 = BOX_COLS * g + 4 * (lane & 7);
    u64 xd[R][DP];
    float ts[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int k = 0; k < DP; ++k) { const float x = rows.crd[k][r0 + r]; xd[r][k] = pack2(x, x); }
        mx[r] = all ? NEG_BIG : rows.ref[r0 + r];
        ts[r] = 0.f; sd[r] = 0.0;
    }
    const float ptop = rows.top[g];
    // this thread's 16-byte piece of a box: row kk, columns qq ..; boxes of more than 32 pieces take a second one
    const int kk = lane >> 3, qq = (lane & 7) * 4;
    const float *src0 = (kk < DP ? colc + kk * cp : colt) + qq, *src1 = colt + qq;
    const bool has0 = kk <= DP, has1 = DP == 4 && lane < 8;
#pragma unroll 1
    for (int s0 = first; s0 < nbox; s0 += 128) {
        // 32 boxes, one per thread: whether the group needs it, and the offset D of the two centres with |D|^2 / 2
        float dl[DP], d2 = 0.f, h2 = 0.f;
        const int J = s0 + 4 * lane < nbox ? s0 + 4 * lane : nbox - 1;
#pragma unroll
        for (int k = 0; k < DP; ++k) {
            const float lo = box[k * nb + J], hi = box[(DP + k) * nb + J];
            const float gap = fmaxf(fmaxf(lo - rows.hi[k][g], rows.lo[k][g] - hi), 0.f);
            d2 = fmaf(gap, gap, d2);
            dl[k] = 0.5f * (rows.lo[k][g] + rows.hi[k][g]) - 0.5f * (lo + hi);
            h2 = fmaf(0.5f * dl[k], dl[k], h2);
        }
        float t = top[halves ? 2 * J : J];
        if (halves) t = fmaxf(t, top[2 * J + 1]);
        const bool need = s0 + 4 * lane < nbox && (all || !(t + ptop - 0.5f * d2 < cut));      // NaN: keep
        const unsigned word = __ballot_sync(0xffffffffu, need);
        const int cnt = __popc(word);
        __syncwarp();                                    // everyone has read what list and ring held before
        if (need) list[__popc(word & ((1u << lane) - 1u))] = (unsigned char)lane;
        __syncwarp();
        auto issue = [&](const int at) {
            if (at < cnt) {
                const int j = (s0 + 4 * list[at]) * BOX_COLS;
                float *dst = ring + (at & 3) * BOX + qq;
                if (has0) cp_async16(dst + kk * BOX_COLS, src0 + j);
                if (has1) cp_async16(dst + DP * BOX_COLS, src1 + j);
            }
            cp_async_commit();
        };
        issue(0); issue(1); issue(2);
#pragma unroll 1
        for (int at = 0; at < cnt; ++at) {
            cp_async_wait<2>();
            __syncwarp();                                // the box is there for every thread, and the one before it is read
            issue(at + 3);
            const int e = list[at];
            const float *bx = ring + (at & 3) * BOX + cs * 8;
            u64 y[DP][NP], E[NP];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int k = 0; k < DP; ++k) {
                    const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(bx + k * BOX_COLS + 4 * h);
                    y[k][2 * h] = t.x; y[k][2 * h + 1] = t.y;
                }
                const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(bx + DP * BOX_COLS + 4 * h);
                E[2 * h] = t.x; E[2 * h + 1] = t.y;
            }
            const float hh = __shfl_sync(0xffffffffu, h2, e);
            float D[DP];
#pragma unroll
            for (int k = 0; k < DP; ++k) {
                D[k] = __shfl_sync(0xffffffffu, dl[k], e);
                const u64 dd = pack2(D[k], D[k]);
#pragma unroll
                for (int p = 0; p < NP; ++p) E[p] = fma2(dd, y[k][p], E[p]);
            }
            // shifted arguments of row r; its reference is mx[r]
            float sh[R], es[R];
            auto args = [&](const int r, u64 (&acc)[NP]) {
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    acc[p] = E[p];
#pragma unroll
                    for (int k = 0; k < DP; ++k) acc[p] = fma2(xd[r][k], y[k][p], acc[p]);
                }
            };
            float worst = 0.f;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                sh[r] = hh;
#pragma unroll
                for (int k = 0; k < DP; ++k) { float x, x_; unpack2(xd[r][k], x, x_); sh[r] = fmaf(D[k], x, sh[r]); }
                const float ref = sh[r] + mx[r];
                const u64 mm = pack2(ref, ref);
                u64 acc[NP];
                float v[2 * NP];
                args(r, acc);
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    float lo, hi;
                    unpack2(sub2(acc[p], mm), lo, hi);
                    v[2 * p] = ex2_fast(lo); v[2 * p + 1] = ex2_fast(hi);
                }
                es[r] = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
                worst += es[r];                          // (infinite or NaN if one is)
            }
            if (!(worst <= 1024.f)) {                    // rare: a reference has to move; the row's own sum decides, never a sibling row's
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (!(es[r] <= 1024.f)) {
                        u64 acc[NP];
                        float v[2 * NP];
                        args(r, acc);
#pragma unroll
                        for (int p = 0; p < NP; ++p) unpack2(acc[p], v[2 * p], v[2 * p + 1]);
                        float mt = v[0];
#pragma unroll
                        for (int p = 1; p < 2 * NP; ++p) mt = fmaxf(mt, v[p]);
                        const float mn = ceilf(mt - sh[r]), fac = pow2i(mx[r] - mn);
                        ts[r] *= fac;
                        sd[r] *= (double)fac;
                        mx[r] = mn;
                        es[r] = 0.f;
#pragma unroll
                        for (int p = 0; p < 2 * NP; ++p) es[r] += ex2_fast(v[p] - (sh[r] + mn));
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) ts[r] += es[r];
            if ((at & 15) == 15 || at + 1 == cnt) {      // at most 128 terms a thread in an fp32 sum
#pragma unroll
                for (int r = 0; r < R; ++r) { sd[r] += (double)ts[r]; ts[r] = 0.f; }
            }
        }
    }
}

// ---------------------------------------------------------------- one pass per cycle
// f-leg and the column sums of the g-leg in one pass over the pairs.  A block takes GROUP_ROWS source points (a group) and the target
// points that matter to it, forms the entries
//     e_ij = 2^(gam_j - |r_i - c_j|^2 / 2 + |r'_i|^2 / 2 - ref_i) = 2^((E_j - ref) + r'_i . c_j + (ref - ref_i)),
//     E_j - ref = ((gam_j - ref) - |c_j|^2 / 2),      c_j relative to the centre of the group's box of 32
// once, adds up its rows, S_i = sum_j e_ij, and - since the plan after the f-leg is a_i e_ij / S_i - its part of the column sums
//     T_j = sum_i (a_i / S_i) e_ij
// from the entries, which it has kept in tensor memory.  Parts are added to the lane's totals as integers (units of
// 2^-44 next to b_j), so the total depends neither on the order of the blocks nor on the launch shape; the g-leg's
// launch turns them into potentials (columns_from_sums).
//
// Which target points: those for which, with the distance d from the point to the group's box, either gam_j + prow - d^2 / 2 (prow
// the largest phi - log2 a of the group) or gam_j - log2 b_j + pcol - d^2 / 2 (pcol the largest phi) reaches the cut of
// update_near_kernel.  They are listed with a margin of CY_MARGIN bits and the list is kept for later cycles: it holds while
// what the target's potentials have risen by since their base (`risen`, by lane, from the g-legs) and what
// prow and pcol have risen by since the list was written are within the margin together.  When the target's have used up half of
// it, all groups list anew from the potentials of that cycle, which become the base.  (Registration: 16 of 300 cycles,
// most of them among the first 50.)  All of it follows from the lane's own values, cycle by cycle.
// Rows whose sum comes out below 2^-6 of the estimate, or above 2^60, start over with the largest argument over all columns as
// their reference.  Columns whose total comes out below 2^-6 of b_j (or beyond its range) are left to the g-leg's own pass.
// What is left out is below 2^-32 of a row's estimated sum, so below 2^-26 of any row sum that is taken.  A column's part is
// bounded with pcol, from before the f-leg, which may raise phi by up to six bits: where it raises group g's beyond what
// its lists have room for, by r_g bits, up to 2^-32 of b_j times the mean of 2^r_g over the groups is missing, and columns are left to
// their own pass below 2^-6 of b_j times that mean already (`overrun`), so that less than 2^-26 of any total that is taken is missing, too.
// (With the largest r_g in place of the mean, which outliers set: registration 76.4 -> 77.1 ms.)
//
// Arguments.  E_j is formed as ((gam_j - ref) - |c_j|^2 / 2), the potential as the sum of two fp32 numbers, c_j relative to the centre of
// the group's box of 32 and ref one row's reference, so what is rounded is small where an entry matters.  Against 64 bits, 16
// registration lanes of 2048 points, legs by themselves -> one pass: potentials 5.1e-7 -> 5.5e-8, residual 1.0e-5 -> 7.2e-6.
//
// Work layout.  Persistent blocks of four warps, four to an SM (128 of the 512 columns of tensor memory each); a warp lists, keeps
// and walks its own boxes, so there is one block barrier a group, for the row sums; the next group's record and the
// heads of its lists are on their way meanwhile.  A thread has four rows and four of a step's 32 points.
// What bounds it: instruction issue (half of the slots; 190 instructions a step of 16 pairs a thread, 86 of them multiply-adds, sums and
// exponentials, and 640 a warp and group) at the 16 warps an SM that tensor memory allows; the special-function unit is a quarter busy.
// Registration workload, f-leg and g-leg -> one pass and g-leg: 32 lanes of 8192 points 212 + 233 -> 200 + 9 us, solve 139 -> 76 ms;
// one lane of 4096 points 14 + 24 -> 7 + 4 us, solve 12.8 -> 6.4 ms.  Steps on the way, 32 lanes: boxes of 8 points tested in every
// cycle 423 us; lists of single points kept over cycles 247 us; persistent blocks, records ahead 234 us; a step's points
// from one record each, no selects 210 us; 32-bit offsets 200 us.  The loop over steps unrolled by eight: slower (instruction fetch).
constexpr int CY_STEPS = 8;                              // steps of 32 target points whose entries a warp keeps in tensor memory
constexpr int CY_TM = 16 * CY_STEPS;                     // ... columns of it: four blocks an SM
constexpr float CY_MARGIN = 2.f;
constexpr float CY_LOW = 0x1p-6f, CY_HIGH = 0x1p60f;

// How far the potentials of 32 target points (a warp's) have risen since their base, or their new base.  Those of a frozen lane, too, whose
// potentials stay: a lane that froze in the cycle of a new base would go without and make its lists in every cycle from then on.
__device__ __forceinline__ void note_rise(const Dev &P, const Ctl &c, const int slot, const int j, const double before, const double now)
{
    if (P.dry_run) return;
    const int home = P.home[slot], at = P.based_at[home];
    const bool has = j < P.m;
    float base = -3.0e38f, rise = 0.f;
    if (at == c.cycle) {                                 // every group has made its list from the potentials before this leg
        float top = base = has ? __double2float_ru(before) : -3.0e38f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
        if (j < P.mp) P.base_gam[(size_t)home * P.mp + j] = base;
        if (j < P.mp && (j & 31) == 0) P.base_top[(size_t)home * P.nby + (j >> 5)] = top;
    } else if (has) base = P.base_gam[(size_t)home * P.mp + j];
    if (has) {
        rise = fmaxf(__fsub_ru(__double2float_ru(now), base), 0.f);
        if (!(rise <= 1.0e30f) || !isfinite(now)) rise = 1.0e30f;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) rise = fmaxf(rise, __shfl_xor_sync(0xffffffffu, rise, off));
    if ((threadIdx.x & 31) == 0) atomicMax(P.risen + home, ((unsigned long long)(unsigned)at << 32) | __float_as_uint(rise));
}

// 2^r of a group whose phi has risen by r bits more than its lists have room for, added up by lane as integers (any order), double-buffered
// like the column totals (the column check's launch zeroes the next cycle's: beside the totals that store cost 5 of 245 us a cycle, in the
// g-leg 1 of 9, in the planner 0.1 us of every batch's cycle); OVERRUN_ALL: those cannot be used.
constexpr float OVERRUN_UNIT = 64.f;
constexpr unsigned OVERRUN_ALL = 1u << 31;               // (2^14 groups, the most that 262 143 points make, of 2^14 + 1 units stay below)

// base + off bytes: a base that is the same for the whole launch and a 32-bit offset (the layout keeps these arrays below 4 GiB)
template <typename T>
__device__ __forceinline__ T *at_bytes(T *base, const unsigned off)
{
    return reinterpret_cast<T *>(const_cast<char *>(reinterpret_cast<const char *>(base)) + off);
}

template <int DP>
__global__ void __launch_bounds__(UPD_THREADS, NEAR_BLOCKS) near_rows_kernel(const Dev P)
{
    constexpr int NW = GROUP_WARPS, GR = GROUP_ROWS, HEAD = CY_STEPS * 32;
    __shared__ GroupRecord rec[2];
    __shared__ __align__(16) unsigned short ids[2][NW][HEAD + 64];        // heads of the lists (and room to look two steps ahead)
    __shared__ float scales[NW][HEAD + 32];              // ... and the points' units
    __shared__ __align__(16) float stage[NW][2][(DP + 1) * 32];
    __shared__ unsigned char boxl[NW][32];
    __shared__ double part[2][NW][GR];
    __shared__ float partm[NW][GR];
    __shared__ __align__(16) float wsm[NW][GR];
    __shared__ float redo_ref[GR];
    __shared__ float allowed[2];                         // the largest phi that the group's lists have room for
    __shared__ uint32_t tm_holder;

    // (programmatic dependent launch as in update_kernel)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Ctl c = *P.ctl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int groups = (P.n + GR - 1) / GR, items = c.n_phys * groups;
    if (c.done || c.static_final || (int)blockIdx.x >= items) {
        if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    if (warp == 0) tc_alloc<CY_TM>(&tm_holder);
    tc_fence_before();

    for (int e = tid; e < 2 * NW * 64; e += UPD_THREADS) ids[e / (NW * 64)][e / 64 % NW][HEAD + e % 64] = 0;

    // items are groups of all lanes in turn; the record of an item and the heads of its lists come by cp.async, an item ahead
    auto fetch = [&](const int home, const int group, const int b) {
        const size_t hg = (size_t)home * groups + group;
        if (8 * lane < P.list_cap) cp_async16(ids[b][warp] + 8 * lane, P.lists + (hg * NW + warp) * P.list_cap + 8 * lane);
        if (warp == 0) cp_async16(reinterpret_cast<char *>(&rec[b]) + 16 * lane, reinterpret_cast<const char *>(&group_record(P, home, group)) + 16 * lane);
        cp_async_commit();
    };
    int item = blockIdx.x;
    const int step = gridDim.x, sstep = step / groups, gstep = step - sstep * groups;
    auto advance = [&](int &slot, int &group) {
        slot += sstep; group += gstep;
        if (group >= groups) { group -= groups; ++slot; }
    };
    int slot = item / groups, group = item - slot * groups, slot1 = slot, group1 = group;
    advance(slot1, group1);
    int home = P.home[slot];
    fetch(home, group, 0);
    int home1 = item + step < items ? P.home[slot1] : 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    unsigned long long risen = P.risen[home];
    cp_async_wait<0>();
    __syncthreads();
    tc_fence_after();
    const uint32_t tk = tm_holder + ((uint32_t)(warp * 32) << 16);
    const int rq = lane & 3, cg = lane >> 2;             // thread (cg, rq): rows 4 rq .. 4 rq + 3 against four of a step's 32 points
    const int rr = lane & (GR - 1);
    const int own = 4 * cg + 2 * (lane & 1) + ((lane >> 1) & 1);               // the step's point whose sum this thread ends up with
    const bool u1 = lane & 1, u2 = lane & 2, u8 = lane & 8, u16 = lane & 16;
    const int nbox = (P.m + BOX_COLS - 1) / BOX_COLS;
    unsigned long long *const acc = P.colacc[c.parity];
    const float limit = 0x1p62f / (float)groups;         // totals stay below 2^62

    int turn = 0;
#pragma unroll 1
    for (int b = 0; item < items; item += step, b ^= 1) {
        const int homen = home1, slotn = slot1, groupn = group1;
        unsigned long long risenn = 0ull;
        // (whoever reads the buffers of the item after this one has passed the barrier of the item before it)
        if (item + step < items) { fetch(homen, groupn, b ^ 1); risenn = P.risen[homen]; }
        advance(slot1, group1);
        if (item + 2 * step < items) home1 = P.home[slot1];
        const GroupRecord &R = rec[b];
        if (P.early_exit && P.state[slot] != 0) {        // (the whole block)
            cp_async_wait<0>();
            __syncthreads();
            home = homen; risen = risenn; slot = slotn; group = groupn;
            continue;
        }
        const int based = (int)(risen >> 32);
        const float rise = __uint_as_float((unsigned)risen);
        const bool rebase = based == 0 || !(rise <= 0.5f * CY_MARGIN);
        float prow = R.prow, pcol = R.pcol, ref = -R.row[rr].x;
        const float wt = R.row[rr].y;
        bool stale = rebase || R.made_from != based || !(prow - R.made_prow <= CY_MARGIN - rise && pcol - R.made_pcol <= CY_MARGIN - rise);
        int len = stale ? 0 : R.len[warp];
        if (tid == 0 && !stale) allowed[b] = R.made_pcol + (CY_MARGIN - rise);
        float gcen[DP], gref = R.row[0].x > NEG_BIG ? -R.row[0].x : 0.f;          // a reference for the whole group
        u64 xn[4][DP], nref[4];
#pragma unroll
        for (int k = 0; k < DP; ++k) {
            gcen[k] = R.centre[k];
            const float4 t = *reinterpret_cast<const float4 *>(&R.crd[k][4 * rq]);
            xn[0][k] = pack2(t.x, t.x); xn[1][k] = pack2(t.y, t.y); xn[2][k] = pack2(t.z, t.z); xn[3][k] = pack2(t.w, t.w);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) { const float f = R.row[4 * rq + r].x + gref; nref[r] = pack2(f, f); }
        unsigned short *list = P.lists + (((size_t)home * groups + group) * NW + warp) * P.list_cap, *id0 = ids[b][warp];
        const unsigned hy = (unsigned)home * (unsigned)(P.mp + 1), hc = (unsigned)home * (unsigned)(P.nby + 1), ha = (unsigned)home * (unsigned)P.mp;
        if (!P.dry_run) {
            // the totals of the next cycle start at zero
            unsigned long long *next = P.colacc[c.parity ^ 1] + (size_t)home * P.mp;
            for (int j = group * UPD_THREADS + tid; j < P.mp; j += groups * UPD_THREADS) next[j] = 0ull;
            if (rebase && group == 0 && tid == 0) P.based_at[home] = c.cycle + 1;
        }

        // lists of the group: warp w takes the boxes w, w + NW, ...
        auto make_list = [&]() {
            const float cutr = -(NEAR_BITS + NEAR_SLACK + CY_MARGIN + (float)(32 - __clz(P.m))), cutc = -(NEAR_BITS + NEAR_SLACK + CY_MARGIN + (float)(32 - __clz(P.n)));
            const float *box32 = P.boxy + (size_t)slot * 2 * DP * P.nby, *lb32 = P.lby + (size_t)home * P.nby;
            const float *top32 = rebase ? P.topy + (size_t)slot * P.nby : P.base_top + (size_t)home * P.nby;
            const float *b16 = P.boxx16 + (size_t)home * 2 * DP * 2 * P.nbx;
            float glo[DP], ghi[DP];
#pragma unroll
            for (int k = 0; k < DP; ++k) { glo[k] = b16[k * 2 * P.nbx + group]; ghi[k] = b16[(DP + k) * 2 * P.nbx + group]; }
            int cnt = 0;
#pragma unroll 1
            for (int s0 = 0; NW * s0 + warp < nbox; s0 += 32) {
                const int J = NW * (s0 + lane) + warp, Jc = min(J, nbox - 1);
                float d2 = 0.f;
#pragma unroll
                for (int k = 0; k < DP; ++k) {
                    const float t = fmaxf(fmaxf(box32[k * P.nby + Jc] - ghi[k], glo[k] - box32[(DP + k) * P.nby + Jc]), 0.f);
                    d2 = fmaf(t, t, d2);
                }
                d2 *= 0.5f;
                const float top = top32[Jc];
                const bool need = J < nbox && (!(top + prow - d2 < cutr) || !(top - lb32[Jc] + pcol - d2 < cutc));       // NaN: keep
                const unsigned word = __ballot_sync(0xffffffffu, need);
                const int nb = __popc(word);
                __syncwarp();
                if (need) boxl[warp][__popc(word & ((1u << lane) - 1u))] = (unsigned char)lane;
                __syncwarp();
#pragma unroll 2
                for (int q = 0; q < nb; ++q) {
                    const int B = NW * (s0 + boxl[warp][q]) + warp, j = BOX_COLS * B + lane;
                    const float4 cr = reinterpret_cast<const float4 *>(P.crdy)[hy + j], ce = reinterpret_cast<const float4 *>(P.ceny)[hc + B];
                    const float cv[4] = {cr.x + ce.x, cr.y + ce.y, cr.z + ce.z, cr.w + ce.w};
                    float e2 = 0.f;
#pragma unroll
                    for (int k = 0; k < DP; ++k) {
                        const float t = fmaxf(fmaxf(cv[k] - ghi[k], glo[k] - cv[k]), 0.f);
                        e2 = fmaf(t, t, e2);
                    }
                    e2 *= 0.5f;
                    const size_t o = (size_t)slot * P.mp + j;
                    const float g = rebase ? __double2float_ru(P.gam[o]) : P.base_gam[(size_t)home * P.mp + j], lb = (float)P.lb2[o];
                    const bool keep = j < P.m && (!(g + prow - e2 < cutr) || !(g - lb + pcol - e2 < cutc));
                    const unsigned w = __ballot_sync(0xffffffffu, keep);
                    const int at = cnt + __popc(w & ((1u << lane) - 1u));
                    if (keep) { list[at] = (unsigned short)j; if (at < HEAD) id0[at] = (unsigned short)j; }
                    cnt += __popc(w);
                }
            }
            // (up to whole steps, and two steps more: the point of weight zero)
            len = (cnt + 31) / 32 * 32;
            for (int at = cnt + lane; at < len + 64; at += 32) { list[at] = (unsigned short)P.mp; if (at < HEAD + 64) id0[at] = (unsigned short)P.mp; }
            GroupRecord &g = group_record(P, home, group);
            if (lane == 0) g.len[warp] = len;
            if (tid == 0) {
                g.made_prow = prow; g.made_pcol = pcol; g.made_from = rebase ? c.cycle + 1 : based;
                allowed[b] = pcol + (rebase ? CY_MARGIN : CY_MARGIN - rise);
            }
            __syncwarp();
        };
        // A step is 32 listed points.  They are shifted to the group's centre once, by the lane they fall to, and go through shared
        // memory: negated coordinates and E_j less the group's reference.
        float4 cr, ce;
        float2 ul;
        float g;
        auto load = [&](const unsigned id) {
            cr = *reinterpret_cast<const float4 *>(at_bytes(P.crdy, 16u * (hy + id)));
            ce = *reinterpret_cast<const float4 *>(at_bytes(P.ceny, 16u * (hc + id / BOX_COLS)));
            g = DP < 4 ? cr.w : *at_bytes(P.gamy, 4u * (hy + id));
            ul = *at_bytes(P.unit_low, 8u * (hy + id));
        };
        auto put = [&](float *dst) {
            const float cv[4] = {cr.x, cr.y, cr.z, cr.w}, cc[4] = {ce.x, ce.y, ce.z, ce.w};
            float h = 0.f;
#pragma unroll
            for (int k = 0; k < DP; ++k) {
                const float nc = (gcen[k] - cc[k]) - cv[k];
                h = fmaf(nc, nc, h);
                dst[32 * k] = nc;
            }
            dst[32 * DP] = fmaf(-0.5f, h, (g - gref) + ul.y);
        };
        // arguments less the references, a[r][p]: row 4 rq + r, points 4 cg + 2 p and the next
        auto arguments = [&](const float *st, u64 (&a)[4][2]) {
            u64 nc[DP][2], E[2];
#pragma unroll
            for (int k = 0; k < DP; ++k) { const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(st + 32 * k); nc[k][0] = t.x; nc[k][1] = t.y; }
            { const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(st + 32 * DP); E[0] = t.x; E[1] = t.y; }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    a[r][p] = add2(E[p], nref[r]);
#pragma unroll
                    for (int k = 0; k < DP; ++k) a[r][p] = fma2(xn[r][k], nc[k][p], a[r][p]);
                }
        };
        // 2^a, as words.  (Words are added up and multiplied one by one from here on: the pairs of packed instructions and the 16
        // consecutive registers of an access to tensor memory would cost a copy each.)
        auto entries = [&](const u64 (&a)[4][2], uint32_t (&w)[16]) {
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    float lo, hi;
                    unpack2(a[r][p], lo, hi);
                    w[4 * r + 2 * p] = __float_as_uint(ex2_fast(lo)); w[4 * r + 2 * p + 1] = __float_as_uint(ex2_fast(hi));
                }
        };
        float *const st_put = stage[warp][0] + lane;
        const float *const st_get = stage[warp][0] + 4 * cg;
        constexpr int ST = (DP + 1) * 32;
        // steps first .. last - 1 of points that which(l) names, whatever their number (and two steps past them)
        auto stream = [&](const int first, const int last, auto &&which, auto &&use) {
            load(which(first));
            unsigned next = which(first + 1);
            __syncwarp();
            put(st_put + (first & 1) * ST);
            __syncwarp();
#pragma unroll 1
            for (int l = first; l < last; ++l) {
                load(next);
                next = which(l + 2);
                u64 a[4][2];
                arguments(st_get + (l & 1) * ST, a);
                use(l, a);
                put(st_put + ((l + 1) & 1) * ST);
                __syncwarp();
            }
        };
        auto tail = [&](const int l) -> unsigned { return list[32 * l + lane]; };

        // ---- rows
        double S = 0.0;                                  // of row lane & 15, in every warp
        bool bad = false;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            if (stale) make_list();
            double sd[4];
            float ts[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) { sd[r] = 0.0; ts[r] = 0.f; }
            const int steps = len / 32;
            auto add_rows = [&](const uint32_t (&w)[16]) {
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    ts[r] += (__uint_as_float(w[4 * r]) + __uint_as_float(w[4 * r + 1])) + (__uint_as_float(w[4 * r + 2]) + __uint_as_float(w[4 * r + 3]));
            };
            auto flush = [&]() {                         // (at most 64 terms in an fp32 sum)
#pragma unroll
                for (int r = 0; r < 4; ++r) { sd[r] += (double)ts[r]; ts[r] = 0.f; }
            };
            // the steps whose entries are kept
            {
                const int held = min(steps, CY_STEPS);
                load(id0[lane]);
                unsigned next = id0[32 + lane];
                __syncwarp();
                put(st_put); scales[warp][lane] = ul.x;
                __syncwarp();
                // (two steps to a turn, so that their buffers are known: addresses cost no instructions)
                const unsigned short *ip = id0 + lane;
                float *sp = scales[warp] + lane;
                uint32_t t = tk;
                auto step_of = [&](auto odd) {
                    constexpr int B = decltype(odd)::value;
                    load(next);
                    next = ip[32 * (B + 2)];
                    u64 a[4][2];
                    uint32_t w[16];
                    arguments(st_get + B * ST, a);
                    entries(a, w);
                    tc_st16_issue(t + 16 * B, w);
                    add_rows(w);
                    put(st_put + (B ^ 1) * ST); sp[32 * (B + 1)] = ul.x;
                    __syncwarp();
                };
#pragma unroll 1
                for (int l = 0; l < held; l += 2, ip += 64, sp += 64, t += 32) {
                    step_of(std::integral_constant<int, 0>());
                    if (l + 1 < held) step_of(std::integral_constant<int, 1>());
                }
            }
            flush();
            if (steps > CY_STEPS) {
                stream(CY_STEPS, steps, tail, [&](const int l, const u64 (&a)[4][2]) {
                    uint32_t w[16];
                    entries(a, w);
                    add_rows(w);
                    if ((l & 15) == 15) flush();
                });
                flush();
            }
            // over the eight threads that hold the same rows: thread (cg, rq) ends up with row 4 rq + 2 (cg bit 2) + (cg bit 1)
            {
                double k0 = u16 ? sd[2] : sd[0], k1 = u16 ? sd[3] : sd[1];
                k0 += __shfl_xor_sync(0xffffffffu, u16 ? sd[0] : sd[2], 16);
                k1 += __shfl_xor_sync(0xffffffffu, u16 ? sd[1] : sd[3], 16);
                double t = u8 ? k1 : k0;
                t += __shfl_xor_sync(0xffffffffu, u8 ? k0 : k1, 8);
                t += __shfl_xor_sync(0xffffffffu, t, 4);
                if (!(lane & 4)) part[b][warp][4 * rq + (u16 ? 2 : 0) + (u8 ? 1 : 0)] = t;
            }
            cp_async_wait<0>();                          // (the next item's record: visible to all after the barrier)
            __syncthreads();
            S = (part[b][0][rr] + part[b][1][rr]) + (part[b][2][rr] + part[b][3][rr]);
            bad = wt > 0.f && !(S >= (double)CY_LOW && S <= (double)CY_HIGH);
            if (pass || !__any_sync(0xffffffffu, bad)) break;                 // (the same in every warp)
            // the estimate was wrong: those rows' largest argument over all columns takes its place
            tc_st_wait();
            float mx[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) { mx[q] = NEG_BIG; nref[q] = 0ull; }
            gref = 0.f;
            stream(0, (nbox - warp + NW - 1) / NW,
                   [&](const int l) -> unsigned { const int j = BOX_COLS * (NW * l + warp) + lane; return (unsigned)min(j, P.mp); },
                   [&](const int, const u64 (&a)[4][2]) {
#pragma unroll
                       for (int q = 0; q < 4; ++q)
#pragma unroll
                           for (int p = 0; p < 2; ++p) {
                               float lo, hi;
                               unpack2(a[q][p], lo, hi);
                               mx[q] = fmaxf(mx[q], fmaxf(lo, hi));
                           }
                   });
#pragma unroll
            for (int q = 0; q < 4; ++q) {
#pragma unroll
                for (int off = 4; off < 32; off <<= 1) mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], off));
                if (cg == 0) partm[warp][4 * rq + q] = mx[q];
            }
            __syncthreads();                             // (part is read, too)
            const float m = fmaxf(fmaxf(partm[0][rr], partm[1][rr]), fmaxf(partm[2][rr], partm[3][rr]));
            if (bad) ref = fabsf(m) < 1.0e29f ? ceilf(m) : 1.0e30f;
            {
                const size_t ro = (size_t)slot * P.np + group * GR + (wt > 0.f ? rr : 0);
                const bool has = wt > 0.f && ref < 1.0e30f;
                const double p = P.la2[ro] + P.sqx[ro] - (double)ref;           // (at most a bit below the potential of a row that was fine)
                prow = has ? __double2float_ru(P.sqx[ro] - (double)ref + (bad ? 0.0 : 1.0)) : -3.0e38f;
                pcol = has ? __double2float_ru(p + (bad ? 0.0 : 1.0)) : -3.0e38f;
            }
#pragma unroll
            for (int off = GR / 2; off > 0; off >>= 1) {
                prow = fmaxf(prow, __shfl_xor_sync(0xffffffffu, prow, off));
                pcol = fmaxf(pcol, __shfl_xor_sync(0xffffffffu, pcol, off));
            }
            if (tid < GR) redo_ref[tid] = -ref;
            stale = true;
            __syncthreads();
            gref = redo_ref[0] > -1.0e30f ? -redo_ref[0] : 0.f;
#pragma unroll
            for (int r = 0; r < 4; ++r) { const float f = redo_ref[4 * rq + r] + gref; nref[r] = pack2(f, f); }
        }

        // ---- this block's part of the column sums
        bool useless = __any_sync(0xffffffffu, bad);
        {
            // 1 / S by a Newton step on the approximation
            const float s = (float)S;
            float r;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s));
            r = fmaf(r, fmaf(-s, r, 1.f), r);
            if (lane < GR) wsm[warp][lane] = wt > 0.f && !bad && !P.dry_run ? wt * r : 0.f;
        }
        __syncwarp();
        const float4 wr = *reinterpret_cast<const float4 *>(wsm[warp] + 4 * rq);
        auto add_part = [&](const uint32_t (&w)[16], const unsigned id, const float sc) {
            auto col = [&](const int q) -> float {
                return fmaf(__uint_as_float(w[12 + q]), wr.w, fmaf(__uint_as_float(w[8 + q]), wr.z, fmaf(__uint_as_float(w[4 + q]), wr.y, __uint_as_float(w[q]) * wr.x)));
            };
            const float s0 = col(0), s1 = col(1), s2 = col(2), s3 = col(3);
            // halving exchange over the four threads that have the other rows
            const float k0 = (u1 ? s2 : s0) + __shfl_xor_sync(0xffffffffu, u1 ? s0 : s2, 1), k1 = (u1 ? s3 : s1) + __shfl_xor_sync(0xffffffffu, u1 ? s1 : s3, 1);
            const float v = ((u2 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, u2 ? k0 : k1, 2)) * sc;
            useless = useless || !(v <= limit);          // (NaN, too)
            // What rounds to nothing is not added.  Nor is a NaN, which the point of weight zero has, too, where a lane is not finite: its
            // number is that of the next lane's first total.  (A total that something above the limit has gone into is not used.)
            asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %2, 0f3f000000;\n\t@p red.global.add.u64 [%0], %1;\n\t}"
                         ::"l"(at_bytes(acc, 8u * (ha + id))), "l"(__float2ull_rn(v)), "f"(v) : "memory");
        };
        tc_st_wait();
        {
            const int steps = len / 32;
            const int held = min(steps, CY_STEPS);
            const unsigned short *ip = id0 + own;
            const float *sp = scales[warp] + own;
            uint32_t w0[16], w1[16], t = tk;
            if (held > 0) { tc_ld16_issue(t, w0); tc_ld16_wait(w0); }
#pragma unroll 1
            for (int l = 0; l < held; l += 2, ip += 64, sp += 64) {
                // (past the last step held: not used)
                tc_ld16_issue(t + 16, w1);
                add_part(w0, ip[0], sp[0]);
                tc_ld16_wait(w1);
                if (l + 1 < held) {
                    if (l + 2 < held) { t += 32; tc_ld16_issue(t, w0); }
                    add_part(w1, ip[32], sp[32]);
                    if (l + 2 < held) tc_ld16_wait(w0);
                }
            }
            // what tensor memory had no room for is formed again
            if (steps > CY_STEPS)
                stream(CY_STEPS, steps, tail, [&](const int l, const u64 (&a)[4][2]) {
                    uint32_t x[16];
                    entries(a, x);
                    const unsigned id = list[32 * l + own];
                    add_part(x, id, P.unit_low[hy + id].x);
                });
        }
        useless = __any_sync(0xffffffffu, useless);
        if (useless && lane == 0 && !P.dry_run) atomicOr(P.overrun + (size_t)c.parity * P.W + home, OVERRUN_ALL);

        // ---- the rows' epilogue: one warp's, while the others go on
        if (warp == (turn++ & (NW - 1))) {
            const bool frozen = (P.mode == MODE_MASKED) && P.state[slot] != 0, writes = !frozen && !P.dry_run;
            const bool in = wt > 0.f;
            const float most = allowed[b];
            const int ri = group * GR + rr;
            const size_t ro = (size_t)slot * P.np + (in ? ri : 0);
            const double p0 = P.phi[c.parity][ro], lw = P.la2[ro], sq = P.sqx[ro];
            double pot = 0.0, term = 0.0;
            unsigned long long fixed = 0ull;
            if (in) row_math((int)FORM_DOT, true, lw, sq, (double)wt, p0, ref, S, 0.f, pot, term);
            if (in && lane < GR) {
                fixed = residual_fixed(P, LEG_F, slot, term, frozen);
                if (writes) {
                    float hi, lo;
                    split_potential<float>((int)FORM_DOT, pot, sq, hi, lo);
                    P.phi[c.parity ^ 1][ro] = pot;
                    reinterpret_cast<float *>(P.ft[c.parity ^ 1])[ro] = hi;
                    reinterpret_cast<float *>(P.fl[c.parity ^ 1])[ro] = lo;
                }
            }
#pragma unroll
            for (int off = GR / 2; off > 0; off >>= 1) fixed += __shfl_xor_sync(0xffffffffu, fixed, off);
            if (writes) {
                float top = in ? __double2float_ru(pot) : -3.0e38f;
#pragma unroll
                for (int off = GR / 2; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
                if (lane == 0) P.topx[c.parity ^ 1][(size_t)slot * 2 * P.nbx + group] = top;
                row_record(P, home, ri, in, pot, lw, sq, wt);                   // (both halves of the warp write the same)
                // (the whole warp asks; at most six bits, or the rows have started over)
                if (top > most && lane == 0)
                    atomicAdd(P.overrun + (size_t)c.parity * P.W + home, (unsigned)(OVERRUN_UNIT * ex2_fast(fminf(top - most, 8.f))) + 1u);
            }
            if (lane == 0 && !P.dry_run) finish_lane_residual(P, LEG_F, slot, fixed);
        }
        home = homen; risen = risenn; slot = slotn; group = groupn;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) { tc_fence_after(); tc_dealloc<CY_TM>(tm_holder); }
}

// The g-leg of RB columns from the totals that near_rows_kernel left.  Returns, a bit for each box of 32, where they cannot be used: the
// caller then goes over the pairs of those.  (By box, not by block: what a column is formed from must not depend on how many
// a launch gives to a block.)  One chain of loads and one barrier before what is written: the launch is latencies throughout, 8.8 us for
// 32 lanes of 8192 columns, and a cycle of theirs took 5 us longer with a barrier in front and one behind.
template <int RB>
__device__ __forceinline__ unsigned columns_from_sums(const Dev &P, const Ctl &c, const int slot, const int base)
{
    constexpr int NB = RB / BOX_COLS;
    __shared__ int low_box[NB];
    const int home = P.home[slot];
    const unsigned over = P.overrun[(size_t)(c.parity ^ 1) * P.W + home];
    const int tid = threadIdx.x, j = base + tid;
    const bool has = tid < RB && j < P.m;
    const size_t o = (size_t)slot * P.mp + (has ? j : 0), ho = (size_t)home * (P.mp + 1) + (has ? j : 0);
    unsigned long long t = 0ull;
    double sq = 0.0, lb = 0.0, before = 0.0;
    float sc = 1.f;
    int low = 0;
    if (has) {
        t = P.colacc[c.parity ^ 1][(size_t)home * P.mp + j];
        sq = P.sqy[o]; lb = P.lb2[o]; sc = P.unit_low[ho].x; before = P.gam[o];
        double least = (double)CY_LOW;                   // of b_j
        if (over)
            least = over >= OVERRUN_ALL ? 1.0e300 : least * (double)(1.f + (float)over / (OVERRUN_UNIT * (float)((P.n + GROUP_ROWS - 1) / GROUP_ROWS)));
        low = !((double)t >= least * P.wb[o] * (double)sc) || t < (1ull << 36) || t >= (1ull << 62);
    }
    low = __any_sync(0xffffffffu, low);
    if (tid < RB && (tid & 31) == 0) low_box[tid / BOX_COLS] = low;
    __syncthreads();
    unsigned left = 0u;
#pragma unroll
    for (int e = 0; e < NB; ++e) left |= low_box[e] ? 1u << e : 0u;
    const bool frozen = (P.mode == MODE_MASKED) && P.state[slot] != 0;
    if (tid < RB && !low && !P.dry_run) {                // whole warps
        double pot = frozen ? before : -1.0e300;
        if (has && !frozen) {
            const int e = (int)(__float_as_uint(sc) >> 23) - 127;
            pot = before + lb - (log2((double)t) - (double)e);
            float hi, lo;
            split_potential<float>((int)FORM_DOT, pot, sq, hi, lo);
            P.gam[o] = pot;
            reinterpret_cast<float *>(P.gt)[o] = hi;
            reinterpret_cast<float *>(P.gl)[o] = lo;
            home_potential(P, home, j, pot);
        }
        float top = __double2float_ru(pot);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
        if ((tid & 31) == 0 && has && !frozen) P.topy[(size_t)slot * P.nby + j / BOX_COLS] = top;
        note_rise(P, c, slot, j, before, pot);
    }
    return left;
}

// A block takes NG groups of 32 rows; its four warps share every group's boxes (box J goes to warp J mod 4), so
// that a group with many boxes - outliers share one with points of a region - does not keep one
// warp busy alone.  Partial results are merged in warp order.
template <int DP, int NG>
__global__ void __launch_bounds__(UPD_THREADS, NEAR_BLOCKS) update_near_kernel(const Dev P, const int leg, const int nlanes)
{
    constexpr int R = 4, CS = 4, RB = BOX_COLS * NG, NW = UPD_THREADS / 32;
    static_assert(RB <= UPD_THREADS, "one thread per row in the epilogue");
    __shared__ LegScratch<RB> sc;
    __shared__ NearRows<DP, RB> rows;
    __shared__ double part_s[NW][RB];
    __shared__ float part_m[NW][RB];
    __shared__ int redo[NG];
    __shared__ unsigned char list[NW][32];
    __shared__ __align__(16) float ring[NW][4 * (DP + 1) * BOX_COLS];

    // (programmatic dependent launch as in update_kernel)
    const bool early = (leg == LEG_F);
    if (leg == LEG_G) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Ctl c = *P.ctl;
    if (leg == LEG_V) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int slot = blockIdx.y, row_base = (int)blockIdx.x * RB;
    if (leg == LEG_V && P.lists && row_base == 0 && slot < c.n_phys && slot < nlanes && threadIdx.x == 0)
        P.overrun[(size_t)(c.parity ^ 1) * P.W + P.home[slot]] = 0u;
    if (leg == LEG_V && (int)blockIdx.y >= nlanes) {
        guard_pool(P, c, nlanes, reinterpret_cast<unsigned long long *>(sc.red));
        return;
    }
    const bool rows_x = (leg == LEG_F);
    const int nrows = rows_x ? P.n : P.m, rp = rows_x ? P.np : P.mp;
    const int ncols = rows_x ? P.m : P.n, cp = rows_x ? P.mp : P.np;
    const bool idle = c.done || slot >= c.n_phys || (P.early_exit && P.state[slot] != 0) || (leg != LEG_V && c.static_final) ||
                      (leg == LEG_V && !(c.static_final || lane_needs_column_check(P, c, slot))) || row_base >= nrows;
    if (idle) {
        if (early && blockIdx.x == 0 && blockIdx.y == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const float *colc = reinterpret_cast<const float *>(rows_x ? P.ys : P.xs) + (size_t)slot * DP * cp;
    const float *colt = rows_x ? reinterpret_cast<const float *>(P.gt) + (size_t)slot * cp : reinterpret_cast<const float *>(P.ft[c.parity]) + (size_t)slot * cp;
    const int nbc = rows_x ? P.nby : P.nbx;
    const float *cbox = (rows_x ? P.boxy : P.boxx) + (size_t)slot * 2 * DP * nbc;
    const float *ctop = rows_x ? P.topy + (size_t)slot * nbc : P.topx[c.parity] + (size_t)slot * (P.lists ? 2 : 1) * nbc;
    double before = 0.0;                                 // this thread's potential
    unsigned own = (1u << NG) - 1u;                      // the groups that go over the pairs
    if (leg == LEG_G && P.lists) {
        own = columns_from_sums<RB>(P, c, slot, row_base);
        if (!own) return;
        if (threadIdx.x < RB && row_base + (int)threadIdx.x < nrows) before = P.gam[(size_t)slot * rp + row_base + threadIdx.x];
    }
    const int nbox = (ncols + BOX_COLS - 1) / BOX_COLS;
    const float cut = -(NEAR_BITS + NEAR_SLACK + (float)(32 - __clz(ncols)));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid < RB) {                                      // (whole warps)
        const float *rowc = reinterpret_cast<const float *>(rows_x ? P.xs : P.ys) + (size_t)slot * DP * rp;
        const int nbr = rows_x ? P.nbx : P.nby, i = row_base + tid, grp = i / BOX_COLS;
        const float *rbox = (rows_x ? P.boxx : P.boxy) + (size_t)slot * 2 * DP * nbr;
        const bool in = i < nrows;
        const size_t o = (size_t)slot * rp + (in ? i : 0);
        const double p = (rows_x ? P.phi[c.parity] : P.gam)[o], lw = (rows_x ? P.la2 : P.lb2)[o], sq = (rows_x ? P.sqx : P.sqy)[o];
        if (in && leg != LEG_G) asm volatile("prefetch.global.L1 [%0];" ::"l"((rows_x ? P.wa : P.wb) + o));
#pragma unroll
        for (int k = 0; k < DP; ++k) rows.crd[k][tid] = in ? rowc[(size_t)k * rp + i] : 0.f;
        const double est = lw + sq - p;
        rows.ref[tid] = in && fabs(est) < 1.0e7 ? ceilf((float)est) : (in ? NEG_BIG : 0.f);
        // the largest phi_i - log2 w_i of the group (a row without an estimate needs every column)
        float top = -3.0e38f;
        if (in) top = fabs(p - lw) + sq < 5.0e6 ? __double2float_ru(p - lw) : 3.0e38f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
        if (lane == 0 && in) {
            rows.top[warp] = top;
#pragma unroll
            for (int k = 0; k < DP; ++k) { rows.lo[k][warp] = rbox[k * nbr + grp]; rows.hi[k][warp] = rbox[(DP + k) * nbr + grp]; }
        }
    }
    if (early) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid < NG) redo[tid] = 0;
    __syncthreads();
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
        for (int g = 0; g < NG; ++g) {
            if (row_base + BOX_COLS * g >= nrows) break;
            if (pass == 1 ? !redo[g] : !(own >> g & 1u)) continue;
            float mx[R];
            double sd[R];
            stream_near<DP, RB>(colc, colt, cp, nbox, cbox, ctop, !rows_x && P.lists, nbc, rows, g, cut, pass == 1, warp, lane, ring[warp], list[warp], mx, sd);
            merge_splits<CS, R>(mx, sd);
            if (lane < 8) {
#pragma unroll
                for (int r = 0; r < R; ++r) { part_m[warp][BOX_COLS * g + lane * R + r] = mx[r]; part_s[warp][BOX_COLS * g + lane * R + r] = sd[r]; }
            }
        }
        __syncthreads();
        // the warps' parts, in warp order; rows far below their estimate start over, from "minus infinity" and over
        // all columns (rows that were fine keep the first pass's result, whatever their group needed)
        int low = 0;
        if (tid < RB && (own >> warp & 1u) && (pass == 0 || sc.row_h[tid] != 0.f)) {
            float m = part_m[0][tid];
            double t = part_s[0][tid];
#pragma unroll
            for (int w = 1; w < NW; ++w) {
                const float mo = part_m[w][tid], mn = fmaxf(m, mo);
                t = t * (double)pow2i(m - mn) + part_s[w][tid] * (double)pow2i(mo - mn);
                m = mn;
            }
            sc.row_m[tid] = m;
            sc.row_s[tid] = t;
            low = pass == 0 && row_base + tid < nrows && m <= rows.ref[tid] && !(t >= NEAR_FLOOR);
            sc.row_h[tid] = low ? 1.f : 0.f;
            if (low) redo[tid / BOX_COLS] = 1;
        }
        if (!__syncthreads_or(low)) break;
    }
    // (row_h is the shift of difference-form rows, which these lanes do not have: all zero by now)
    finish_rows<float, RB, UPD_THREADS, true>(P, c, leg, slot, (int)FORM_DOT, sc.row_m, sc.row_s, sc.row_h, sc.red, row_base, own);
    if (leg == LEG_G && P.lists && tid < RB && (own >> warp & 1u)) {
        const int j = row_base + tid;
        if (j < nrows) home_potential(P, P.home[slot], j, P.gam[(size_t)slot * rp + j]);
        note_rise(P, c, slot, j, before, j < nrows ? P.gam[(size_t)slot * rp + j] : 0.0);
    }
}

template <int DP>
static int launch_near_dp(const Dev &P, int leg, int width, cudaStream_t st)
{
    const int nrows = (leg == LEG_F) ? P.n : P.m, lanes = width < 1 ? 1 : width;
    const bool pool_on = leg == LEG_V && P.guard > 0.0;
    if (leg == LEG_F && P.lists) {
        const long long items = (long long)((P.n + GROUP_ROWS - 1) / GROUP_ROWS) * lanes;
        launch_pdl(near_rows_kernel<DP>, dim3((unsigned)(items < 148 * NEAR_BLOCKS ? items : 148 * NEAR_BLOCKS)), dim3(UPD_THREADS), 0, st, P);
        return 0;
    }
    // blocks of 32 rows where blocks of 64 would leave SMs without a full set (same bits)
    if ((long long)((nrows + 63) / 64) * lanes < 148 * NEAR_BLOCKS) {
        const int per = (nrows + 31) / 32, pool = guard_pool_rows(per, pool_on, lanes);
        launch_pdl(update_near_kernel<DP, 1>, dim3(per, lanes + pool), dim3(UPD_THREADS), 0, st, P, leg, lanes);
        return pool > 0;
    }
    const int per = (nrows + 63) / 64, pool = guard_pool_rows(per, pool_on, lanes);
    launch_pdl(update_near_kernel<DP, 2>, dim3(per, lanes + pool), dim3(UPD_THREADS), 0, st, P, leg, lanes);
    return pool > 0;
}

int launch_near(const Dev &P, int leg, int width, cudaStream_t st)
{
    return P.DP == 2 ? launch_near_dp<2>(P, leg, width, st) : (P.DP == 3 ? launch_near_dp<3>(P, leg, width, st) : launch_near_dp<4>(P, leg, width, st));
}

}  // namespace skb
