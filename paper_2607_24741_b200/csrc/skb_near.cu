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
#include "skb_update.cuh"
#include "skb_host.h"

namespace skb {

constexpr int SORT_CHUNK = 8192;                    // points ordered together (by one block, in shared memory)
constexpr int SORT_LEAF = 16;
constexpr float NEAR_BITS = 32.f, NEAR_SLACK = 0.5f;
constexpr double NEAR_FLOOR = 0x1p-6;
// Points of the larger cloud from which the order pays: at 1024 points (16 lanes, eps 0.01) a leg is 13.7 -> 10.3 us and
// a solve of 60 cycles 2.5 -> 2.3 ms, ordering included; the boxes of smaller clouds are too wide to skip much.
constexpr int NEAR_MIN = 1024;
constexpr int NEAR_BLOCKS = 4;                      // blocks per SM (127 registers); five and six spill: 225 and 224 us a leg

bool near_shape(int f64, int DP, int CS, int n, int m)
{
    return !f64 && DP > 0 && DP <= 4 && CS == 4 && (n > m ? n : m) >= NEAR_MIN;
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
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
        }
        if (lane == 0) { box[k * nb + b32] = lo; box[(P.DP + k) * nb + b32] = hi; }
        const float rel = in ? (float)(v - (double)(0.5f * (lo + hi))) : 0.f;
        crd[(size_t)k * pp + i] = rel;
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
    } else {
        for (int e = 0; e < 2; ++e) {
            reinterpret_cast<float *>(P.ft[e])[o] = hi0; reinterpret_cast<float *>(P.fl[e])[o] = 0.f; P.phi[e][o] = 0.0;
            if (lane == 0) P.topx[e][(size_t)slot * nb + b32] = 0.f;
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
    if (lane) return;
    if (side) P.topy[(size_t)slot * nb + (i >> 5)] = top;
    else { P.topx[0][(size_t)slot * nb + (i >> 5)] = top; P.topx[1][(size_t)slot * nb + (i >> 5)] = top; }
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
                                            const int nb, const NearRows<DP, RB> &rows, const int g, const float cut, const bool all,
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
        const bool need = s0 + 4 * lane < nbox && (all || !(top[J] + ptop - 0.5f * d2 < cut));      // NaN: keep
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
    const float *ctop = (rows_x ? P.topy : P.topx[c.parity]) + (size_t)slot * nbc;
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
            if (pass == 1 && !redo[g]) continue;
            float mx[R];
            double sd[R];
            stream_near<DP, RB>(colc, colt, cp, nbox, cbox, ctop, nbc, rows, g, cut, pass == 1, warp, lane, ring[warp], list[warp], mx, sd);
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
        if (tid < RB && (pass == 0 || sc.row_h[tid] != 0.f)) {
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
    finish_rows<float, RB, UPD_THREADS, true>(P, c, leg, slot, (int)FORM_DOT, sc.row_m, sc.row_s, sc.row_h, sc.red, row_base);
}

template <int DP>
static int launch_near_dp(const Dev &P, int leg, int width, cudaStream_t st)
{
    const int nrows = (leg == LEG_F) ? P.n : P.m, lanes = width < 1 ? 1 : width;
    const bool pool_on = leg == LEG_V && P.guard > 0.0;
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
