// Set-up, audit planning, retirement/compaction and read-back kernels.
//
//  prep       inputs -> the kernels' layout (scaled dimension-major coordinates, squared
//             norms, log2 weights, cold potentials f = g = 0); validates values.
//  plan       one CTA per audit: turns the per-lane flags into the retire list by a warp
//             ballot / prefix-sum scan, records depth, status and residuals of retirees
//             (completion depth l_t, Eq. 6), pairs every hole left below the new width
//             with a survivor from above it, and advances the counters of Eq. 7.
//  warm       replaces the cold potentials by a caller's proposal (Section "Initialization and
//             repeated couplings"), before the first cycle.
//  emit_move  writes retirees' potentials to the result buffers in the caller's units and
//             moves every slot-indexed array of a paired survivor into the hole it fills
//             (Section "Screen, verify, and compact").  Holes and sources are disjoint slot
//             sets, so the in-place copies cannot race.
//  gather     potentials in original lane order (retired lanes from the result buffers,
//             running lanes from their slots).
#include "skb_device.cuh"
#include "skb_host.h"
#include "skb_pairs64.cuh"

namespace skb {

// ---------------------------------------------------------------- prep
// One CTA per lane: joint centroid of the two clouds, the largest scaled squared distance
// from it, and from that the cost form the lane will use.
// Lanes come in as a block of problems: input problem q goes to slot slot0 + q as lane lane0 + q
// (create: slot0 = lane0 = 0, all W; a refill: the first free slot, the next unused lane number).

// Per-slot state of a lane that comes in; r2: largest squared distance of a point from the centre.  One thread.
__device__ __forceinline__ void lane_enters(const Dev &P, const float *eps, const int q, const int slot, const int lane0, const int cycle0,
                                            const double r2)
{
    const double e = (double)eps[q];
    const bool eps_ok = (e > 0.0) && isfinite(e);
    const double s = eps_ok ? 1.4426950408889634 / e : 1.0;
    if (!eps_ok) atomicOr(&P.ctl->error, ERR_VALUE);
    P.scale[slot] = s;
    P.lane_id[slot] = lane0 + q;
    P.start[slot] = cycle0;
    // whatever an earlier lane left in the slot
    P.nonfinite[slot] = 0; P.state[slot] = 0; P.flag[slot] = 0; P.verdict[slot] = 0;
    P.rsum_row[slot] = 0ull; P.rsum_col[slot] = 0ull; P.rsum_row64[slot] = 0ull; P.esc[slot] = 0;
    P.ret_at[slot] = 0; P.n_checks[slot] = 0;
    P.absorbed[slot] = eps_ok && 4.0 * s * r2 <= SC_COLD_BITS; P.cyc_log[slot] = 0;
    // (lanes in spatial order have a form of their own, which shares the expanded form's scale and terms)
    int form = P.permx ? FORM_DOT : P.cost_form == 1 ? FORM_DOT : (P.cost_form == 2 ? FORM_DIFF : (s * r2 > P.form_threshold ? FORM_DIFF : FORM_DOT));
    P.form[slot] = form;
    atomicMax(&P.ctl->max_radius_bits, (unsigned long long)__double_as_longlong(eps_ok ? s * r2 : 0.0));
}

// d <= 32.  Eight dimensions at a time: every thread sums its points in all of them, then one warp per dimension
// adds the 256 partial sums up, in the order of a binary tree over the threads.  (One dimension after the other,
// each with a tree of eight barriers, was a chain of some 15 us on the lanes of the sensor workload, d = 15.)
__global__ void __launch_bounds__(256) lane_stats_kernel(const Dev P, const void *xin, const void *yin, const float *eps,
                                                         const int slot0, const int lane0, const int cycle0)
{
    __shared__ double part[8][256];
    __shared__ double cen[32];
    const int q = blockIdx.x, slot = slot0 + q, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tot = P.n + P.m;
    for (int k0 = 0; k0 < P.d; k0 += 8) {
        double s[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = 0.0;
        for (int p = tid; p < tot; p += 256) {
            const bool isx = p < P.n;
            const size_t idx = (isx ? ((size_t)q * P.n + p) : ((size_t)q * P.m + (p - P.n))) * P.d + k0;
#pragma unroll
            for (int k = 0; k < 8; ++k) if (k0 + k < P.d) s[k] += (double)load_raw(P, isx ? xin : yin, idx + k);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) part[k][tid] = s[k];
        __syncthreads();
        // pairs 128, 64, 32 apart, then 16 .. 1
        const double *r = part[warp];
        double v = ((r[lane] + r[lane + 128]) + (r[lane + 64] + r[lane + 192])) + ((r[lane + 32] + r[lane + 160]) + (r[lane + 96] + r[lane + 224]));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0 && k0 + warp < P.d) cen[k0 + warp] = v / (double)tot;
        __syncthreads();
    }
    double mxr = 0.0;
    for (int p = tid; p < tot; p += 256) {
        const bool isx = p < P.n;
        const size_t base = isx ? ((size_t)q * P.n + p) * P.d : ((size_t)q * P.m + (p - P.n)) * P.d;
        double r2 = 0.0;
        for (int k = 0; k < P.d; ++k) { const double v = (double)load_raw(P, isx ? xin : yin, base + k) - cen[k]; r2 += v * v; }
        mxr = fmax(mxr, r2);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mxr = fmax(mxr, __shfl_xor_sync(0xffffffffu, mxr, off));
    if (lane == 0) part[0][warp] = mxr;
    __syncthreads();
    for (int k = tid; k < P.DP; k += 256) P.center[(size_t)slot * P.DP + k] = k < P.d ? cen[k] : 0.0;
    if (tid == 0) {
        for (int w = 1; w < 8; ++w) mxr = fmax(mxr, part[0][w]);
        lane_enters(P, eps, q, slot, lane0, cycle0, mxr);
    }
}

// Deep lanes (32 < d <= 1024): a cluster of blocks per lane, each with a share of the points.  A warp reads 256 dimensions of
// a row at a time (whole sectors) and keeps a sum per dimension; the blocks read each other's sums through shared
// memory, in block order.  Then a warp per point for the distances.  (One block per lane read 134 MB of the feature
// workload - 64 lanes of 1024 x 1024, d = 512 - from 64 SMs: 713 us.)
constexpr int STATS_BLOCKS = 8, STATS_WARPS = 8;
__global__ void __cluster_dims__(STATS_BLOCKS, 1, 1) __launch_bounds__(32 * STATS_WARPS)
lane_stats_deep_kernel(const Dev P, const void *xin, const void *yin, const float *eps, const int slot0, const int lane0, const int cycle0)
{
    __shared__ double part[STATS_WARPS][256];
    __shared__ double sums[1024], cen[1024], far[1];
    const int q = blockIdx.y, slot = slot0 + q, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x;
    const int tot = P.n + P.m, per = (tot + STATS_BLOCKS - 1) / STATS_BLOCKS, p0 = b * per, p1 = min(tot, p0 + per);
    auto row = [&](const int p, const void *&base) -> size_t {
        const bool isx = p < P.n;
        base = isx ? xin : yin;
        return (isx ? (size_t)q * P.n + p : (size_t)q * P.m + (p - P.n)) * P.d;
    };
    for (int k0 = 0; k0 < P.d; k0 += 256) {
        double s[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] = 0.0;
#pragma unroll 2
        for (int p = p0 + warp; p < p1; p += STATS_WARPS) {
            const void *base;
            const size_t o = row(p, base);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = k0 + 32 * e + lane;
                if (k < P.d) s[e] += (double)load_raw(P, base, o + k);
            }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) part[warp][32 * e + lane] = s[e];
        __syncthreads();
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < STATS_WARPS; ++w) t += part[w][tid];
        if (k0 + tid < P.d) sums[k0 + tid] = t;
        __syncthreads();
    }
    cluster_sync_all();
    for (int k = tid; k < P.d; k += 32 * STATS_WARPS) {
        double t = 0.0;
#pragma unroll
        for (int r = 0; r < STATS_BLOCKS; ++r) t += ld_cluster(&sums[k], r);
        cen[k] = t / (double)tot;
    }
    __syncthreads();
    double mxr = 0.0;
#pragma unroll 2
    for (int p = p0 + warp; p < p1; p += STATS_WARPS) {
        const void *base;
        const size_t o = row(p, base);
        double r2 = 0.0;
#pragma unroll 8
        for (int k = lane; k < P.d; k += 32) { const double v = (double)load_raw(P, base, o + k) - cen[k]; r2 = fma(v, v, r2); }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, off);
        mxr = fmax(mxr, r2);
    }
    if (lane == 0) part[0][warp] = mxr;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < STATS_WARPS; ++w) mxr = fmax(mxr, part[0][w]);
        far[0] = mxr;
    }
    if (b == 0) for (int k = tid; k < P.DP; k += 32 * STATS_WARPS) P.center[(size_t)slot * P.DP + k] = k < P.d ? cen[k] : 0.0;
    cluster_sync_all();
    if (b == 0 && tid == 0) {
        for (int r = 1; r < STATS_BLOCKS; ++r) mxr = fmax(mxr, ld_cluster(&far[0], r));
        lane_enters(P, eps, q, slot, lane0, cycle0, mxr);
    }
    cluster_sync_all();                                   // nobody's sums go while another may read them
}

// Zero potentials absorbed, scalings 1 (arrays that share memory with the streamed terms are written after those).
__device__ __forceinline__ void cold_scalings(const Dev &P, const int side, const size_t o)
{
    if (!P.phi0) return;
    if (side) { P.gam0[o] = 0.0; P.vv[o] = 1.0; }
    else { P.phi0[o] = 0.0; P.uu[0][o] = 1.0; P.uu[1][o] = 1.0; }
}

template <typename T>
__global__ void prep_kernel(const Dev P, const void *xin, const void *yin, const float *a, const float *b, const int slot0)
{
    const int q = blockIdx.y, slot = slot0 + q;
    const int side = blockIdx.z;                     // 0: x / a, 1: y / b
    const int npts = side ? P.m : P.n, pp = side ? P.mp : P.np;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= pp) return;
    const double s = P.scale[slot];
    const int form = (sizeof(T) == 8) ? (int)FORM_DOT : P.form[slot];
    T *crd = reinterpret_cast<T *>(side ? P.ys : P.xs) + (size_t)slot * P.DP * pp;
    const size_t o = (size_t)slot * pp + i;
    T *hi0 = side ? reinterpret_cast<T *>(P.gt) : reinterpret_cast<T *>(P.ft[0]);
    T *lo0 = side ? reinterpret_cast<T *>(P.gl) : reinterpret_cast<T *>(P.fl[0]);
    double *sq = side ? P.sqy : P.sqx, *lw = side ? P.lb2 : P.la2, *wt = side ? P.wb : P.wa;
    T hi, lo = T(0);
    if (i >= npts) {                                  // padding points
        for (int k = 0; k < P.DP; ++k) crd[(size_t)k * pp + i] = T(0);
        hi = T(NEG_BIG);
        sq[o] = 0.0; lw[o] = 0.0; wt[o] = 0.0;
    } else {
        const double sc = sqrt(form == FORM_DOT ? 2.0 * s : s);
        const size_t ibase = ((size_t)q * npts + i) * P.d;
        const double *cen = P.center + (size_t)slot * P.DP;
        double nrm = 0.0;
        bool ok = true;
        for (int k = 0; k < P.DP; ++k) {
            T v = T(0);
            if (k < P.d) {
                const float raw = load_raw(P, side ? yin : xin, ibase + k);
                ok = ok && isfinite(raw);
                v = (T)(sc * ((double)raw - cen[k]));
            }
            crd[(size_t)k * pp + i] = v;
            nrm += (double)v * (double)v;
        }
        nrm = form == FORM_DOT ? 0.5 * nrm : 0.0;
        const float w = (side ? b : a)[(size_t)q * npts + i];
        ok = ok && (w > 0.0f) && isfinite(w);
        if (!ok) atomicOr(&P.ctl->error, ERR_VALUE);
        sq[o] = nrm;
        lw[o] = ok ? log2((double)w) : 0.0;
        wt[o] = ok ? (double)w : 0.0;
        if (P.phi0 && ok && w < SC_COLD_WEIGHT) atomicMin(&P.absorbed[slot], w < SC_MIN_WEIGHT ? SC_NO_MATRIX : 0);
        hi = (T)(-nrm);                                // cold start: phi = gam = 0
    }
    hi0[o] = hi; lo0[o] = lo;
    if (!side) {
        reinterpret_cast<T *>(P.ft[1])[o] = hi; reinterpret_cast<T *>(P.fl[1])[o] = lo;
        P.phi[0][o] = 0.0; P.phi[1][o] = 0.0;
    } else {
        P.gam[o] = 0.0;
    }
    cold_scalings(P, side, o);
}

// Layout of tensor-core lanes: their coordinates stay raw (the tiled bf16 copies), so a point leaves only its
// scaled squared norm, weight and cold potentials here.  Eight threads per point, 64 dimensions in 16-byte pieces at a
// time (d is a multiple of 64; with two-byte loads it took 65 us on the feature workload).
__global__ void __launch_bounds__(256) prep_tensor_kernel(const Dev P, const void *xin, const void *yin, const float *a, const float *b, const int slot0)
{
    const int q = blockIdx.y, slot = slot0 + q, side = blockIdx.z, sub = threadIdx.x & 7;
    const int npts = side ? P.m : P.n, pp = side ? P.mp : P.np;
    const int i = blockIdx.x * 32 + (threadIdx.x >> 3);
    const size_t o = (size_t)slot * pp + i;
    float hi = NEG_BIG;                                    // padding points
    double nrm = 0.0, lw = 0.0, wt = 0.0;
    bool ok = true;
    const double sc = sqrt(2.0 * P.scale[slot]);
    if (i < npts) {
        const uint4 *src = reinterpret_cast<const uint4 *>(reinterpret_cast<const unsigned short *>(side ? yin : xin) + ((size_t)q * npts + i) * P.d) + sub;
#pragma unroll 4
        for (int k = 0; k < P.d / 64; ++k) {
            const uint4 t = src[8 * k];
            const unsigned w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float raw = __uint_as_float(e & 1 ? w[e / 2] & 0xffff0000u : w[e / 2] << 16);
                ok = ok && isfinite(raw);
                const double v = sc * (double)raw;
                nrm = fma(v, v, nrm);
            }
        }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, off);
    ok = (__ballot_sync(0xffffffffu, ok) >> (threadIdx.x & 24) & 0xffu) == 0xffu;
    if (i >= pp || sub != 0) return;
    if (i < npts) {
        nrm *= 0.5;
        const float w = (side ? b : a)[(size_t)q * npts + i];
        ok = ok && (w > 0.0f) && isfinite(w);
        if (!ok) atomicOr(&P.ctl->error, ERR_VALUE);
        lw = ok ? log2((double)w) : 0.0;
        wt = ok ? (double)w : 0.0;
        if (P.phi0 && ok && w < SC_COLD_WEIGHT) atomicMin(&P.absorbed[slot], w < SC_MIN_WEIGHT ? SC_NO_MATRIX : 0);
        hi = (float)(-nrm);                                // cold start: phi = gam = 0
    }
    (side ? P.sqy : P.sqx)[o] = nrm; (side ? P.lb2 : P.la2)[o] = lw; (side ? P.wb : P.wa)[o] = wt;
    if (side) {
        reinterpret_cast<float *>(P.gt)[o] = hi; reinterpret_cast<float *>(P.gl)[o] = 0.f; P.gam[o] = 0.0;
    } else {
        for (int e = 0; e < 2; ++e) {
            reinterpret_cast<float *>(P.ft[e])[o] = hi; reinterpret_cast<float *>(P.fl[e])[o] = 0.f; P.phi[e][o] = 0.0;
        }
    }
    cold_scalings(P, side, o);
}

// Warm proposal: potentials in the caller's units -> the kernels' representation of both buffers
// (same formulas as the cold start in prep_kernel, with phi = s f0 and gam = s g0 instead of 0).
// Runs before the first cycle, when slot t still holds lane t.
template <typename T>
__global__ void warm_kernel(const Dev P, const double *f0, const double *g0)
{
    const int slot = blockIdx.y, side = blockIdx.z;
    const int npts = side ? P.m : P.n, pp = side ? P.mp : P.np;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npts) return;
    const double *src = side ? g0 : f0;
    if (!src) return;
    const int *perm = side ? P.permy : P.permx;
    const double v = src[(size_t)slot * npts + (perm ? perm[(size_t)P.lane_id[slot] * pp + i] : i)];
    if (!isfinite(v)) { atomicOr(&P.ctl->error, ERR_VALUE); return; }
    if (P.phi0 && P.absorbed[slot] > 0) P.absorbed[slot] = 0;      // (every writer stores the same value)
    const int form = (sizeof(T) == 8) ? (int)FORM_DOT : P.form[slot];
    const size_t o = (size_t)slot * pp + i;
    const double pot = P.scale[slot] * v;
    T hi, lo;
    if (form == FORM_DOT) { hi = (T)(pot - (side ? P.sqy : P.sqx)[o]); lo = T(0); }
    else { hi = (T)pot; lo = (T)(pot - (double)hi); }
    if (!side) {
        P.phi[0][o] = pot; P.phi[1][o] = pot;
        reinterpret_cast<T *>(P.ft[0])[o] = hi; reinterpret_cast<T *>(P.ft[1])[o] = hi;
        reinterpret_cast<T *>(P.fl[0])[o] = lo; reinterpret_cast<T *>(P.fl[1])[o] = lo;
    } else {
        P.gam[o] = pot;
        reinterpret_cast<T *>(P.gt)[o] = hi; reinterpret_cast<T *>(P.gl)[o] = lo;
    }
}

// ---------------------------------------------------------------- plan
constexpr int PLAN_THREADS = 1024;   // upper bound; the launch sizes the block to the width

// exclusive prefix sums of up to three 0/1 flags over the block, by warp ballot + popc
__device__ __forceinline__ void block_scan3(int f0, int f1, int f2, int (&ex)[3], int (&tot)[3], int (*wsum)[3])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned b0 = __ballot_sync(0xffffffffu, f0), b1 = __ballot_sync(0xffffffffu, f1),
                   b2 = __ballot_sync(0xffffffffu, f2);
    ex[0] = __popc(b0 & lt); ex[1] = __popc(b1 & lt); ex[2] = __popc(b2 & lt);
    __syncthreads();
    if (lane == 0) { wsum[warp][0] = __popc(b0); wsum[warp][1] = __popc(b1); wsum[warp][2] = __popc(b2); }
    __syncthreads();
    int run[3] = {0, 0, 0};
    const int nwarp = blockDim.x >> 5;
    for (int w = 0; w < nwarp; ++w) {
        if (w == warp) { ex[0] += run[0]; ex[1] += run[1]; ex[2] += run[2]; }
        run[0] += wsum[w][0]; run[1] += wsum[w][1]; run[2] += wsum[w][2];
    }
    tot[0] = run[0]; tot[1] = run[1]; tot[2] = run[2];
}

template <typename T>
__device__ __forceinline__ void emit_move_one(const Dev &P, const Ctl &c, const int r, const int tid, const int nth);

// FUSE: the same block also emits and moves the lanes it retires (see launch_plan).
template <typename T, bool FUSE>
__global__ void __launch_bounds__(PLAN_THREADS) plan_kernel(const Dev P)
{
    __shared__ int wsum[PLAN_THREADS / 32][3];
    pdl_enter();
    Ctl c = *P.ctl;
    const int tid = threadIdx.x, NT = blockDim.x;
    if (c.done) { if (tid == 0) P.ctl->n_retire = 0; return; }
    const int k = c.cycle;                           // cycles completed by the audited state
    const int A = c.n_phys;
    // a lane has used up its cycles when ITS OWN count reaches max_iter (lanes that replaced finished
    // ones came in later; everywhere else start is 0)
    auto at_limit = [&](int s) { return k - P.start[s] >= P.max_iter; };

    if (P.mode == MODE_STATIC && c.static_final) {   // emit every lane at the common boundary
        for (int s = tid; s < P.W; s += NT) {
            P.ret_slot[s] = s; P.ret_lane[s] = s; P.ret_src[s] = -1; P.ret_scale[s] = P.scale[s];
            // the closing column check ran no f-leg: r_row is the last screen's value
            P.res_row[s] = P.rrow[s]; P.res_col[s] = (double)P.rsum_col[s] * (1.0 / RSUM_SCALE);
            P.rsum_col[s] = 0ull;
            if (P.nonfinite[s]) P.status[s] = LANE_NONFINITE;
        }
        if (tid == 0) {
            Ctl *g = P.ctl;
            g->n_retire = FUSE ? 0 : P.W; g->emit_parity = c.parity; g->n_running = 0; g->done = 1;
            g->pair_terms += (long long)P.W * P.n * P.m;      // the final column check
        }
        if (FUSE) {
            __syncthreads();
            Ctl cc = c;
            cc.emit_parity = c.parity;
            for (int r = 0; r < P.W; ++r) emit_move_one<T>(P, cc, r, tid, NT);
        }
        return;
    }

    // which running lanes leave at this audit
    auto decide_vals = [&](bool held, int nf, int fl, int vd, bool limit, int &ret, int &st) {
        ret = 0; st = LANE_RUNNING;
        if (held) return;
        if (nf) { ret = 1; st = LANE_NONFINITE; }
        else if (fl && vd) { ret = 1; st = LANE_DONE; }
        else if (limit) { ret = 1; st = LANE_ITER_LIMIT; }
    };
    auto decide = [&](int s, int &ret, int &st) {
        ret = 0; st = LANE_RUNNING;
        if (s >= A) return;
        const bool held = (P.mode != MODE_ACTIVE) && P.state[s] != 0;   // frozen / already passed
        decide_vals(held, P.nonfinite[s], P.flag[s], P.verdict[s], at_limit(s), ret, st);
    };

    // pass 1.  The legs left each lane's residuals as exact fixed-point sums: turn them into the
    // values, the screen flag and the two-sided verdict (Eq. 5), clear the sums for the next
    // cycle, and count retirees and screen-positive lanes on the way.
    int cnt = 0, nflag = 0;
    for (int s = tid; s < A; s += NT) {
        const int fl = lane_flag(P, c, s) ? 1 : 0;
        const int nf = P.nonfinite[s];
        const bool held = (P.mode != MODE_ACTIVE) && P.state[s] != 0;
        const double rr = lane_row_residual(P, s);
        const double rc = (double)P.rsum_col[s] * (1.0 / RSUM_SCALE);
        const int vd = (!nf && fmax(rr, rc) <= P.tol_stop) ? 1 : 0;
        P.rsum_row[s] = 0ull; P.rsum_col[s] = 0ull; P.rsum_row64[s] = 0ull; P.esc[s] = 0;
        P.rrow[s] = rr; P.rcol[s] = rc;
        P.flag[s] = fl; P.verdict[s] = vd;
        int r, st; decide_vals(held, nf, fl, vd, at_limit(s), r, st);
        cnt += r;
        nflag += fl;
    }
    for (int off = 16; off > 0; off >>= 1) {
        cnt += __shfl_down_sync(0xffffffffu, cnt, off);
        nflag += __shfl_down_sync(0xffffffffu, nflag, off);
    }
    if ((tid & 31) == 0) { wsum[tid >> 5][0] = cnt; wsum[tid >> 5][1] = nflag; }
    __syncthreads();
    int nret = 0, nflagged = 0;
    for (int w = 0; w < (NT >> 5); ++w) { nret += wsum[w][0]; nflagged += wsum[w][1]; }
    __syncthreads();
    const int Anew = (P.mode == MODE_ACTIVE) ? A - nret : A;

    // pass 2: ordered lists (retirees, holes below Anew, survivors at or above Anew);
    // most audits retire nobody and skip it
    int base[3] = {0, 0, 0};
    for (int s0 = 0; s0 < (nret > 0 ? A : 0); s0 += NT) {
        const int s = s0 + tid;
        int r, st; decide(s, r, st);
        const int hole = (P.mode == MODE_ACTIVE) && r && s < Anew;
        const int fill = (P.mode == MODE_ACTIVE) && !r && s >= Anew && s < A;
        int ex[3], tot[3];
        block_scan3(r, hole, fill, ex, tot, wsum);
        if (r) {
            const int idx = base[0] + ex[0];
            const int lane = P.lane_id[s];
            P.ret_slot[idx] = s; P.ret_lane[idx] = lane; P.ret_scale[idx] = P.scale[s];
            P.ret_src[idx] = hole ? -(base[1] + ex[1]) - 2 : -1;      // hole ordinal, resolved below
            if (P.mode != MODE_STATIC || st != LANE_DONE) {            // STATIC keeps residuals for the end
                P.res_row[lane] = P.rrow[s];
                P.res_col[lane] = P.flag[s] ? P.rcol[s] : __longlong_as_double(0x7ff8000000000000LL);
            }
            P.depth[lane] = at_limit(s) && st != LANE_DONE ? P.max_iter : k - P.start[s];
            P.status[lane] = st;
            if (P.mode != MODE_ACTIVE) P.state[s] = 1;
        }
        if (hole) P.hole_list[base[1] + ex[1]] = s;
        if (fill) P.fill_list[base[2] + ex[2]] = s;
        base[0] += tot[0]; base[1] += tot[1]; base[2] += tot[2];
        __syncthreads();
    }
    __threadfence_block();
    __syncthreads();
    const int nholes = base[1];
    // resolve each hole's source, then move the per-slot scalars
    for (int r = tid; r < nret; r += NT) {
        const int code = P.ret_src[r];
        if (code <= -2) P.ret_src[r] = P.fill_list[-(code + 2)];
    }
    __syncthreads();
    for (int h = tid; h < nholes; h += NT) {
        const int dst = P.hole_list[h], src = P.fill_list[h];
        P.lane_id[dst] = P.lane_id[src];
        P.start[dst] = P.start[src];
        P.scale[dst] = P.scale[src];
        P.form[dst] = P.form[src];
        P.absorbed[dst] = P.absorbed[src];
        P.cyc_log[dst] = P.cyc_log[src];
        if (P.home) { const int t = P.home[dst]; P.home[dst] = P.home[src]; P.home[src] = t; }
        P.nonfinite[dst] = 0;
    }
    if (tid == 0) {
        Ctl *g = P.ctl;
        g->n_retire = (P.mode == MODE_STATIC || FUSE) ? 0 : nret;      // what is left for the emit/move kernel
        g->emit_parity = c.parity;
        // lanes whose pair terms were really evaluated (the early-exit arm skips frozen lanes)
        const int worked = P.early_exit ? c.n_running : A;
        g->pair_terms += (long long)worked * P.n * P.m         // the f-leg that produced this screen
                         + (long long)nflagged * P.n * P.m;    // column checks
        bool go_on;
        if (P.mode == MODE_ACTIVE) {
            g->n_phys = Anew; g->n_running = Anew; go_on = Anew > 0;
        } else if (P.mode == MODE_MASKED) {
            g->n_running = c.n_running - nret; go_on = g->n_running > 0;
        } else {
            g->n_passed = c.n_passed + nret;
            go_on = g->n_passed < P.W;
            if (!go_on) g->static_final = 1;
        }
        if (go_on) {
            const int width = (P.mode == MODE_ACTIVE) ? Anew : (P.early_exit ? g->n_running : P.W);
            g->cycle = k + 1;
            g->parity = c.parity ^ 1;
            g->slots += width;
            g->pair_terms += (long long)width * P.n * P.m;     // the g-leg that completes cycle k+1
            if (k < P.widths_cap) P.widths[k] = width;
        } else if (P.mode != MODE_STATIC) {
            g->done = 1;
        }
    }
    if (FUSE && P.mode != MODE_STATIC && nret > 0) {
        __syncthreads();                                  // the lists and per-slot scalars above are this block's own writes
        Ctl cc = c;
        cc.emit_parity = c.parity;
        for (int r = 0; r < nret; ++r) emit_move_one<T>(P, cc, r, tid, NT);
    }
}

// Planner after a multi-cycle launch (lane_cycles_kernel): the lanes that passed inside the launch
// have written their own depth, status, residuals and potentials; what is left is the accounting of
// Eq. 6-8 for all `K` cycles of the launch at once - widths A_k, slots, pair terms - the pairing of
// holes below the new width with survivors from above it, and the advance of the control block.
template <typename T, bool FUSE>
__global__ void __launch_bounds__(PLAN_THREADS) plan_cycles_kernel(const Dev P, const int K)
{
    __shared__ int wsum[PLAN_THREADS / 32][3];
    // lanes that left at the audit of the state after k0 + j cycles (a word between 32 of them: threads read runs of a power of two)
    __shared__ int left_[MAX_CYCLES_IN_LAUNCH + MAX_CYCLES_IN_LAUNCH / 32];
    auto left_at = [&](const int j) -> int & { return left_[j + (j >> 5)]; };
    __shared__ int checks_s, nret_s, last_s, ran_s;
    __shared__ unsigned long long slots_s, terms_s;
    pdl_enter();
    const Ctl c = *P.ctl;
    const int tid = threadIdx.x, NT = blockDim.x;
    if (c.done) { if (tid == 0) P.ctl->n_retire = 0; return; }
    const int k0 = c.cycle, A = c.n_phys;
    for (int j = tid; j < K; j += NT) left_at(j) = 0;
    if (tid == 0) { checks_s = nret_s = ran_s = 0; last_s = 0; slots_s = terms_s = 0ull; }
    __syncthreads();
    int nchk = 0;
    for (int s = tid; s < A; s += NT) {
        const int r = P.ret_at[s];
        if (r > 0) { atomicAdd(&left_at(r - 1 - k0), 1); atomicAdd(&nret_s, 1); atomicMax(&last_s, r - 1 - k0); }
        nchk += P.n_checks[s];
        P.rsum_row[s] = 0ull; P.rsum_col[s] = 0ull;      // between launches the residual sums are zero
        P.rsum_row64[s] = 0ull; P.esc[s] = 0;
    }
    for (int off = 16; off > 0; off >>= 1) nchk += __shfl_down_sync(0xffffffffu, nchk, off);
    if ((tid & 31) == 0 && nchk) atomicAdd(&checks_s, nchk);
    __syncthreads();
    const int nret = nret_s;
    const bool compact = P.mode == MODE_ACTIVE;      // MASKED: lanes stay where they are, frozen or not
    const int Anew = compact ? A - nret : A;
    const int parity_new = c.parity ^ (K & 1);       // survivors ran all K cycles
    // ordered lists: holes below the new width, survivors at or above it
    int base[3] = {0, 0, 0};
    for (int s0 = 0; s0 < (nret > 0 && compact ? A : 0); s0 += NT) {
        const int s = s0 + tid;
        const int r = (s < A && P.ret_at[s] > 0) ? 1 : 0;
        const int hole = r && s < Anew;
        const int fill = (s < A) && !r && s >= Anew;
        int ex[3], tot[3];
        block_scan3(r, hole, fill, ex, tot, wsum);
        if (hole) P.hole_list[base[1] + ex[1]] = s;
        if (fill) P.fill_list[base[2] + ex[2]] = s;
        base[0] += tot[0]; base[1] += tot[1]; base[2] += tot[2];
        __syncthreads();
    }
    __threadfence_block();
    __syncthreads();
    const int nholes = base[1];
    for (int h = tid; h < nholes; h += NT) {
        const int dst = P.hole_list[h], src = P.fill_list[h];
        P.ret_slot[h] = dst; P.ret_lane[h] = -1; P.ret_src[h] = src; P.ret_scale[h] = 1.0;   // move only
        P.lane_id[dst] = P.lane_id[src];
        P.start[dst] = P.start[src];
        P.scale[dst] = P.scale[src];
        P.form[dst] = P.form[src];
        P.absorbed[dst] = P.absorbed[src];
        P.cyc_log[dst] = P.cyc_log[src];
        P.nonfinite[dst] = 0;
        P.rrow[dst] = P.rrow[src]; P.rcol[dst] = P.rcol[src]; P.flag[dst] = P.flag[src];
    }
    // the audit that counts as the most recent one: the launch's last, or the one at which the last lane left.  A lane
    // that froze at that very audit shows what it was decided from; one that froze before shows a frozen lane's values
    const int jl = nret == c.n_running ? last_s : K - 1;
    for (int s = tid; s < A; s += NT) {
        if (P.mode == MODE_MASKED) {
            const int r = P.ret_at[s];
            if (r > 0 && r - 1 - k0 == jl) {
                const double rc = P.res_col[P.lane_id[s]];
                P.rrow[s] = P.res_row[P.lane_id[s]];
                P.flag[s] = !isnan(rc);
                P.rcol[s] = isnan(rc) ? 0.0 : rc;
            } else if (P.early_exit && P.state[s]) { P.rrow[s] = 0.0; P.rcol[s] = 0.0; P.flag[s] = 0; }
        }
        P.ret_at[s] = 0; P.n_checks[s] = 0;
    }
    // The widths of the launch's cycles and what they add up to: every thread takes a run of consecutive cycles, the
    // lanes that left before it from a scan over the threads.
    {
        const bool full = P.mode == MODE_MASKED && !P.early_exit;
        const int per = (K + NT - 1) / NT, j0 = tid * per, j1 = min(K, j0 + per);
        int mine = 0;
        for (int j = j0; j < j1; ++j) mine += left_at(j);
        int incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) { const int o = __shfl_up_sync(0xffffffffu, incl, off); if ((tid & 31) >= off) incl += o; }
        if ((tid & 31) == 31) wsum[tid >> 5][0] = incl;
        __syncthreads();
        int w = c.n_running - (incl - mine), ran = 0;   // running lanes before cycle k0 + j0
        for (int e = 0; e < (tid >> 5); ++e) w -= wsum[e][0];
        unsigned long long slots = 0ull, legs = 0ull;
        for (int j = j0; j < j1 && w > 0; ++j) {
            legs += full ? A : w;                        // the f-leg whose epilogue screened the state after k0 + j cycles
            w -= left_at(j);
            if (w == 0) break;
            const int width = full ? A : w;              // the launch's width is the running lanes', or W under a mask
            if (k0 + j < P.widths_cap) P.widths[k0 + j] = width;      // cycle k0 + j + 1 ran at this width
            slots += width;
            legs += width;                               // its g-leg
            ++ran;
        }
        if (legs) { atomicAdd(&slots_s, slots); atomicAdd(&terms_s, legs); atomicAdd(&ran_s, ran); }
        __syncthreads();
    }
    if (tid == 0) {
        Ctl *g = P.ctl;
        const long long nm = (long long)P.n * P.m, slots = (long long)slots_s, terms = ((long long)terms_s + checks_s) * nm;
        const int ran = ran_s;
        g->cycle = k0 + ran;
        g->parity = parity_new;
        g->emit_parity = parity_new ^ 1;             // the move copies the OTHER buffer: the survivors' current row potentials
        g->n_phys = Anew; g->n_running = c.n_running - nret;
        g->n_retire = FUSE ? 0 : nholes;
        g->slots += slots;
        g->pair_terms += terms;
        g->mask_left = g->mask_last = 0;
        if (c.n_running == nret) g->done = 1;
    }
    if (FUSE && nholes > 0) {
        __syncthreads();
        Ctl cc = c;
        cc.emit_parity = parity_new ^ 1;
        for (int r = 0; r < nholes; ++r) emit_move_one<T>(P, cc, r, tid, NT);
    }
}

// Planner of a STATIC batch between the two halves of a multi-cycle launch (scaling_kernel).  In the first half the
// lanes that had not passed ran up to K cycles, each stopping at the state it passed at.  If some lane has still
// not passed, every lane goes on to cycle k0 + K; otherwise the batch ends at the cycle of the last one to pass.  The
// second half (SC_CATCH_UP) takes the passed lanes there, and in the end writes everyone's outputs.  Whole lanes
// are independent problems, so the order in which their cycles run changes no bit, and each runs every cycle once.
__global__ void __launch_bounds__(PLAN_THREADS) plan_static_kernel(const Dev P, const int K)
{
    __shared__ int nret_s, checks_s, last_s;
    pdl_enter();
    const Ctl c = *P.ctl;
    const int tid = threadIdx.x, NT = blockDim.x;
    if (c.done) return;
    const int k0 = c.cycle;
    if (tid == 0) nret_s = checks_s = last_s = 0;
    __syncthreads();
    int nret = 0, nchk = 0, last = 0;
    for (int s = tid; s < P.W; s += NT) {
        const int r = P.ret_at[s];                       // (left for SC_CATCH_UP, which clears it)
        if (r > 0) { ++nret; last = max(last, r - 1 - k0); }
        nchk += P.n_checks[s];
        P.n_checks[s] = 0;
    }
    for (int off = 16; off > 0; off >>= 1) {
        nret += __shfl_down_sync(0xffffffffu, nret, off);
        nchk += __shfl_down_sync(0xffffffffu, nchk, off);
        last = max(last, __shfl_down_sync(0xffffffffu, last, off));
    }
    if ((tid & 31) == 0) { atomicAdd(&nret_s, nret); atomicAdd(&checks_s, nchk); atomicMax(&last_s, last); }
    __syncthreads();
    const bool all = c.n_passed + nret_s == P.W;
    const int ran = all ? last_s : K;
    for (int j = tid; j < ran; j += NT) if (k0 + j < P.widths_cap) P.widths[k0 + j] = P.W;
    if (tid == 0) {
        Ctl *g = P.ctl;
        const long long nm = (long long)P.n * P.m;
        g->prev_cycle = k0;
        g->cycle = k0 + ran;
        g->parity = c.parity ^ (ran & 1);
        g->n_passed = c.n_passed + nret_s;
        g->n_retire = 0;
        g->slots += (long long)ran * P.W;
        // both legs of every cycle, the f-leg that screened the last state, the column checks, the closing one
        g->pair_terms += ((2ll * ran + (all ? 2 : 0)) * P.W + checks_s) * nm;
        if (all) { g->static_final = 1; g->n_running = 0; g->done = 1; }
    }
}
void launch_plan_static(const Dev &P, int cycles, cudaStream_t st)
{
    const int nt = P.W >= PLAN_THREADS ? PLAN_THREADS : (P.W + 31) / 32 * 32;
    launch_pdl(plan_static_kernel, dim3(1), dim3(nt), 0, st, P, cycles);
}

// ---------------------------------------------------------------- emit + move
template <typename T>
__global__ void __launch_bounds__(256) emit_move_kernel(const Dev P)
{
    pdl_enter();
    const Ctl c = *P.ctl;
    const int nret = c.n_retire;
    if (nret <= 0) return;
    // The launch's blocks are dealt out among the retirees of this audit (usually one or two): a move
    // is a plain copy of up to a few MB and should have the whole machine's loads in flight.
    const int nb = gridDim.x, b = blockIdx.x;
    const int per = nb / nret;
    if (per >= 1) {
        const int r = b / per;
        if (r < nret) emit_move_one<T>(P, c, r, (b % per) * blockDim.x + threadIdx.x, per * blockDim.x);
    } else {
        for (int r = b; r < nret; r += nb) emit_move_one<T>(P, c, r, threadIdx.x, blockDim.x);
    }
}

// Retiree r of the list: `nth` threads (this one is number `tid`) write its outputs and, if its slot
// is a hole below the new width, copy the paired survivor's state into it.
template <typename T>
__device__ __forceinline__ void emit_move_one(const Dev &P, const Ctl &c, const int r, const int tid, const int nth)
{
    const int slot = P.ret_slot[r], lane = P.ret_lane[r], src = P.ret_src[r];
    const double inv_s = 1.0 / P.ret_scale[r];
    const int ep = c.emit_parity;
    // emit: potentials of the audited state in the caller's units (f = phi / s); lane < 0: the lane
    // in the hole wrote its own outputs when it left (multi-cycle launches), only the move is left
    if (lane >= 0)
        for (int i = tid; i < P.n; i += nth)
            P.f_out[(size_t)lane * P.n + (P.permx ? P.permx[(size_t)lane * P.np + i] : i)] = P.phi[ep][(size_t)slot * P.np + i] * inv_s;
    for (int j = tid; j < P.m; j += nth) {
        // the hole's own g is read before the survivor's g is copied over it (same thread)
        if (lane >= 0) P.g_out[(size_t)lane * P.m + (P.permy ? P.permy[(size_t)lane * P.mp + j] : j)] = P.gam[(size_t)slot * P.mp + j] * inv_s;
        if (src >= 0) P.gam[(size_t)slot * P.mp + j] = P.gam[(size_t)src * P.mp + j];
    }
    if (tid == 0 && lane >= 0) P.emitted[lane] = 1;
    if (src < 0) return;
    // Move the survivor in slot `src` into the hole `slot`: all of its slot-indexed arrays as ONE list
    // of 16-byte vectors, so that a thread's loads in flight span arrays (array after array, each
    // with its own loop, cost one DRAM round trip per array: ~15 us for any lane size).
    __shared__ const uint4 *seg_src[24];
    __shared__ uint4 *seg_dst[24];
    __shared__ unsigned seg_end[24];          // running total of vectors up to and including the segment
    __shared__ int seg_n;
    __syncthreads();                          // the table may still be in use by this block's previous retiree
    if (threadIdx.x == 0) {
        int ns = 0;
        unsigned run = 0;
        auto add = [&](void *base, size_t bytes_per_lane) {
            if (!base || bytes_per_lane == 0) return;
            seg_src[ns] = reinterpret_cast<const uint4 *>((const char *)base + (size_t)src * bytes_per_lane);
            seg_dst[ns] = reinterpret_cast<uint4 *>((char *)base + (size_t)slot * bytes_per_lane);
            run += (unsigned)(bytes_per_lane / 16);
            seg_end[ns++] = run;
        };
        const int np_ = ep ^ 1;   // buffer that holds the survivors' current row potentials
        if (P.dots) {
            // the tiled copies stay behind: nothing reads those of a lane whose products are stored
            add(P.dots, (size_t)P.np * P.mp * 4);
        } else if (P.tensor) {
            add(P.xb, (size_t)((P.n + 127) / 128) * P.d * 256);      // tiled copies: 128-point tiles x d bf16
            add(P.yb, (size_t)((P.m + 127) / 128) * P.d * 256);
        } else {
            add(P.xs, (size_t)P.DP * P.np * sizeof(T));
            add(P.ys, (size_t)P.DP * P.mp * sizeof(T));
        }
        if (P.guard > 0.0) {                                          // raw input copies of the guard band
            add(P.xraw, P.xraw_stride);
            add(P.yraw, P.yraw_stride);
        }
        add(P.sqx, (size_t)P.np * 8); add(P.sqy, (size_t)P.mp * 8);
        add(P.la2, (size_t)P.np * 8); add(P.lb2, (size_t)P.mp * 8);
        add(P.wa, (size_t)P.np * 8); add(P.wb, (size_t)P.mp * 8);
        add(P.phi[np_], (size_t)P.np * 8);
        if (P.phi0) {                                                 // lanes on the scaling kernel have no streamed terms
            add(P.phi0, (size_t)P.np * 8); add(P.gam0, (size_t)P.mp * 8);
            add(P.uu[np_], (size_t)P.np * 8); add(P.vv, (size_t)P.mp * 8);
        } else {
            add(P.ft[np_], (size_t)P.np * sizeof(T));
            add(P.fl[np_], (size_t)P.np * sizeof(T));
            add(P.gt, (size_t)P.mp * sizeof(T));
            add(P.gl, (size_t)P.mp * sizeof(T));
        }
        if (P.topy) {                                                 // lanes in spatial order (the order itself is kept by lane)
            add(P.boxx, (size_t)2 * P.DP * P.nbx * 4); add(P.boxy, (size_t)2 * P.DP * P.nby * 4);
            add(P.topx[np_], (size_t)(P.lists ? 2 : 1) * P.nbx * 4); add(P.topy, (size_t)P.nby * 4);
        }
        seg_n = ns;
    }
    __syncthreads();
    const int ns = seg_n;
    const unsigned total = seg_end[ns - 1];
    for (unsigned v = tid; v < total; v += 4u * (unsigned)nth) {       // four loads in flight per thread
        uint4 a[4];
        uint4 *d[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned idx = v + (unsigned)u * (unsigned)nth;
            d[u] = nullptr;
            if (idx < total) {
                int sg = 0;
                while (idx >= seg_end[sg]) ++sg;
                const unsigned off = idx - (sg ? seg_end[sg - 1] : 0u);
                a[u] = seg_src[sg][off];
                d[u] = seg_dst[sg] + off;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) if (d[u]) *d[u] = a[u];
    }
}

// ---------------------------------------------------------------- gather (read-back)
template <typename O>
__global__ void gather_kernel(const Dev P, O *f, O *g)
{
    const Ctl c = *P.ctl;
    const int y = blockIdx.x;                         // lanes along x: up to twice 65535 of them
    const int tid = blockIdx.y * blockDim.x + threadIdx.x, nth = gridDim.y * blockDim.x;
    if (y < P.L) {                                    // emitted lanes, by lane id
        const int lane = y;
        if (!P.emitted[lane]) return;
        if (f) for (int i = tid; i < P.n; i += nth) f[(size_t)lane * P.n + i] = (O)P.f_out[(size_t)lane * P.n + i];
        if (g) for (int j = tid; j < P.m; j += nth) g[(size_t)lane * P.m + j] = (O)P.g_out[(size_t)lane * P.m + j];
    } else {                                          // lanes still held in a slot
        const int slot = y - P.L;
        if (c.done || slot >= c.n_phys) return;
        if (P.mode == MODE_MASKED && P.state[slot]) return;
        const int lane = P.lane_id[slot];
        if (P.emitted[lane]) return;
        const double inv_s = 1.0 / P.scale[slot];
        if (f) for (int i = tid; i < P.n; i += nth)
            f[(size_t)lane * P.n + (P.permx ? P.permx[(size_t)lane * P.np + i] : i)] = (O)(P.phi[c.parity][(size_t)slot * P.np + i] * inv_s);
        if (g) for (int j = tid; j < P.m; j += nth)
            g[(size_t)lane * P.m + (P.permy ? P.permy[(size_t)lane * P.mp + j] : j)] = (O)(P.gam[(size_t)slot * P.mp + j] * inv_s);
    }
}

__global__ void gather_small_kernel(const Dev P, int *depth, int *status, float *rrow, float *rcol)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= P.L) return;
    if (depth) depth[t] = P.depth[t];
    if (status) status[t] = P.status[t];
    if (rrow) rrow[t] = (float)P.res_row[t];
    if (rcol) rcol[t] = (float)P.res_col[t];
}

// What the most recent audit measured for the lanes still held in a slot (one-launch-per-leg path).
__global__ void gather_audit_kernel(const Dev P, float *rrow, float *rcol, int *flagged)
{
    const Ctl c = *P.ctl;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= P.W || s >= c.n_phys) return;
    const int lane = P.lane_id[s];
    if (rrow) rrow[lane] = (float)P.rrow[s];
    if (rcol) rcol[lane] = P.flag[s] ? (float)P.rcol[s] : __int_as_float(0x7fc00000);
    if (flagged) flagged[lane] = P.flag[s];
}
void launch_gather_audit(const Dev &P, float *rrow, float *rcol, int *flagged, cudaStream_t st)
{
    gather_audit_kernel<<<(P.W + 255) / 256, 256, 0, st>>>(P, rrow, rcol, flagged);
}

// ---------------------------------------------------------------- plan application
// out[t, i, :] = sum_j pi_ij v[t, j, :] with pi = exp((f + g - C)/eps) from the potentials the batch
// holds for lane t (Eq. 3's plan, never stored): the coupling applied to caller-supplied values, e.g.
// v = y gives a_i times the barycentric image of x_i.  One warp per row, float64 throughout, cost from
// the caller's raw coordinates.  After a g-leg every pi_ij <= b_j <= 1, so the exponentials need no shift.
constexpr int APPLY_MAX_DV = 16;
__global__ void __launch_bounds__(128) apply_plan_kernel(const Dev P, const void *x, const void *y, const float *eps,
                                                         const float *v, const int dv, float *out)
{
    const int lane_t = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * 4 + warp;
    if (i >= P.n || !P.emitted[lane_t]) return;
    const double inv_eps = 1.0 / (double)eps[lane_t];
    const double fi = P.f_out[(size_t)lane_t * P.n + i];
    const double *g = P.g_out + (size_t)lane_t * P.m;
    const size_t xb = ((size_t)lane_t * P.n + i) * P.d;
    double acc[APPLY_MAX_DV];
#pragma unroll
    for (int c = 0; c < APPLY_MAX_DV; ++c) acc[c] = 0.0;
    for (int j = lane; j < P.m; j += 32) {
        const size_t yb = ((size_t)lane_t * P.m + j) * P.d;
        double cst = 0.0;
        for (int k = 0; k < P.d; ++k) {
            const double t = (double)load_raw(P, x, xb + k) - (double)load_raw(P, y, yb + k);
            cst = fma(t, t, cst);
        }
        const double pij = exp((fi + g[j] - cst) * inv_eps);
        const float *vj = v + ((size_t)lane_t * P.m + j) * dv;
#pragma unroll
        for (int c = 0; c < APPLY_MAX_DV; ++c) if (c < dv) acc[c] = fma(pij, (double)vj[c], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < APPLY_MAX_DV; ++c) {
        if (c < dv) {
            double a = acc[c];
            for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
            if (lane == 0) out[((size_t)lane_t * P.n + i) * dv + c] = (float)a;
        }
    }
}
// The wide tiles' part of R rows (skb_pairs64.cuh), by differences; every NC-th of the columns.  Out of line:
// its registers would come off the tiled loop's.
template <int DM, int DV, int R, int NC>
__device__ __noinline__ void apply_wide_tiles(const bool bf16, const int n, const int m, const int d, double *tile, const double *org, const void *x,
                                              const void *y, const float *v, const int i0, const double k2, const double *f,
                                              const double *g, const int dv, const int cs, const bool row_wide, double *out)
{
    auto raw = [bf16](const void *base, size_t i) -> float {
        return bf16 ? __uint_as_float((unsigned)reinterpret_cast<const unsigned short *>(base)[i] << 16) : reinterpret_cast<const float *>(base)[i];
    };
    for (int e = 0; e < R * DV; ++e) out[e] = 0.0;
    for (int j0 = 0; j0 < m; j0 += P64_TJ) {
        __syncthreads();
        P64Part<DM, 128> part;
        p64_fetch(part, j0, m, d, [&](int j, int k) { return raw(y, (size_t)j * d + k); }, [&](int j) { return g[j]; });
        const bool wide = p64_tile<DM, 128>(tile, org, j0, m, d, k2, part);
        if (!__syncthreads_or(wide || row_wide)) continue;
        for (int j = j0 + cs; j < m && j < j0 + P64_TJ; j += NC)
            for (int r = 0; r < R; ++r) {
                const int i = i0 + r < n ? i0 + r : n - 1;
                const double t = p64_entry(d, k2, f[i] + g[j], [&](int k) { return raw(x, (size_t)i * d + k); }, [&](int k) { return raw(y, (size_t)j * d + k); });
                for (int c = 0; c < dv; ++c) out[r * DV + c] = fma(t, (double)v[(size_t)j * dv + c], out[r * DV + c]);
            }
    }
}
// The same for d <= 32 by column tiles in shared memory (skb_pairs64.cuh); DV: values per point, rounded up.
// 8 lanes of 4096 x 4096 points, d = dv = 3: 966 us with one warp per row, 414 us so with CUDA's exp2 and two rows a thread,
// 281 us with p64_exp2 and four.
constexpr int P64_APPLY_ROWS = 32;                       // rows of a block (64: the last wave is emptier, 301 against 281 us)
template <int DM, int DV>
__global__ void __launch_bounds__(128, DM <= 4 && DV <= 3 ? 4 : 1) apply_plan_tiled_kernel(const Dev P, const void *x, const void *y, const float *eps,
                                                               const float *v, const int dv, float *out)
{
    // (four rows to a thread halve what it reads from shared memory per pair; more values a point want the registers)
    constexpr int R = DM <= 4 && DV <= 4 ? 4 : 2, RW = P64_APPLY_ROWS / 4, NC = 32 / (RW / R);
    __shared__ double tile[P64_TILE<DM, 128>];
    __shared__ double vals[DV * P64_TJ];                  // (a tile's values, float64)
    __shared__ double org[DM];
    const int lane_t = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (!P.emitted[lane_t]) return;
    const int cs = lane / (RW / R), i0 = blockIdx.x * (4 * RW) + warp * RW + lane % (RW / R) * R;
    const double k2 = 1.4426950408889634 / (double)eps[lane_t], entry = p64_table();
    const double *f = P.f_out + (size_t)lane_t * P.n, *g = P.g_out + (size_t)lane_t * P.m;
    const size_t xb = (size_t)lane_t * P.n * P.d, yb = (size_t)lane_t * P.m * P.d;
    if (threadIdx.x < DM) org[threadIdx.x] = threadIdx.x < P.d ? (double)load_raw(P, x, xb + (size_t)blockIdx.x * (4 * RW) * P.d + threadIdx.x) : 0.0;
    __syncthreads();
    double xr[R][DM], ri[R], acc[R][DV];
    bool row_wide = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = i0 + r < P.n ? i0 + r : P.n - 1;
        double q = 0.0;
#pragma unroll
        for (int k = 0; k < DM; ++k) { xr[r][k] = k < P.d ? (double)load_raw(P, x, xb + (size_t)i * P.d + k) - org[k] : 0.0; q = fma(xr[r][k], xr[r][k], q); }
        ri[r] = k2 * (f[i] - q);
        row_wide = row_wide || p64_wide(k2, q);
#pragma unroll
        for (int c = 0; c < DV; ++c) acc[r][c] = 0.0;
    }
    bool any_wide = false;
    auto load = [&](int j, int k) { return load_raw(P, y, yb + (size_t)j * P.d + k); };
    auto pot = [&](int j) { return g[j]; };
    constexpr int NV = (P64_TJ * DV + 127) / 128;
    float vn[NV];
    auto fetch_vals = [&](const int j0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const int e = threadIdx.x + 128 * q, j = j0 + e % P64_TJ, c = e / P64_TJ;
            vn[q] = (j < P.m && c < dv) ? v[((size_t)lane_t * P.m + j) * dv + c] : 0.f;
        }
    };
    P64Part<DM, 128> part;
    if (P64_AHEAD<DM>) { p64_fetch(part, 0, P.m, P.d, load, pot); fetch_vals(0); }
    for (int j0 = 0; j0 < P.m; j0 += P64_TJ) {
        if (!P64_AHEAD<DM>) { p64_fetch(part, j0, P.m, P.d, load, pot); fetch_vals(j0); }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NV; ++q)
            if (P64_TJ * DV % 128 == 0 || threadIdx.x + 128 * q < P64_TJ * DV) vals[threadIdx.x + 128 * q] = (double)vn[q];
        const bool wide = p64_tile<DM, 128>(tile, org, j0, P.m, P.d, k2, part);
        if (P64_AHEAD<DM>) { p64_fetch(part, j0 + P64_TJ, P.m, P.d, load, pot); fetch_vals(j0 + P64_TJ); }
        if (__syncthreads_or(wide || row_wide)) { any_wide = true; continue; }
        const int end = P.m - j0 < P64_TJ ? P.m - j0 : P64_TJ;                 // (whole warps go on together past it)
#pragma unroll 2
        for (int jj = cs; jj < P64_TJ; jj += NC) {
            double t[R];
            const double c0 = tile[DM * P64_TJ + jj];
#pragma unroll
            for (int r = 0; r < R; ++r) t[r] = c0 + ri[r];
#pragma unroll
            for (int k = 0; k < DM; ++k) {
                const double yk = tile[k * P64_TJ + jj];
#pragma unroll
                for (int r = 0; r < R; ++r) t[r] = fma(xr[r][k], yk, t[r]);
            }
            p64_exp2(t, entry);
            if (end < P64_TJ && jj >= end)
#pragma unroll
                for (int r = 0; r < R; ++r) t[r] = 0.0;
#pragma unroll
            for (int c = 0; c < DV; ++c) {
                const double vc = vals[c * P64_TJ + jj];
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r][c] = fma(t[r], vc, acc[r][c]);
            }
        }
    }
    if (any_wide) {
        double more[R][DV];
        const size_t es = P.xy_bf16 ? 2 : 4;
        apply_wide_tiles<DM, DV, R, NC>(P.xy_bf16 != 0, P.n, P.m, P.d, tile, org, (const char *)x + xb * es, (const char *)y + yb * es,
                                    v + (size_t)lane_t * P.m * dv, i0, k2, f, g, dv, cs, row_wide, &more[0][0]);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < DV; ++c) acc[r][c] += more[r][c];
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < DV; ++c) {
            double a = acc[r][c];
#pragma unroll
            for (int off = RW / R; off < 32; off *= 2) a += __shfl_xor_sync(0xffffffffu, a, off);
            if (cs == 0 && i0 + r < P.n && c < dv) out[((size_t)lane_t * P.n + i0 + r) * dv + c] = (float)a;
        }
}
template <int DM>
static void launch_apply_tiled(const Dev &P, const void *x, const void *y, const float *eps, const float *v, int dv, float *out, int lanes, cudaStream_t st)
{
    const dim3 grid((P.n + P64_APPLY_ROWS - 1) / P64_APPLY_ROWS, lanes);
    if constexpr (DM <= 4)
        if (dv <= 3) { apply_plan_tiled_kernel<DM, 3><<<grid, 128, 0, st>>>(P, x, y, eps, v, dv, out); return; }
    if (dv <= 4) apply_plan_tiled_kernel<DM, 4><<<grid, 128, 0, st>>>(P, x, y, eps, v, dv, out);
    else apply_plan_tiled_kernel<DM, APPLY_MAX_DV><<<grid, 128, 0, st>>>(P, x, y, eps, v, dv, out);
}
// Few blocks of rows leave SMs empty while the threads of the tiled kernel walk 16 times the columns: up to the counts of blocks of 64
// below a warp per row is faster (us, tiled <-> warp per row; d = 8, dv = 1: 500 points 43 <- 39, 1000 64 <- 58, 1300 75 <- 73, 1600 82 -> 83,
// 2000 101 -> 112; wide values, d = dv = 5, two lanes of 1000 72 <- 56; dv = 12, d = 3, 500 points 42 <- 39).  Not where the tiles hold four
// rows a thread (d = dv = 3: one lane of 500 points 35 -> 39, of 4096 100 -> 165, of 5000 139 -> 345), nor for narrow values of
// more dimensions (d = 30, dv = 3, 8 blocks 61 -> 78).
void launch_apply_plan(const Dev &P, const void *x, const void *y, const float *eps, const float *v, int dv, float *out,
                       int lanes, cudaStream_t st)
{
    const long long blocks = (long long)((P.n + 63) / 64) * lanes;
    const bool narrow = dv <= 4 ? P.d > 4 && P.d <= 8 && blocks <= 24 : blocks <= (P.d <= 8 && dv <= 8 ? 80 : 8);
    if (P.d > P64_MAX_D || narrow) { apply_plan_kernel<<<dim3((P.n + 3) / 4, lanes), 128, 0, st>>>(P, x, y, eps, v, dv, out); return; }
    if (P.d <= 3) { launch_apply_tiled<3>(P, x, y, eps, v, dv, out, lanes, st); return; }
    if (P.d <= 4) { launch_apply_tiled<4>(P, x, y, eps, v, dv, out, lanes, st); return; }
    if (P.d <= 16) { launch_apply_tiled<16>(P, x, y, eps, v, dv, out, lanes, st); return; }
    launch_apply_tiled<P64_MAX_D>(P, x, y, eps, v, dv, out, lanes, st);
}

// Slots by falling scale (smallest eps first, equal ones as they come).
__global__ void __launch_bounds__(128) order_kernel(const Dev P, int *order)
{
    const int s = blockIdx.x * 128 + threadIdx.x;
    if (s >= P.W) return;
    const double mine = P.scale[s];
    int rank = 0;
    for (int t = 0; t < P.W; ++t) { const double x = P.scale[t]; rank += x > mine || (x == mine && t < s); }
    order[rank] = s;
}
void launch_order(const Dev &P, int *order, cudaStream_t st) { order_kernel<<<(P.W + 127) / 128, 128, 0, st>>>(P, order); }

// ---------------------------------------------------------------- launchers
void launch_lane_stats(const Dev &P, const void *x, const void *y, const float *eps, int slot0, int lane0, int count,
                       int cycle0, cudaStream_t st)
{
    if (P.d <= 32) lane_stats_kernel<<<count, 256, 0, st>>>(P, x, y, eps, slot0, lane0, cycle0);
    else lane_stats_deep_kernel<<<dim3(STATS_BLOCKS, count), 32 * STATS_WARPS, 0, st>>>(P, x, y, eps, slot0, lane0, cycle0);
}
void launch_prep(const Dev &P, const void *x, const void *y, const float *a, const float *b, int slot0, int count, cudaStream_t st)
{
    const int pp = P.np > P.mp ? P.np : P.mp;
    dim3 grid((pp + 127) / 128, count, 2);
    if (P.permx) launch_prep_near(P, x, y, a, b, slot0, count, st);
    else if (P.tensor) prep_tensor_kernel<<<dim3((pp + 31) / 32, count, 2), 256, 0, st>>>(P, x, y, a, b, slot0);
    else if (P.compute_f64) prep_kernel<double><<<grid, 128, 0, st>>>(P, x, y, a, b, slot0);
    else prep_kernel<float><<<grid, 128, 0, st>>>(P, x, y, a, b, slot0);
}
// New lanes have come in: the control block takes them into the width (between cycles, ACTIVE only).
__global__ void refill_ctl_kernel(const Dev P, const int count)
{
    Ctl *g = P.ctl;
    g->n_phys += count; g->n_running += count; g->done = 0; g->n_retire = 0;
}
void launch_refill_ctl(const Dev &P, int count, cudaStream_t st) { refill_ctl_kernel<<<1, 1, 0, st>>>(P, count); }
void launch_warm(const Dev &P, const double *f0, const double *g0, cudaStream_t st)
{
    const int pp = P.n > P.m ? P.n : P.m;
    dim3 grid((pp + 127) / 128, P.W, 2);
    if (P.compute_f64) warm_kernel<double><<<grid, 128, 0, st>>>(P, f0, g0);
    else warm_kernel<float><<<grid, 128, 0, st>>>(P, f0, g0);
}
// Bytes one retirement can move (a survivor's whole state into the hole) plus what it emits.
static size_t lane_state_bytes(const Dev &P)
{
    const size_t ts = P.compute_f64 ? 8 : 4;
    size_t coords = (size_t)P.DP * (P.np + P.mp) * ts;
    if (P.tensor) coords = P.dots ? (size_t)P.np * P.mp * 4 : ((size_t)((P.n + 127) / 128) + (size_t)((P.m + 127) / 128)) * P.d * 256;
    if (P.guard > 0.0) coords += P.xraw_stride + P.yraw_stride;
    return coords + (size_t)(P.np + P.mp) * (4 * 8 + (P.phi0 ? 16 : 2 * ts) + 8);
}
// When even the retirement of every lane at once would move little (narrow batches of small
// lanes), the planner's own block emits and moves, and the emit/move kernel is not launched:
// one kernel less in the chain of dependent launches that bounds a narrow cycle.  Same device
// functions either way, so the results do not depend on the choice.
static bool plan_fuses_move(const Dev &P, int width)
{
    const int lanes = (P.mode == MODE_STATIC) ? P.W : (width < 1 ? 1 : width);
    if (lanes == 1) return (size_t)(P.n + P.m) * 16 <= ((size_t)512 << 10);      // (a last lane is emitted, nothing moves)
    return (size_t)lanes * lane_state_bytes(P) <= ((size_t)512 << 10);
}
int launch_plan(const Dev &P, int width, cudaStream_t st)
{
    int nt = (width + 31) / 32 * 32;
    if (P.mode == MODE_STATIC) nt = (P.W + 31) / 32 * 32;
    const bool fuse = plan_fuses_move(P, width);
    nt = nt < (fuse ? 256 : 128) ? (fuse ? 256 : 128) : (nt > PLAN_THREADS ? PLAN_THREADS : nt);
    if (fuse) {
        if (P.compute_f64) launch_pdl(plan_kernel<double, true>, dim3(1), dim3(nt), 0, st, P);
        else launch_pdl(plan_kernel<float, true>, dim3(1), dim3(nt), 0, st, P);
    } else {
        launch_pdl(plan_kernel<float, false>, dim3(1), dim3(nt), 0, st, P);
    }
    return 1;
}
int launch_plan_cycles(const Dev &P, int width, int cycles, cudaStream_t st)
{
    int nt = (width + 31) / 32 * 32;
    const bool fuse = plan_fuses_move(P, width);
    nt = nt < (fuse ? 256 : 128) ? (fuse ? 256 : 128) : (nt > PLAN_THREADS ? PLAN_THREADS : nt);
    if (fuse) {
        if (P.compute_f64) launch_pdl(plan_cycles_kernel<double, true>, dim3(1), dim3(nt), 0, st, P, cycles);
        else launch_pdl(plan_cycles_kernel<float, true>, dim3(1), dim3(nt), 0, st, P, cycles);
    } else {
        launch_pdl(plan_cycles_kernel<float, false>, dim3(1), dim3(nt), 0, st, P, cycles);
    }
    return 1;
}
int launch_emit_move(const Dev &P, int width, cudaStream_t st)
{
    if (plan_fuses_move(P, width)) return 0;
    if (width < 1) width = 1;
    // one block per 16 KB of a lane's state (four 16-byte vectors per thread and pass), at least one
    // block per lane that could retire at once, at most four blocks per SM
    long long blocks = (long long)((lane_state_bytes(P) + 16383) / 16384);
    if (blocks < (width > 128 ? 128 : width)) blocks = width > 128 ? 128 : width;
    if (blocks > 148 * 4) blocks = 148 * 4;
    if (P.compute_f64) launch_pdl(emit_move_kernel<double>, dim3((unsigned)blocks), dim3(256), 0, st, P);
    else launch_pdl(emit_move_kernel<float>, dim3((unsigned)blocks), dim3(256), 0, st, P);
    return 1;
}
void launch_gather(const Dev &P, void *f, void *g, bool f64, cudaStream_t st)
{
    const int mx = P.n > P.m ? P.n : P.m;
    int gx = (mx + 1023) / 1024; if (gx > 16) gx = 16;
    dim3 grid(P.L + P.W, gx);
    if (f64) gather_kernel<double><<<grid, 256, 0, st>>>(P, (double *)f, (double *)g);
    else gather_kernel<float><<<grid, 256, 0, st>>>(P, (float *)f, (float *)g);
}
void launch_gather_small(const Dev &P, int *depth, int *status, float *rrow, float *rcol, cudaStream_t st)
{
    gather_small_kernel<<<(P.L + 255) / 256, 256, 0, st>>>(P, depth, status, rrow, rcol);
}

// Guard strips: one block per strip, one 32-bit word per thread.  fill = 1 writes the pattern,
// fill = 0 compares and lowers *bad (all ones on entry) to 1 + the index of a damaged strip.
__global__ void __launch_bounds__(GUARD_STRIP_BYTES / 4) guard_strips_kernel(unsigned char *base, const GuardList gl, const int fill, unsigned *bad)
{
    const int strip = blockIdx.x;
    if (strip >= gl.count) return;
    unsigned *w = reinterpret_cast<unsigned *>(base + (size_t)gl.off256[strip] * 256u);
    const unsigned want = 0xA5C3F00Du ^ ((unsigned)strip * 0x9E3779B9u) ^ threadIdx.x;
    if (fill) { w[threadIdx.x] = want; return; }
    if (w[threadIdx.x] != want) atomicMin(bad, (unsigned)strip + 1u);
}
void launch_guard_strips(void *base, const GuardList &gl, bool fill, int *bad, cudaStream_t st)
{
    if (gl.count < 1) return;
    guard_strips_kernel<<<gl.count, GUARD_STRIP_BYTES / 4, 0, st>>>((unsigned char *)base, gl, fill ? 1 : 0, (unsigned *)bad);
}

}  // namespace skb
