// Float64 pair sums over small dimensions: plan entries pi_ij = 2^(k (f_i + g_j - |x_i - y_j|^2)), k = log2(e) / eps,
// for a block of rows against column tiles in shared memory.  Used by the row residual of given potentials and
// by the application of the plan; both need the sum (or a weighted sum) of a row's entries, not its maximum.
//
// Coordinates are taken relative to the block's first row (`org`; in float64 the difference of two fp32 values is
// exact to 2^-53 of itself), so a common offset of the clouds does not enter.  A tile's columns are converted and
// scaled once per block (y' = 2 k (y - org), c = k (g - |y - org|^2)) and then serve every row, so a pair costs d
// multiply-adds, one addition and an exp2.  The argument's rounding error grows with k |x - org|^2 and
// k |y - org|^2 instead of with the cost itself: a tile in which one of them is above P64_WIDE is summed by
// differences, term by term (the caller's own loop).  Below it the terms are at most 2^17 and the d + 2 roundings
// of an argument add up to less than 2^-32 (d = 32), 2^-8 of the rounding of an fp32 result.
// A warp holds 8 or 16 rows, two or four to a thread; the threads that hold the same rows share the columns out, and their partial
// sums are added by xor-shuffles.
//
// What bounds it: issue and the latency of dependent float64 operations at 3.2 warps a scheduler.  Plan application at d = 3: 17 float64
// operations of 38 instructions a pair, the float64 pipe and the issue slots both half busy.  The next tile's coordinates are fetched into registers
// before the pair loop of the present one (up to eight dimensions: beyond, the rows' own coordinates need the registers).
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>

namespace skb {

constexpr int P64_TJ = 64;          // columns per tile
constexpr int P64_MAX_D = 32;

constexpr double P64_WIDE = 32768.0;

// k |p - org|^2 is too large for the expanded form (NaN and infinity included)
__device__ __forceinline__ bool p64_wide(const double k2, const double sq) { return !(k2 * sq <= P64_WIDE); }

// 2^t for R arguments of every thread of a warp, good to about an ulp: t = k / 32 + r, |r| <= 1/64, 2^(k mod 32 / 32) from a table of
// one entry a thread (`entry`: 2^(lane / 32)), 2^r from its Taylor series (degree 6: truncation 4e-18); the table method of
// P. Tang, ACM TOMS 15, 1989, with the table read by shuffles.  Ten float64 operations, some twenty in CUDA's exp2, which
// takes the arguments that leave [-1022, 1022], except that those below -1080 are zero.  Called by whole warps.
__device__ __forceinline__ double p64_table() { return exp2((double)(threadIdx.x & 31) / 32.0); }
template <int R>
__device__ __forceinline__ void p64_exp2(double (&t)[R], const double entry)
{
    bool odd = false;
#pragma unroll
    for (int r = 0; r < R; ++r) odd = odd || ((unsigned)__double2hiint(t[r]) & 0x7fffffffu) >= 0x408ff000u;         // |t| >= 1022 or NaN
    double v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const double magic = 211106232532992.0;          // 1.5 * 2^47: the sum's low word is k
        const double m = t[r] + magic, x = t[r] - (m - magic);
        const int k = __double2loint(m);
        const int lo = __shfl_sync(0xffffffffu, __double2loint(entry), k), hi = __shfl_sync(0xffffffffu, __double2hiint(entry), k);
        const double s = __hiloint2double(hi + (k >> 5 << 20), lo);
        double q = 1.5403530393381609e-4;                // ln(2)^6 / 720 ...
        q = fma(q, x, 1.3333558146428443e-3);
        q = fma(q, x, 9.6181291076284772e-3);
        q = fma(q, x, 5.5504108664821580e-2);
        q = fma(q, x, 2.4022650695910072e-1);
        q = fma(q, x, 6.9314718055994531e-1);
        v[r] = fma(s, q * x, s);
    }
    if (odd) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const unsigned h = (unsigned)__double2hiint(t[r]);
            if ((h & 0x7fffffffu) >= 0x408ff000u) v[r] = h >= 0xc090e000u && h <= 0xfff00000u ? 0.0 : exp2(t[r]);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) t[r] = v[r];
}

// One entry of a wide tile, from coordinate differences.
template <typename LoadX, typename LoadY>
__device__ __forceinline__ double p64_entry(const int d, const double k2, const double fg, LoadX x, LoadY y)
{
    double c = 0.0;
    for (int k = 0; k < d; ++k) { const double e = (double)x(k) - (double)y(k); c = fma(e, e, c); }
    return exp2((fg - c) * k2);
}

template <int DM> constexpr bool P64_AHEAD = DM <= 8;
// What a thread converts of a tile: every THREADS / TJ-th coordinate of one column, and the column's potential.
template <int DM, int THREADS>
struct P64Part {
    static constexpr int STEP = THREADS / P64_TJ, NK = (DM + STEP - 1) / STEP;
    float c[NK];
    double pot;
};
// `load(j, k)` is coordinate k of column j as fp32, `pot(j)` its potential.
template <int DM, int THREADS, typename Load, typename Pot>
__device__ __forceinline__ void p64_fetch(P64Part<DM, THREADS> &p, const int j0, const int m, const int d, Load load, Pot pot)
{
    const int j = j0 + (int)threadIdx.x % P64_TJ;
#pragma unroll
    for (int e = 0; e < P64Part<DM, THREADS>::NK; ++e) {
        const int k = e * P64Part<DM, THREADS>::STEP + (int)threadIdx.x / P64_TJ;
        p.c[e] = j < m && k < d ? load(j, k) : 0.f;
    }
    p.pot = threadIdx.x < P64_TJ && j < m ? pot(j) : 0.0;
}
// Tile of columns j0 .. j0 + TJ - 1: y' as [DM][TJ], then c, then scratch.  Columns past the end get c = -inf (entries
// of zero).  A thread keeps the sum of its coordinates' squares, so the norms cost no second pass over them.
// Contains a barrier, needs one after it.  True if a column of this thread is wide.
template <int DM, int THREADS> constexpr int P64_TILE = (DM + 1) * P64_TJ + THREADS;       // doubles
template <int DM, int THREADS>
__device__ __forceinline__ bool p64_tile(double *sm, const double *org, const int j0, const int m, const int d, const double k2, const P64Part<DM, THREADS> &p)
{
    static_assert(THREADS % P64_TJ == 0, "whole groups of threads per coordinate");
    double *part = sm + (DM + 1) * P64_TJ;
    const int jj = threadIdx.x % P64_TJ, j = j0 + jj;
    double s = 0.0;
#pragma unroll
    for (int e = 0; e < P64Part<DM, THREADS>::NK; ++e) {
        const int k = e * P64Part<DM, THREADS>::STEP + (int)threadIdx.x / P64_TJ;
        const double v = j < m && k < d ? (double)p.c[e] - org[k] : 0.0;
        if (DM % P64Part<DM, THREADS>::STEP == 0 || k < DM) sm[k * P64_TJ + jj] = 2.0 * k2 * v;
        s = fma(v, v, s);
    }
    part[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x >= P64_TJ) return false;
#pragma unroll
    for (int h = 1; h < P64Part<DM, THREADS>::STEP; ++h) s += part[threadIdx.x + h * P64_TJ];
    sm[DM * P64_TJ + jj] = j < m ? k2 * (p.pot - s) : -CUDART_INF;
    return j < m && p64_wide(k2, s);
}

}  // namespace skb
