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
// A warp holds 16 rows, two to a thread; its four quarters take every fourth column, so a quarter-warp reads one
// shared-memory address.  The partial sums of the quarters are added by xor-shuffles.
//
// What bounds it: the latency of dependent float64 operations (d + 1 and exp2 per pair) at 3.3 warps a scheduler; the float64
// pipe is busy half of the time (52 % at d = 3, 49 % at d = 15).  The next tile's coordinates are fetched into registers
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
