// Float64 pair sums over small dimensions: plan entries pi_ij = 2^(k (f_i + g_j - |x_i - y_j|^2)), k = log2(e) / eps,
// for a block of rows against column tiles in shared memory.  Used by the row residual of given potentials and
// by the application of the plan; both need the sum (or a weighted sum) of a row's entries, not its maximum.
//
// A tile's columns are converted to float64 and scaled once per block (y' = 2 k y, c = k (g - |y|^2)) and then
// serve every row, so a pair costs d multiply-adds, one addition and an exp2.  (|x|^2 + |y|^2 - 2 x.y in float64:
// the products of fp32 coordinates are exact, the rounding error of the argument is 1e-16 of its terms.)
// A warp holds 16 rows, two to a thread; its four quarters take every fourth column, so a quarter-warp reads one
// shared-memory address.  The partial sums of the quarters are added by xor-shuffles.
//
// What bounds it: the float64 pipe (d + 1 operations and exp2 per pair).
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>

namespace skb {

constexpr int P64_TJ = 64;          // columns per tile
constexpr int P64_MAX_D = 32;

// Tile of columns j0 .. j0 + TJ - 1: y' as [DM][TJ], then c.  `load(j, k)` is coordinate k of column j as fp32,
// `pot(j)` its potential.  Columns past the end get c = -inf (entries of zero).
template <int DM, int THREADS, typename Load, typename Pot>
__device__ __forceinline__ void p64_tile(double *sm, const int j0, const int m, const int d, const double k2, Load load, Pot pot)
{
    for (int e = threadIdx.x; e < P64_TJ * DM; e += THREADS) {
        const int jj = e % P64_TJ, k = e / P64_TJ, j = j0 + jj;
        sm[k * P64_TJ + jj] = (j < m && k < d) ? 2.0 * k2 * (double)load(j, k) : 0.0;
    }
    for (int jj = threadIdx.x; jj < P64_TJ; jj += THREADS) {
        const int j = j0 + jj;
        double c = -CUDART_INF;
        if (j < m) {
            double s = 0.0;
            for (int k = 0; k < d; ++k) { const double v = (double)load(j, k); s = fma(v, v, s); }
            c = k2 * (pot(j) - s);
        }
        sm[DM * P64_TJ + jj] = c;
    }
}

}  // namespace skb
