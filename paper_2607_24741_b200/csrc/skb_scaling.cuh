// Lanes whose kernel matrix stays on chip: formed once per launch, kept in registers or in tensor memory.  Lanes of mixed and,
// under the automatic choice, fp32 arithmetic (exponents from float64 coordinates) and deep lanes (from stored dot products).
//
// With potentials (phi0, gam0) absorbed into the matrix,
//     K_ij = 2^(phi0_i + gam0_j - s C_ij) / (a_i b_j),      phi = phi0 + log2 u,   gam = gam0 + log2 v,
// the two legs of Eq. 3 are the scaling updates
//     u_i = 1 / sum_j K_ij b_j v_j,        v_j = 1 / sum_i K_ij a_i u_i,
// one fp32 multiply-add per pair and leg instead of a d-term float64 distance and an exponential.
// Exponents are float64 (rounded once, after the integer part has been split off), K is fp32, sums are
// fp32 over at most 32 terms and float64 beyond, u, v and the potentials are float64: what the
// log-domain kernels of the mixed arithmetic hold in 32 and in 64 bits is held so here.
//
// Range.  fp32 K has no entries below 2^-124.  An update that would take a u or v out of 2^+-45 is not
// taken: the leg is done again in the log domain (log_rows / log_cols: per-row or per-column maximum,
// then the sum, both passes over the distances), after which the new potentials are absorbed and K is
// formed anew.  A lane whose u or v has left 2^+-30 after a cycle is absorbed too.  So what K does not hold is
// below 2^-124 sum_j b_j v_j <= 2^(-124 + 30) of a row sum 1 / u_i >= 2^-45, and below 2^-124 sum_i a_i u_i <=
// 2^(-124 + 45) of a column sum 1 / v_j >= 2^-45: at most 2^-34 of the sum, whatever the weights (K divided by both
// of them: with a_i alone the column bound would carry a factor a_i / b_j).  The operands a u and b v stay normal
// fp32 numbers, and K = P / (a_i b_j) <= 1 / a_i within its range, while no weight is below 2^-80: a lane with a
// smaller one (SC_NO_MATRIX, found when its layout is written) stays in the log domain for all of its cycles.
// A cold lane whose entries before any potential are above 2^-SC_COLD_BITS, with weights from SC_COLD_WEIGHT on, starts with zero
// potentials absorbed; the first cycle of the others, and of a warm start, is a log-domain cycle.  All of these decisions are taken per lane from the lane's own values, and K is a function of
// (phi0, gam0) alone, which are part of the lane's state: a lane's bits depend neither on how its cycles
// were shared out among launches nor on the mode.
//
// Work layout.  A cluster of NC blocks owns the lane; a block of NW warps owns NW * RW rows, a warp RW of
// them, and a thread the entries of its warp's rows in CL columns: E = RW * CL values, in registers or, where a
// lane would otherwise need several blocks, in tensor memory, which holds as much again as the register file and is
// read as fast as the multiply-adds go (256 words of 256 threads: 770 clk alone, 1020 with one packed
// multiply-add per pair of words, 960 for the multiply-adds alone).  Row
// sums are reduced by a halving exchange over the 32 threads; column sums go through shared memory and, where a lane has
// several blocks, by bulk copies between their shared memories that report to an mbarrier of the receiver.  Every block forms all
// of v by itself.  A cycle takes two block barriers, four in a cluster, and one more in the blocks that add up a share
// of the columns (two-step exchange); there is no cluster barrier in it.  The column sums of the next state are formed before
// the row residual has been decided on, and dropped where the lane leaves.
//
// What bounds it: the chain of dependent steps of a cycle (two rounds of multiply-adds, the exchange of row
// sums, two float64 reciprocals, the column parts through shared memory, the exchange between blocks), not a
// unit: the multiply-adds of a 256 x 256 lane are 256 clk of packed fp32 per scheduler, a cycle is 3700.
// Measured per cycle in long launches: 8 lanes of 64 x 64, d = 2: 0.75 us; 96 of 100 x 77: 1.2 us; one lane of
// 256 x 256, d = 8, K in registers of a cluster of four blocks -> in tensor memory of one block: 1.7 -> 1.5 us; 148 of
// them 5.4 -> 1.55 us (four blocks of a cluster per SM waited for each other's exchanges); all 1024 of the sweep workload
// 27 -> 10 us, 24 -> 10.9 ms per solve at tol 1e-3.  512 x 512, clusters of eight blocks, registers -> of four, tensor memory:
// 5.6 -> 3.5 us.  16 warps of 16 rows instead of 8 of 32: 2.2 us.
// Forming K costs 10 to 35 us per wave of a launch (latency: two warps per scheduler), so a caller that steps one cycle per call
// pays mostly for that: 28 us on one lane of 256 x 256, 156 us on 1024; 290 us on 256 lanes of 512 x 512, d = 15, and 295 us on 64 of
// 1024 x 1024, d = 512, where two streamed legs take 120 and 130 us.  From three to four cycles per call on it is the faster way
// (362 and 417 against 481 and 519 us), at 64 by 3 to 4 times.  The formation is a loop in every variant:
// unrolled, as it has to be to index registers, it was 100 KB of instructions that ran once per launch, and
// fetching them took longer than running them (256 x 256: 43 -> 25 us per call; 96 lanes of 100 x 77: 30 -> 20 us).
// The exchange between blocks: a cluster barrier 2.9 us a cycle of 256 x 256 in four blocks, remote stores that report to a
// barrier of the receiver 2.4; now bulk copies, see SC_WAIT_CLOCKS.  128-thread blocks (two of different lanes per SM)
// instead of 256: 58 -> 47 us per cycle of 1024 lanes, together with the rows' order that spares the selects of the exchange.
#pragma once
#include "skb_update.cuh"
#include "skb_host.h"
#include "skb_tmem.cuh"

namespace skb {

constexpr int SC_TAKE = 45, SC_KEEP = 30;               // bands of log2 u and log2 v: update taken / K kept
constexpr int SC_BAD = 1, SC_DRIFT = 2, SC_NF = 4, SC_LEAVE = 8;

// 2^arg for a float64 argument: integer part split off in float64, the remainder (|.| <= 1/2) rounded
// to fp32 and put through the Taylor series of e^(x ln 2) (degree 7: truncation 5e-9), so the result is
// good to about an ulp whatever the size of the argument.  Zero below 2^-124, 2^100 from there on.
// WORDS: the range tested on the argument's high word, by integers, instead of by two float64 comparisons and
// selects.  Same results; the launches of one leg are faster so, the launches of whole cycles slower (96 lanes of
// 100 x 77: 4.1 -> 5.1 ms a solve: it changes what the cycle loop keeps in registers).
template <bool WORDS = false>
__device__ __forceinline__ float exp2_split(const double arg)
{
    const double x = WORDS ? arg : fmin(fmax(arg, -200.0), 100.0);
    const double magic = 6755399441055744.0;             // 1.5 * 2^52: the sum's low word is the integer part
    const double t = x + magic;
    const int ni = __double2loint(t);
    const float f = (float)(x - (t - magic));
    float q = 1.5252734e-5f;
    q = fmaf(q, f, 1.5403530e-4f);
    q = fmaf(q, f, 1.3333558e-3f);
    q = fmaf(q, f, 9.6181291e-3f);
    q = fmaf(q, f, 5.5504109e-2f);
    q = fmaf(q, f, 2.4022651e-1f);
    q = fmaf(q, f, 6.9314718e-1f);
    const float p = fmaf(q, f, 1.0f);
    const float r = __int_as_float(__float_as_int(p) + (ni << 23));
    if constexpr (!WORDS) return ni >= -124 ? r : 0.0f;
    else {
        const int hi = __double2hiint(arg);
        const float z = (unsigned)hi <= 0xc05f4000u && ni >= -124 ? r : 0.0f;         // -125
        return hi < 0x40590000 ? z : 0x1p100f;                                        // 100
    }
}

__device__ __forceinline__ u64 mul2(u64 a, u64 b)
{
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// fp32 -> float64 and back (towards zero) by integers, for positive normal fp32 numbers: the conversion unit is slow and
// far away.  Zero and subnormal numbers become something below 2^-125, infinities and NaN something from 2^128 on.
__device__ __forceinline__ double widen(const float x)
{
    const unsigned u = __float_as_uint(x);
    return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}
__device__ __forceinline__ float narrow(const double x)
{
    return __uint_as_float(__funnelshift_l((unsigned)__double2loint(x), (unsigned)__double2hiint(x) - 0x38000000u, 3));
}
// 1 / s to float64 accuracy: a third-order step on the fp32 approximation (relative error 2^-23, cubed).  For s outside
// 2^+-SC_SUMS the result is meaningless: the caller asks out_of_band() about s too.
constexpr int SC_SUMS = 100;
__device__ __forceinline__ double rcp64(const double s)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(narrow(s)));
    const double x = widen(r), e = fma(-s, x, 1.0);
    return fma(x * e, e, fma(x, e, x));
}
// x (u or v) is not within 2^+-BAND: negative, zero, infinite and NaN included
template <int BAND>
__device__ __forceinline__ bool out_of_band(const double x)
{
    return ((unsigned)__double2hiint(x) >> 20) - (unsigned)(1023 - BAND) >= (unsigned)(2 * BAND);
}

// TM: a thread's E values of K are in tensor memory, which is used as storage of its own (32x32b accesses: a warp's
// lane and column range belong to the same threads throughout), instead of in registers.
enum ScalingSource : int { SRC_F64, SRC_DOTS };          // float64 coordinates; the stored dot products of deep lanes
template <int NW_, int CL_, int RW_, bool TM_ = false>
struct ScalingShape {
    static constexpr int NW = NW_, CL = CL_, RW = RW_;
    static constexpr bool TM = TM_;
    static constexpr int TM_COLS = TM ? CL * RW * NW / 4 : 32;       // tensor memory columns of a block
    static constexpr int THREADS = 32 * NW, COLS = 32 * CL, RB = NW * RW;
    static constexpr int NQ = (COLS + THREADS - 1) / THREADS;        // columns a thread owns in the column steps
    static constexpr int G = (CL >= 16 || CL * RW == 64) ? 2 : 4;    // rows whose distances are formed together
    static constexpr int GW = G * CL;                                // ... and their entries of K
    // Wide lanes exchange column sums in two steps: every block adds up the parts of a share of the columns and sends the
    // totals to the others (all parts to all blocks, as the narrower ones do it, would be 128 KB a block and cycle).
    static constexpr bool TWO_STEP = CL >= 32;
    static constexpr int RANKS = TWO_STEP ? 16 : MAX_CLUSTER_RANKS;  // blocks of a cluster at most
    static constexpr int MIN_BLOCKS = TWO_STEP ? 4 : 1;
    // log2 of the blocks that add columns up
    __host__ __device__ static constexpr int owner_bits(int nc) { return nc >= 16 ? 4 : (nc >= 8 ? 3 : 2); }
    static constexpr int SHARE = 32 / RW;                            // threads that end up with the same row's sum
    // K in registers: 255 of them a thread for the narrow tiles, too, which spill in every cycle with 128 although the entries
    // are 32 or 64 of those (drain of lanes of 64 x 64, d = 2, 128 -> 255: one lane 573 -> 460 us, 256 602 -> 493, 1200
    // 1054 -> 736; of 100 x 60 870 -> 674, 993 -> 750, 2169 -> 1681; 168 registers lie between).
    // K in 256 columns of tensor memory, in 32 registers, or in 64 of clusters of two columns a thread: two kernels, blocks() an SM with 128
    // registers a thread and half as many that do not spill (ROOMY); cycles_kernel has the rule.
    static constexpr int blocks(bool cluster) { return TM ? 512 / TM_COLS : (CL * RW == 32 || (cluster && CL == 2) ? 512 : 256) / THREADS; }
    static constexpr bool has_roomy(bool cluster) { return blocks(cluster) * THREADS > 256; }
    static constexpr int ROOMY_BLOCKS = TM ? 1 : 256 / THREADS;
    // Launches of one leg do not hold K: 128 registers.  Lanes of 512 columns and more, whose G rows of distances are 64 registers
    // and up, form their entries in a loop and take 255: unrolled, the entries' instructions run once and are
    // fetched for longer, and at 128 registers they spill (f-leg of 64 lanes of 1024 x 1024 1224 -> 310 us, of 256 lanes of
    // 512 x 512, d = 15, 344 -> 298 us; narrower lanes are faster unrolled: 1024 of 256 x 256 119 against 150 us).
    static constexpr bool LEG_ROLLED = CL >= 16;
    static constexpr int LEG_BLOCKS = (LEG_ROLLED ? 256 : 512) / THREADS;
    static constexpr int FP32_COLS = CL <= 4 ? 8 : 32;               // columns a row's sum holds before it becomes float64
    static constexpr int FP32_WARPS = CL >= 8 && RW <= 16 ? 2 : 1;   // warps' column parts added in fp32 (at most 32 rows)
    static_assert(RW >= 8 && RW <= 32 && CL >= 2 && CL <= 32, "unsupported tile");
    static_assert(!TM || (NW % 4 == 0 && GW % 32 == 0 && TM_COLS <= 512 && 512 / TM_COLS <= 4), "unsupported tile in tensor memory");
    static_assert(!TWO_STEP || COLS == 4 * THREADS, "the two-step exchange has one thread to a column where four blocks share them");
    // dynamic shared memory: column parts of every warp; the exchange buffers: what goes out, what comes in (TWO_STEP: parts
    // of the own columns, totals of all; totals that go out); where K is in registers, the words it is formed in
    static constexpr size_t PARTS = sizeof(double) * NW * COLS;
    __host__ __device__ static constexpr size_t exchange(int nc)
    {
        return sizeof(double) * 2 * (COLS + (TWO_STEP ? (size_t)nc * (COLS >> owner_bits(nc)) + COLS + THREADS : (size_t)nc * COLS));
    }
    static size_t smem(int nc) { return PARTS + exchange(nc) + (TM ? 0 : sizeof(float) * (size_t)RW * CL * THREADS); }
};

// What the exponents of a lane are formed from.
struct ScalingOperand {
    const double *xs, *ys;                               // SRC_F64: scaled coordinates, dimension-major
    const float *dots;                                   // SRC_DOTS: x_i . y_j of the raw points, rows of mp
    double two_s;
    int np, mp, d;
};
// acc += x_i . y_j of the scaled coordinates for G consecutive rows and this thread's CL columns
// (2 lane, 2 lane + 1, + 64, ...).  Rows and columns past the end read row / column 0; their results are
// masked by the additive terms.
template <int SRC, int CL, int G>
__device__ __forceinline__ void dot_tile(const ScalingOperand &o, const int i0, const int lane, double (&acc)[G][CL])
{
    const int first = i0 < o.np ? i0 : 0;
    int yo[CL / 2];
#pragma unroll
    for (int h = 0; h < CL / 2; ++h) { const int j = h * 64 + 2 * lane; yo[h] = j < o.mp ? j : 0; }
    if constexpr (SRC == SRC_DOTS) {
        const float *row = o.dots + (size_t)first * o.mp;
        float2 t[G][CL / 2];
#pragma unroll
        for (int r = 0; r < G; ++r)
#pragma unroll
            for (int h = 0; h < CL / 2; ++h) t[r][h] = *reinterpret_cast<const float2 *>(row + (size_t)r * o.mp + yo[h]);
#pragma unroll
        for (int r = 0; r < G; ++r)
#pragma unroll
            for (int h = 0; h < CL / 2; ++h) {
                acc[r][2 * h] = fma(o.two_s, (double)t[r][h].x, acc[r][2 * h]);
                acc[r][2 * h + 1] = fma(o.two_s, (double)t[r][h].y, acc[r][2 * h + 1]);
            }
    } else {
        const double *xp = o.xs + first;
#pragma unroll 1
        for (int k = 0; k < o.d; ++k) {
            double x[G];
#pragma unroll
            for (int r = 0; r < G; r += 2) {
                const double2 t = *reinterpret_cast<const double2 *>(xp + (size_t)k * o.np + r);
                x[r] = t.x; x[r + 1] = t.y;
            }
#pragma unroll
            for (int h = 0; h < CL / 2; ++h) {
                const double2 y = *reinterpret_cast<const double2 *>(o.ys + (size_t)k * o.mp + yo[h]);
#pragma unroll
                for (int r = 0; r < G; ++r) {
                    acc[r][2 * h] = fma(x[r], y.x, acc[r][2 * h]);
                    acc[r][2 * h + 1] = fma(x[r], y.y, acc[r][2 * h + 1]);
                }
            }
        }
    }
}

// Halving exchange: RW per-thread partial sums (one per row of the warp) -> the sum over the 32 threads of
// row lane / SHARE.  Sums are fp32 while they hold at most LIM columns, float64 from there on.
// PERM: threads hold the rows in an order of their own - local row r is row r ^ (lane / SHARE & ~3) - in
// which the half to keep always comes first, so that the wide steps need no selects.
template <int CL, int LIM, bool PERM, int OFF, int CNT, typename V>
__device__ __forceinline__ double row_exchange(V (&s)[CNT], const int lane)
{
    constexpr int COLS_IN = CL * (32 / (2 * OFF));                 // columns a partial sum holds already
    if constexpr (sizeof(V) == 4 && COLS_IN >= LIM) {
        double t[CNT];
#pragma unroll
        for (int r = 0; r < CNT; ++r) t[r] = widen(s[r]);
        return row_exchange<CL, LIM, PERM, OFF, CNT, double>(t, lane);
    } else {
        if constexpr (CNT > 1) {
            V h[CNT / 2];
            const bool up = (lane & OFF) != 0;
#pragma unroll
            for (int r = 0; r < CNT / 2; ++r) {
                const bool swap = !(PERM && CNT / 2 >= 4) && up;
                const V keep = swap ? s[r + CNT / 2] : s[r], give = swap ? s[r] : s[r + CNT / 2];
                h[r] = keep + __shfl_xor_sync(0xffffffffu, give, OFF);
            }
            if constexpr (OFF == 1) return (double)h[0];
            else return row_exchange<CL, LIM, PERM, OFF / 2, CNT / 2, V>(h, lane);
        } else {
            V h[1] = {s[0] + __shfl_xor_sync(0xffffffffu, s[0], OFF)};
            if constexpr (OFF == 1) return (double)h[0];
            else return row_exchange<CL, LIM, PERM, OFF / 2, 1, V>(h, lane);
        }
    }
}

// Log-domain row step for the RW rows of a warp: integer-valued reference M >= every argument - 1 and
// S = sum_j 2^(arg_ij - M), arg_ij = colB_j + x_i . y_j, of row lane / SHARE.  Two passes over the
// distances; runs in the first cycle of lanes that do not start absorbed and where an update leaves the range of K.
template <int SRC, int NW, int CL, int RW>
__device__ __noinline__ void log_rows(const ScalingOperand &o, const int i0,
                                      const double *colB, double *S, double *M)
{
    typedef ScalingShape<NW, CL, RW> L;
    const int lane = threadIdx.x & 31;
    double mine = 0.0;
    float part[RW];                                      // (indexed in a rolled loop, so on the stack)
#pragma unroll 1
    for (int g = 0; g < RW / L::G; ++g) {
        double acc[L::G][CL], mr[L::G];
#pragma unroll
        for (int r = 0; r < L::G; ++r)
#pragma unroll
            for (int e = 0; e < CL; ++e) acc[r][e] = colB[(e / 2) * 64 + 2 * lane + (e & 1)];
        dot_tile<SRC, CL, L::G>(o, i0 + g * L::G, lane, acc);
#pragma unroll
        for (int r = 0; r < L::G; ++r) {
            double t = -1.0e300;
#pragma unroll
            for (int e = 0; e < CL; ++e) t = fmax(t, acc[r][e]);
            for (int off = 16; off > 0; off >>= 1) t = fmax(t, __shfl_xor_sync(0xffffffffu, t, off));
            mr[r] = ceil(t);
            if (lane / L::SHARE == g * L::G + r) mine = mr[r];
            float s = 0.f;
#pragma unroll
            for (int e = 0; e < CL; ++e) s += exp2_split(acc[r][e] - mr[r]);
            part[g * L::G + r] = s;
        }
    }
    *S = row_exchange<CL, L::FP32_COLS, false, 16, RW, float>(part, lane);
    *M = mine;
}

// Column counterpart of log_rows, first half: the maximum of rowA_i + x_i . y_j over the warp's rows.
template <int SRC, int NW, int CL, int RW>
__device__ __noinline__ void log_cols_max(const ScalingOperand &o, const int i0,
                                          const double *rowA, double *out)
{
    typedef ScalingShape<NW, CL, RW> L;
    const int lane = threadIdx.x & 31;
    double mc[CL];
#pragma unroll
    for (int e = 0; e < CL; ++e) mc[e] = -1.0e300;
#pragma unroll 1
    for (int g = 0; g < RW / L::G; ++g) {
        double acc[L::G][CL];
#pragma unroll
        for (int r = 0; r < L::G; ++r)
#pragma unroll
            for (int e = 0; e < CL; ++e) acc[r][e] = rowA[g * L::G + r];
        dot_tile<SRC, CL, L::G>(o, i0 + g * L::G, lane, acc);
#pragma unroll
        for (int r = 0; r < L::G; ++r)
#pragma unroll
            for (int e = 0; e < CL; ++e) mc[e] = fmax(mc[e], acc[r][e]);
    }
#pragma unroll
    for (int e = 0; e < CL; ++e) out[(e / 2) * 64 + 2 * lane + (e & 1)] = mc[e];
}
// ... second half: sums of 2^(rowA_i + x_i . y_j - M_j) over the warp's rows.
template <int SRC, int NW, int CL, int RW>
__device__ __noinline__ void log_cols_sum(const ScalingOperand &o, const int i0,
                                          const double *rowA, const double *colM, float *out)
{
    typedef ScalingShape<NW, CL, RW> L;
    const int lane = threadIdx.x & 31;
    float s[CL];
#pragma unroll
    for (int e = 0; e < CL; ++e) s[e] = 0.f;
#pragma unroll 1
    for (int g = 0; g < RW / L::G; ++g) {
        double acc[L::G][CL];
#pragma unroll
        for (int r = 0; r < L::G; ++r)
#pragma unroll
            for (int e = 0; e < CL; ++e) acc[r][e] = rowA[g * L::G + r] - colM[(e / 2) * 64 + 2 * lane + (e & 1)];
        dot_tile<SRC, CL, L::G>(o, i0 + g * L::G, lane, acc);
#pragma unroll
        for (int r = 0; r < L::G; ++r)
#pragma unroll
            for (int e = 0; e < CL; ++e) s[e] += exp2_split(acc[r][e]);
    }
#pragma unroll
    for (int e = 0; e < CL; ++e) out[(e / 2) * 64 + 2 * lane + (e & 1)] = s[e];
}

// Float64 re-evaluation of a block's rows (guard band); out of line so that its registers stay out of the
// cycle loop's allocation.
template <int NW>
__device__ __noinline__ unsigned long long scaling_reeval(const Dev *P, const int slot, const int r0, const int r1, const double *pot,
                                                          unsigned long long *red, int *bad)
{
    // direct_rows_block, four rows of a warp side by side: the same terms in the same order, with the latencies of
    // their distances, exponentials and shuffles shared (one row after the other 60 us a lane of 100 x 77)
    constexpr int R = 4, U = 2;
    const Dev &D = *P;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double s = D.scale[slot];
    const double *gam = D.gam + (size_t)slot * D.mp;
    const void *xl = (const char *)D.xraw + (size_t)slot * D.xraw_stride, *yl = (const char *)D.yraw + (size_t)slot * D.yraw_stride;
    unsigned long long part = 0ull;
    int nf = 0;
    for (int i0 = r0 + warp; i0 < r1; i0 += R * NW) {
        int row[R];
        double phi[R], sum[R];
#pragma unroll
        for (int r = 0; r < R; ++r) { row[r] = min(i0 + r * NW, r1 - 1); phi[r] = pot[row[r] - r0]; sum[r] = 0.0; }
        for (int j0 = lane; j0 < D.m; j0 += 32 * U) {
            double c[R][U], gj[U];
            size_t yb[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int j = j0 + 32 * u < D.m ? j0 + 32 * u : D.m - 1;
                yb[u] = (size_t)j * D.d;
                gj[u] = __ldcg(gam + j);
#pragma unroll
                for (int r = 0; r < R; ++r) c[r][u] = 0.0;
            }
            for (int k = 0; k < D.d; ++k) {
                double y[U];
#pragma unroll
                for (int u = 0; u < U; ++u) y[u] = (double)load_raw(D, yl, yb[u] + k);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const double x = (double)load_raw(D, xl, (size_t)row[r] * D.d + k);
#pragma unroll
                    for (int u = 0; u < U; ++u) { const double t = x - y[u]; c[r][u] = fma(t, t, c[r][u]); }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const double v = exp2(phi[r] + gj[u] - s * c[r][u]);
                    sum[r] += j0 + 32 * u < D.m ? v : 0.0;
                }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int r = 0; r < R; ++r) sum[r] += __shfl_xor_sync(0xffffffffu, sum[r], off);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (i0 + r * NW >= r1) continue;
            const double term = fabs(sum[r] - D.wa[(size_t)slot * D.np + row[r]]);
            if (!isfinite(term)) nf = 1;
            else if (lane == 0) part += __double2ull_rn(fmin(term, RSUM_ROW_MAX) * RSUM_SCALE);
        }
    }
    nf = __syncthreads_or(nf);
    if (lane == 0) red[warp] = part;
    __syncthreads();
    unsigned long long all = 0ull;
    if (threadIdx.x == 0) for (int w = 0; w < NW; ++w) all += red[w];
    __syncthreads();
    *bad = nf;
    return all;
}

// Exchange between the blocks of a cluster without a cluster barrier: bulk copies from shared memory to shared memory
// that report their bytes to a barrier of the receiver, which waits on it.  (A cluster barrier's release waits until
// all of the block's remote stores have been acknowledged, and remote stores of 16 bytes a thread go out one by one.
// A cycle of 24 lanes of 500 x 333, four blocks: 4.2 -> 3.3 us; sent by all warps, of 64 lanes of 1024 x 1024, sixteen
// blocks: 2.9 -> 2.4 us per four lanes.)  The wait is bounded like every wait of this library.
constexpr long long SC_WAIT_CLOCKS = 2000000000LL;
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned peer_addr(const unsigned a, const unsigned rank)
{
    unsigned x;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(x) : "r"(a), "r"(rank));
    return x;
}
// `bytes` (a multiple of 16) of this block's shared memory into a peer's, reported to the peer's barrier
__device__ __forceinline__ void copy_to_peer(const void *dst, const void *src, const unsigned bytes, const void *bar, const unsigned rank)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(peer_addr(smem_addr(dst), rank)), "r"(smem_addr(src)), "r"(bytes), "r"(peer_addr(smem_addr(bar), rank)) : "memory");
}
__device__ __forceinline__ void expect_bytes(const void *bar, const unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// this thread's writes to shared memory become visible to copies issued after the next block barrier
__device__ __forceinline__ void fence_for_copies() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ bool bar_try_wait(const unsigned a, const unsigned parity)
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(a), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool bar_wait(const unsigned a, const unsigned parity)
{
    if (bar_try_wait(a, parity)) return true;
    const long long t0 = clock64();
    while (!bar_try_wait(a, parity))
        if (clock64() - t0 > SC_WAIT_CLOCKS) return false;
    return true;
}

template <bool CLU>
__device__ __forceinline__ void scaling_barrier()
{
    if constexpr (CLU) cluster_sync_all();
    else __syncthreads();
}

// KIND = SC_CYCLES: up to `cycles` whole cycles of every lane.  SC_CATCH_UP: the passed lanes of a STATIC batch go on to
// the cycle that the others have reached (plan_static_kernel).  SC_LEG: leg = LEG_F / LEG_V / LEG_G as a launch of its
// own, for phase timing and dry runs: an entry of K is formed where it is used, with the same bits, and never kept.
// CLU = 0: a lane has one block (its rows fit), and nothing of the cluster machinery is in the way.
// ROOMY: with 255 registers a thread where there is a kernel with 128, too (same arithmetic).
template <int SRC, int NW, int CL, int RW, bool CLU, bool TMEM, int KIND, bool ROOMY = false>
__global__ void __launch_bounds__(32 * NW, (KIND == SC_LEG ? ScalingShape<NW, CL, RW, TMEM>::LEG_BLOCKS : (ROOMY ? ScalingShape<NW, CL, RW, TMEM>::ROOMY_BLOCKS : ScalingShape<NW, CL, RW, TMEM>::blocks(CLU))))
scaling_kernel(const __grid_constant__ Dev P, const int leg, const int cycles)
{
    typedef ScalingShape<NW, CL, RW, TMEM> L;
    constexpr bool LEG = KIND == SC_LEG, ROLLED = LEG && L::LEG_ROLLED, catch_up = KIND == SC_CATCH_UP, TM = TMEM && !LEG;
    constexpr int THREADS = L::THREADS, COLS = L::COLS, RB = L::RB, NQ = L::NQ, SHARE = L::SHARE;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long swr[NW];
    __shared__ __align__(16) unsigned long long sw[2][NW];          // ... what this block sends
    __shared__ __align__(16) unsigned long long xw[2][L::RANKS * NW];  // residual part and flags of every warp of the cluster
    __shared__ int sflag;                                // column flags
    // Two words, because no block barrier lies between the last read of the one and the first write of the other within a
    // cycle: a warp that reads late would take a column that has left the band, found by a warp ahead of it, for a wait that ran out.
    __shared__ volatile int vflag;                       // a column has left the band
    __shared__ volatile int wflag;                       // a wait ran out (never cleared)
    __shared__ __align__(16) double colB[COLS], rowA[RB];       // additive terms of columns / own rows
    __shared__ __align__(16) float vs[COLS];             // b v of all columns
    __shared__ __align__(16) float2 uas[RB];             // a u of own rows, in both halves
    __shared__ __align__(8) unsigned long long xbar[2];  // arrival of an exchange's stores, one per buffer
    __shared__ __align__(8) unsigned long long tbar[2];  // ... and of its totals (TWO_STEP)
    __shared__ uint32_t tm_holder;

    pdl_enter();
    const Ctl c = *P.ctl;
    const int slot = P.order ? P.order[blockIdx.y] : (int)blockIdx.y;
    // every exit here is taken by the whole cluster
    const int lane_id = P.lane_id[slot < c.n_phys ? slot : 0];
    if ((c.done && !catch_up) || slot >= c.n_phys) return;
    if (P.early_exit && P.state[slot] != 0) return;
    int par = c.parity, k = c.cycle, todo = cycles;
    bool just_passed = false;
    if constexpr (LEG) {
        if (leg != LEG_V && c.static_final) return;
        if (leg == LEG_V && !(c.static_final || lane_needs_column_check(P, c, slot))) return;
    } else if (P.mode == MODE_STATIC) {
        if ((P.state[slot] != 0) != catch_up) return;
        if (catch_up) {
            if (P.emitted[lane_id]) return;
            const int left = P.ret_at[slot];             // passed in the launch just run, or before it
            k = left > 0 ? left - 1 : c.prev_cycle;
            todo = c.cycle - k;
            just_passed = left > 0 && todo == 0;         // at the state that is the last one: its audit stands
            par = c.parity ^ (todo & 1);
        }
    }
    const bool closing = catch_up && c.static_final;     // every lane has passed: this one's outputs are written at c.cycle
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = CLU ? (int)blockIdx.x : 0, NC = CLU ? (int)gridDim.x : 1;
    double *partd = reinterpret_cast<double *>(smem_raw);                // column parts of every warp
    float *partf = reinterpret_cast<float *>(partd);
    // TWO_STEP: the first `own` blocks add up `share` columns each, 2^tpb threads to a column
    const int ob = L::owner_bits(NC), own = 1 << ob, share = COLS >> ob, tpb = ob - 2;
    double *xbuf = reinterpret_cast<double *>(smem_raw + L::PARTS);      // [2][NC][COLS] column parts of every block; TWO_STEP: [2][NC][share]
    double *tbuf = xbuf + (size_t)2 * NC * share;                        // TWO_STEP: [2][COLS] totals
    double *sbuf = L::TWO_STEP ? tbuf + 2 * COLS : xbuf + (size_t)2 * NC * COLS;         // [2][COLS] what this block sends
    double *ubuf = sbuf + 2 * COLS;                                      // TWO_STEP: [2][THREADS] totals it sends
    u64 *kstage = reinterpret_cast<u64 *>(smem_raw + L::PARTS + L::exchange(NC));   // K on its way into the registers
    int xch = 0;                                                         // exchanges so far: their buffer alternates

    ScalingOperand o;
    o.np = P.np; o.mp = P.mp; o.d = P.d;
    if constexpr (SRC == SRC_DOTS) { o.dots = P.dots + (size_t)slot * P.np * P.mp; o.two_s = 2.0 * P.scale[slot]; }
    else {
        o.xs = reinterpret_cast<const double *>(P.xs) + (size_t)slot * P.DP * P.np;
        o.ys = reinterpret_cast<const double *>(P.ys) + (size_t)slot * P.DP * P.mp;
    }
    const int i0 = b * RB + warp * RW;                   // first row of this warp
    const int lr = warp * RW + lane / SHARE;             // this thread's row (SHARE threads hold the same one)
    const int perm = lane / SHARE & ~3;                  // order of the rows in K (see row_exchange)
    const int i = b * RB + lr;
    const bool rok = i < P.n, rown = rok && lane % SHARE == 0;
    const int j0 = tid * NQ;                             // this thread's columns in the column steps: NQ adjacent ones
    const bool cown = COLS >= THREADS || tid < COLS;
    const size_t ro = (size_t)slot * P.np + (rok ? i : 0), co = (size_t)slot * P.mp;
    const int start = P.start[slot];
    const double inv_s = 1.0 / P.scale[slot];
    const double a_i = rok ? P.wa[ro] : 0.0, a_fix = a_i * RSUM_SCALE;
    bool frozen = P.mode == MODE_MASKED && P.state[slot] != 0;

    // state: `us`, `vsd` are u and v while `ab` (potentials absorbed into K), the potentials themselves before
    bool ab = P.absorbed[slot] > 0;
    const bool no_matrix = P.absorbed[slot] < 0;
    // (the absorbed potentials stay in registers: every block holds all columns', and global memory gets them
    // back only at the end, when no block of the cluster can still be reading)
    double us = ab ? 1.0 : 0.0, phi0 = 0.0, vsd[NQ], gam0[NQ], bq[NQ];
    if (rok) { us = ab ? P.uu[par][ro] : P.phi[par][ro]; phi0 = P.phi0[ro]; }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int j = j0 + q;
        const bool has = cown && j < P.m;
        vsd[q] = has ? (ab ? P.vv[co + j] : P.gam[co + j]) : 0.0;
        gam0[q] = has ? P.gam0[co + j] : 0.0;
        bq[q] = has ? P.wb[co + j] : 0.0;
    }
    // residual totals above this (fixed point) can neither pass the screen nor lie in the guard band
    unsigned long long near_tot;
    {
        double t = P.tol_screen;
        if (P.guard > 0.0) {
            t = fmax(t, P.tol_screen + fmax(P.guard * P.tol_screen, GUARD_ABS_FLOOR));
            t = fmax(t, P.tol_stop + fmax(P.guard * P.tol_stop, GUARD_ABS_FLOOR));
        }
        near_tot = (unsigned long long)fmin(t * 1.000001 * RSUM_SCALE, 1.0e18) + 2ull;
    }
    if (tid == 0) {
        sflag = 0; vflag = 0; wflag = 0;
        if constexpr (CLU) {
            for (int e = 0; e < 2; ++e) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&xbar[e])) : "memory");
                if constexpr (L::TWO_STEP) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&tbar[e])) : "memory");
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }
    unsigned xphase = 0u;                                // phase of each buffer's barrier
    bool dead = false;                                   // a bounded wait ran out
    if constexpr (TM) { if (warp == 0) tc_alloc<L::TM_COLS>(&tm_holder); tc_fence_before(); }
    scaling_barrier<CLU>();                              // every block's shared memory is there
    uint32_t tk = 0u;                                    // this warp's part of tensor memory
    if constexpr (TM) { tc_fence_after(); tk = tm_holder + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * (RW * CL)); }

    // entries of K for G of the warp's rows, from rowA and colB
    auto form = [&](const int g, u64 (&kk)[L::G][CL / 2]) {
        double acc[L::G][CL];
#pragma unroll
        for (int r = 0; r < L::G; ++r) {
            const double ra = rowA[warp * RW + ((g * L::G) ^ perm) + r];
#pragma unroll
            for (int e = 0; e < CL; ++e) acc[r][e] = ra + colB[(e / 2) * 64 + 2 * lane + (e & 1)];
        }
        dot_tile<SRC, CL, L::G>(o, i0 + ((g * L::G) ^ perm), lane, acc);
#pragma unroll
        for (int r = 0; r < L::G; ++r)
#pragma unroll
            for (int h = 0; h < CL / 2; ++h) kk[r][h] = pack2(exp2_split<LEG || TM>(acc[r][2 * h]), exp2_split<LEG || TM>(acc[r][2 * h + 1]));
    };
    u64 K[LEG || TM ? 1 : RW][CL / 2];                   // pairs of columns
    // use(r, k) for every group of G rows, k[q][h] the entries of row r + q, with the next group's on their way
    auto each_rows = [&](auto &&use) {
        if constexpr (TM) {
            uint32_t ra[L::GW / 32][32], rb[L::GW / 32][32];
            auto fetch = [&](const int g, uint32_t (&w)[L::GW / 32][32]) {
#pragma unroll
                for (int e = 0; e < L::GW / 32; ++e) tc_ld32_issue(tk + (uint32_t)(g * L::GW + 32 * e), w[e]);
            };
            auto arrive = [&](uint32_t (&w)[L::GW / 32][32]) {
#pragma unroll
                for (int e = 0; e < L::GW / 32; ++e) tc_ld_wait(w[e]);
            };
            auto pass = [&](const int g, const uint32_t (&w)[L::GW / 32][32]) {
                u64 kk[L::G][CL / 2];
#pragma unroll
                for (int q = 0; q < L::G; ++q)
#pragma unroll
                    for (int h = 0; h < CL / 2; ++h) {
                        const int x = q * CL + 2 * h;
                        kk[q][h] = pack2(__uint_as_float(w[x / 32][x % 32]), __uint_as_float(w[x / 32][x % 32 + 1]));
                    }
                use(g * L::G, kk);
            };
            constexpr int NG = RW / L::G;
            static_assert(NG % 2 == 0, "groups are taken in pairs");
            fetch(0, ra);
            arrive(ra);
#pragma unroll
            for (int g = 0; g < NG; g += 2) {
                fetch(g + 1, rb);
                pass(g, ra);
                arrive(rb);
                if (g + 2 < NG) fetch(g + 2, ra);
                pass(g + 1, rb);
                if (g + 2 < NG) arrive(ra);
            }
        } else if constexpr (ROLLED) {
#pragma unroll 1
            for (int r = 0; r < RW; r += L::G) {
                u64 kk[L::G][CL / 2];
                form(r / L::G, kk);
                use(r, kk);
            }
        } else {
#pragma unroll
            for (int r = 0; r < RW; r += L::G) {
                u64 kk[L::G][CL / 2];
                if constexpr (LEG) form(r / L::G, kk);
                else {
#pragma unroll
                    for (int q = 0; q < L::G; ++q)
#pragma unroll
                        for (int h = 0; h < CL / 2; ++h) kk[q][h] = K[r + q][h];
                }
                use(r, kk);
            }
        }
    };
    auto row_phi = [&](const double x) -> double { return ab ? phi0 + log2(x) : x; };
    auto col_gam = [&](const int q) -> double { return ab ? gam0[q] + log2(vsd[q]) : vsd[q]; };
    // column parts of sum_i K_ij w_i, w in uas: one row of partf per warp
    auto col_parts = [&]() {
        // (two sums of half the rows each where a warp has 32: shorter sums, smaller errors)
        constexpr int NA = RW > 16 ? 2 : 1;
        static_assert(!ROLLED || NA == 1, "a rolled loop has one set of sums");
        u64 acc[NA][CL / 2];
        if constexpr (ROLLED) {
#pragma unroll
            for (int h = 0; h < CL / 2; ++h) acc[0][h] = 0ull;
        }
        each_rows([&](const int r, const u64 (&kk)[L::G][CL / 2]) {
            const int e = ROLLED ? 0 : r / (RW / NA), first = !ROLLED && r % (RW / NA) == 0;
#pragma unroll
            for (int q = 0; q < L::G; q += 2) {
                const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(uas + warp * RW + ((r + q) ^ perm));
#pragma unroll
                for (int h = 0; h < CL / 2; ++h) {
                    acc[e][h] = q || !first ? fma2(kk[q][h], w.x, acc[e][h]) : mul2(kk[q][h], w.x);
                    acc[e][h] = fma2(kk[q + 1][h], w.y, acc[e][h]);
                }
            }
        });
#pragma unroll
        for (int h = 0; h < CL / 2; ++h) {
            if constexpr (NA == 2) acc[0][h] = add2(acc[0][h], acc[1][h]);
            *reinterpret_cast<u64 *>(partf + warp * COLS + h * 64 + 2 * lane) = acc[0][h];
        }
    };
    // this block's part of the thread's columns: fp32 up to 32 rows, float64 beyond, as a tree
    auto block_cols = [&](double (&t)[NQ]) {
        constexpr int NP = NW / L::FP32_WARPS;
        double p[NP][NQ];
        auto part = [&](const int w, float (&x)[NQ]) {
            const float *src = partf + w * COLS + (cown ? j0 : 0);
            if constexpr (NQ == 4) { const float4 y = *reinterpret_cast<const float4 *>(src); x[0] = y.x; x[1] = y.y; x[2] = y.z; x[3] = y.w; }
            else if constexpr (NQ == 2) { const float2 y = *reinterpret_cast<const float2 *>(src); x[0] = y.x; x[1] = y.y; }
            else x[0] = src[0];
        };
#pragma unroll
        for (int w = 0; w < NP; ++w) {
            float x[NQ];
            part(w * L::FP32_WARPS, x);
            if constexpr (L::FP32_WARPS == 2) {
                float y[NQ];
                part(w * 2 + 1, y);
#pragma unroll
                for (int q = 0; q < NQ; ++q) x[q] += y[q];
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) p[w][q] = widen(x[q]);
        }
#pragma unroll
        for (int step = 1; step < NP; step *= 2)
#pragma unroll
            for (int w = 0; w + step < NP; w += 2 * step)
#pragma unroll
                for (int q = 0; q < NQ; ++q) p[w][q] += p[w + step][q];
#pragma unroll
        for (int q = 0; q < NQ; ++q) t[q] = cown ? p[0][q] : 0.0;
    };
    auto put_vs = [&](const double (&v)[NQ]) {
        if (!cown) return;
        if constexpr (NQ == 4) *reinterpret_cast<float4 *>(vs + j0) = make_float4((float)(bq[0] * v[0]), (float)(bq[1] * v[1]), (float)(bq[2] * v[2]), (float)(bq[3] * v[3]));
        else if constexpr (NQ == 2) *reinterpret_cast<float2 *>(vs + j0) = make_float2((float)(bq[0] * v[0]), (float)(bq[1] * v[1]));
        else vs[j0] = (float)(bq[0] * v[0]);
    };
    // exact sum over a warp of fixed-point terms below 2^47, valid in every thread
    auto warp_fixed = [&](const unsigned long long x) -> unsigned long long {
        const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)x & 0x3ffffffu);
        const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 26));
        return (unsigned long long)lo + ((unsigned long long)hi << 26);
    };
    // a term of a residual, scaled to the fixed point and clamped (never NaN), as an integer
    auto to_fixed = [&](const double t) -> unsigned long long {
        const double z = fmin(t, RSUM_ROW_MAX * RSUM_SCALE) + 0x1p52;
        return ((unsigned long long)(__double2hiint(z) & 0xfffff) << 32) | (unsigned)__double2loint(z);
    };
    // every warp's residual part and flags (bits 60 and up) go to every block ...
    auto rows_word = [&](const unsigned long long fx, const int flags) -> unsigned long long {
        unsigned long long word = warp_fixed(fx);
        if (__any_sync(0xffffffffu, flags)) word |= (unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)flags) << 60;
        return word;
    };
    auto send_rows = [&](const unsigned long long fx, const int flags) {
        const unsigned long long word = rows_word(fx, flags);
        if constexpr (CLU) { if (lane < NC) st_cluster<unsigned long long>(&xw[xch & 1][b * NW + warp], lane, word); }
        else if (lane == 0) xw[xch & 1][warp] = word;
    };
    // ... and are added up by everyone, after the exchange's barrier
    auto recv_rows = [&](int &flags) -> unsigned long long {
        const unsigned long long low = (1ull << 60) - 1ull;
        if constexpr (!CLU) {
            unsigned long long t = 0ull, f = 0ull;
#pragma unroll
            for (int w = 0; w < NW; ++w) { const unsigned long long x = xw[xch & 1][w]; t += x & low; f |= x; }
            flags = (int)(f >> 60);
            return t;
        } else {
            // split so that neither half of 64 (128: RW is 8) words overflows
            constexpr int CUT = L::RANKS * NW > 64 ? 25 : 26;
            static_assert(L::RANKS * NW <= 64 || RW <= 16, "the upper halves of a clamped residual have to fit");
            unsigned lo = 0u, hi = 0u, f = 0u;
            for (int e = lane; e < NC * NW; e += 32) {
                const unsigned long long w = xw[xch & 1][e];
                lo += (unsigned)w & ((1u << CUT) - 1u);
                hi += (unsigned)((w & low) >> CUT);
                f |= (unsigned)(w >> 60);
            }
            lo = __reduce_add_sync(0xffffffffu, lo);
            hi = __reduce_add_sync(0xffffffffu, hi);
            flags = __any_sync(0xffffffffu, f) ? (int)__reduce_or_sync(0xffffffffu, f) : 0;
            return (unsigned long long)lo + ((unsigned long long)hi << CUT);
        }
    };
    // Logical mask: a frozen lane works on until the batch is over, which is when the last lane has passed and this one has
    // run as many cycles.  Every 64th cycle one thread of the lane asks, and tells the others with the flags.  (Off the usual path: asked
    // there with the flags of every cycle, it cost lanes without a mask 4 %.)
    auto mask_over = [&](const int k) -> int {
        if (b != 0 || tid != 0) return 0;
        const volatile Ctl *now = P.ctl;
        if (now->mask_left < c.n_running) return 0;
        __threadfence();
        return k >= now->mask_last ? SC_LEAVE : 0;
    };
    // TWO_STEP: this thread's column of the block's share, its total (or maximum) from the parts in xbuf
    auto share_total = [&](const bool is_max) -> double {
        const double *src = xbuf + (size_t)(xch & 1) * NC * share + (tid >> tpb);
        double t = is_max ? -1.0e300 : 0.0;
#pragma unroll
        for (int e = 0; e < L::RANKS / 2; ++e) {
            const int rk = (e << tpb) + (tid & ((1 << tpb) - 1));
            const double x = rk < NC ? src[(size_t)rk * share] : (is_max ? -1.0e300 : 0.0);
            t = is_max ? fmax(t, x) : t + x;
        }
        for (int off = 1; off < (1 << tpb); off <<= 1) {
            const double x = __shfl_xor_sync(0xffffffffu, t, off);
            t = is_max ? fmax(t, x) : t + x;
        }
        return t;
    };
    // one value per owned column and block -> their sum (or maximum) over the blocks, in every block; with barriers, for the
    // steps off the usual path.  The caller counts the exchange up when it has read what else came with it.
    auto exchange_cols = [&](double (&val)[NQ], const bool is_max) {
        if constexpr (L::TWO_STEP) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int j = j0 + q;
                st_cluster<double>(xbuf + ((size_t)(xch & 1) * NC + b) * share + j % share, j / share, val[q]);
            }
            scaling_barrier<CLU>();
            if (b < own) {
                const double t = share_total(is_max);
                for (int rk = tid & ((1 << tpb) - 1); rk < NC; rk += 1 << tpb) st_cluster<double>(tbuf + (size_t)(xch & 1) * COLS + b * share + (tid >> tpb), rk, t);
            }
            scaling_barrier<CLU>();
#pragma unroll
            for (int q = 0; q < NQ; ++q) val[q] = tbuf[(size_t)(xch & 1) * COLS + j0 + q];
        } else {
            double *dst = xbuf + ((size_t)(xch & 1) * NC + b) * COLS;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int j = j0 + q;
                if (cown) {
                    if constexpr (!CLU) dst[j] = val[q];
                    else for (int rk = 0; rk < NC; ++rk) st_cluster<double>(dst + j, rk, val[q]);
                }
            }
            scaling_barrier<CLU>();
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                if (!cown) continue;
                const double *src = xbuf + (size_t)(xch & 1) * NC * COLS + j0 + q;
                val[q] = src[0];
                for (int rk = 1; rk < NC; ++rk) { const double x = src[(size_t)rk * COLS]; val[q] = is_max ? fmax(val[q], x) : val[q] + x; }
            }
        }
    };
    // log-domain column step from row potentials `phi`: the potential of every owned column that makes its
    // marginal equal to its weight
    auto log_cols = [&](const double phi, double (&pnew)[NQ]) {
        if (lane % SHARE == 0) rowA[lr] = rok ? phi - P.sqx[ro] : -1.0e30;
        __syncwarp();
        log_cols_max<SRC, NW, CL, RW>(o, i0, rowA + warp * RW, partd + warp * COLS);
        __syncthreads();
        double val[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int j = j0 + q;
            val[q] = -1.0e300;
            if (cown) for (int w = 0; w < NW; ++w) val[q] = fmax(val[q], partd[w * COLS + j]);
        }
        exchange_cols(val, true);
        double mc[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int j = j0 + q;
            mc[q] = 0.0;
            if (cown) { mc[q] = ceil(val[q]); colB[j] = mc[q]; }
        }
        ++xch;
        __syncthreads();
        log_cols_sum<SRC, NW, CL, RW>(o, i0, rowA + warp * RW, colB, partf + warp * COLS);
        __syncthreads();
        block_cols(val);
        exchange_cols(val, false);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int j = j0 + q;
            pnew[q] = 0.0;
            if (cown && j < P.m) pnew[q] = P.lb2[co + j] + P.sqy[co + j] - (mc[q] + log2(val[q]));
        }
        ++xch;
        __syncthreads();
    };

    int it = 0, checks = 0, retired_at = 0, fl = 0;
    int nf = !LEG && !frozen ? P.nonfinite[slot] : 0;
    double rr = 0.0, rc = 0.0;
    bool need_build = true, near = false;
    for (;;) {
        if (need_build && ab) {
            if (lane % SHARE == 0) rowA[lr] = rok ? phi0 - P.la2[ro] - P.sqx[ro] : -1.0e30;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int j = j0 + q;
                if (cown) {
                    colB[j] = j < P.m ? gam0[q] - P.lb2[co + j] - P.sqy[co + j] : -1.0e30;
                    vs[j] = (float)(bq[q] * vsd[q]);
                }
            }
            __syncthreads();
            if constexpr (!LEG) {
#pragma unroll 1
                for (int g = 0; g < RW / L::G; ++g) {
                    u64 kk[L::G][CL / 2];
                    form(g, kk);
                    if constexpr (TM) {
                        uint32_t w[L::GW / 32][32];
#pragma unroll
                        for (int r = 0; r < L::G; ++r)
#pragma unroll
                            for (int h = 0; h < CL / 2; ++h) {
                                const int x = r * CL + 2 * h;
                                float k0, k1;
                                unpack2(kk[r][h], k0, k1);
                                w[x / 32][x % 32] = __float_as_uint(k0); w[x / 32][x % 32 + 1] = __float_as_uint(k1);
                            }
#pragma unroll
                        for (int e = 0; e < L::GW / 32; ++e) tc_st32_issue(tk + (uint32_t)(g * L::GW + 32 * e), w[e]);
                    } else {
#pragma unroll
                        for (int r = 0; r < L::G; ++r)
#pragma unroll
                            for (int h = 0; h < CL / 2; ++h) kstage[((g * L::G + r) * (CL / 2) + h) * THREADS + tid] = kk[r][h];
                    }
                }
                if constexpr (TM) tc_st_wait();
                else {
#pragma unroll
                    for (int r = 0; r < RW; ++r)
#pragma unroll
                        for (int h = 0; h < CL / 2; ++h) K[r][h] = kstage[(r * (CL / 2) + h) * THREADS + tid];
                }
                __syncthreads();
            }
        }
        need_build = false;

        // ---------------- whole cycles on K while nothing needs a decision; the f-leg yields the row residual
        // of the state before it, and the column sums of the state after it are formed beside it
        bool scal = ab, done = false;
        double unew = 0.0, T[NQ];
        unsigned long long tot = 0ull;
        int all = SC_BAD;                            // "the f-leg is still to be done, in the log domain"
        if (ab && (!LEG || leg == LEG_F)) {
#pragma unroll 1
            for (;;) {
                {
                    u64 v[CL / 2];
                    float s[RW];
#pragma unroll
                    for (int h = 0; h < CL / 2; ++h) v[h] = *reinterpret_cast<const u64 *>(vs + h * 64 + 2 * lane);
                    each_rows([&](const int r, const u64 (&kk)[L::G][CL / 2]) {
#pragma unroll
                        for (int q = 0; q < L::G; ++q) {
                            u64 t = mul2(kk[q][0], v[0]);
                            if constexpr (CL >= 32) {                // (shorter chains, shorter sums)
                                u64 t2 = mul2(kk[q][1], v[1]);
#pragma unroll
                                for (int h = 2; h < CL / 2; h += 2) { t = fma2(kk[q][h], v[h], t); t2 = fma2(kk[q][h + 1], v[h + 1], t2); }
                                t = add2(t, t2);
                            } else {
#pragma unroll
                                for (int h = 1; h < CL / 2; ++h) t = fma2(kk[q][h], v[h], t);
                            }
                            float s0, s1;
                            unpack2(t, s0, s1);
                            s[r + q] = s0 + s1;
                        }
                    });
                    const double S = row_exchange<CL, L::FP32_COLS, true, 16, RW, float>(s, lane);
                    unew = rok ? rcp64(S) : 1.0;
                    const double term = rown ? a_fix * fabs(fma(us, S, -1.0)) : 0.0;
                    const int flags = (rok && out_of_band<SC_SUMS>(S)) || out_of_band<SC_TAKE>(unew) ? SC_BAD | SC_DRIFT : (out_of_band<SC_KEEP>(unew) ? SC_DRIFT : 0);
                    const unsigned long long fx = to_fixed(term);
                    if constexpr (LEG) {
                        send_rows(fx, flags);
                        scaling_barrier<CLU>();
                        tot = recv_rows(all);
                        ++xch;
                        break;
                    }
                    if (lane % SHARE == 0) { const float w = (float)(a_i * unew); uas[lr] = make_float2(w, w); }
                    __syncwarp();
                    col_parts();
                    const unsigned long long word = rows_word(fx, flags);
                    if (lane == 0) (CLU ? sw[xch & 1] : xw[xch & 1])[warp] = word;
                }
                __syncthreads();
                block_cols(T);
                if constexpr (CLU) {
                    const int e = xch & 1;
                    double *out = sbuf + e * COLS;
                    if (cown) {
                        if constexpr (NQ == 1) out[j0] = T[0];
                        else {
#pragma unroll
                            for (int q = 0; q < NQ; q += 2) *reinterpret_cast<double2 *>(out + j0 + q) = make_double2(T[q], T[q + 1]);
                        }
                    }
                    fence_for_copies();
                    if (tid == 0) {
                        expect_bytes(&xbar[e], (unsigned)(NC * ((!L::TWO_STEP ? COLS : (b < own ? share : 0)) + NW) * 8));
                        if constexpr (L::TWO_STEP) expect_bytes(&tbar[e], (unsigned)(COLS * 8));
                    }
                    __syncthreads();
                    // a warp sends to the ranks warp, warp + NW, ...: one after the other from one warp they took 1000 clk
                    for (int rk = warp; rk < NC; rk += NW) {
                        if (lane == 0) {
                            if constexpr (!L::TWO_STEP) copy_to_peer(xbuf + ((size_t)e * NC + b) * COLS, out, COLS * 8, &xbar[e], rk);
                            else if (rk < own) copy_to_peer(xbuf + ((size_t)e * NC + b) * share, out + rk * share, share * 8, &xbar[e], rk);
                            copy_to_peer(&xw[e][b * NW], sw[e], NW * 8, &xbar[e], rk);
                        }
                    }
                    __syncwarp();
                    const unsigned phase = (xphase >> e) & 1u;
                    bool ok = bar_wait(smem_addr(&xbar[e]), phase);
                    if constexpr (L::TWO_STEP) {
                        if (b < own) {                       // (the same for the whole block)
                            const double t = share_total(false);
                            if ((tid & ((1 << tpb) - 1)) == 0) ubuf[e * THREADS + (tid >> tpb)] = t;
                            fence_for_copies();
                            __syncthreads();
                            for (int rk = warp; rk < NC; rk += NW)
                                if (lane == 0) copy_to_peer(tbuf + (size_t)e * COLS + b * share, ubuf + e * THREADS, share * 8, &tbar[e], rk);
                            __syncwarp();
                        }
                        ok = bar_wait(smem_addr(&tbar[e]), phase) && ok;
                    }
                    xphase ^= 1u << e;
                    if (!ok) wflag = 1;
                    __syncthreads();
                    if (wflag) { dead = true; break; }
                }
                if constexpr (CLU && L::TWO_STEP) {
                    const double *src = tbuf + (size_t)(xch & 1) * COLS + j0;
#pragma unroll
                    for (int q = 0; q < NQ; q += 2) { const double2 t = *reinterpret_cast<const double2 *>(src + q); T[q] = t.x; T[q + 1] = t.y; }
                } else if constexpr (CLU) {
                    if (cown) {
                        const double *src = xbuf + (size_t)(xch & 1) * NC * COLS + j0;
#pragma unroll
                        for (int rk = 0; rk < MAX_CLUSTER_RANKS; ++rk) {
                            if (rk >= NC) continue;
                            if constexpr (NQ == 2) {
                                const double2 t = *reinterpret_cast<const double2 *>(src + rk * COLS);
                                T[0] = rk ? T[0] + t.x : t.x; T[1] = rk ? T[1] + t.y : t.y;
                            } else T[0] = rk ? T[0] + src[rk * COLS] : src[rk * COLS];
                        }
                    }
                }
                // g-leg, on its way while the words are added up
                double vn[NQ];
                int flags = 0;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    vn[q] = 0.0;
                    if (cown && j0 + q < P.m) {
                        vn[q] = rcp64(T[q]);
                        flags |= out_of_band<SC_KEEP>(vn[q]) | out_of_band<SC_SUMS>(T[q]);
                    }
                }
                tot = recv_rows(all);
                ++xch;
                if (all || (frozen ? (k & 63) == 0 : tot <= near_tot && !catch_up) || nf || (k - start >= P.max_iter && !catch_up) || (closing && it == todo)) break;
                if (!frozen) put_vs(vn);
                if (flags) vflag = 1;
                __syncthreads();
                if (vflag) {                             // (read by all before it is cleared, cleared before it is set again)
                    __syncthreads();
                    if (tid == 0) vflag = 0;
                    break;
                }
                if (!frozen) {
                    us = unew;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) vsd[q] = vn[q];
                }
                ++k;
                par ^= 1;
                if (++it >= todo && !closing) { done = true; break; }
            }
        }
        if (dead) {
            if (tid == 0) atomicOr(&P.ctl->error, ERR_WAIT);
            break;
        }
        if (done) {
            // (the last audit was that of the state before this launch's last cycle, and it flagged nothing)
            rr = (double)tot * (1.0 / RSUM_SCALE);
            rc = 0.0;
            fl = 0;
            break;
        }

        if (KIND == SC_CYCLES && frozen && (k & 63) == 0) {
            send_rows(0ull, mask_over(k));
            scaling_barrier<CLU>();
            int over;
            recv_rows(over);
            ++xch;
            if (over & SC_LEAVE) {
                // (a frozen lane's last audit flags nothing and has the residual of the state it froze at)
                if (!(all & SC_BAD)) rr = (double)tot * (1.0 / RSUM_SCALE);
                else if (it == 0) rr = P.rrow[slot];
                rc = 0.0;
                fl = 0;
                par = c.parity ^ (todo & 1);                 // where the lanes that go on have theirs
                break;
            }
        }

        // ---------------- f-leg in the log domain, where K cannot be used
        if (!LEG || leg == LEG_F) {
            if (all & SC_BAD) {
                scal = false;
                double term = 0.0;                       // in units of the fixed point
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int j = j0 + q;
                    if (cown) colB[j] = j < P.m ? col_gam(q) - P.sqy[co + j] : -1.0e30;
                }
                __syncthreads();
                double S, M;
                log_rows<SRC, NW, CL, RW>(o, i0, colB, &S, &M);
                unew = 0.0;
                if (rok) row_math((int)FORM_DOT, true, P.la2[ro], P.sqx[ro], a_i, row_phi(us), (float)M, S, 0.f, unew, term);
                const int flags = !isfinite(unew) || !isfinite(term) ? SC_NF : 0;
                send_rows(rown && !flags ? to_fixed(term * RSUM_SCALE) : 0ull, flags);
                scaling_barrier<CLU>();
                tot = recv_rows(all);
                ++xch;
            }
            if (all & SC_NF) nf = 1;
            near = tot <= near_tot;
            rr = (double)tot * (1.0 / RSUM_SCALE);
            if (scal && (all & SC_DRIFT)) need_build = true;
            if constexpr (LEG) {
                if (!P.dry_run) {
                    if (rown && !frozen) {
                        P.phi[par ^ 1][ro] = scal ? phi0 + log2(unew) : unew;
                        P.uu[par ^ 1][ro] = unew;
                    }
                    if (b == 0 && tid == 0) {
                        P.rsum_row[slot] += tot;
                        P.cyc_log[slot] = scal ? 0 : 1;
                        if (nf && !frozen) P.nonfinite[slot] = 1;
                    }
                }
                break;
            }
        }

        // ---------------- audit of the state before the f-leg
        const bool close_now = closing && it == todo;
        if constexpr (!LEG) { fl = 0; rc = 0.0; }
        if (!LEG && near && !frozen && !catch_up) {
            const bool audited = lane_audited(P, k, start);
            if (audited && !nf && in_guard_band(P, rr)) {
                // guard band: decide from a float64 re-evaluation of the row residual; it reads the column
                // potentials from global memory
                if (lane % SHARE == 0) rowA[lr] = rok ? row_phi(us) : 0.0;
                if (b == 0) {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) { const int j = j0 + q; if (cown && j < P.m) P.gam[co + j] = col_gam(q); }
                }
                scaling_barrier<CLU>();
                __syncthreads();
                int bad;
                const unsigned long long mine = scaling_reeval<NW>(&P, slot, b * RB, min(b * RB + RB, P.n), rowA, swr, &bad);
                send_rows(tid == 0 ? mine : 0ull, bad ? SC_NF : 0);
                scaling_barrier<CLU>();
                int all;
                const unsigned long long tot = recv_rows(all);
                ++xch;
                rr = (double)tot * (1.0 / RSUM_SCALE);
                if (all & SC_NF) nf = 1;
            }
            fl = audited && !nf && rr <= P.tol_screen;
        }
        if ((LEG && leg == LEG_V) || (!LEG && (fl || close_now))) {
            // column half of the two-sided check: the marginals of the audited state, genuinely measured
            double term[NQ];
            if (ab) {
                if (lane % SHARE == 0) { const float w = (float)(a_i * us); uas[lr] = make_float2(w, w); }
                __syncwarp();
                col_parts();
                __syncthreads();
                double val[NQ];
                block_cols(val);
                exchange_cols(val, false);
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int j = j0 + q;
                    term[q] = (cown && j < P.m) ? bq[q] * fabs(fma(vsd[q], val[q], -1.0)) : 0.0;
                }
                ++xch;
            } else {
                double pn[NQ];
                log_cols(us, pn);
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int j = j0 + q;
                    term[q] = (cown && j < P.m) ? bq[q] * fabs(expm1((vsd[q] - pn[q]) * 0.6931471805599453)) : 0.0;
                }
            }
            unsigned long long fx = 0ull;
            int bad = 0;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                if (!isfinite(term[q])) bad = 1;
                else fx += to_fixed(term[q] * RSUM_SCALE);
            }
            bad = __syncthreads_or(bad);
            const unsigned long long ws = warp_fixed(fx);
            if (lane == 0) swr[warp] = ws;
            __syncthreads();
            unsigned long long totc = 0ull;                           // every block has all columns: the same total
            for (int w = 0; w < NW; ++w) totc += swr[w];
            __syncthreads();
            if (bad) nf = 1;
            rc = (double)totc * (1.0 / RSUM_SCALE);
            ++checks;
            if constexpr (LEG) {
                if (b == 0 && tid == 0 && !P.dry_run) { P.rsum_col[slot] += totc; if (bad) P.nonfinite[slot] = 1; }
                break;
            }
        }
        if (close_now) {
            // the common last cycle of a STATIC batch.  A lane that passed at this very state keeps the row residual its
            // decision was taken from
            if (rown) P.f_out[(size_t)lane_id * P.n + i] = row_phi(us) * inv_s;
            if (b == 0) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) { const int j = j0 + q; if (cown && j < P.m) P.g_out[(size_t)lane_id * P.m + j] = col_gam(q) * inv_s; }
                if (tid == 0) {
                    P.res_row[lane_id] = just_passed ? P.rrow[slot] : rr;
                    P.res_col[lane_id] = rc;
                    if (nf) P.status[lane_id] = LANE_NONFINITE;
                    P.emitted[lane_id] = 1;
                }
            }
            break;
        }
        if (!LEG && !frozen && !catch_up && (near || nf || k - start >= P.max_iter)) {
            const bool vd = !nf && fmax(rr, rc) <= P.tol_stop;
            const bool limit = k - start >= P.max_iter;
            int st = LANE_RUNNING;
            if (nf) st = LANE_NONFINITE;
            else if (fl && vd) st = LANE_DONE;
            else if (limit) st = LANE_ITER_LIMIT;
            if (st != LANE_RUNNING && P.mode == MODE_STATIC) {
                // the lane waits here until the others are known to go on (SC_CATCH_UP)
                if (b == 0 && tid == 0) {
                    P.depth[lane_id] = (limit && st != LANE_DONE) ? P.max_iter : k - start;
                    P.status[lane_id] = st;
                    P.state[slot] = 1;
                }
                retired_at = k + 1;
                break;
            }
            if (st != LANE_RUNNING) {
                if (rown) P.f_out[(size_t)lane_id * P.n + i] = row_phi(us) * inv_s;
                if (b == 0) {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) { const int j = j0 + q; if (cown && j < P.m) P.g_out[(size_t)lane_id * P.m + j] = col_gam(q) * inv_s; }
                    if (tid == 0) {
                        P.res_row[lane_id] = rr;
                        P.res_col[lane_id] = fl ? rc : __longlong_as_double(0x7ff8000000000000LL);
                        P.depth[lane_id] = (limit && st != LANE_DONE) ? P.max_iter : k - start;
                        P.status[lane_id] = st;
                        P.emitted[lane_id] = 1;
                        if (P.mode == MODE_MASKED) {
                            P.state[slot] = 1;
                            atomicMax(&P.ctl->mask_last, k);
                            __threadfence();
                            atomicAdd(&P.ctl->mask_left, 1);
                        }
                    }
                }
                retired_at = k + 1;
                if (P.mode == MODE_ACTIVE || P.early_exit) break;
                frozen = true;                           // logical mask: the work goes on, nothing is stored
            }
        }

        // ---------------- g-leg
        double vnew[NQ];
        bool log_g = false;
        if constexpr (LEG) {
            // us is what the f-leg left (u, or the row potential where it ran in the log domain)
            log_g = !ab || P.cyc_log[slot] != 0;
            unew = us;
            scal = !log_g;
            if (scal) {
                if (lane % SHARE == 0) { const float w = rok ? (float)(a_i * unew) : 0.f; uas[lr] = make_float2(w, w); }
                __syncwarp();
                col_parts();
                send_rows(0ull, rok && out_of_band<SC_KEEP>(unew) ? SC_DRIFT : 0);
                __syncthreads();
                double val[NQ];
                block_cols(val);
                exchange_cols(val, false);
                int all;
                recv_rows(all);
#pragma unroll
                for (int q = 0; q < NQ; ++q) T[q] = cown ? val[q] : 0.0;
                ++xch;
                need_build = (all & SC_DRIFT) != 0;
            }
        }
        if (scal) {
            int flags = 0;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int j = j0 + q;
                vnew[q] = 0.0;
                if (cown) {
                    if (j < P.m) {
                        vnew[q] = rcp64(T[q]);
                        flags |= out_of_band<SC_SUMS>(T[q]) || out_of_band<SC_TAKE>(vnew[q]) ? SC_BAD | SC_DRIFT : (out_of_band<SC_KEEP>(vnew[q]) ? SC_DRIFT : 0);
                    }
                    if (!frozen) vs[j] = (float)(bq[q] * vnew[q]);
                }
            }
            if (flags) atomicOr(&sflag, flags);
            __syncthreads();
            const int all = sflag;
            if (all) { __syncthreads(); if (tid == 0) sflag = 0; }
            if (all & SC_DRIFT) need_build = true;
            if (all & SC_BAD) log_g = true;
        } else log_g = true;
        double phinew = unew;                            // row potential, where the column step needs it
        if (log_g) {
            if (scal) phinew = rok ? phi0 + log2(unew) : 0.0;
            log_cols(phinew, vnew);
            need_build = true;
            bool bad = false;
#pragma unroll
            for (int q = 0; q < NQ; ++q) bad = bad || !isfinite(vnew[q]);
            if (__syncthreads_or(bad ? 1 : 0) && !frozen) nf = 1;
        }
        if (!frozen) {
            if (need_build && no_matrix) {
                us = phinew;                             // (every leg of such a lane has run in the log domain)
#pragma unroll
                for (int q = 0; q < NQ; ++q) vsd[q] = vnew[q];
            } else if (need_build) {
                // absorb the new potentials: K is formed anew from them
                if (!log_g) {
                    phinew = rok ? phi0 + log2(unew) : 0.0;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) { const int j = j0 + q; if (cown && j < P.m) vnew[q] = gam0[q] + log2(vnew[q]); }
                }
                ab = true;
                us = 1.0;
                phi0 = phinew;
#pragma unroll
                for (int q = 0; q < NQ; ++q) gam0[q] = vnew[q];
#pragma unroll
                for (int q = 0; q < NQ; ++q) { const int j = j0 + q; vsd[q] = (cown && j < P.m) ? 1.0 : 0.0; }
            } else {
                us = unew;
#pragma unroll
                for (int q = 0; q < NQ; ++q) vsd[q] = vnew[q];
            }
        } else need_build = false;
        if constexpr (LEG) {
            if (!P.dry_run && !frozen) {
                if (nf && b == 0 && tid == 0) P.nonfinite[slot] = 1;
                if (need_build && ab && rown) { P.uu[par][ro] = 1.0; P.phi0[ro] = phi0; }
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int j = j0 + q;
                    if (b == 0 && cown && j < P.m) {
                        P.vv[co + j] = vsd[q];
                        P.gam0[co + j] = gam0[q];
                        P.gam[co + j] = col_gam(q);
                    }
                }
                if (b == 0 && tid == 0 && ab) P.absorbed[slot] = 1;
            }
            break;
        }
        ++k;
        par ^= 1;
        if (++it >= todo && !closing) break;
    }
    if constexpr (!LEG) {
        if (b == 0 && tid == 0) {
            P.ret_at[slot] = retired_at;
            P.n_checks[slot] = catch_up ? 0 : checks;
            if (!just_passed) { P.rrow[slot] = rr; P.rcol[slot] = catch_up ? 0.0 : rc; P.flag[slot] = fl; }
        }
        if (!retired_at || P.mode != MODE_ACTIVE) {
            // the lane goes back out; a frozen one keeps the state it froze with
            if (rown) {
                P.phi[par][ro] = row_phi(us);
                P.uu[par][ro] = us;
                P.phi0[ro] = phi0;
            }
            if (b == 0) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int j = j0 + q;
                    if (cown && j < P.m) { P.gam[co + j] = col_gam(q); P.vv[co + j] = vsd[q]; P.gam0[co + j] = gam0[q]; }
                }
                if (tid == 0) { P.absorbed[slot] = ab ? 1 : (no_matrix ? SC_NO_MATRIX : 0); if (nf) P.nonfinite[slot] = 1; }
            }
        }
    }
    if constexpr (TM) {
        tc_fence_before();
        __syncthreads();
        if (warp == 0) { tc_fence_after(); tc_dealloc<L::TM_COLS>(tm_holder); }
    }
    if constexpr (CLU) cluster_sync_all();               // no block leaves while another may still write into its memory
}

// ---------------------------------------------------------------- host side
constexpr int SMEM_PER_SM = 226 << 10;                   // shared by the blocks of an SM (each is charged 1 KB more)
struct ScalingVariant {
    int threads, cols, rb;
    bool cluster;                                        // lanes of several blocks
    int min_blocks, max_blocks;
    const void *kernel[3], *roomy[2];                    // by ScalingKind; of SC_CYCLES and SC_CATCH_UP, where there are any
    int tm_cols;                                         // tensor memory columns (0: K in registers)
    size_t (*smem)(int nc);
};
#define SKB_SC(SRC, NW, CL, RW, CLU, TM) { 32 * NW, 32 * CL, NW * RW, CLU, ScalingShape<NW, CL, RW, TM>::MIN_BLOCKS, ScalingShape<NW, CL, RW, TM>::RANKS, \
    {(const void *)&scaling_kernel<SRC, NW, CL, RW, CLU, TM, SC_CYCLES>, (const void *)&scaling_kernel<SRC, NW, CL, RW, CLU, TM, SC_CATCH_UP>, \
     (const void *)&scaling_kernel<SRC, NW, CL, RW, CLU, TM, SC_LEG>}, \
    {(const void *)&scaling_kernel<SRC, NW, CL, RW, CLU, TM, SC_CYCLES, ScalingShape<NW, CL, RW, TM>::has_roomy(CLU)>, \
     (const void *)&scaling_kernel<SRC, NW, CL, RW, CLU, TM, SC_CATCH_UP, !TM && ScalingShape<NW, CL, RW, TM>::has_roomy(CLU)>}, TM ? ScalingShape<NW, CL, RW, TM>::TM_COLS : 0, &ScalingShape<NW, CL, RW, TM>::smem }

// Variants by the source of their exponents, narrowest column count first, then fewest rows per block.
struct ScalingTable { const ScalingVariant *v; int count; };
ScalingTable scaling_table_f64();                        // skb_scaling.cu
ScalingTable scaling_table_dots();                       // skb_scaling_dots.cu

}  // namespace skb
