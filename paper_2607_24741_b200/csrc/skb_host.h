// Host-side declarations shared by the translation units of the library.
#pragma once
#include <cuda_runtime.h>
#include "skb_device.cuh"

namespace skb {

// Launch with programmatic stream serialization allowed (the kernel must call pdl_enter()).
//
// Invariants the kernels of a cycle rely on (f-leg, column check, plan, emit/move, g-leg, in that
// order on one stream):
//  - every kernel executes griddepcontrol.wait in at least one block before it completes, so that
//    "my predecessor has completed" implies "everything earlier in the stream has completed";
//  - the control block is written by the plan kernel only, coordinates and the per-slot scalars by
//    the plan and emit/move kernels only;
//  - a kernel that reads state BEFORE its own wait (the SIMT f-leg: control block, row coordinates,
//    row potentials; the column check: control block) may do so because the kernel that released it
//    is a g-leg (of this batch or of another batch sharing the stream), and g-legs release their
//    dependents only after their own wait: by then the plan and emit/move kernels before it are
//    complete, and nothing between them and the early reader writes what it reads early;
//  - kernels launched without the attribute (set-up, read-back, a caller's own kernels) neither
//    start early nor release early, so they may sit anywhere in the stream.
template <typename... KArgs, typename... Args>
inline void launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Update-kernel variant: compute type, padded dimension, rows per thread, column split.
struct Variant {
    int f64, xf, DP, R, CS;   // xf: float64 arguments with fp32 special-function exponentials
    int rows_per_cta;
    size_t smem;
    int (*launch)(const Dev &, int leg, int width, cudaStream_t);   // 1: the guard band's pool rode in a column-check launch
    // several whole cycles per launch, one thread-block cluster per lane; null where there is none
    void (*launch_cycles)(const Dev &, int cycles, int width, cudaStream_t);
    // does a lane of n x m points fit the shared-memory-resident version of the multi-cycle kernel?
    bool (*lane_fits_shared)(int n, int m);
};
constexpr int MAX_CLUSTER_BLOCKS = MAX_CLUSTER_RANKS;   // a lane needs at most this many row blocks
// Upper bound on the cycles one multi-cycle launch runs.  Lanes are independent and leave a launch when they pass, so a
// long launch keeps the SMs full where a series of short ones waits for its slowest lanes after each.  A drain waits for every launch
// before it enqueues the next, 12 to 17 us with an idle GPU, which lanes deeper than this pay.
constexpr int MAX_CYCLES_IN_LAUNCH = 8192;
// ... of those that a caller's number of cycles is cut into (enqueued one behind the other)
constexpr int STEP_CYCLES_IN_LAUNCH = 2048;
// ... and under a logical mask, whose lanes work on until the last one has passed, however early they do.  Lanes that wait for a
// place on the GPU cannot pass, so a launch of more lanes than fit works on to its end: what a caller asks for
// beyond the last lane's depth costs at most the rest of one launch (launches after it return at once).
constexpr int MASK_CYCLES_IN_LAUNCH = 256;
// Picks the variant for a shape (depends on the static shape only, so that every mode
// and every run of the same batch uses the same reduction order).  Null if unsupported.
// (lanes: those that the batch can take in, which decides about the spatial order)
const Variant *choose_variant(int W, int lanes, int n, int m, int d, bool f64, bool fast_exp, int force_cs, bool spatial);
int padded_dim(int d);

void launch_lane_stats(const Dev &P, const void *x, const void *y, const float *eps, int slot0, int lane0, int count,
                       int cycle0, cudaStream_t st);
void launch_prep(const Dev &P, const void *x, const void *y, const float *a, const float *b, int slot0, int count, cudaStream_t st);
void launch_refill_ctl(const Dev &P, int count, cudaStream_t st);
void launch_warm(const Dev &P, const double *f0, const double *g0, cudaStream_t st);
int launch_plan(const Dev &P, int width, cudaStream_t st);        // both return the number of kernels launched
// tensor-core update kernel (bf16 inputs, d a multiple of 64 up to 512)
bool tc_eligible(int d, bool bf16);
const char *tc_make_map(void *out_map, void *base, int W, int npts, int d);
size_t tc_tiled_bytes(int W, int npts, int d);
void launch_retile(const void *src, void *dst, int W, int npts, int d, cudaStream_t st);
void launch_wait_probe(int *out, long long budget_clocks, cudaStream_t st);
void launch_guard_pool(const Dev &P, cudaStream_t st);
void launch_guard_strips(void *base, const GuardList &gl, bool fill, int *bad, cudaStream_t st);
void launch_update_tc(const Dev &P, const void *maps, int leg, int width, cudaStream_t st);
void launch_gram(const Dev &P, const void *maps, int slot0, int count, cudaStream_t st);
int launch_emit_move(const Dev &P, int width, cudaStream_t st);
// lanes kept in spatial order, whose legs skip the boxes of columns that are too far away to matter
bool near_shape(int f64, int DP, int CS, int n, int m, int lanes);    // lanes: that a batch with room for lists can take in, else 1
constexpr int NEAR_PAIRS = 4096;        // pairs per lane that launch_near_estimate counts into Ctl::near_kept
void launch_near_estimate(const Dev &P, const void *x, const void *y, int lanes, cudaStream_t st);
void launch_spatial_sort(const Dev &P, const void *x, const void *y, int slot0, int count, cudaStream_t st);
void launch_prep_near(const Dev &P, const void *x, const void *y, const float *a, const float *b, int slot0, int count, cudaStream_t st);
void launch_near_tops(const Dev &P, cudaStream_t st);
int launch_near(const Dev &P, int leg, int width, cudaStream_t st);     // 1: the guard band's pool rode in a column-check launch
int guard_pool_rows(int per_row, bool on, int lanes);
// lanes small enough for their kernel matrix to stay on chip (dots: deep lanes, formed from stored dot products): whole
// cycles, or one leg as a launch of its own
bool scaling_fits(bool dots, int n, int m);
enum ScalingKind : int { SC_CYCLES, SC_CATCH_UP, SC_LEG };      // see scaling_kernel; `leg` counts for SC_LEG only
void launch_scaling(const Dev &P, ScalingKind kind, int leg, int cycles, int width, cudaStream_t st);
int launch_plan_cycles(const Dev &P, int width, int cycles, cudaStream_t st);
void launch_order(const Dev &P, int *order, cudaStream_t st);
bool scaling_shares_sm(const Dev &P, int width);       // lanes that fewer of them would not
int scaling_blocks(const Dev &P);          // blocks of a lane
int scaling_resident(const Dev &P);        // lanes that are on the GPU at the same time, at least
void launch_plan_static(const Dev &P, int cycles, cudaStream_t st);
void launch_gather(const Dev &P, void *f, void *g, bool f64, cudaStream_t st);
void launch_gather_audit(const Dev &P, float *rrow, float *rcol, int *flagged, cudaStream_t st);
void launch_apply_plan(const Dev &P, const void *x, const void *y, const float *eps, const float *v, int dv, float *out,
                       int lanes, cudaStream_t st);
void launch_gather_small(const Dev &P, int *depth, int *status, float *rrow, float *rcol, cudaStream_t st);

}  // namespace skb
