// Kernel matrices on chip: the variants formed from float64 coordinates, the choice of a variant and the launch.
#include "skb_scaling.cuh"

namespace skb {

static const ScalingVariant g_scaling[] = {
    SKB_SC(SRC_F64, 2, 2, 8, false, false), SKB_SC(SRC_F64, 4, 2, 16, false, false), SKB_SC(SRC_F64, 4, 2, 32, false, false), SKB_SC(SRC_F64, 4, 2, 32, true, false),
    SKB_SC(SRC_F64, 4, 4, 16, false, false), SKB_SC(SRC_F64, 4, 4, 32, false, false), SKB_SC(SRC_F64, 4, 4, 32, true, false),
    SKB_SC(SRC_F64, 4, 8, 16, false, false), SKB_SC(SRC_F64, 8, 8, 16, false, true), SKB_SC(SRC_F64, 8, 8, 32, false, true), SKB_SC(SRC_F64, 4, 8, 16, true, false),
    SKB_SC(SRC_F64, 8, 16, 16, true, true),
};
ScalingTable scaling_table_f64() { return {g_scaling, (int)(sizeof(g_scaling) / sizeof(g_scaling[0]))}; }

// The variant of a lane shape: the narrowest column tile that holds the columns; of its row tiles the
// smallest that needs the fewest blocks.  Depends on the shape alone (the order of the sums follows from
// it), so every mode and every launch of a batch uses the same one.  Null: the lane is too large.
static int blocks_of(const ScalingVariant &v, int n)
{
    const int nc = (n + v.rb - 1) / v.rb;
    return nc < v.min_blocks ? v.min_blocks : nc;
}
static const ScalingVariant *scaling_variant(bool dots, int n, int m)
{
    const ScalingTable t = dots ? scaling_table_dots() : scaling_table_f64();
    const ScalingVariant *best = nullptr;
    int best_nc = 0;
    for (int i = 0; i < t.count; ++i) {
        const ScalingVariant &v = t.v[i];
        if (m > v.cols || (best && v.cols > best->cols)) continue;
        const int nc = blocks_of(v, n);
        if (nc > (v.cluster ? v.max_blocks : 1)) continue;
        if (!best || nc < best_nc) { best = &v; best_nc = nc; }
    }
    return best;
}

bool scaling_fits(bool dots, int n, int m) { return scaling_variant(dots, n, m) != nullptr; }

// (clusters of 200 KB of shared memory or tensor memory that fit, measured: 74 of two blocks, 33 of four, 15 of eight, 7 of sixteen)
int scaling_resident(const Dev &P)
{
    const int nc = scaling_blocks(P);
    return nc <= 1 ? 148 : (nc <= 2 ? 74 : (nc <= 4 ? 33 : (nc <= 8 ? 15 : 7)));
}
// The kernel with 128 or the one with 255 registers a thread, for `blocks` blocks.
static const void *cycles_kernel(const ScalingVariant *v, ScalingKind kind, const Dev &P, long long blocks)
{
    if (kind == SC_LEG) return v->kernel[kind];
    const bool mask = P.mode == MODE_MASKED && !P.early_exit;
    // Lanes in half of the tensor memory: alone on their SM with all of its registers while that makes two rounds at most.  Drain
    // of lanes of 128 x 160, d = 8, two blocks an SM -> one: 1 lane 994 -> 887 us, 148 1003 -> 905, 256 1105 -> 900, 400 1290 <- 1365,
    // 1200 3073 <- 3519.  One round under a mask, whose lanes all work to the end: 149 3822 <- 4128, 220 4532 <- 4749, 296 4608 <- 5143.
    if (v->tm_cols) return blocks <= (mask ? 148 : 2 * 148) ? v->roomy[kind] : v->kernel[kind];
    // K in 32 registers: 255 wherever lanes leave.  Where all work to the end (STATIC) or launches end together (a mask), what
    // counts beyond one round of 296 blocks is how full the last one is.  60 x 60 and 30 x 30, 128 -> 255, STATIC: 296 lanes 2033 -> 1718, 320
    // 2310 -> 2204 and 2103 <-> 2102, 360 2326 <- 2419, 592 2579 <- 2733, 1500 4715 <- 5243; mask: 296 1988 -> 1618, 320 2400 <- 2596,
    // 400 2498 <- 2687, 450 2846 -> 2718, 700 3981 -> 3722, 1500 6761 -> 6701.
    // Clusters of 64 registers, 250 x 60, 128 -> 255: STATIC 296 lanes 7632 -> 7387, 512 11.3 -> 10.8 ms, 750 14.1 -> 14.0 and 15.1 <- 15.3, 900 15.1 <- 16.5,
    // 1200 20.0 <- 23.2; a mask 27.4 -> 21.2 at 900.
    const long long places = 148 * 256 / v->threads;
    if (v->cluster) return P.mode == MODE_STATIC && blocks > 5 * places ? v->kernel[kind] : v->roomy[kind];
    const bool shared = P.mode == MODE_STATIC ? blocks > places + places / 8 : mask && blocks > places && blocks <= places + 2 * places / 5;
    return shared ? v->kernel[kind] : v->roomy[kind];
}
// Does a launch of `width` lanes take the kernel that shares an SM, where one of fewer lanes would take the one that has it alone?
bool scaling_shares_sm(const Dev &P, int width)
{
    const ScalingVariant *v = scaling_variant(P.dots != nullptr, P.n, P.m);
    return cycles_kernel(v, SC_CYCLES, P, (long long)blocks_of(*v, P.n) * width) != v->roomy[SC_CYCLES];
}
int scaling_blocks(const Dev &P) { return blocks_of(*scaling_variant(P.dots != nullptr, P.n, P.m), P.n); }

void launch_scaling(const Dev &P, ScalingKind kind, int leg, int cycles, int width, cudaStream_t st)
{
    const ScalingVariant *v = scaling_variant(P.dots != nullptr, P.n, P.m);
    const int nc = blocks_of(*v, P.n);
    const void *kernel = cycles_kernel(v, kind, P, (long long)nc * width);
    // No block may take its place on an SM and then wait there for tensor memory while blocks of its cluster hold theirs.
    // Blocks that take the whole register file are alone anyway.  Others ask for shared memory in proportion to their tensor
    // memory; without a cluster they may wait, and ask for as much as keeps one block too many away.  (No more
    // than that: what is left is the cache that spilled registers live in; with all of it asked for, a solve of 64
    // lanes of 1024 x 1024, d = 512, takes 5.9 ms instead of 5.3.)
    size_t smem = v->smem(nc), most = v->smem(v->cluster ? v->max_blocks : nc);
    if (v->tm_cols && kind != SC_LEG) {
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return;        // (the caller looks at cudaGetLastError)
        const bool alone = (fa.numRegs + 7) / 8 * 8 * v->threads >= 65536;
        const size_t share = alone ? 0 : v->cluster ? (size_t)SMEM_PER_SM * v->tm_cols / 512 : (size_t)SMEM_PER_SM / (512 / v->tm_cols + 1) + 1024;
        if (share > fa.sharedSizeBytes + smem) smem = share - fa.sharedSizeBytes;
        if (smem > most) most = smem;
    }
    // (with the fixed arrays some variants are beyond the 48 KB that need no permission; the attributes belong to the
    // current device, so they are set with every launch, to the variant's limits whatever the lane: another
    // host thread may launch the same variant for lanes of fewer blocks in between)
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (v->max_blocks > MAX_CLUSTER_RANKS) cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nc, width < 1 ? 1 : width);
    cfg.blockDim = dim3(v->threads);
    cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = nc; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = v->cluster ? 2 : 1;
    Dev dev = P;
    void *args[3] = {&dev, &leg, &cycles};
    cudaLaunchKernelExC(&cfg, kernel, args);
}

}  // namespace skb
