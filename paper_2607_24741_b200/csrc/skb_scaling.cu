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
int scaling_blocks(const Dev &P) { return blocks_of(*scaling_variant(P.dots != nullptr, P.n, P.m), P.n); }

void launch_scaling(const Dev &P, ScalingKind kind, int leg, int cycles, int width, cudaStream_t st)
{
    const ScalingVariant *v = scaling_variant(P.dots != nullptr, P.n, P.m);
    const void *kernel = v->kernel[kind];
    const int nc = blocks_of(*v, P.n);
    // Lanes in half of the tensor memory: alone on their SM with all of its registers while that makes two rounds at most.  Drain
    // of lanes of 128 x 160, d = 8, two blocks an SM -> one: 1 lane 994 -> 887 us, 148 1003 -> 905, 256 1105 -> 900, 400 1290 <- 1365,
    // 1200 3073 <- 3519.
    if (kind == SC_CYCLES && nc * width <= 2 * 148) kernel = v->roomy;
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
