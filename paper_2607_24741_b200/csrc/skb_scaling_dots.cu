// Kernel matrices on chip: the variants for deep lanes, whose exponents come from stored dot products.
#include "skb_scaling.cuh"

namespace skb {

static const ScalingVariant g_scaling_dots[] = {
    SKB_SC(SRC_DOTS, 4, 4, 32, false, false), SKB_SC(SRC_DOTS, 4, 4, 32, true, false),
    SKB_SC(SRC_DOTS, 8, 8, 16, false, true), SKB_SC(SRC_DOTS, 8, 8, 32, false, true), SKB_SC(SRC_DOTS, 8, 8, 32, true, true),
    SKB_SC(SRC_DOTS, 8, 16, 16, true, true),
    SKB_SC(SRC_DOTS, 8, 32, 8, true, true),
};
ScalingTable scaling_table_dots() { return {g_scaling_dots, (int)(sizeof(g_scaling_dots) / sizeof(g_scaling_dots[0]))}; }

}  // namespace skb
