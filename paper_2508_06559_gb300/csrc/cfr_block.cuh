// The block sweep: all T iterations of one work item (a root and a run of its score slots) in one
// thread block, its state on chip.  Host-side declarations and the layout shared with cfr_sweep.cuh.
#pragma once

#include "pasur_internal.cuh"

namespace pasur {

constexpr int kBlockSlots = 6;        // most score slots of one item
constexpr int kBlockMaxThreads = 512;

struct BlockParams {
    const BlockItem *items;
    const TreeView *views;
    const float *dcfr;  // per iteration: regret factor if R > 0, if R <= 0, strategy-sum factor
    int iters;
    int64_t t0;
    float tau;          // dead zone: a regret counts as positive above tau * t * Umax(root)
    int32_t *err;
};

// byte offsets of an item's arrays in shared memory: the warps' segments (16 B; per level step at most
// one per warp and one per run) at 0, entries (8 B), then per (node, slot) regrets, strategy sums and
// values (one node more: the reach of the root's mover)
struct BlockOffsets {
    uint32_t ent, R, S, V, end;
};
__host__ __device__ __forceinline__ BlockOffsets block_offsets(int64_t L, int64_t nA, int64_t nr, int W, int warps) {
    auto up = [](int64_t x) { return (uint32_t)((x + 15) & ~(int64_t)15); };
    BlockOffsets o;
    o.ent = (uint32_t)(2 * nr + 15 * warps) * 16;
    o.R = o.ent + up(nA * 8);
    o.S = o.R + up(L * W * 4);
    o.V = o.S + up(L * W * 4);
    o.end = o.V + up((L + 1) * W * 4);
    return o;
}

// the kernels for items of W slots (one translation unit per W)
const void *block_kernel(int variant, int W);
const void *cluster_kernel(int variant, int W);
#define PASUR_SWEEP_KERNELS(W)                   \
    const void *block_kernel_w##W(int variant);  \
    const void *cluster_kernel_w##W(int variant);
PASUR_SWEEP_KERNELS(1)
PASUR_SWEEP_KERNELS(2)
PASUR_SWEEP_KERNELS(3)
PASUR_SWEEP_KERNELS(4)
PASUR_SWEEP_KERNELS(5)
PASUR_SWEEP_KERNELS(6)
#undef PASUR_SWEEP_KERNELS

}  // namespace pasur
