// Kernel of the block sweep; one translation unit per slot count W.
#pragma once

#include "cfr_sweep.cuh"

namespace pasur {
namespace {

// One item per block: its state from device memory, all iterations, and back.
template <int VARIANT, int W>
__global__ void __launch_bounds__(kBlockMaxThreads, 1) k_cfr_block(BlockParams p) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ SweepShared sh;
    const int tid = threadIdx.x;
    const BlockItem it = p.items[blockIdx.x];
    const TreeView &tv = p.views[it.tree];
    const CfrRoot &cr = tv.roots[it.root];
    const int L = cr.ls[9];
    const int64_t slot0 = tv.fgt_off0[it.root] + it.s0;
    SweepAt at;
    at.root = tv.broots + it.root;
    at.runs = tv.b_run + at.root->run_off;
    at.term = tv.b_term + cr.loc_off;
    at.place(sm, block_offsets(L, cr.as[9], at.root->rs[8], W, blockDim.x >> 5));
    if (tid < W) sh.tu[tid] = 0.f;
    int64_t base[W];
    int32_t str[W];
    float um[W];
#pragma unroll
    for (int w = 0; w < W; w++) {
        base[w] = tv.slot_base[slot0 + w];
        str[w] = tv.slot_str[slot0 + w];
        um[w] = 0.f;
    }
    __syncthreads();
    load_state<W>(at, tv, cr, cr, base, str, it.s0, um);
#pragma unroll
    for (int w = 0; w < W; w++) atomicMax((unsigned *)&sh.tu[w], __float_as_uint(um[w]));
    if (tid < W) sts(at.v + (L * W + tid) * 4, 1.f);  // the reach of the root's mover
    make_programs<W>(sh, at, 0, 15, true, 0);
    float tu[W];
#pragma unroll
    for (int w = 0; w < W; w++) tu[w] = p.tau * sh.tu[w];
    double acc = 0.0;
    const uint32_t root = at.v + 4 * tid;  // the root's value (tid < W)
    if (sh.n == 0) {
        // no active node: the root's value is its one leaf's
        if (tid < W)
            for (int il = 0; il < p.iters; il++) acc += (double)lds(root);
    } else {
        Cursor c;
        c.place<W>();
        c.start<W>(at.seg + 16 * sh.first[tid >> 5], at.seg + 16 * sh.first[(tid >> 5) + 1]);
        for (int il = 0; il < p.iters; il++) {
            const float tf = (float)(p.t0 + il + 1);
            StepFactors f{0.f, 0.f, 0.f};
            if (VARIANT == 1) f = {p.dcfr[3 * il], p.dcfr[3 * il + 1], p.dcfr[3 * il + 2]};
            float thr[W];
#pragma unroll
            for (int w = 0; w < W; w++) thr[w] = tu[w] * tf;
            run_program<VARIANT, W>(c, at, thr, f);
            // the root's value (its step is warp 0's alone), then its reach 1 in the value's place
            // again: the next top-down steps are warp 0's too, up to a block barrier
            if (tid < W) {
                acc += (double)lds(root);
                sts(root, 1.f);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    if (tid < W) {
        if (!isfinite(acc)) atomicOr(p.err, 1);
        tv.uacc[slot0 + tid] += acc;
    }
    store_state<W>(at, tv, cr, base, str);
}

template <int W>
const void *block_kernel_of(int variant) {
    return variant == 1 ? (const void *)k_cfr_block<1, W> : (const void *)k_cfr_block<0, W>;
}

}  // namespace
}  // namespace pasur
