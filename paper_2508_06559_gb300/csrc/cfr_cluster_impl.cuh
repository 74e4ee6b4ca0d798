// Kernel of the cluster sweep: a root subtree too large for one block, split over the distributed
// shared memory of a thread-block cluster; one translation unit per slot count W.
//
// CTA r of the cluster holds part r (subtrees of active level-ell nodes); CTA 0 also holds the top
// levels 0..ell-1.  Per iteration: CTA 0 runs the top-down steps of the top and pushes every active
// level-ell node's reach and its parent's reach into the owning CTA; cluster barrier; every CTA runs
// both passes over its part and pushes the node values back to CTA 0; cluster barrier; CTA 0 runs the
// bottom-up steps of the top.  Every node's arithmetic is the block sweep's.
#pragma once

#include "cfr_sweep.cuh"

namespace pasur {
namespace {

__device__ __forceinline__ uint32_t cl_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cl_id() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}
// All threads of all CTAs of the cluster; shared::cluster writes before it are visible after it.  The
// warp converges first, and the barrier is the form that does not ask for it: the compiler is free to
// leave lanes apart after a loop.
__device__ __forceinline__ void cl_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    __syncwarp();
}
// the address of this CTA's shared byte a in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cl_map(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_st(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ float cl_ld(uint32_t a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}

template <int VARIANT, int W>
__global__ void __launch_bounds__(kBlockMaxThreads, 1) k_cfr_cluster(BlockParams p, const ClusterItem *__restrict__ clu) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ SweepShared sh;
    __shared__ float s_qmax[kMaxClusterCtas][W];
    __shared__ uint32_t s_v[kMaxClusterCtas];  // per part: its values' offset in its CTA's shared memory
    const int tid = threadIdx.x, nth = blockDim.x, nw = nth >> 5;
    const uint32_t q = cl_rank();
    const ClusterItem c = clu[cl_id()];
    const TreeView &tv = p.views[c.tree];
    const CfrRoot &cr = tv.roots[c.root];
    const ClusterPart *parts = tv.cparts + c.part0;  // [0] the top, [1 + r] part r
    const CfrRoot &tr = tv.roots[parts[0].root], &pr = tv.roots[parts[1 + q].root];
    const int64_t slot0 = tv.fgt_off0[c.root] + c.s0;
    auto offsets = [&](int root) {
        const CfrRoot &r = tv.roots[root];
        return block_offsets(r.ls[9], r.as[9], tv.broots[root].rs[8], W, nw);
    };
    auto region = [&](SweepAt &at, int root, const unsigned char *from) {
        at.root = tv.broots + root;
        at.runs = tv.b_run + at.root->run_off;
        at.term = tv.b_term + tv.roots[root].loc_off;
        at.place(from, offsets(root));
    };
    // CTA 0: part 0 at offset 0, the top right after it
    const BlockOffsets o0 = offsets(parts[1].root), ot = offsets(parts[0].root);
    SweepAt at, top;
    region(at, parts[1 + q].root, sm);
    if (q == 0) region(top, parts[0].root, sm + o0.end);
    const uint32_t base = smem_addr(sm), top_v = base + o0.end + ot.V;
    if (tid < W) sh.tu[tid] = 0.f;
    if (tid < c.nparts) s_v[tid] = offsets(parts[1 + tid].root).V;
    int64_t sbase[W];
    int32_t str[W];
    float um[W];
#pragma unroll
    for (int w = 0; w < W; w++) {
        sbase[w] = tv.slot_base[slot0 + w];
        str[w] = tv.slot_str[slot0 + w];
        um[w] = 0.f;
    }
    __syncthreads();
    load_state<W>(at, tv, pr, cr, sbase, str, c.s0, um);
    if (q == 0) load_state<W>(top, tv, tr, cr, sbase, str, c.s0, um);
#pragma unroll
    for (int w = 0; w < W; w++) atomicMax((unsigned *)&sh.tu[w], __float_as_uint(um[w]));
    if (q == 0 && tid < W) sts(top.v + (tr.ls[9] * W + tid) * 4, 1.f);  // the reach of the root's mover
    // the programs of the part, and of the top's two passes (this warp's segments of each)
    const int warp = tid >> 5;
    make_programs<W>(sh, at, 0, 15, false, 0);
    const uint32_t pa = at.seg + 16 * sh.first[warp], pz = at.seg + 16 * sh.first[warp + 1];
    uint32_t da = 0, dz = 0, ua = 0, uz = 0;
    if (q == 0) {
        const int n = make_programs<W>(sh, top, 0, 7, false, 0);
        da = top.seg + 16 * sh.first[warp];
        dz = top.seg + 16 * sh.first[warp + 1];
        make_programs<W>(sh, top, 7, 15, false, n);
        ua = top.seg + 16 * sh.first[warp];
        uz = top.seg + 16 * sh.first[warp + 1];
    }
    Cursor cur;
    cur.place<W>();
    cl_sync();  // every CTA runs: its shared memory may be addressed
    if (tid < W) cl_st(cl_map(smem_addr(&s_qmax[q][tid]), 0), sh.tu[tid]);
    cl_sync();
    float tu[W];
#pragma unroll
    for (int w = 0; w < W; w++) {
        float m = 0.f;
        for (int r = 0; r < c.nparts; r++) m = fmaxf(m, cl_ld(cl_map(smem_addr(&s_qmax[r][w]), 0)));
        tu[w] = p.tau * m;
    }
    const int32_t *cx = tv.cx + 5 * c.x0;
    const int x0 = parts[1 + q].x_begin, x1 = parts[1 + q].x_end;
    const uint32_t root = top_v + 4 * tid;  // CTA 0: the root's value (tid < W)
    double acc = 0.0;
    for (int il = 0; il < p.iters; il++) {
        const float tf = (float)(p.t0 + il + 1);
        StepFactors f{0.f, 0.f, 0.f};
        if (VARIANT == 1) f = {p.dcfr[3 * il], p.dcfr[3 * il + 1], p.dcfr[3 * il + 2]};
        float thr[W];
#pragma unroll
        for (int w = 0; w < W; w++) thr[w] = tu[w] * tf;
        if (q == 0) {
            cur.start<W>(da, dz);
            run_program<VARIANT, W>(cur, top, thr, f);
            // reaches of the active level-ell nodes and of their parents, into their owners
            for (int j = tid; j < c.nx * W; j += nth) {
                const int32_t *e = cx + 5 * (j / W);
                const int w4 = j % W * 4;
                const uint32_t r = (uint32_t)e[0], v = base + s_v[r] + w4;
                cl_st(cl_map(v + e[3] * (W * 4), r), lds(top_v + e[1] * (W * 4) + w4));
                cl_st(cl_map(v + e[4] * (W * 4), r), lds(top_v + e[2] * (W * 4) + w4));
            }
        }
        cl_sync();
        cur.start<W>(pa, pz);
        run_program<VARIANT, W>(cur, at, thr, f);
        // values of the part's level-ell nodes, into the top
        for (int j = x0 * W + tid; j < x1 * W; j += nth) {
            const int32_t *e = cx + 5 * (j / W);
            const int w4 = j % W * 4;
            cl_st(cl_map(top_v + e[1] * (W * 4) + w4, 0), lds(at.v + e[3] * (W * 4) + w4));
        }
        cl_sync();
        if (q == 0) {
            cur.start<W>(ua, uz);
            run_program<VARIANT, W>(cur, top, thr, f);
            // the root's value, then its reach 1 in the value's place again (the top's next steps begin
            // on warp 0 too)
            if (tid < W) {
                acc += (double)lds(root);
                sts(root, 1.f);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    store_state<W>(at, tv, pr, sbase, str);
    if (q == 0) {
        store_state<W>(top, tv, tr, sbase, str);
        if (tid < W) {
            if (!isfinite(acc)) atomicOr(p.err, 1);
            tv.uacc[slot0 + tid] += acc;
        }
    }
    cl_sync();  // no CTA leaves while another may still address its shared memory
}

template <int W>
const void *cluster_kernel_of(int variant) {
    return variant == 1 ? (const void *)k_cfr_cluster<1, W> : (const void *)k_cfr_cluster<0, W>;
}

}  // namespace
}  // namespace pasur
