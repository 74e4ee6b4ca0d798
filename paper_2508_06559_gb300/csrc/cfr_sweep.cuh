// The sweep of one item (a root, or a part of one, and W of its score slots) whose state lies in one
// block's shared memory: device code shared by the block sweep and the cluster sweep.
//
// What bounds it: the instructions and the latency of one level step, not a bandwidth.  So
//  - a lane holds one node with all W slots: entry words, addresses, branches and loops are paid once
//    per node, and the slots' dependent chains overlap;
//  - the entries of a level are ordered by degree and a warp's chunk is 32 nodes of one degree (no
//    divergence); the children of a run lie child-major (child a of the run's i-th node at
//    c0 + a * n + i, slots innermost), so a warp's accesses to regrets, strategy sums and values are
//    consecutive;
//  - everything that does not change over the iterations is resolved once per item into shared-memory
//    byte addresses, as one program per warp (a list of segments);
//  - nodes whose children are all terminals take no top-down step, and a node's reach lies in its
//    value's place until the bottom-up pass replaces it: 12 bytes of state per (node, slot).
// A pair (active node, slot) and iteration costs an SM 2.1 ns with one slot, 1.56 with two, 1.21 with four; one
// (node, slot) per thread with the entries decoded in every iteration and 16 bytes of state cost 4 to 5.  One final
// round's root (1000 iterations on one SM) took 9.7 ms so and takes 4.7; the final round of the largest deal (15,900
// roots) 0.90 and 0.41 s.
#pragma once

#include "cfr_block.cuh"
#include "cfr_node.cuh"

namespace pasur {
namespace {

// ---- shared memory by 32-bit address -----------------------------------------------------------

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint4 lds4u(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint2 lds2u(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float lds(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }

// slots w0..w0+N-1 of the W slots at a: the widest accesses the slots' alignment allows
template <int W, int w0, int N>
__device__ __forceinline__ void lds_n(uint32_t a, float *x) {
    if constexpr (W % 4 == 0 && w0 % 4 == 0 && N % 4 == 0) {
#pragma unroll
        for (int i = 0; i < N; i += 4)
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(x[i]), "=f"(x[i + 1]), "=f"(x[i + 2]), "=f"(x[i + 3])
                         : "r"(a + (w0 + i) * 4)
                         : "memory");
    } else if constexpr (W % 2 == 0 && w0 % 2 == 0 && N % 2 == 0) {
#pragma unroll
        for (int i = 0; i < N; i += 2)
            asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x[i]), "=f"(x[i + 1]) : "r"(a + (w0 + i) * 4) : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < N; i++) x[i] = lds(a + (w0 + i) * 4);
    }
}
template <int W, int w0, int N>
__device__ __forceinline__ void sts_n(uint32_t a, const float *x) {
    if constexpr (W % 4 == 0 && w0 % 4 == 0 && N % 4 == 0) {
#pragma unroll
        for (int i = 0; i < N; i += 4)
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a + (w0 + i) * 4), "f"(x[i]), "f"(x[i + 1]),
                         "f"(x[i + 2]), "f"(x[i + 3])
                         : "memory");
    } else if constexpr (W % 2 == 0 && w0 % 2 == 0 && N % 2 == 0) {
#pragma unroll
        for (int i = 0; i < N; i += 2)
            asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a + (w0 + i) * 4), "f"(x[i]), "f"(x[i + 1]) : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < N; i++) sts(a + (w0 + i) * 4, x[i]);
    }
}

// ---- one node ----------------------------------------------------------------------------------

struct StepFactors {
    float fpos, fneg, fs;
};

// a node's addresses: its first child's regret and value, its parent's and its own value, bytes from
// one child to the next; sof: from a regret to its strategy sum
struct NodeAt {
    uint32_t r, v, up, me, stride, sof;
};

// slots of a D-degree node handled at once, bounded by the registers their children take
__host__ __device__ constexpr int slot_group(int W, int D) {
    const int cap = D <= 2 ? 6 : 3;
    const int g = (W + (W + cap - 1) / cap - 1) / ((W + cap - 1) / cap);
    return g > 1 && W % 2 == 0 && g % 2 == 1 ? g - 1 : g;
}

// Top-down: the reaches of the active children (regret matching, eq. RM).  A terminal child keeps its
// value and needs no reach.
template <int D, int W, int w0 = 0>
__device__ __forceinline__ void td_node(const NodeAt &n, unsigned mask, const float *thr) {
    constexpr int g = slot_group(W, D), G = W - w0 < g ? W - w0 : g;
    float own[G], r[D][G], x[D][G];
    lds_n<W, w0, G>(n.up, own);
#pragma unroll
    for (int a = 0; a < D; a++) lds_n<W, w0, G>(n.r + a * n.stride, r[a]);
#pragma unroll
    for (int w = 0; w < G; w++) {
        float rw[D], xw[D];
#pragma unroll
        for (int a = 0; a < D; a++) rw[a] = r[a][w];
        if constexpr (D == 1) xw[0] = own[w];
        else rm_reach<D>(rw, own[w], thr[w0 + w], xw);
#pragma unroll
        for (int a = 0; a < D; a++) x[a][w] = xw[a];
    }
#pragma unroll
    for (int a = 0; a < D; a++)
        if (mask >> a & 1u) sts_n<W, w0, G>(n.v + a * n.stride, x[a]);
    if constexpr (w0 + G < W) td_node<D, W, w0 + G>(n, mask, thr);
}

// Bottom-up: the node's value, and the regret and strategy-sum updates of its child edges (bu_vals)
template <int VARIANT, int D, int W, int w0 = 0>
__device__ __forceinline__ void bu_node(const NodeAt &n, bool alex, const float *thr, const StepFactors &f) {
    constexpr int g = slot_group(W, D), G = W - w0 < g ? W - w0 : g;
    float pp[G], po[G], r[D][G], v[D][G], s[D][G], vh[G];
    lds_n<W, w0, G>(n.up, pp);
    lds_n<W, w0, G>(n.me, po);
#pragma unroll
    for (int a = 0; a < D; a++) {
        lds_n<W, w0, G>(n.r + a * n.stride, r[a]);
        lds_n<W, w0, G>(n.v + a * n.stride, v[a]);
        lds_n<W, w0, G>(n.r + n.sof + a * n.stride, s[a]);
    }
#pragma unroll
    for (int w = 0; w < G; w++) {
        float rw[D], vw[D], sw[D];
#pragma unroll
        for (int a = 0; a < D; a++) {
            rw[a] = r[a][w];
            vw[a] = v[a][w];
            sw[a] = s[a][w];
        }
        vh[w] = bu_vals<VARIANT, D>(rw, vw, sw, pp[w], alex ? po[w] : -po[w], thr[w0 + w], f.fpos, f.fneg, f.fs);
#pragma unroll
        for (int a = 0; a < D; a++) {
            r[a][w] = rw[a];
            s[a][w] = sw[a];
        }
    }
    sts_n<W, w0, G>(n.me, vh);
#pragma unroll
    for (int a = 0; a < D; a++) {
        sts_n<W, w0, G>(n.r + a * n.stride, r[a]);
        sts_n<W, w0, G>(n.r + n.sof + a * n.stride, s[a]);
    }
    if constexpr (w0 + G < W) bu_node<VARIANT, D, W, w0 + G>(n, alex, thr, f);
}

// A node of more than 8 children, one slot.  term[a * nn]: whether child a is a terminal.
__device__ __noinline__ void td_any(NodeAt n, int d, float thr, const uint8_t *term, int nn) {
    const float own = lds(n.up);
    float sum = 0.f;
    for (int a = 0; a < d; a++) {
        const float r = lds(n.r + a * n.stride);
        sum += r > thr ? r : 0.f;
    }
    const float iv = sum > 0.f ? rcp_pos(sum) : 0.f, u = own * (1.f / (float)d);
    for (int a = 0; a < d; a++) {
        const float r = lds(n.r + a * n.stride);
        const float x = sum > 0.f ? (r > thr ? own * (r * iv) : 0.f) : u;
        if (!term[a * nn]) sts(n.v + a * n.stride, x);
    }
}
template <int VARIANT>
__device__ __noinline__ void bu_any(NodeAt n, int d, bool alex, float thr, StepFactors f) {
    const float pp = lds(n.up), po = lds(n.me), spo = alex ? po : -po;
    float sum = 0.f;
    for (int a = 0; a < d; a++) {
        const float r = lds(n.r + a * n.stride);
        sum += r > thr ? r : 0.f;
    }
    const float inv = sum > 0.f ? rcp_pos(sum) : 0.f, u = 1.f / (float)d;
    const float v0 = lds(n.v);
    float vh = v0;
    for (int a = 1; a < d; a++) {
        const float r = lds(n.r + a * n.stride);
        vh += (sum > 0.f ? (r > thr ? r * inv : 0.f) : u) * (lds(n.v + a * n.stride) - v0);
    }
    for (int a = 0; a < d; a++) {
        float r = lds(n.r + a * n.stride), s = lds(n.r + n.sof + a * n.stride);
        const float sg = sum > 0.f ? (r > thr ? r * inv : 0.f) : u;
        const float inst = spo * (lds(n.v + a * n.stride) - vh);
        if (VARIANT == 1) {
            r = r * (r > 0.f ? f.fpos : f.fneg) + inst;
            s = s * f.fs + pp * sg;
        } else {
            r = r + inst;
            s = s + pp * sg;
        }
        sts(n.r + a * n.stride, r);
        sts(n.r + n.sof + a * n.stride, s);
    }
    sts(n.me, vh);
}

// ---- the warps' programs -----------------------------------------------------------------------

// A warp's program is a list of segments: each a run's nodes (or part of them) in one level step, and
// what follows it: another segment, a warp barrier or a block barrier.
// x = address of its first node's first child's regret, y = bytes from one child to the next, z =
// address of its first entry, w = nodes | degree (255: 255 or more) << 16 | flags << 24.
// An entry: address of the node's value; low 24 bits of its parent's value's address | mask of its active
// children (the first 8) << 24.  (In a cluster the bits above hold the CTA's rank.)
// A segment's lanes hold a node each with all its slots, or (kSegSpread) one (node, slot) each.
constexpr uint32_t kSegUp = 1, kSegAlex = 2, kSegSyncWarp = 4, kSegSync = 8, kSegSpread = 16;
constexpr int kSegSolo = 256, kSegSmall = 512;  // of a level step: warp 0's alone, few nodes (not stored in segments)
// Most chunks of a step that is warp 0's alone.  With one, a final round of 1000 iterations, the last four rounds, six
// rounds and 64 deals take 5.6, 23.1, 48.1 and 165 ms; with none 5.9, 24.2, 48.9, 168; with two 5.6, 24.2, 49.6, 170; with
// four 7.4, -, 58.6, 193.  (Here and below: one comparison on one GPU; from one to another the longer ones differ by up to 8 %.)
constexpr int kSoloChunks = 1;

struct SweepShared {
    int r0[16], r1[16], fl[16], n;  // level steps: runs, flags
    int first[33];                  // first segment of every warp
    float tu[8];
};

// where a sweep's arrays lie (see BlockOffsets) and the root's tables
struct SweepAt {
    uint32_t seg, ent, r, v, sof, vof, hi;  // vof: from a regret to its value; hi: the addresses' bits above 23
    const BlockRun *runs;
    const BlockRoot *root;
    const uint8_t *term;  // per block index: 1 for a terminal (global memory)
    __device__ __forceinline__ void place(const void *sm, const BlockOffsets &o) {
        seg = smem_addr(sm);
        ent = seg + o.ent;
        r = seg + o.R;
        v = seg + o.V;
        sof = o.S - o.R;
        vof = o.V - o.R;
        hi = seg & 0xFF000000u;
        // opaque: kept in registers instead of being derived from the block's shared window again
        asm volatile("" : "+r"(seg), "+r"(ent), "+r"(r), "+r"(v), "+r"(sof), "+r"(vof), "+r"(hi));
    }
};

// whether the lanes of a run's chunks hold one (node, slot) each: nodes of many children (their slots
// would run one after the other), and steps with too few nodes to occupy the warps
template <int W>
__device__ __forceinline__ bool run_spread(const BlockRun &r, bool small) { return W > 1 && (r.d > 4 || small); }
template <int W>
__device__ __forceinline__ int run_tile(const BlockRun &r, bool small) { return run_spread<W>(r, small) ? 32 / W : 32; }
template <int W>
__device__ __forceinline__ int run_chunks(const BlockRun &r, bool small) {
    const int t = run_tile<W>(r, small);
    return (r.n + t - 1) / t;
}
// the weight of one of its chunks: about its issue slots
template <int W>
__device__ __forceinline__ int run_weight(const BlockRun &r, bool small) {
    return run_spread<W>(r, small) ? 6 + 3 * min((int)r.d, 64) : 6 + (W + 2) * (int)min((int)r.d, 64);
}

// The chunks of a level step (runs r0..r1-1 in order) shared out by weight: the place (run, chunk)
// where warp i's part of nw begins.
template <int W>
__device__ __forceinline__ int2 step_cut(const BlockRun *runs, int r0, int r1, bool small, int64_t total, int i, int nw) {
    int64_t at = total * i / nw;
    for (int r = r0; r < r1; r++) {
        const int m = run_chunks<W>(runs[r], small), w = run_weight<W>(runs[r], small);
        if (at < (int64_t)m * w) return make_int2(r, (int)(at / w));
        at -= (int64_t)m * w;
    }
    return make_int2(r1, 0);
}

// Level steps i0..i1-1 of one iteration (i < 7 the top-down levels 0..6 over the runs with an active
// child, i >= 7 the bottom-up levels 7..0 over all; empty ones left out) as the warps' programs, from
// segment `base` on (the end is returned).  A step of few chunks is warp 0's alone; after it a warp
// barrier suffices where the next one is too (cyclic: the last step's next is the first).
template <int W>
__device__ __forceinline__ int make_programs(SweepShared &sh, const SweepAt &at, int i0, int i1, bool cyclic, int base) {
    const int tid = threadIdx.x, warp = tid >> 5, nw = blockDim.x >> 5, i = tid & 31;
    const BlockRoot &br = *at.root;
    __syncthreads();
    if (tid == 0) {
        int n = 0;
        for (int x = i0; x < i1; x++) {
            const int k = x < 7 ? x : 14 - x, r0 = br.rs[k], r1 = x < 7 ? br.rt[k] : br.rs[k + 1];
            if (r1 <= r0) continue;
            int m = 0;
            for (int r = r0; r < r1; r++) m += (at.runs[r].n + 31) >> 5;
            const bool small = m <= nw / 2;  // half the warps idle (a quarter: 64 deals 168 ms, all: 165, this: 165)
            m = 0;
            for (int r = r0; r < r1; r++) m += run_chunks<W>(at.runs[r], small);
            sh.r0[n] = r0;
            sh.r1[n] = r1;
            sh.fl[n++] = (x < 7 ? 0 : kSegUp) | ((k & 1) == 0 ? kSegAlex : 0) | (m <= kSoloChunks ? kSegSolo : 0) | (small ? kSegSmall : 0);
        }
        sh.n = n;
        for (int x = 0; x < n; x++) {
            const bool end = x + 1 == n;
            const bool solo = (sh.fl[x] & kSegSolo) && (!end || cyclic) && (sh.fl[end ? 0 : x + 1] & kSegSolo);
            sh.fl[x] |= solo ? kSegSyncWarp : kSegSync;
        }
        sh.first[0] = base;
    }
    __syncthreads();
    // lane l of a warp takes step l of the warp's program: counted first, then written in step order
    const int n_steps = sh.n;
    int2 a = make_int2(0, 0), z = make_int2(0, 0);
    int cnt = 0, fl = 0;
    bool small = false;
    if (i < n_steps) {
        fl = sh.fl[i];
        small = fl & kSegSmall;
        const int r0 = sh.r0[i], r1 = sh.r1[i];
        if (fl & kSegSolo) {
            a = warp == 0 ? make_int2(r0, 0) : make_int2(r1, 0);
            z = make_int2(r1, 0);
        } else {
            int64_t total = 0;
            for (int r = r0; r < r1; r++) total += (int64_t)run_chunks<W>(at.runs[r], small) * run_weight<W>(at.runs[r], small);
            a = step_cut<W>(at.runs, r0, r1, small, total, warp, nw);
            z = step_cut<W>(at.runs, r0, r1, small, total, warp + 1, nw);
        }
        cnt = a.x == z.x ? (z.y > a.y ? 1 : 0) : z.x - a.x + (z.y > 0 ? 1 : 0);
        if (cnt <= 0) cnt = fl & kSegSync ? 1 : 0;  // without work: the barrier alone
    }
    int pre = cnt;
    for (int s = 1; s < 32; s <<= 1) {
        const int u = __shfl_up_sync(0xFFFFFFFFu, pre, s);
        if (i >= s) pre += u;
    }
    if (i == 31) sh.first[warp + 1] = pre;
    __syncthreads();
    if (tid == 0)
        for (int x = 0; x < nw; x++) sh.first[x + 1] += sh.first[x];
    __syncthreads();
    uint32_t out = at.seg + 16 * (sh.first[warp] + pre - cnt);
    const uint32_t keep = (uint32_t)fl & (kSegUp | kSegAlex), sync = (uint32_t)fl & (kSegSync | kSegSyncWarp);
    auto put = [&](uint32_t x, uint32_t y, uint32_t zz, uint32_t w) {
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(out), "r"(x), "r"(y), "r"(zz), "r"(w) : "memory");
        out += 16;
    };
    int n = 0;
    for (int r = a.x; i < n_steps && (r < z.x || (r == z.x && z.y > (r == a.x ? a.y : 0))); r++) {
        const BlockRun run = at.runs[r];
        const int tile = run_tile<W>(run, small), from = (r == a.x ? a.y : 0) * tile, to = r == z.x ? z.y * tile : run.n;
        const uint32_t spread = run_spread<W>(run, small) ? kSegSpread : 0u;
        n++;
        put(at.r + (run.c0 + from) * W * 4, run.n * W * 4, at.ent + (run.e0 + from) * 8,
            (uint32_t)(min(to, (int)run.n) - from) | (uint32_t)min((int)run.d, 255) << 16 | (keep | spread | (n == cnt ? sync : 0u)) << 24);
    }
    if (n == 0 && cnt == 1) put(0, 0, 0, sync << 24);
    __syncthreads();
    return sh.first[nw];
}

__device__ __noinline__ int run_degree(const BlockRun *runs, int n_runs, int e) {
    for (int r = 0; r < n_runs; r++)
        if (e >= runs[r].e0 && e < runs[r].e0 + runs[r].n) return runs[r].d;
    return 0;
}

// A warp's place in its program: the current segment and its first entry, read ahead (they never
// change) so that nothing but the entry's load is left between a segment's work and its barrier.
struct Cursor {
    uint32_t first, last, pa;
    uint4 sg;
    uint2 en;
    // the lane's place where a lane holds one (node, slot): node, slot * 4
    uint32_t lane, q, w4;
    template <int W>
    __device__ __forceinline__ void place() {
        lane = threadIdx.x & 31;
        q = lane < 32 / W * W ? lane / W : 1u << 16;
        w4 = lane < 32 / W * W ? lane % W * 4 : 0;
        asm volatile("" : "+r"(lane), "+r"(q), "+r"(w4));
    }
    template <int W>
    __device__ __forceinline__ void entry() {
        const uint32_t node = W > 1 && (sg.w & kSegSpread << 24) ? q : lane;
        if (node < (sg.w & 0xFFFFu)) en = lds2u(sg.z + 8 * node);
    }
    template <int W>
    __device__ __forceinline__ void start(uint32_t seg0, uint32_t seg1) {
        first = pa = seg0;
        last = seg1;
        if (first != last) {
            sg = lds4u(pa);
            entry<W>();
        }
    }
};

// A segment's chunks of nodes of d children.  M: slots a lane holds (W, or 1 with the slots spread
// over the lanes).
template <int VARIANT, int W, int M>
__device__ __forceinline__ void run_segment(const SweepAt &at, uint32_t ctl, const uint4 &sg, uint2 en, uint32_t node, uint32_t w4,
                                            uint32_t ofs, const float *thr, const StepFactors &f) {
    constexpr int T = M == W ? 32 : 32 / W;
    const uint32_t flags = ctl >> 24, d = ctl >> 16 & 255u;
    const bool alex = flags & kSegAlex;
    int chunks = ((int)(ctl & 0xFFFFu) + T - 1) / T;
    int left = (int)(ctl & 0xFFFFu) - (int)node;  // the lane has a node while it is positive
    uint32_t ea = sg.z + 8 * node;
    NodeAt n{sg.x + ofs, 0, 0, 0, sg.y, at.sof};
    n.v = n.r + at.vof;
    auto each = [&](auto body) {
        do {
            if (left > 0) {
                n.me = en.x;
                n.up = (en.y & 0xFFFFFFu) | at.hi;
                if constexpr (M != W) {
                    n.me += w4;
                    n.up += w4;
                }
                body();
            }
            left -= T;
            if (--chunks == 0) break;
            ea += 8 * T;
            n.r += T * W * 4;
            n.v += T * W * 4;
            if (left > 0) en = lds2u(ea);
        } while (true);
    };
    if (!(flags & kSegUp)) {
        if (d == 2) each([&]() { td_node<2, M>(n, en.y >> 24, thr); });
        else if (d == 3) each([&]() { td_node<3, M>(n, en.y >> 24, thr); });
        else if (d == 4) each([&]() { td_node<4, M>(n, en.y >> 24, thr); });
        else if (d == 1) each([&]() { td_node<1, M>(n, en.y >> 24, thr); });
        else if constexpr (M == 1) {
            if (d == 5) each([&]() { td_node<5, 1>(n, en.y >> 24, thr); });
            else if (d == 6) each([&]() { td_node<6, 1>(n, en.y >> 24, thr); });
            else if (d == 7) each([&]() { td_node<7, 1>(n, en.y >> 24, thr); });
            else if (d == 8) each([&]() { td_node<8, 1>(n, en.y >> 24, thr); });
            else
                each([&]() {
                    const int dd = d < 255 ? (int)d : run_degree(at.runs, at.root->rs[8], (int)(ea - at.ent) / 8);
                    td_any(n, dd, thr[0], at.term + (n.r - at.r) / (W * 4), n.stride / (W * 4));
                });
        }
    } else {
        if (d == 2) each([&]() { bu_node<VARIANT, 2, M>(n, alex, thr, f); });
        else if (d == 3) each([&]() { bu_node<VARIANT, 3, M>(n, alex, thr, f); });
        else if (d == 4) each([&]() { bu_node<VARIANT, 4, M>(n, alex, thr, f); });
        else if (d == 1) each([&]() { bu_node<VARIANT, 1, M>(n, alex, thr, f); });
        else if constexpr (M == 1) {
            if (d == 5) each([&]() { bu_node<VARIANT, 5, 1>(n, alex, thr, f); });
            else if (d == 6) each([&]() { bu_node<VARIANT, 6, 1>(n, alex, thr, f); });
            else if (d == 7) each([&]() { bu_node<VARIANT, 7, 1>(n, alex, thr, f); });
            else if (d == 8) each([&]() { bu_node<VARIANT, 8, 1>(n, alex, thr, f); });
            else
                each([&]() {
                    const int dd = d < 255 ? (int)d : run_degree(at.runs, at.root->rs[8], (int)(ea - at.ent) / 8);
                    bu_any<VARIANT>(n, dd, alex, thr[0], f);
                });
        }
    }
}

// One pass through a warp's program.
template <int VARIANT, int W>
__device__ __forceinline__ void run_program(Cursor &c, const SweepAt &at, const float *thr, const StepFactors &f) {
    if (c.first == c.last) return;
    float thr1 = thr[0];
    if constexpr (W > 1) {
#pragma unroll
        for (int w = 1; w < W; w++)
            if (c.w4 == 4 * w) thr1 = thr[w];
    }
    do {
        // the same in every lane: a reduction tells the compiler, whose branches on it are uniform
        const uint32_t ctl = __reduce_or_sync(0xFFFFFFFFu, c.sg.w);
        const uint4 sg = c.sg;
        const uint2 en = c.en;
        c.pa = c.pa + 16 == c.last ? c.first : c.pa + 16;
        c.sg = lds4u(c.pa);
        if (ctl >> 16 & 255u) {
            if (W > 1 && (ctl & kSegSpread << 24)) run_segment<VARIANT, W, 1>(at, ctl, sg, en, c.q, c.w4, c.lane * 4, &thr1, f);
            else run_segment<VARIANT, W, W>(at, ctl, sg, en, c.lane, 0, c.lane * (W * 4), thr, f);
        }
        c.entry<W>();
        if (ctl & kSegSync << 24) __syncthreads();
        else if (ctl & kSegSyncWarp << 24) __syncwarp();
    } while (c.pa != c.first);
}

// Entries as addresses; regrets and strategy sums from their places in device memory; values of the
// terminals (constant over the iterations), other values 1 (the root's reach; the others are written
// before they are read); per slot the largest |terminal value| into um (per thread).  xr: the root or
// pseudo-root, cr: the root whose local nodes it is made of (nodes without one, inv < 0, have no
// regret of their own here).
template <int W>
__device__ __forceinline__ void load_state(const SweepAt &at, const TreeView &tv, const CfrRoot &xr, const CfrRoot &cr,
                                           const int64_t *base, const int32_t *str, int64_t s0, float *um) {
    const int tid = threadIdx.x, nth = blockDim.x, L = xr.ls[9], nA = xr.as[9];
    const uint32_t *ge = tv.b_ent + xr.act_off;
    const uint8_t *gm = tv.b_msk + xr.act_off;
    for (int i = tid; i < nA; i += nth) {
        const uint32_t e = ge[i], up = e >> 16 == 0xFFFFu ? (uint32_t)L : e >> 16;
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(at.ent + 8 * i), "r"(at.v + (e & 0xFFFFu) * (W * 4)),
                     "r"((at.v + up * (W * 4) & 0xFFFFFFu) | (uint32_t)gm[i] << 24)
                     : "memory");
    }
    const int32_t *inv = tv.b_inv + xr.loc_off;
    const int64_t *tq = tv.loc_tq + cr.loc_off;
    for (int x = tid; x < L; x += nth) {
        const int l = inv[x];
        const int64_t q = l < 0 ? -1 : tq[l];
#pragma unroll
        for (int w = 0; w < W; w++) {
            const int64_t g = base[w] + (int64_t)l * str[w];
            sts(at.r + (x * W + w) * 4, l < 0 ? 0.f : tv.R[g]);
            sts(at.r + at.sof + (x * W + w) * 4, l < 0 ? 0.f : tv.S[g]);
            float v = 1.f;
            if (q >= 0) {
                v = tv.leaf_v[q + s0 + w];
                um[w] = fmaxf(um[w], fabsf(v));
            }
            sts(at.v + (x * W + w) * 4, v);
        }
    }
}

template <int W>
__device__ __forceinline__ void store_state(const SweepAt &at, const TreeView &tv, const CfrRoot &xr, const int64_t *base,
                                            const int32_t *str) {
    const int32_t *inv = tv.b_inv + xr.loc_off;
    for (int x = threadIdx.x; x < xr.ls[9]; x += blockDim.x) {
        const int l = inv[x];
        if (l < 0) continue;
#pragma unroll
        for (int w = 0; w < W; w++) {
            const int64_t g = base[w] + (int64_t)l * str[w];
            tv.R[g] = lds(at.r + (x * W + w) * 4);
            tv.S[g] = lds(at.r + at.sof + (x * W + w) * 4);
        }
    }
}

}  // namespace
}  // namespace pasur
