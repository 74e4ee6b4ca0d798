// CFR over an unfolded round (section "CFR Algorithm"; eq. RM, eq. avsigma; DCFR eqs.
// DFCR_REG / DFCR_AVG).
//
// Round roots are independent (open hands: every FGT node is its own information set and root
// reach is 1), so the round is cut into work items: one GT root and a run of W of its score
// slots.  One thread block runs all T iterations of an item (cfr_sweep.cuh): per iteration a top-down
// pass over levels 0..6 (regret matching and reach) and a bottom-up pass over levels 7..0 (values,
// regret and strategy-sum updates), with a block barrier between levels (a warp barrier between levels
// of one chunk each, which one warp steps through); an (active node, slot) pair belongs to one thread in
// each pass, so the updates of a node's child edges need no atomics.
//
// Forced-move chains are resolved once: a node whose whole subtree is one path of single moves
// has sigma = 1 and zero regret on every edge below it and the value of its one leaf, so only the
// "active" nodes (a local node that is not such a chain) are swept, and state is kept only for
// local nodes (the root and the children of active nodes).  The item's regrets R, strategy sums
// S, values V and reaches live in shared memory for all T iterations (no DRAM traffic per
// iteration).  A root whose state does not fit one block is split over a thread-block cluster
// (distributed shared memory) or, beyond a cluster, swept level by level over every SM with its
// state in device memory.  Between calls R and S lie in device memory, local node index times slots,
// slot-minor; the local nodes of each level are numbered in the order of their parents' entries, so
// the children of consecutive entries are consecutive.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <memory>
#include <new>
#include <string>

#include "cfr_block.cuh"
#include "cfr_node.cuh"
#include "cfr_split.cuh"
#include "pasur_internal.cuh"

namespace pasur {
namespace {

// forked streams: the level-streaming sweep, then the cluster and block launches in turn (the first of them takes the
// context's own stream)
constexpr int kAuxStream = 0, kAuxSweep = 1;
// solved slots per SM and per slot of an item: below it items take fewer slots, so that the GPU has blocks (1 and 4
// measured the same: rounds have either many slots or few)
constexpr int64_t kSlotsPerSm = 2;

struct CfrParams {
    const CfrItem *items;
    const TreeView *views;
    const float *dcfr;  // per iteration: regret factor if R > 0, if R <= 0, strategy-sum factor
    int iters;
    int64_t t0;
    float tau;  // dead zone: a regret counts as positive above tau * t * Umax(root)
    int32_t *err;
};

// whether W slots of a root fit one block of the sweep (node indices and the root's mark in 16 bits)
bool block_fits(const CfrRoot &cr, const BlockRoot &br, int W, size_t limit) {
    return cr.ls[9] < 65535 && block_offsets(cr.ls[9], cr.as[9], br.rs[8], W, kBlockMaxThreads / 32).end <= limit;
}

// Index of child edge a of a node whose first child is local node c, at slot w of an item of
// 2^sh slots (slot-minor layout; every item's slot count is a power of two).
__device__ __forceinline__ int at(int c, int a, int sh, int w) {
    return ((c + a) << sh) + w;
}

// Regret matching at one (active node, slot) with D children and the reach of the children.
// X[n] holds the reach of the player who moved into node n; own = the mover's reach at the node.
template <int D>
__device__ __forceinline__ void td_node(int c, int sh, int w, float own, const float *__restrict__ R, float *__restrict__ X,
                                        float thr) {
    if constexpr (D == 1) {
        X[at(c, 0, sh, w)] = own;
        return;
    } else {
        float r[D], x[D];
#pragma unroll
        for (int a = 0; a < D; a++) r[a] = R[at(c, a, sh, w)];
        rm_reach<D>(r, own, thr, x);
#pragma unroll
        for (int a = 0; a < D; a++) X[at(c, a, sh, w)] = x[a];
    }
}

__device__ __forceinline__ void td_node_any(int c, int d, int sh, int w, float own, const float *__restrict__ R,
                                            float *__restrict__ X, float thr) {
    float sum = 0.f;
    for (int a = 0; a < d; a++) {
        const float r = R[at(c, a, sh, w)];
        sum += r > thr ? r : 0.f;
    }
    if (sum > 0.f) {
        const float inv = rcp_pos(sum);
        for (int a = 0; a < d; a++) {
            const float r = R[at(c, a, sh, w)];
            X[at(c, a, sh, w)] = r > thr ? own * (r * inv) : 0.f;
        }
    } else {
        const float u = own * (1.f / (float)d);
        for (int a = 0; a < d; a++) X[at(c, a, sh, w)] = u;
    }
}

// Value of one (active node, slot) with D children and the updates of its child edges (bu_vals)
// in R and S.  Returns v(h).
template <int VARIANT, int D>
__device__ __forceinline__ float bu_node(int c, int sh, int w, float pp, float spo, float *__restrict__ R,
                                         float *__restrict__ S, const float *__restrict__ V, float thr, float fpos,
                                         float fneg, float fs) {
    float r[D], v[D], s[D];
#pragma unroll
    for (int a = 0; a < D; a++) {
        const int q = at(c, a, sh, w);
        r[a] = R[q];
        v[a] = V[q];
        s[a] = S[q];
    }
    const float vh = bu_vals<VARIANT, D>(r, v, s, pp, spo, thr, fpos, fneg, fs);
#pragma unroll
    for (int a = 0; a < D; a++) {
        const int q = at(c, a, sh, w);
        R[q] = r[a];
        S[q] = s[a];
    }
    return vh;
}

template <int VARIANT>
__device__ __forceinline__ float bu_node_any(int c, int d, int sh, int w, float pp, float spo, float *__restrict__ R,
                                             float *__restrict__ S, const float *__restrict__ V, float thr, float fpos,
                                             float fneg, float fs) {
    float sum = 0.f;
    for (int a = 0; a < d; a++) {
        const float r = R[at(c, a, sh, w)];
        sum += r > thr ? r : 0.f;
    }
    const float inv = sum > 0.f ? rcp_pos(sum) : 0.f, u = 1.f / (float)d;
    const float v0 = V[at(c, 0, sh, w)];
    float vh = v0;
    for (int a = 1; a < d; a++) {
        const float r = R[at(c, a, sh, w)];
        vh += (sum > 0.f ? (r > thr ? r * inv : 0.f) : u) * (V[at(c, a, sh, w)] - v0);
    }
    for (int a = 0; a < d; a++) {
        const int q = at(c, a, sh, w);
        const float r = R[q];
        const float sg = sum > 0.f ? (r > thr ? r * inv : 0.f) : u;
        const float inst = spo * (V[q] - vh);
        if (VARIANT == 1) {
            R[q] = r * (r > 0.f ? fpos : fneg) + inst;
            S[q] = S[q] * fs + pp * sg;
        } else {
            R[q] = r + inst;
            S[q] = S[q] + pp * sg;
        }
    }
    return vh;
}

template <int VARIANT>
__device__ __forceinline__ void dcfr_factors(const CfrParams &p, int il, float &fpos, float &fneg, float &fs) {
    fpos = fneg = fs = 0.f;
    if (VARIANT == 1) {
        fpos = p.dcfr[3 * il];
        fneg = p.dcfr[3 * il + 1];
        fs = p.dcfr[3 * il + 2];
    }
}

// ---- class 5: a level-streaming sweep over every SM --------------------------------------------
//
// Items whose state lives in device memory are not given one block each: every level step of an
// iteration is one launch over the (entry, slot) pairs of that level of all such items of the
// plan, spread over the whole grid (the launch boundary is the level barrier).  A pair runs the
// same node code as in a block, so the results are the block sweep's bit for bit.

struct StreamPlan {
    const int64_t *pairs;  // [8][n + 1] exclusive prefix of (entry, slot) pairs per level
    const int64_t *locs;   // [n + 1] of (local node, slot) pairs
    const int64_t *slots;  // [n + 1] of slots
    uint32_t *tu;          // per slot: largest |terminal value| (float bits)
    double *acc;           // per slot: sum of the root values of the current call
    int64_t n;
    const StreamDesc *desc;  // [n] per item
};

// j with pre[j] <= x < pre[j + 1] (pre[0] = 0 <= x < pre[n])
__device__ __forceinline__ int64_t stream_item(const int64_t *pre, int64_t n, int64_t x) {
    int64_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (pre[mid] <= x) lo = mid;
        else hi = mid;
    }
    return lo;
}

// the prefixes and descriptors of a plan's class-5 items (one thread; once per plan)
__global__ void k_stream_plan(const CfrItem *items, int64_t n, const TreeView *views, int64_t *pairs, int64_t *locs,
                              const int64_t *slots, StreamDesc *desc) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    int64_t pk[8] = {0}, pl = 0;
    for (int64_t j = 0; j < n; j++) {
        const CfrItem it = items[j];
        const TreeView &tv = views[it.tree];
        const CfrRoot &cr = tv.roots[it.root];
        for (int k = 0; k < 8; k++) {
            pairs[(int64_t)k * (n + 1) + j] = pk[k];
            pk[k] += (int64_t)(cr.as[k + 1] - cr.as[k]) * it.ns;
        }
        locs[j] = pl;
        pl += (int64_t)cr.ls[9] * it.ns;
        StreamDesc sd;
        sd.R = tv.R + it.data_base;
        sd.S = tv.S + it.data_base;
        sd.V = tv.V + it.scratch_base;
        sd.X = tv.X + it.scratch_base;
        sd.li = tv.act_li + cr.act_off;
        sd.pl = tv.act_pl + cr.act_off;
        sd.cs = tv.act_cs + cr.act_off;
        sd.d = tv.act_d + cr.act_off;
        for (int k = 0; k < 9; k++) sd.as[k] = cr.as[k];
        sd.ns = it.ns;
        sd.sh = __ffs(it.ns) - 1;
        sd.slot = slots[j];
        desc[j] = sd;
    }
    for (int k = 0; k < 8; k++) pairs[(int64_t)k * (n + 1) + n] = pk[k];
    locs[n] = pl;
}

// terminal values and the dead-zone scale per slot, root reach 1, sums cleared
__global__ void k_stream_setup(CfrParams p, StreamPlan sp) {
    const int64_t total = sp.locs[sp.n];
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = stream_item(sp.locs, sp.n, x);
        const CfrItem it = p.items[j];
        const TreeView &tv = p.views[it.tree];
        const CfrRoot &cr = tv.roots[it.root];
        const int sh = __ffs(it.ns) - 1;
        const int64_t r = x - sp.locs[j];
        const int li = (int)(r >> sh), w = (int)(r & (it.ns - 1));
        float *V = tv.V + it.scratch_base, *X = tv.X + it.scratch_base;
        const int64_t q = tv.loc_tq[cr.loc_off + li];
        if (q >= 0) {
            const float v = tv.leaf_v[q + it.s0 + w];
            V[r] = v;
            atomicMax(&sp.tu[sp.slots[j] + w], __float_as_uint(fabsf(v)));
        }
        if (li == 0) {
            X[w] = 1.f;
            sp.acc[sp.slots[j] + w] = 0.0;
        }
    }
}

// One (entry, slot) pair of level k of a streamed item: the block sweep's node code on the item's
// arrays in device memory.
template <int VARIANT, bool TD>
__device__ __forceinline__ void stream_pair(const StreamDesc &sd, int k, int64_t r, const StreamPlan &sp, float tau,
                                            float tf, bool alex, float fpos, float fneg, float fs) {
    const int sh = sd.sh;
    const int e = sd.as[k] + (int)(r >> sh), w = (int)(r & (sd.ns - 1));
    const int c = sd.cs[e], d = sd.d[e], li = sd.li[e], pl = sd.pl[e];
    float *R = sd.R, *S = sd.S, *V = sd.V, *X = sd.X;
    // the dead zone rounded as in the block sweep: (tau * Umax) * t
    const float thr = (tau * __uint_as_float(sp.tu[sd.slot + w])) * tf;
    if (TD) {
        const float own = pl < 0 ? 1.f : X[(pl << sh) + w];
        switch (d) {
            case 1: td_node<1>(c, sh, w, own, R, X, thr); break;
            case 2: td_node<2>(c, sh, w, own, R, X, thr); break;
            case 3: td_node<3>(c, sh, w, own, R, X, thr); break;
            case 4: td_node<4>(c, sh, w, own, R, X, thr); break;
            case 5: td_node<5>(c, sh, w, own, R, X, thr); break;
            case 6: td_node<6>(c, sh, w, own, R, X, thr); break;
            case 7: td_node<7>(c, sh, w, own, R, X, thr); break;
            case 8: td_node<8>(c, sh, w, own, R, X, thr); break;
            default: td_node_any(c, d, sh, w, own, R, X, thr);
        }
    } else {
        const float pp = pl < 0 ? 1.f : X[(pl << sh) + w];
        const float po = X[(li << sh) + w];
        const float spo = alex ? po : -po;
        float vh;
        switch (d) {
            case 1: vh = bu_node<VARIANT, 1>(c, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs); break;
            case 2: vh = bu_node<VARIANT, 2>(c, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs); break;
            case 3: vh = bu_node<VARIANT, 3>(c, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs); break;
            case 4: vh = bu_node<VARIANT, 4>(c, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs); break;
            case 5: vh = bu_node<VARIANT, 5>(c, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs); break;
            case 6: vh = bu_node<VARIANT, 6>(c, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs); break;
            case 7: vh = bu_node<VARIANT, 7>(c, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs); break;
            case 8: vh = bu_node<VARIANT, 8>(c, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs); break;
            default: vh = bu_node_any<VARIANT>(c, d, sh, w, pp, spo, R, S, V, thr, fpos, fneg, fs);
        }
        V[(li << sh) + w] = vh;
        if (k == 0) sp.acc[sd.slot + w] += (double)vh;  // the root (one entry per item)
    }
}

constexpr int kStreamThreads = 256;

// One level step (level k; top-down or bottom-up) of iteration il of every class-5 item: a
// grid-stride loop over the level's (entry, slot) pairs of all items (consecutive threads on
// consecutive slots and entries); each pair finds its item by a binary search over the level's
// prefix (a few cached loads) and reads what it needs from the item's descriptor.
template <int VARIANT, bool TD>
__global__ void __launch_bounds__(kStreamThreads, TD ? 4 : 3) k_stream_level(CfrParams p, StreamPlan sp, int k, int il) {
    const int64_t *pre = sp.pairs + (int64_t)k * (sp.n + 1);
    const int64_t total = pre[sp.n];
    const float tf = (float)(p.t0 + il + 1);
    float fpos, fneg, fs;
    dcfr_factors<VARIANT>(p, il, fpos, fneg, fs);
    const bool alex = (k & 1) == 0;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = stream_item(pre, sp.n, x);
        stream_pair<VARIANT, TD>(sp.desc[j], k, x - pre[j], sp, p.tau, tf, alex, fpos, fneg, fs);
    }
}

// the call's root values into the running sums (a root without moves keeps its terminal value)
__global__ void k_stream_finalize(CfrParams p, StreamPlan sp) {
    const int64_t total = sp.slots[sp.n];
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = stream_item(sp.slots, sp.n, x);
        const CfrItem it = p.items[j];
        const TreeView &tv = p.views[it.tree];
        const CfrRoot &cr = tv.roots[it.root];
        const int w = (int)(x - sp.slots[j]);
        double acc = sp.acc[x];
        if (cr.as[1] == cr.as[0]) {
            const float v = tv.V[it.scratch_base + w];
            acc = 0.0;
            for (int il = 0; il < p.iters; il++) acc += (double)v;
        }
        if (!isfinite(acc)) atomicOr(p.err, 1);
        tv.uacc[tv.fgt_off0[it.root] + it.s0 + w] += acc;
    }
}

struct LevelPtrs {
    const int64_t *fgt[9];
    const int64_t *child[9];
    int64_t base[9];  // offset of level k in the concatenated edge output (levels 1..8)
};

__global__ void k_fill(float *out, int64_t n, float v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) out[i] = v;
}

// average strategy of the child edges of every active node, canonical FGT order, one or more blocks per
// item (every other edge lies below a forced move and has average strategy 1)
__global__ void k_export_sigma(const CfrItem *items, int64_t n_items, const CfrRoot *roots, const int32_t *act_cs,
                               const uint16_t *act_d, const int64_t *act_gt, const float *Sg, LevelPtrs lp, float *out) {
    for (int64_t id = blockIdx.x; id < n_items; id += gridDim.x) {
        const CfrItem it = items[id];
        const CfrRoot &cr = roots[it.root];
        const int W = it.ns;
        const int64_t n = (int64_t)cr.as[8] * W;
        const float *S = Sg + it.data_base;
        int k = 0;
        for (int64_t x = (int64_t)cr.as[0] * W + blockIdx.y * blockDim.x + threadIdx.x; x < n; x += blockDim.x * gridDim.y) {
            const int e = (int)(x / W), w = (int)(x % W);
            while (e >= cr.as[k + 1]) k++;
            const int c = act_cs[cr.act_off + e], d = act_d[cr.act_off + e];
            const int64_t j = act_gt[cr.act_off + e];
            const int64_t c0 = lp.child[k][j], base = lp.base[k + 1] + it.s0 + w;
            float sum = 0.f;
#pragma unroll 4
            for (int a = 0; a < d; a++) sum += S[(c + a) * W + w];
#pragma unroll 4
            for (int a = 0; a < d; a++) {
                float sb = sum > 0.f ? S[(c + a) * W + w] / sum : 1.f / (float)d;
                out[base + lp.fgt[k + 1][c0 + a]] = sb;
            }
        }
    }
}

__global__ void k_export_util(const double *uacc, const int64_t *cidx0, int64_t n, double inv_t, float *out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (float)(uacc[cidx0[i]] * inv_t);
}

// One level of sum_e m_e (a_e - b_e)^2 over the solved edges e of the level (m_e: full slots that
// solved slot stands for), one warp per GT node, lanes over its solved slots; block sums in f64
// added to *acc.
__global__ void k_sigma_sqdiff(const int32_t *__restrict__ root, int64_t m, const int64_t *__restrict__ cfgt_off,
                               const int64_t *__restrict__ csoff, const int32_t *__restrict__ cmult,
                               const float *__restrict__ a, const float *__restrict__ b, double *acc) {
    __shared__ double part[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    double sum = 0.0;
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < m; j += nw) {
        const int32_t g = root[j];
        const int64_t c0 = cfgt_off[j], ns = cfgt_off[j + 1] - c0, w0 = csoff[g];
        for (int64_t x = lane; x < ns; x += 32) {
            const double d = (double)a[c0 + x] - (double)b[c0 + x];
            sum += (double)cmult[w0 + x] * d * d;
        }
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xFFFFFFFFu, sum, o);
    if (lane == 0) part[wid] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) s += part[i];
        atomicAdd(acc, s);
    }
}

// The average strategies of every full slot from those of the solved slots: full slot s of root g reads solved
// slot cidx0[score_off[g] + s] - csoff[g] of the same node.  All levels in one launch, eight lanes to a node (a
// root has some 5 to 20 full slots); a launch per level with a warp to a node left most lanes idle and made the
// exports of small rounds a chain of launches (sampled games through three rounds: 400 us, 295 so, 232 with the
// solved slots' export shared out over blocks).
struct ExpandLevels {
    const int32_t *root[9];
    const int64_t *fgt[9], *cfgt[9];
    int64_t first[10];       // nodes of the levels 1 .. k-1
    int64_t out[9], in[9];   // where a level's edges start
};

__global__ void k_expand_edges(const ExpandLevels L, const int64_t *__restrict__ score_off, const int64_t *__restrict__ csoff,
                               const int64_t *__restrict__ cidx0, const float *__restrict__ in, float *__restrict__ out) {
    const int lane = threadIdx.x & 7;
    const int64_t step = (int64_t)gridDim.x * (blockDim.x >> 3);
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3; i < L.first[9]; i += step) {
        int k = 1;
        while (i >= L.first[k + 1]) k++;
        const int64_t j = i - L.first[k];
        const int32_t g = L.root[k][j];
        const int64_t q0 = L.fgt[k][j], ns = L.fgt[k][j + 1] - q0, c0 = L.in[k] + L.cfgt[k][j] - csoff[g], s0 = score_off[g];
        for (int64_t s = lane; s < ns; s += 8) out[L.out[k] + q0 + s] = in[c0 + cidx0[s0 + s]];
    }
}

// The layout's kernels run over all levels at once: level k's M[k] nodes and one more element (for the scans'
// totals) at off[k].  With a launch, or three, per level, 121 launches of some 3 us made up most of a small round's
// set-up (1.15 ms of the 5.85 of a final round of 1000 iterations; 0.9 of 5.6 so).
struct LayoutLevels {
    const int64_t *child[9], *parent[9];  // child[8], parent[0]: unused
    const int32_t *root[9];
    int64_t off[10];
};

// level of element i, i - off in j; nodes of that level
__device__ __forceinline__ int level_of(const LayoutLevels &L, int64_t i, int64_t &j) {
    int k = 0;
    while (i >= L.off[k + 1]) k++;
    j = i - L.off[k];
    return k;
}

// Local and active flags.  A node is active when its subtree is more than one path of forced moves (then none of its
// ancestors' is one either); local when it is a root or its parent is active.
__global__ void k_flags(const LayoutLevels L, int32_t *__restrict__ local, int32_t *__restrict__ active) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < L.off[9]; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t j;
        const int k = level_of(L, i, j);
        if (i == L.off[k + 1] - 1) {
            local[i] = active[i] = 0;
            continue;
        }
        bool path = true;
        int64_t x = j;
        for (int kk = k; kk < 8 && path; kk++) {
            const int64_t c = L.child[kk][x];
            path = L.child[kk][x + 1] - c == 1;
            x = c;
        }
        active[i] = !path;
        bool loc = k == 0 || !path;
        if (!loc) {
            const int64_t p = L.parent[k][j];
            loc = L.child[k - 1][p + 1] - L.child[k - 1][p] > 1;
        }
        local[i] = loc;
    }
}

struct RankPtrs {
    const int64_t *loc[9];
    const int64_t *act[9];
};

// per root and level: global local-rank and active-rank at the root's first node
__global__ void k_root_ranks(const int64_t *bounds, int64_t n_roots, RankPtrs rp, int64_t *out) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g <= n_roots; g += (int64_t)gridDim.x * blockDim.x)
        for (int k = 0; k < 9; k++) {
            int64_t b = bounds[g * 9 + k];
            out[g * 18 + k] = rp.loc[k][b];
            out[g * 18 + 9 + k] = rp.act[k][b];
        }
}

__global__ void k_fill_layout(const LayoutLevels L, const int32_t *__restrict__ local, const int32_t *__restrict__ active,
                              const int64_t *__restrict__ loc_rank, const int64_t *__restrict__ act_rank,
                              const int64_t *__restrict__ fgt_off8, const CfrRoot *__restrict__ roots, int64_t *loc_tq, int32_t *act_li,
                              int32_t *act_pl, int32_t *act_cs, uint16_t *act_d, int64_t *act_gt, uint64_t *act_key, int32_t *act_rk,
                              int32_t *err) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < L.off[9]; i += (int64_t)gridDim.x * blockDim.x) {
        if (!local[i]) continue;
        int64_t j;
        const int k = level_of(L, i, j);
        const int32_t g = L.root[k][j];
        const CfrRoot &cr = roots[g];
        const int64_t li = cr.ls[k] + (loc_rank[i] - cr.locbase[k]);
        if (active[i]) {
            loc_tq[cr.loc_off + li] = -1;
            const int64_t e = cr.act_off + cr.as[k] + (act_rank[i] - cr.actbase[k]);
            const int64_t c0 = L.child[k][j], d = L.child[k][j + 1] - c0;
            if (d > 65535) atomicOr(err, 2);
            act_li[e] = (int32_t)li;
            act_pl[e] = k == 0 ? -1 : (int32_t)(cr.ls[k - 1] + (loc_rank[L.off[k - 1] + L.parent[k][j]] - cr.locbase[k - 1]));
            act_cs[e] = (int32_t)(cr.ls[k + 1] + (loc_rank[L.off[k + 1] + c0] - cr.locbase[k + 1]));
            act_d[e] = (uint16_t)d;
            act_gt[e] = j;
            // sort key: the (root, level) segment, then degree descending
            act_key[e] = ((uint64_t)(cr.act_off + cr.as[k]) << 16) | (uint64_t)(0xFFFF - (d > 0xFFFF ? 0xFFFF : d));
            act_rk[e] = (g << 3) | k;
        } else {
            int64_t x = j;
            for (int kk = k; kk < 8; kk++) x = L.child[kk][x];  // follow the forced moves to the leaf
            loc_tq[cr.loc_off + li] = fgt_off8[x];
        }
    }
}

// the entries in sorted order
struct EntryArrays {
    int32_t *li, *pl, *cs, *rk;
    uint16_t *d;
    int64_t *gt;
};

__global__ void k_gather_entries(const EntryArrays in, const int64_t *__restrict__ perm, int64_t n, EntryArrays out, int32_t *deg) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = perm[i];
        out.li[i] = in.li[e];
        out.pl[i] = in.pl[e];
        out.cs[i] = in.cs[e];
        out.rk[i] = in.rk[e];
        out.gt[i] = in.gt[e];
        deg[i] = out.d[i] = in.d[e];
    }
}

// pos: exclusive scan of the degrees over the sorted entries.  The children of the entries of
// root g at level k, in entry order, are the local nodes of level k+1 of that root: child a of
// entry e becomes local node ls[k+1] + (pos[e] - pos[first entry of (g, k)]) + a.  lmap[old
// global local index] = new global local index.
__global__ void k_renumber_map(int64_t n, const int32_t *act_rk, const CfrRoot *roots, const int64_t *pos,
                               const int32_t *act_cs, const uint16_t *act_d, int64_t *lmap) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t g = act_rk[e] >> 3, k = act_rk[e] & 7;
        const CfrRoot &cr = roots[g];
        const int64_t first = cr.ls[k + 1] + (pos[e] - pos[cr.act_off + cr.as[k]]);
        const int d = act_d[e];
        for (int a = 0; a < d; a++) lmap[cr.loc_off + act_cs[e] + a] = cr.loc_off + first + a;
    }
}

__global__ void k_renumber_roots(int64_t nr, const CfrRoot *roots, int64_t *lmap) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < nr; g += (int64_t)gridDim.x * blockDim.x)
        if (roots[g].ls[9] > 0) lmap[roots[g].loc_off] = roots[g].loc_off;
}

__global__ void k_renumber_apply(int64_t n, const int32_t *act_rk, const CfrRoot *roots, const int64_t *pos, const int64_t *lmap,
                                 int32_t *act_li, int32_t *act_pl, int32_t *act_cs) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t g = act_rk[e] >> 3, k = act_rk[e] & 7;
        const CfrRoot &cr = roots[g];
        act_li[e] = (int32_t)(lmap[cr.loc_off + act_li[e]] - cr.loc_off);
        if (act_pl[e] >= 0) act_pl[e] = (int32_t)(lmap[cr.loc_off + act_pl[e]] - cr.loc_off);
        act_cs[e] = (int32_t)(cr.ls[k + 1] + (pos[e] - pos[cr.act_off + cr.as[k]]));
    }
}

__global__ void k_renumber_tq(int64_t n, const int64_t *lmap, const int64_t *tq_old, int64_t *tq) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
        tq[lmap[x]] = tq_old[x];
}

// ---- the block sweep's order (BlockRun, BlockRoot) ---------------------------------------------

// 1 for an active entry whose children are all terminals
__global__ void k_block_bottom(int64_t n, const int32_t *act_rk, const CfrRoot *roots, const int32_t *act_cs, const uint16_t *act_d,
                               const int64_t *loc_tq, int32_t *bottom) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t *tq = loc_tq + roots[act_rk[e] >> 3].loc_off + act_cs[e];
        int b = 1;
        for (int a = 0; a < act_d[e]; a++) b &= tq[a] >= 0;
        bottom[e] = b;
    }
}

// stable partition of every (root, level) segment: entries with an active child first
// (brank: exclusive scan of the bottom flags); src = entry at each place, deg its degree
__global__ void k_block_order(int64_t n, const int32_t *act_rk, const CfrRoot *roots, const int32_t *bottom, const int64_t *brank,
                              const uint16_t *act_d, int64_t *src, int32_t *deg) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const CfrRoot &cr = roots[act_rk[e] >> 3];
        const int k = act_rk[e] & 7;
        const int64_t a = cr.act_off + cr.as[k], b = cr.act_off + cr.as[k + 1];
        const int64_t before = brank[e] - brank[a], all = brank[b] - brank[a];
        const int64_t i = bottom[e] ? a + (b - a - all) + before : e - before;
        src[i] = e;
        deg[i] = act_d[e];
    }
}

// 1 at the first place of every run of one (root, level), bottom flag and degree
__global__ void k_block_runs(int64_t n, const int64_t *src, const int32_t *act_rk, const int32_t *bottom, const int32_t *deg,
                             int32_t *first) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int f = 1;
        if (i > 0) {
            const int64_t e = src[i], p = src[i - 1];
            f = act_rk[e] != act_rk[p] || bottom[e] != bottom[p] || deg[i] != deg[i - 1];
        }
        first[i] = f;
    }
}

// run_at[r] = first place of run r (runs numbered by the exclusive scan `run` of `first`); run_at[runs] = n
__global__ void k_block_run_starts(int64_t n, const int32_t *first, const int64_t *run, int64_t *run_at) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += (int64_t)gridDim.x * blockDim.x)
        if (i == n || first[i]) run_at[run[i]] = i;
}

// the runs, and the block index of every child (bmap: local -> block index, per root).  dpos:
// exclusive scan of deg over the places.  Indices of roots with more than 65535 nodes are cut to
// 16 bits: such roots are not solved in a block.
__global__ void k_block_children(int64_t n, const int64_t *src, const int32_t *act_rk, const CfrRoot *roots, const int32_t *first,
                                 const int64_t *run, const int64_t *run_at, const int64_t *dpos, const int32_t *deg,
                                 const int32_t *act_cs, int32_t *bmap, BlockRun *runs) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = src[i], r = run[i] + first[i] - 1, a = run_at[r];
        const int m = (int)(run_at[r + 1] - a), d = deg[i];
        const CfrRoot &cr = roots[act_rk[e] >> 3];
        const int k = act_rk[e] & 7;
        const int c0 = cr.ls[k + 1] + (int)(dpos[a] - dpos[cr.act_off + cr.as[k]]);
        int32_t *bm = bmap + cr.loc_off + act_cs[e];
        for (int x = 0; x < d; x++) bm[x] = c0 + x * m + (int)(i - a);
        if (first[i]) runs[r] = BlockRun{(uint16_t)c0, (uint16_t)(i - cr.act_off), (uint16_t)m, (uint16_t)d};
        if (k == 0) bmap[cr.loc_off] = 0;
    }
}

// entries and masks at their places
__global__ void k_block_entries(int64_t n, const int64_t *src, const int32_t *act_rk, const CfrRoot *roots, const int32_t *act_li,
                                const int32_t *act_pl, const int32_t *act_cs, const uint16_t *act_d, const int64_t *loc_tq,
                                const int32_t *bmap, uint32_t *ent, uint8_t *msk) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = src[i];
        const CfrRoot &cr = roots[act_rk[e] >> 3];
        const int32_t *bm = bmap + cr.loc_off;
        const uint32_t li = (uint32_t)bm[act_li[e]], pl = act_pl[e] < 0 ? 0xFFFFu : (uint32_t)bm[act_pl[e]];
        ent[i] = (li & 0xFFFFu) | (pl << 16);
        unsigned mk = 0;
        const int64_t *tq = loc_tq + cr.loc_off + act_cs[e];
        for (int x = 0; x < act_d[e] && x < 8; x++) mk |= (tq[x] < 0 ? 1u : 0u) << x;
        msk[i] = (uint8_t)mk;
    }
}

// inv: block -> local index; term: terminals by block index; roots without an active node keep their one local node at 0
// (blockIdx.y: blocks to a root, where the roots are few and large)
__global__ void k_block_inverse(const int32_t *bmap, const CfrRoot *roots, int64_t nr, const int64_t *loc_tq, int32_t *inv,
                                uint8_t *term) {
    for (int64_t g = (int64_t)blockIdx.x; g < nr; g += gridDim.x) {
        const CfrRoot &cr = roots[g];
        const int L = cr.ls[9];
        for (int l = blockIdx.y * blockDim.x + threadIdx.x; l < L; l += gridDim.y * blockDim.x) {
            const int64_t b = cr.loc_off + (cr.as[9] == 0 ? l : bmap[cr.loc_off + l]);
            inv[b] = l;
            term[b] = loc_tq[cr.loc_off + l] >= 0;
        }
    }
}

__global__ void k_block_roots(int64_t nr, const CfrRoot *roots, const int64_t *run, const int64_t *brank, BlockRoot *out) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < nr; g += (int64_t)gridDim.x * blockDim.x) {
        const CfrRoot &cr = roots[g];
        BlockRoot br;
        br.run_off = run[cr.act_off];
        for (int k = 0; k < 9; k++) br.rs[k] = (int32_t)(run[cr.act_off + cr.as[k]] - br.run_off);
        for (int k = 0; k < 7; k++) {
            const int64_t a = cr.act_off + cr.as[k], b = cr.act_off + cr.as[k + 1];
            br.rt[k] = (int32_t)(run[b - (brank[b] - brank[a])] - br.run_off);
        }
        out[g] = br;
    }
}

__global__ void k_iota(int64_t *out, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) out[i] = i;
}

unsigned grid_for(int64_t threads, int block) {
    int64_t b = (threads + block - 1) / block;
    if (b < 1) b = 1;
    if (b > (1 << 20)) b = 1 << 20;
    return (unsigned)b;
}

// Several device temporaries carved from one allocation (pieces 256-byte aligned, n + 1 elements
// each): one allocator call instead of one per array.
struct Slab {
    size_t total = 0;
    std::vector<std::pair<void **, size_t>> want;
    template <typename T>
    void add(T **p, int64_t n) {
        want.push_back({(void **)p, total});
        total += (sizeof(T) * (size_t)(n + 1) + 255) & ~(size_t)255;
    }
    int alloc(pasur_ctx *ctx, std::vector<std::pair<void *, size_t>> &tmp) {
        char *base = nullptr;
        PASUR_TRY(dev_alloc(ctx, (void **)&base, total));
        tmp.push_back({(void *)base, total});
        for (auto &w : want) *w.first = base + w.second;
        return PASUR_OK;
    }
};

// The block sweep's order of the tree's entries: runs, entries, masks, index maps and per-root
// ranges (act_rk: root << 3 | level per entry).
int build_block_order(pasur_tree *t, const int32_t *act_rk) {
    pasur_ctx *ctx = t->ctx;
    const int64_t n = t->n_active, nr = t->n_roots;
    std::vector<std::pair<void *, size_t>> tmp;
    struct Guard {
        pasur_ctx *c;
        std::vector<std::pair<void *, size_t>> *v;
        ~Guard() {
            for (auto &x : *v) dev_free(c, x.first, x.second);
        }
    } guard{ctx, &tmp};
    int32_t *bottom, *deg, *first, *bmap;
    int64_t *brank, *src, *run, *run_at, *dpos;
    Slab sl;
    sl.add(&bottom, n);
    sl.add(&deg, n);
    sl.add(&first, n);
    sl.add(&bmap, t->n_local);
    sl.add(&brank, n);
    sl.add(&src, n);
    sl.add(&run, n);
    sl.add(&run_at, n + 1);
    sl.add(&dpos, n);
    PASUR_TRY(sl.alloc(ctx, tmp));
    PASUR_TRY(tree_alloc(t, (void **)&t->b_ent, sizeof(uint32_t) * (size_t)(n + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->b_msk, sizeof(uint8_t) * (size_t)(n + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->b_inv, sizeof(int32_t) * (size_t)(t->n_local + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->b_term, sizeof(uint8_t) * (size_t)(t->n_local + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->broots_d, sizeof(BlockRoot) * (size_t)(nr + 1)));
    const unsigned grid = grid_for(n, 256);
    auto launched = [&]() -> int {
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        return PASUR_OK;
    };
    if (n > 0) {
        k_block_bottom<<<grid, 256, 0, ctx->stream>>>(n, act_rk, t->croots_d, t->act_cs, t->act_d, t->loc_tq, bottom);
        PASUR_TRY(launched());
    }
    PASUR_TRY(exclusive_scan_i32(ctx, bottom, brank, n));
    if (n > 0) {
        k_block_order<<<grid, 256, 0, ctx->stream>>>(n, act_rk, t->croots_d, bottom, brank, t->act_d, src, deg);
        PASUR_TRY(launched());
        k_block_runs<<<grid, 256, 0, ctx->stream>>>(n, src, act_rk, bottom, deg, first);
        PASUR_TRY(launched());
    }
    PASUR_TRY(exclusive_scan_i32(ctx, deg, dpos, n));
    PASUR_TRY(exclusive_scan_i32(ctx, first, run, n));
    k_block_run_starts<<<grid_for(n + 1, 256), 256, 0, ctx->stream>>>(n, first, run, run_at);
    PASUR_TRY(launched());
    int64_t n_runs = 0;
    PASUR_TRY(read_i64(ctx, run + n, &n_runs));
    t->n_runs = n_runs;
    PASUR_TRY(tree_alloc(t, (void **)&t->b_run, sizeof(BlockRun) * (size_t)(n_runs + 1)));
    if (n > 0) {
        k_block_children<<<grid, 256, 0, ctx->stream>>>(n, src, act_rk, t->croots_d, first, run, run_at, dpos, deg, t->act_cs, bmap,
                                                        t->b_run);
        PASUR_TRY(launched());
        k_block_entries<<<grid, 256, 0, ctx->stream>>>(n, src, act_rk, t->croots_d, t->act_li, t->act_pl, t->act_cs, t->act_d,
                                                       t->loc_tq, bmap, t->b_ent, t->b_msk);
        PASUR_TRY(launched());
    }
    t->broots_h.resize((size_t)nr);
    if (nr > 0) {
        dim3 g((unsigned)std::min<int64_t>(nr, 65535));
        g.y = (unsigned)std::min<int64_t>(64, (8 * (int64_t)ctx->num_sms + g.x - 1) / g.x);
        k_block_inverse<<<g, 256, 0, ctx->stream>>>(bmap, t->croots_d, nr, t->loc_tq, t->b_inv, t->b_term);
        PASUR_TRY(launched());
        k_block_roots<<<grid_for(nr, 256), 256, 0, ctx->stream>>>(nr, t->croots_d, run, brank, t->broots_d);
        PASUR_TRY(launched());
        PASUR_CUDA(ctx, cudaMemcpyAsync(t->broots_h.data(), t->broots_d, sizeof(BlockRoot) * (size_t)nr, cudaMemcpyDeviceToHost,
                                        ctx->stream));
    }
    return PASUR_OK;
}

int build_layout(pasur_tree *t) {
    pasur_ctx *ctx = t->ctx;
    std::vector<std::pair<void *, size_t>> tmp, rk_tmp;  // rk_tmp: what the block order needs too
    struct Guard {
        pasur_ctx *c;
        std::vector<std::pair<void *, size_t>> *v;
        ~Guard() { drop(); }
        void drop() {
            for (auto &x : *v) dev_free(c, x.first, x.second);
            v->clear();
        }
    } guard{ctx, &tmp}, rk_guard{ctx, &rk_tmp};
    int32_t *local = nullptr, *active = nullptr;
    int64_t *lrank = nullptr, *arank = nullptr, *ranks = nullptr;
    const int64_t nr = t->n_roots;
    LayoutLevels L{};
    for (int k = 0; k < 9; k++) {
        L.child[k] = k < 8 ? t->child_off[k] : nullptr;
        L.parent[k] = k > 0 ? t->parent[k] : nullptr;
        L.root[k] = t->root[k];
        L.off[k + 1] = L.off[k] + t->M[k] + 1;
    }
    const int64_t n_all = L.off[9];
    {
        Slab sl, flags;
        sl.add(&local, n_all);
        sl.add(&lrank, n_all);
        sl.add(&arank, n_all);
        PASUR_TRY(sl.alloc(ctx, tmp));
        flags.add(&active, n_all);
        flags.add(&ranks, 18 * (nr + 1));
        PASUR_TRY(flags.alloc(ctx, tmp));
    }
    k_flags<<<grid_for(n_all, 256), 256, 0, ctx->stream>>>(L, local, active);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    PASUR_TRY(exclusive_scan_i32(ctx, local, lrank, n_all));
    PASUR_TRY(exclusive_scan_i32(ctx, active, arank, n_all));
    RankPtrs rp;
    for (int k = 0; k < 9; k++) {
        rp.loc[k] = lrank + L.off[k];
        rp.act[k] = arank + L.off[k];
    }
    k_root_ranks<<<grid_for(nr + 1, 256), 256, 0, ctx->stream>>>(t->bounds_d, nr, rp, ranks);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    std::vector<int64_t> hr((size_t)18 * (nr + 1));
    PASUR_CUDA(ctx, cudaMemcpyAsync(hr.data(), ranks, sizeof(int64_t) * hr.size(), cudaMemcpyDeviceToHost, ctx->stream));
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    t->croots_h.assign((size_t)nr, CfrRoot{});
    int64_t loc_off = 0, act_off = 0;
    for (int64_t g = 0; g < nr; g++) {
        CfrRoot &cr = t->croots_h[(size_t)g];
        const int64_t *a = &hr[(size_t)g * 18], *b = &hr[(size_t)(g + 1) * 18];
        int64_t l = 0, n = 0;
        for (int k = 0; k < 9; k++) {
            cr.locbase[k] = a[k];
            cr.actbase[k] = a[9 + k];
            cr.ls[k] = (int32_t)l;
            cr.as[k] = (int32_t)n;
            l += b[k] - a[k];
            n += b[9 + k] - a[9 + k];
        }
        if (l > INT32_MAX / 64) return set_err(ctx, PASUR_EOVERFLOW, "a root's local subtree is too large");
        cr.ls[9] = (int32_t)l;
        cr.as[9] = (int32_t)n;
        cr.loc_off = loc_off;
        cr.act_off = act_off;
        loc_off += l;
        act_off += n;
    }
    t->n_local = loc_off;
    t->n_active = act_off;
    if (nr > 0) {
        PASUR_TRY(tree_alloc(t, (void **)&t->croots_d, sizeof(CfrRoot) * (size_t)nr));
        PASUR_CUDA(ctx, cudaMemcpyAsync(t->croots_d, t->croots_h.data(), sizeof(CfrRoot) * (size_t)nr, cudaMemcpyHostToDevice,
                                        ctx->stream));
    }
    PASUR_TRY(tree_alloc(t, (void **)&t->loc_tq, sizeof(int64_t) * (size_t)(loc_off + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->act_li, sizeof(int32_t) * (size_t)(act_off + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->act_pl, sizeof(int32_t) * (size_t)(act_off + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->act_cs, sizeof(int32_t) * (size_t)(act_off + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->act_d, sizeof(uint16_t) * (size_t)(act_off + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->act_gt, sizeof(int64_t) * (size_t)(act_off + 1)));
    // the entries as found (f) and what orders them; once the ranks have been read, the sort's permutation, the
    // degrees and their scan take their place
    uint64_t *act_key = nullptr;
    EntryArrays f{}, sorted{t->act_li, t->act_pl, t->act_cs, nullptr, t->act_d, t->act_gt};
    int64_t *f_tq = nullptr, *lmap = nullptr;
    {
        Slab sl;
        sl.add(&act_key, act_off);
        sl.add(&f.li, act_off);
        sl.add(&f.pl, act_off);
        sl.add(&f.cs, act_off);
        sl.add(&f.rk, act_off);
        sl.add(&f.d, act_off);
        sl.add(&f.gt, act_off);
        sl.add(&f_tq, loc_off);
        sl.add(&lmap, loc_off);
        PASUR_TRY(sl.alloc(ctx, tmp));
        Slab rk;
        rk.add(&sorted.rk, act_off);
        PASUR_TRY(rk.alloc(ctx, rk_tmp));
    }
    int64_t *perm = lrank, *pos = arank;
    int32_t *deg = local, *act_rk = sorted.rk;
    PASUR_CUDA(ctx, cudaMemsetAsync(ctx->errflag, 0, sizeof(int32_t), ctx->stream));
    k_fill_layout<<<grid_for(n_all, 256), 256, 0, ctx->stream>>>(L, local, active, lrank, arank, t->cfgt_off[8], t->croots_d, f_tq, f.li,
                                                                f.pl, f.cs, f.d, f.gt, act_key, f.rk, ctx->errflag);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    int32_t ef = 0;
    PASUR_CUDA(ctx, cudaMemcpyAsync(&ef, ctx->errflag, sizeof ef, cudaMemcpyDeviceToHost, ctx->stream));
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (ef) return set_err(ctx, PASUR_EOVERFLOW, "a node has more than 65535 legal moves");
    dev_free(ctx, tmp[1].first, tmp[1].second);  // the active flags: done with, before the sort takes its own memory
    tmp.erase(tmp.begin() + 1);
    // order the active entries of every (root, level) by degree, largest first, so that the lanes
    // of a warp mostly run the same unrolled path
    if (act_off > 0) {
        k_iota<<<grid_for(act_off, 256), 256, 0, ctx->stream>>>(perm, act_off);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        int bits = 16;
        while (((int64_t)1 << (bits - 16)) <= act_off) bits++;
        PASUR_TRY(radix_sort_pairs(ctx, act_key, perm, act_off, bits));
        k_gather_entries<<<grid_for(act_off, 256), 256, 0, ctx->stream>>>(f, perm, act_off, sorted, deg);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
    }
    // renumber the local nodes of every level after the first in the order of their parents'
    // entries: the children of consecutive entries become consecutive nodes (a warp's child
    // accesses fall on few shared-memory banks and few device-memory sectors).  Child a of an
    // entry stays child a, so every node's arithmetic is unchanged.
    if (act_off > 0) {
        PASUR_TRY(exclusive_scan_i32(ctx, deg, pos, act_off));
        k_renumber_map<<<grid_for(act_off, 256), 256, 0, ctx->stream>>>(act_off, act_rk, t->croots_d, pos, t->act_cs, t->act_d,
                                                                        lmap);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        k_renumber_roots<<<grid_for(nr, 256), 256, 0, ctx->stream>>>(nr, t->croots_d, lmap);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        k_renumber_apply<<<grid_for(act_off, 256), 256, 0, ctx->stream>>>(act_off, act_rk, t->croots_d, pos, lmap, t->act_li,
                                                                          t->act_pl, t->act_cs);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        // terminal leaf links follow their nodes
        k_renumber_tq<<<grid_for(loc_off, 256), 256, 0, ctx->stream>>>(loc_off, lmap, f_tq, t->loc_tq);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
    } else if (loc_off > 0) {
        PASUR_CUDA(ctx, cudaMemcpyAsync(t->loc_tq, f_tq, sizeof(int64_t) * (size_t)loc_off, cudaMemcpyDeviceToDevice, ctx->stream));
    }
    guard.drop();  // the block order's temporaries take their place
    PASUR_TRY(build_block_order(t, act_rk));
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return PASUR_OK;
}

}  // namespace

// ---- roots split over thread-block clusters ----------------------------------------------------

namespace {

// A root split over a cluster: its top and its parts as pseudo-roots; offsets relative to the arrays
// here until they are placed after the tree's own.
struct RootSplit {
    bool done = false;
    int W = 1, ell = 0, nparts = 0;
    size_t smem = 0;  // largest CTA need (CTA 0: part 0 + top)
    CfrRoot top{};
    BlockRoot top_runs{};
    std::vector<CfrRoot> parts;
    std::vector<BlockRoot> part_runs;
    std::vector<uint32_t> ent;
    std::vector<uint8_t> msk, term;
    std::vector<int32_t> inv;
    std::vector<BlockRun> runs;
    std::vector<int32_t> cx, x_at;  // exchange entries (5 ints each); first one of every part
    int32_t top_root = 0;           // pseudo-root ids: the top, then the parts
    int64_t x0 = 0;                 // place of its exchange entries
    std::string msg;
};

constexpr int kSplitRuns = 96;  // runs a part is assumed to have while it is planned (checked after)

// the most slots of one item when S slots are shared out evenly over items of at most cap slots
int64_t even_slots(int64_t S, int64_t cap) {
    const int64_t n = (S + cap - 1) / cap;
    return (S + n - 1) / n;
}

// Split the roots whose state fits no block (or above cfg->split_bytes): subtrees of the active
// level-ell nodes packed (in GT order) into parts that each fit one block; CTA 0 also holds the top
// levels.  split[g] stays undone where no split is needed or none is found.
int plan_splits(pasur_tree *t, const pasur_config *cfg, size_t limit, const std::vector<char> &streamed,
                std::vector<RootSplit> &split) {
    pasur_ctx *ctx = t->ctx;
    const int64_t nr = t->n_roots;
    std::vector<int64_t> cand;
    for (int64_t g = 0; g < nr; g++) {
        const CfrRoot &cr = t->croots_h[(size_t)g];
        const int64_t Sg = t->csoff_h[(size_t)g + 1] - t->csoff_h[(size_t)g];
        const int64_t L = cr.ls[9], nA = cr.as[9];
        if (Sg == 0 || L == 0 || nA < 2 || streamed[(size_t)g] || !t->in_range(g)) continue;
        const bool fits = block_fits(cr, t->broots_h[(size_t)g], 1, limit);
        if (!fits || (cfg->split_bytes > 0 && resident_bytes(L, nA, 1) > (size_t)cfg->split_bytes)) cand.push_back(g);
    }
    split.clear();
    if (cand.empty()) return PASUR_OK;
    split.resize((size_t)nr);
    PhaseTimer pt(ctx->stream, "cluster splits");
    // host copies of the layout
    const int64_t NA = t->n_active, NL = t->n_local;
    std::vector<int32_t> hli((size_t)NA), hpl((size_t)NA), hcs((size_t)NA);
    std::vector<uint16_t> hd((size_t)NA);
    std::vector<int64_t> htq((size_t)NL);
    PASUR_CUDA(ctx, cudaMemcpy(hli.data(), t->act_li, sizeof(int32_t) * (size_t)NA, cudaMemcpyDeviceToHost));
    PASUR_CUDA(ctx, cudaMemcpy(hpl.data(), t->act_pl, sizeof(int32_t) * (size_t)NA, cudaMemcpyDeviceToHost));
    PASUR_CUDA(ctx, cudaMemcpy(hcs.data(), t->act_cs, sizeof(int32_t) * (size_t)NA, cudaMemcpyDeviceToHost));
    PASUR_CUDA(ctx, cudaMemcpy(hd.data(), t->act_d, sizeof(uint16_t) * (size_t)NA, cudaMemcpyDeviceToHost));
    PASUR_CUDA(ctx, cudaMemcpy(htq.data(), t->loc_tq, sizeof(int64_t) * (size_t)NL, cudaMemcpyDeviceToHost));
    pt.mark("host copies");
    const size_t target = cfg->split_bytes > 0 ? std::min<size_t>((size_t)cfg->split_bytes, limit) : limit;
    const bool verbose = getenv("PASUR_VERBOSE") != nullptr;
    const int warps = kBlockMaxThreads / 32;
    // the split of one root for items of W slots over at most qmax CTAs
    auto split_one = [&](int64_t g, int W, int qmax, LevelCut *cuts, RootSplit &o) {
        const CfrRoot cr = t->croots_h[(size_t)g];
        const BlockRoot &br = t->broots_h[(size_t)g];
        const int64_t L = cr.ls[9], nA = cr.as[9];
        const int32_t *li = hli.data() + cr.act_off, *pl = hpl.data() + cr.act_off, *cs = hcs.data() + cr.act_off;
        const uint16_t *dd = hd.data() + cr.act_off;
        const int64_t *tq = htq.data() + cr.loc_off;
        auto bytes = [&](int64_t l, int64_t a) { return (size_t)block_offsets(l, a, kSplitRuns, W, warps).end; };
        for (int ell = 1; ell <= 6; ell++) {
            if (cr.as[ell + 1] - cr.as[ell] < 2) continue;
            const size_t top_bytes = block_offsets(cr.ls[ell + 1], cr.as[ell], br.rs[ell], W, warps).end;
            if (top_bytes >= limit) break;
            cuts[ell].make(cr, ell, li, cs, dd);
            const LevelCut &cut = cuts[ell];
            const std::vector<int32_t> &heads = cut.heads, &sub = cut.sub;
            const int ns = (int)heads.size();
            // the target size sets the starting count of parts, a block's shared memory is the hard
            // limit of every part
            const size_t need = bytes(L, nA);
            const int q0 = (int)std::min<size_t>((size_t)qmax, std::max<size_t>(2, (need + target - 1) / target));
            const PartPacking<decltype(bytes)> packing{cut, bytes, limit, top_bytes};
            const int fewest = packing.fewest();
            std::vector<int> first;
            for (int Q = std::max(q0, fewest); fewest > 0 && Q <= qmax; Q++) {
                if (!packing.balanced(Q, first)) continue;
                const int np = (int)first.size();
                if (np < 2 || ctx->clusters_of[np] == 0) continue;
                first.push_back(ns);
                o = RootSplit{};
                o.W = W;
                o.ell = ell;
                o.nparts = np;
                // the top: the root's own entries and nodes, cut at level ell
                o.top = cr;
                o.top_runs = br;
                for (int k = ell; k < 9; k++) o.top_runs.rs[k] = br.rs[ell];
                for (int k = ell; k < 7; k++) o.top_runs.rt[k] = br.rs[ell];
                for (int k = ell + 1; k < 10; k++) o.top.as[k] = cr.as[ell];
                for (int k = ell + 2; k < 10; k++) o.top.ls[k] = cr.ls[ell + 1];
                std::vector<int32_t> part_of((size_t)ns);
                for (int q = 0; q < np; q++)
                    for (int i = first[(size_t)q]; i < first[(size_t)q + 1]; i++) part_of[(size_t)i] = q;
                std::vector<int32_t> bidx((size_t)L, -1), ent_of((size_t)cr.ls[ell + 1], -1);
                for (int32_t e = cr.as[ell]; e < cr.as[ell + 1]; e++) ent_of[(size_t)li[e]] = e;
                // entries part by part and level by level
                std::vector<std::vector<std::vector<int32_t>>> ents((size_t)np, std::vector<std::vector<int32_t>>(8));
                for (int k = ell; k < 8; k++)
                    for (int32_t e = cr.as[k]; e < cr.as[k + 1]; e++) {
                        const int32_t sid = sub[(size_t)li[e]];
                        if (sid >= 0) ents[(size_t)part_of[(size_t)sid]][(size_t)k].push_back(e);
                    }
                for (int q = 0; q < np; q++) {
                    CfrRoot pr{};
                    BlockRoot pb{};
                    pr.loc_off = (int64_t)o.inv.size();
                    pr.act_off = (int64_t)o.ent.size();
                    pb.run_off = (int64_t)o.runs.size();
                    const int h0 = first[(size_t)q], h = first[(size_t)q + 1] - h0;
                    int32_t n = h, m = 0, r = 0;
                    for (int i = 0; i < h; i++) bidx[(size_t)heads[(size_t)(h0 + i)]] = i;
                    o.inv.insert(o.inv.end(), (size_t)h, -1);  // their regrets are the top's
                    // level by level: entries with an active child first, runs of one degree, the runs'
                    // children numbered child by child
                    for (int k = ell; k < 8; k++) {
                        std::vector<int32_t> &el = ents[(size_t)q][(size_t)k];
                        auto active = [&](int32_t e) {
                            for (int a = 0; a < dd[e]; a++)
                                if (tq[cs[e] + a] < 0) return true;
                            return false;
                        };
                        const size_t mid = (size_t)(std::stable_partition(el.begin(), el.end(), active) - el.begin());
                        pb.rs[k] = r;
                        for (size_t i = 0; i < el.size();) {
                            size_t z = i;
                            const size_t end = i < mid ? mid : el.size();
                            while (z < end && dd[el[z]] == dd[el[i]]) z++;
                            const int32_t len = (int32_t)(z - i), d = dd[el[i]];
                            o.runs.push_back(BlockRun{(uint16_t)n, (uint16_t)m, (uint16_t)len, (uint16_t)d});
                            r++;
                            o.inv.resize((size_t)(pr.loc_off + n + len * d));
                            for (int32_t y = 0; y < len; y++)
                                for (int a = 0; a < d; a++) {
                                    const int32_t b = n + a * len + y, x = cs[el[i + (size_t)y]] + a;
                                    bidx[(size_t)x] = b;
                                    o.inv[(size_t)(pr.loc_off + b)] = x;
                                }
                            n += len * d;
                            m += len;
                            i = z;
                            if (k < 7 && i == mid) pb.rt[k] = r;
                        }
                        if (k < 7 && mid == 0) pb.rt[k] = pb.rs[k];
                    }
                    pb.rs[8] = r;
                    const int32_t g0 = n;  // the ghosts: the parents' reaches
                    n += h;
                    o.inv.insert(o.inv.end(), (size_t)h, -1);
                    for (int k = ell; k < 8; k++)
                        for (int32_t e : ents[(size_t)q][(size_t)k]) {
                            const int32_t up = k == ell ? g0 + bidx[(size_t)li[e]] : bidx[(size_t)pl[e]];
                            o.ent.push_back((uint32_t)bidx[(size_t)li[e]] | (uint32_t)up << 16);
                            uint8_t mk = 0;
                            for (int a = 0; a < dd[e] && a < 8; a++) mk |= (uint8_t)((tq[cs[e] + a] < 0 ? 1 : 0) << a);
                            o.msk.push_back(mk);
                        }
                    for (int32_t b = 0; b < n; b++) {
                        const int32_t x = o.inv[(size_t)(pr.loc_off + b)];
                        o.term.push_back(x >= 0 && tq[x] >= 0 ? 1 : 0);
                    }
                    pr.ls[9] = n;
                    pr.as[9] = m;
                    pr.W = W;
                    pr.cls = kClsCluster;
                    size_t b = block_offsets(n, m, r, W, warps).end;
                    if (q == 0) b += top_bytes;
                    o.smem = std::max(o.smem, n >= 65535 ? limit + 1 : b);
                    o.parts.push_back(pr);
                    o.part_runs.push_back(pb);
                    // exchange entries: the part's level-ell nodes
                    o.x_at.push_back((int32_t)(o.cx.size() / 5));
                    for (int i = 0; i < h; i++) {
                        const int32_t x = heads[(size_t)(h0 + i)], e = ent_of[(size_t)x];
                        // block indices of the top: set below from the root's own
                        o.cx.push_back(q);
                        o.cx.push_back(x);
                        o.cx.push_back(pl[e]);
                        o.cx.push_back(i);
                        o.cx.push_back(g0 + i);
                    }
                }
                o.x_at.push_back((int32_t)(o.cx.size() / 5));
                if (o.smem > limit) continue;
                o.done = true;
                return;
            }
            if (verbose) {
                int64_t big = 0;
                for (int i = 0; i < ns; i++) big = std::max<int64_t>(big, (int64_t)bytes(cut.sl[(size_t)i] + 1, cut.sa[(size_t)i]));
                char line[256];
                snprintf(line, sizeof line, "[pasur] root %lld (L %lld, active %lld), %d slots: no split at level %d: %d subtrees, top "
                                            "%zu B, largest subtree %lld B, part limit %zu B\n",
                         (long long)g, (long long)L, (long long)nA, W, ell, ns, top_bytes, (long long)big, limit);
                o.msg += line;
            }
        }
    };
    // roots are independent: split them on host threads; as many slots per item as clusters of up to 8
    // CTAs hold, one slot over up to 16
    const bool ok = on_threads(cand.size(), [&](size_t i) {
        const int64_t g = cand[i];
        const int64_t Sg = t->csoff_h[(size_t)g + 1] - t->csoff_h[(size_t)g];
        RootSplit &o = split[(size_t)g];
        LevelCut cuts[7];
        std::string msg;
        for (int64_t W = even_slots(Sg, cfg->slots_per_item > 0 ? std::min(cfg->slots_per_item, kBlockSlots) : kBlockSlots);
             W >= 1 && !o.done; W = W > 1 ? even_slots(Sg, W - 1) : 0) {
            split_one(g, (int)W, W > 1 && cfg->split_bytes == 0 ? 8 : kMaxClusterCtas, cuts, o);
            if (!o.done) msg += o.msg;
            o.msg.clear();
        }
        o.msg = msg;
    });
    if (!ok) return set_err(ctx, PASUR_ENOMEM, "cluster split: host allocation failed");
    pt.mark("per-root splits");
    for (int64_t g : cand)
        if (!split[(size_t)g].done && !split[(size_t)g].msg.empty()) fputs(split[(size_t)g].msg.c_str(), stderr);
    return PASUR_OK;
}

// the first nodes of several roots in block order, a root to a block: inv[from[b] ..] to out[to[b] .. to[b + 1])
__global__ void k_gather_tops(const int32_t *__restrict__ inv, const int64_t *__restrict__ from, const int64_t *__restrict__ to,
                              int32_t *__restrict__ out) {
    const int64_t a = from[blockIdx.x], o = to[blockIdx.x], n = to[blockIdx.x + 1] - o;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) out[o + i] = inv[a + i];
}

// The parts' entries, runs and index maps after the tree's own (device), the pseudo-roots after the
// real roots, and the exchange entries.  Host threads copy them into place and give back the splits' own
// arrays: 4410 split roots of 3.2e8 nodes in 65 ms (507 one root after the other).
int place_splits(pasur_tree *t, std::vector<RootSplit> &split) {
    pasur_ctx *ctx = t->ctx;
    const int64_t NA = t->n_active, NL = t->n_local, NR = t->n_runs;
    // the split roots; where each one's entries, nodes, runs, exchange entries and top nodes begin
    std::vector<int64_t> roots, from;
    for (size_t g = 0; g < split.size(); g++)
        if (split[g].done) roots.push_back((int64_t)g);
    if (roots.empty()) return PASUR_OK;
    const size_t n = roots.size();
    std::vector<int64_t> e_at(n + 1, 0), l_at(n + 1, 0), r_at(n + 1, 0), x_at(n + 1, 0), t_at(n + 1, 0);
    for (size_t i = 0; i < n; i++) {
        const size_t g = (size_t)roots[i];
        RootSplit &o = split[g];
        from.push_back(t->croots_h[g].loc_off);
        e_at[i + 1] = e_at[i] + (int64_t)o.ent.size();
        l_at[i + 1] = l_at[i] + (int64_t)o.inv.size();
        r_at[i + 1] = r_at[i] + (int64_t)o.runs.size();
        x_at[i + 1] = x_at[i] + (int64_t)o.cx.size();
        t_at[i + 1] = t_at[i] + o.top.ls[9];
        o.top_root = (int32_t)t->croots_h.size();
        o.x0 = x_at[i] / 5;
        t->croots_h.push_back(o.top);
        t->broots_h.push_back(o.top_runs);
        for (size_t q = 0; q < o.parts.size(); q++) {
            CfrRoot pr = o.parts[q];
            BlockRoot pb = o.part_runs[q];
            pr.loc_off += NL + l_at[i];
            pr.act_off += NA + e_at[i];
            pb.run_off += NR + r_at[i];
            t->croots_h.push_back(pr);
            t->broots_h.push_back(pb);
        }
    }
    std::vector<int32_t> tops((size_t)t_at[n]);
    {
        int64_t *from_d = nullptr, *to_d = nullptr;
        int32_t *tops_d = nullptr;
        std::vector<std::pair<void *, size_t>> tmp;
        struct Guard {
            pasur_ctx *c;
            std::vector<std::pair<void *, size_t>> *v;
            ~Guard() {
                for (auto &x : *v) dev_free(c, x.first, x.second);
            }
        } guard{ctx, &tmp};
        Slab sl;
        sl.add(&from_d, (int64_t)n);
        sl.add(&to_d, (int64_t)n);
        sl.add(&tops_d, t_at[n]);
        PASUR_TRY(sl.alloc(ctx, tmp));
        PASUR_CUDA(ctx, cudaMemcpyAsync(from_d, from.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, ctx->stream));
        PASUR_CUDA(ctx, cudaMemcpyAsync(to_d, t_at.data(), sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, ctx->stream));
        k_gather_tops<<<(unsigned)n, 256, 0, ctx->stream>>>(t->b_inv, from_d, to_d, tops_d);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        PASUR_CUDA(ctx, cudaMemcpyAsync(tops.data(), tops_d, sizeof(int32_t) * tops.size(), cudaMemcpyDeviceToHost, ctx->stream));
        PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    }
    const size_t ne = (size_t)e_at[n], nl = (size_t)l_at[n], nrun = (size_t)r_at[n];
    std::unique_ptr<uint32_t[]> ent(new (std::nothrow) uint32_t[ne + 1]);
    std::unique_ptr<uint8_t[]> msk(new (std::nothrow) uint8_t[ne + 1]), term(new (std::nothrow) uint8_t[nl + 1]);
    std::unique_ptr<int32_t[]> inv(new (std::nothrow) int32_t[nl + 1]);
    std::unique_ptr<BlockRun[]> runs(new (std::nothrow) BlockRun[nrun + 1]);
    if (!ent || !msk || !term || !inv || !runs) return set_err(ctx, PASUR_ENOMEM, "cluster split: host allocation failed");
    t->cx_h.resize((size_t)x_at[n]);
    const bool ok = on_threads(n, [&](size_t i) {
        RootSplit &o = split[(size_t)roots[i]];
        // block index of the top's nodes: the inverse of their order
        const int32_t *own = tops.data() + t_at[i];
        std::vector<int32_t> back((size_t)o.top.ls[9], 0);
        for (size_t b = 0; b < back.size(); b++) back[(size_t)own[b]] = (int32_t)b;
        int32_t *cx = std::copy(o.cx.begin(), o.cx.end(), t->cx_h.data() + x_at[i]) - (ptrdiff_t)o.cx.size();
        for (size_t x = 0; x < o.cx.size(); x += 5) {
            cx[x + 1] = back[(size_t)cx[x + 1]];
            cx[x + 2] = back[(size_t)cx[x + 2]];
        }
        auto place = [](auto &v, auto *to) {
            std::copy(v.begin(), v.end(), to);
            v = {};
            v.shrink_to_fit();
        };
        place(o.ent, ent.get() + e_at[i]);
        place(o.msk, msk.get() + e_at[i]);
        place(o.term, term.get() + l_at[i]);
        place(o.inv, inv.get() + l_at[i]);
        place(o.runs, runs.get() + r_at[i]);
    });
    if (!ok) return set_err(ctx, PASUR_ENOMEM, "cluster split: host allocation failed");
    auto grow = [&](void **p, int64_t n_old, size_t size, const void *more, size_t n_more) -> int {
        void *x = nullptr;
        PASUR_TRY(tree_alloc(t, &x, size * ((size_t)n_old + n_more + 1)));
        PASUR_CUDA(ctx, cudaMemcpyAsync(x, *p, size * (size_t)n_old, cudaMemcpyDeviceToDevice, ctx->stream));
        PASUR_CUDA(ctx, cudaMemcpyAsync((char *)x + size * (size_t)n_old, more, size * n_more, cudaMemcpyHostToDevice, ctx->stream));
        *p = x;
        return PASUR_OK;
    };
    auto upload = [&]() -> int {
        PASUR_TRY(grow((void **)&t->b_ent, NA, sizeof(uint32_t), ent.get(), ne));
        PASUR_TRY(grow((void **)&t->b_msk, NA, sizeof(uint8_t), msk.get(), ne));
        PASUR_TRY(grow((void **)&t->b_term, NL, sizeof(uint8_t), term.get(), nl));
        PASUR_TRY(grow((void **)&t->b_inv, NL, sizeof(int32_t), inv.get(), nl));
        PASUR_TRY(grow((void **)&t->b_run, NR, sizeof(BlockRun), runs.get(), nrun));
        PASUR_TRY(tree_alloc(t, (void **)&t->croots_d, sizeof(CfrRoot) * t->croots_h.size()));
        PASUR_TRY(tree_alloc(t, (void **)&t->broots_d, sizeof(BlockRoot) * t->broots_h.size()));
        PASUR_CUDA(ctx, cudaMemcpyAsync(t->broots_d, t->broots_h.data(), sizeof(BlockRoot) * t->broots_h.size(),
                                        cudaMemcpyHostToDevice, ctx->stream));
        return PASUR_OK;
    };
    const int rc = upload();
    // the uploads read arrays of this call, also where a later one was refused
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return rc;
}

}  // namespace

// Largest dynamic shared memory a block of the sweep may request: the per-block opt-in limit minus
// the kernels' own static shared memory (largest over the variants).
int cfr_dyn_smem_limit(pasur_ctx *ctx, size_t *limit) {
    size_t st = 0;
    cudaFuncAttributes fa;
    for (int v = 0; v < 2; v++)
        for (int w = 1; w <= kBlockSlots; w++) {
            PASUR_CUDA(ctx, cudaFuncGetAttributes(&fa, block_kernel(v, w)));
            st = std::max(st, fa.sharedSizeBytes);
            PASUR_CUDA(ctx, cudaFuncGetAttributes(&fa, cluster_kernel(v, w)));
            st = std::max(st, fa.sharedSizeBytes);
        }
    *limit = ctx->smem_optin > st ? ctx->smem_optin - st : 0;
    return PASUR_OK;
}

const void *block_kernel(int variant, int W) {
    switch (W) {
        case 1: return block_kernel_w1(variant);
        case 2: return block_kernel_w2(variant);
        case 3: return block_kernel_w3(variant);
        case 4: return block_kernel_w4(variant);
        case 5: return block_kernel_w5(variant);
        default: return block_kernel_w6(variant);
    }
}
const void *cluster_kernel(int variant, int W) {
    switch (W) {
        case 1: return cluster_kernel_w1(variant);
        case 2: return cluster_kernel_w2(variant);
        case 3: return cluster_kernel_w3(variant);
        case 4: return cluster_kernel_w4(variant);
        case 5: return cluster_kernel_w5(variant);
        default: return cluster_kernel_w6(variant);
    }
}

namespace {

void sweep_launch_config(const SweepLaunch &l, cudaLaunchConfig_t *lc, cudaLaunchAttribute *at) {
    lc->gridDim = dim3((unsigned)((l.end - l.begin) * l.ctas));
    lc->blockDim = dim3((unsigned)l.threads);
    lc->dynamicSmemBytes = l.smem;
    if (l.ctas > 1) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)l.ctas;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        lc->attrs = at;
        lc->numAttrs = 1;
    }
}

// Once per context: the kernels' attributes (global per kernel: the largest dynamic size any plan can
// ask for, so that plans prepared later never lower it under an earlier plan's need) and the cluster
// sizes the device can hold with a whole SM's shared memory per CTA.
int raise_limits(pasur_ctx *ctx, size_t limit) {
    if (ctx->cfr_smem_raised) return PASUR_OK;
    for (int v = 0; v < 2; v++)
        for (int w = 1; w <= kBlockSlots; w++) {
            PASUR_CUDA(ctx, cudaFuncSetAttribute(block_kernel(v, w), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit));
            PASUR_CUDA(ctx, cudaFuncSetAttribute(cluster_kernel(v, w), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit));
            PASUR_CUDA(ctx, cudaFuncSetAttribute(cluster_kernel(v, w), cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        }
    for (int q = 2; q <= kMaxClusterCtas; q++) {
        SweepLaunch l;
        l.ctas = q;
        l.end = 1;
        l.threads = kBlockMaxThreads;
        l.smem = limit;
        cudaLaunchConfig_t lc{};
        cudaLaunchAttribute at[1];
        sweep_launch_config(l, &lc, at);
        if (cudaOccupancyMaxActiveClusters(&ctx->clusters_of[q], cluster_kernel(0, kBlockSlots), &lc) != cudaSuccess) {
            cudaGetLastError();
            ctx->clusters_of[q] = 0;
        }
    }
    ctx->cfr_smem_raised = true;
    return PASUR_OK;
}

}  // namespace

int cfr_setup_tree(pasur_tree *t, const pasur_config *cfg, int tree, std::vector<CfrItem> *cls_items,
                   std::vector<ClusterItem> *clu) {
    pasur_ctx *ctx = t->ctx;
    PhaseTimer pt(ctx->stream, "cfr plan");
    PASUR_TRY(build_layout(t));
    pt.mark("layout");
    size_t limit = 0;
    PASUR_TRY(cfr_dyn_smem_limit(ctx, &limit));
    PASUR_TRY(raise_limits(ctx, limit));
    const Storage storage(ctx->smem_optin, cfg->slots_per_item);
    t->layout_cfg = *cfg;
    t->croots_h.resize((size_t)t->n_roots);
    t->broots_h.resize((size_t)t->n_roots);
    t->cparts_h.clear();
    t->cx_h.clear();
    // roots streamed over every SM (class 5): those above cfg->stream_bytes, and those too large
    // for one block that have enough score slots to fill the streaming sweep's warps with
    // consecutive slots; roots that fit neither a block nor a cluster reach class 5 below too
    std::vector<char> streamed((size_t)t->n_roots, 0);
    for (int64_t g = 0; g < t->n_roots; g++) {
        const CfrRoot &cr = t->croots_h[(size_t)g];
        const int64_t Sg = t->csoff_h[(size_t)g + 1] - t->csoff_h[(size_t)g];
        if (Sg == 0 || cr.ls[9] == 0 || !t->in_range(g)) continue;
        streamed[(size_t)g] = (cfg->stream_bytes > 0 && resident_bytes(cr.ls[9], cr.as[9], 1) > (size_t)cfg->stream_bytes) ||
                              (Sg >= kStreamMinSlots && !block_fits(cr, t->broots_h[(size_t)g], 1, limit));
    }
    // roots too large for one block (or above cfg->split_bytes) go to thread-block clusters
    std::vector<RootSplit> split;
    PASUR_TRY(plan_splits(t, cfg, limit, streamed, split));
    PASUR_TRY(place_splits(t, split));
    pt.mark("cluster splits");
    std::vector<int64_t> &sbase = t->slot_base_h;
    std::vector<int32_t> &sstr = t->slot_str_h;
    sbase.assign((size_t)t->csoff_h[(size_t)t->n_roots] + 1, 0);
    sstr.assign(sbase.size(), 0);
    int64_t data = 0, scratch = 0;
    for (int64_t g = 0; g < t->n_roots; g++) {
        CfrRoot &cr = t->croots_h[(size_t)g];
        const int64_t Sg = t->csoff_h[(size_t)g + 1] - t->csoff_h[(size_t)g];
        const int64_t L = cr.ls[9], nA = cr.as[9];
        cr.W = 0;
        cr.cls = -1;
        if (Sg == 0 || L == 0 || !t->in_range(g)) continue;
        int64_t w = 1;
        int cls = kClsGlobal, store = kClsGlobal;
        if (!split.empty() && split[(size_t)g].done) {
            const RootSplit &o = split[(size_t)g];
            cls = store = kClsCluster;
            ClusterItem ci{};
            ci.tree = tree;
            ci.root = (int32_t)g;
            ci.part0 = (int64_t)t->cparts_h.size();
            ci.x0 = o.x0;
            ci.nx = (int32_t)(o.cx.size() / 5);
            ci.nparts = o.nparts;
            ci.smem = o.smem;
            t->cparts_h.push_back(ClusterPart{o.top_root, 0, 0});
            for (int q = 0; q < o.nparts; q++)
                t->cparts_h.push_back(ClusterPart{o.top_root + 1 + q, o.x_at[(size_t)q], o.x_at[(size_t)q + 1]});
            const int64_t n = (Sg + o.W - 1) / o.W;
            for (int64_t i = 0, s0 = 0; i < n; i++) {
                ci.s0 = (int32_t)s0;
                ci.ns = (int32_t)(Sg / n + (i < Sg % n ? 1 : 0));
                ci.cost = nA * ci.ns;
                clu->push_back(ci);
                s0 += ci.ns;
            }
        } else {
            w = storage.width(L, nA, Sg, streamed[(size_t)g], &store);
            // the sweep's blocks hold more than the storage classes: a root beyond those may still fit
            cls = store;
            if (cls == kClsGlobal && !streamed[(size_t)g] && block_fits(cr, t->broots_h[(size_t)g], 1, limit)) cls = kClsGlobal - 1;
        }
        cr.W = (int32_t)w;
        cr.cls = cls;
        for (int64_t s0 = 0, ns = w; s0 < Sg; s0 += ns) {
            while (ns > Sg - s0) ns /= 2;
            CfrItem it{};
            it.root = (int32_t)g;
            it.tree = tree;
            it.ns = (int32_t)ns;
            it.s0 = s0;
            it.data_base = data;
            for (int64_t x = 0; x < ns; x++) {
                sbase[(size_t)(t->csoff_h[(size_t)g] + s0 + x)] = data + x;
                sstr[(size_t)(t->csoff_h[(size_t)g] + s0 + x)] = (int32_t)ns;
            }
            data += L * it.ns;
            it.scratch_base = -1;
            if (cls == kClsGlobal) {
                it.scratch_base = scratch;
                scratch += L * it.ns;
            }
            it.cost = std::max<int64_t>(nA, 1) * it.ns;
            cls_items[cls].push_back(it);
        }
    }
    t->data_size = data;
    t->scratch_size = scratch;
    t->swept_edges = t->swept_pairs = 0;
    for (int64_t g = 0; g < t->n_roots; g++) {
        const CfrRoot &cr = t->croots_h[(size_t)g];
        if (cr.ls[9] > 1 && t->in_range(g)) {
            const int64_t ns = t->csoff_h[(size_t)g + 1] - t->csoff_h[(size_t)g];
            t->swept_edges += (int64_t)(cr.ls[9] - 1) * ns;
            t->swept_pairs += (int64_t)cr.as[9] * ns;
        }
    }
    if (!t->cparts_h.empty()) {
        PASUR_TRY(tree_alloc(t, (void **)&t->cparts_d, sizeof(ClusterPart) * (t->cparts_h.size() + 1)));
        PASUR_TRY(tree_alloc(t, (void **)&t->cx_d, sizeof(int32_t) * (t->cx_h.size() + 1)));
        PASUR_CUDA(ctx, cudaMemcpyAsync(t->cparts_d, t->cparts_h.data(), sizeof(ClusterPart) * t->cparts_h.size(),
                                        cudaMemcpyHostToDevice, ctx->stream));
        PASUR_CUDA(ctx, cudaMemcpyAsync(t->cx_d, t->cx_h.data(), sizeof(int32_t) * t->cx_h.size(), cudaMemcpyHostToDevice,
                                        ctx->stream));
    }
    if (!t->croots_h.empty())
        PASUR_CUDA(ctx, cudaMemcpyAsync(t->croots_d, t->croots_h.data(), sizeof(CfrRoot) * t->croots_h.size(),
                                        cudaMemcpyHostToDevice, ctx->stream));
    PASUR_TRY(tree_alloc(t, (void **)&t->R, sizeof(float) * (size_t)(data + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->S, sizeof(float) * (size_t)(data + 1)));
    PASUR_CUDA(ctx, cudaMemsetAsync(t->R, 0, sizeof(float) * (size_t)(data + 1), ctx->stream));
    PASUR_CUDA(ctx, cudaMemsetAsync(t->S, 0, sizeof(float) * (size_t)(data + 1), ctx->stream));
    if (scratch) {
        PASUR_TRY(tree_alloc(t, (void **)&t->V, sizeof(float) * (size_t)scratch));
        PASUR_TRY(tree_alloc(t, (void **)&t->X, sizeof(float) * (size_t)scratch));
    }
    PASUR_TRY(tree_alloc(t, (void **)&t->uacc, sizeof(double) * (size_t)(t->cQ[0] + 1)));
    PASUR_CUDA(ctx, cudaMemsetAsync(t->uacc, 0, sizeof(double) * (size_t)(t->cQ[0] + 1), ctx->stream));
    PASUR_TRY(tree_alloc(t, (void **)&t->slot_base, sizeof(int64_t) * sbase.size()));
    PASUR_TRY(tree_alloc(t, (void **)&t->slot_str, sizeof(int32_t) * sstr.size()));
    PASUR_CUDA(ctx, cudaMemcpyAsync(t->slot_base, sbase.data(), sizeof(int64_t) * sbase.size(), cudaMemcpyHostToDevice, ctx->stream));
    PASUR_CUDA(ctx, cudaMemcpyAsync(t->slot_str, sstr.data(), sizeof(int32_t) * sstr.size(), cudaMemcpyHostToDevice, ctx->stream));
    TreeView &v = t->view;
    v.broots = t->broots_d;
    v.b_run = t->b_run;
    v.b_ent = t->b_ent;
    v.b_msk = t->b_msk;
    v.b_inv = t->b_inv;
    v.b_term = t->b_term;
    v.slot_base = t->slot_base;
    v.slot_str = t->slot_str;
    v.roots = t->croots_d;
    v.act_li = t->act_li;
    v.act_pl = t->act_pl;
    v.act_cs = t->act_cs;
    v.act_d = t->act_d;
    v.loc_tq = t->loc_tq;
    v.leaf_v = t->leaf_v;
    v.fgt_off0 = t->cfgt_off[0];
    v.R = t->R;
    v.S = t->S;
    v.V = t->V;
    v.X = t->X;
    v.uacc = t->uacc;
    v.cparts = t->cparts_d;
    v.cx = t->cx_d;
    t->iters_done = 0;
    pt.mark("items and state");
    return PASUR_OK;
}

// The cluster and block sweeps' items and launches: the clusters' items, and every root of the storage
// classes 0..4 of the trees in a block.
int plan_sweeps(pasur_ctx *ctx, CfrPlan &plan, const std::vector<pasur_tree *> &trees, const pasur_config *cfg,
                const std::vector<ClusterItem> &clu, std::vector<std::pair<void *, size_t>> &owned) {
    plan.blk_h.clear();
    plan.launches.clear();
    size_t lim = 0;
    PASUR_TRY(cfr_dyn_smem_limit(ctx, &lim));
    const int full = cfg->threads > 0 ? std::min(cfg->threads, kBlockMaxThreads) : kBlockMaxThreads;
    // clusters: one launch per parts and slots, the largest first
    plan.clu_h = clu;
    std::stable_sort(plan.clu_h.begin(), plan.clu_h.end(), [](const ClusterItem &a, const ClusterItem &b) {
        if (a.nparts != b.nparts) return a.nparts > b.nparts;
        if (a.ns != b.ns) return a.ns > b.ns;
        return a.cost > b.cost;
    });
    for (size_t i = 0; i < plan.clu_h.size(); i++) {
        const ClusterItem &x = plan.clu_h[i];
        if (i == 0 || x.nparts != plan.clu_h[i - 1].nparts || x.ns != plan.clu_h[i - 1].ns) {
            SweepLaunch l;
            l.ctas = x.nparts;
            l.W = x.ns;
            l.threads = full;
            l.begin = (int64_t)i;
            plan.launches.push_back(l);
        }
        plan.launches.back().end = (int64_t)i + 1;
        plan.launches.back().smem = std::max(plan.launches.back().smem, x.smem);
    }
    if (!plan.clu_h.empty()) {
        const size_t b = sizeof(ClusterItem) * plan.clu_h.size();
        PASUR_TRY(dev_alloc(ctx, (void **)&plan.clu_d, b));
        owned.push_back({plan.clu_d, b});
        PASUR_CUDA(ctx, cudaMemcpyAsync(plan.clu_d, plan.clu_h.data(), b, cudaMemcpyHostToDevice, ctx->stream));
    }
    auto in_block = [&](const pasur_tree *t, int64_t g) {
        const int c = t->croots_h[(size_t)g].cls;
        return c >= 0 && c < kClsGlobal;
    };
    int64_t slots = 0;
    for (const pasur_tree *t : trees)
        for (int64_t g = 0; g < t->n_roots; g++)
            if (in_block(t, g)) slots += t->csoff_h[(size_t)g + 1] - t->csoff_h[(size_t)g];
    if (slots == 0) return PASUR_OK;
    // slots per item: as many as a block holds, but with few slots in all rather more blocks than more
    // slots per block
    int64_t wcap = std::max<int64_t>(1, std::min<int64_t>(kBlockSlots, slots / (kSlotsPerSm * ctx->num_sms)));
    if (cfg->slots_per_item > 0) wcap = std::min(cfg->slots_per_item, kBlockSlots);
    // blocks per SM by shared memory (228 KB per SM, 1 KB reserved per block, some static)
    auto per_sm = [&](size_t smem) {
        for (int n = 6; n > 1; n--)
            if ((smem + 1024 + (ctx->smem_optin - lim)) * (size_t)n <= 228 * 1024) return n;
        return 1;
    };
    struct Tagged {
        BlockItem it;
        int per, chunks;
        size_t smem;
    };
    std::vector<Tagged> all;
    for (size_t ti = 0; ti < trees.size(); ti++) {
        const pasur_tree *t = trees[ti];
        for (int64_t g = 0; g < t->n_roots; g++) {
            if (!in_block(t, g)) continue;
            const CfrRoot &cr = t->croots_h[(size_t)g];
            const BlockRoot &br = t->broots_h[(size_t)g];
            const int64_t S = t->csoff_h[(size_t)g + 1] - t->csoff_h[(size_t)g], L = cr.ls[9], nA = cr.as[9], nR = br.rs[8];
            int64_t w = std::min<int64_t>(S, wcap);
            while (w > 1 && !block_fits(cr, br, (int)w, lim)) w--;
            const int64_t n = (S + w - 1) / w;
            int chunks = 1;
            for (int k = 0; k < 8; k++) chunks = std::max(chunks, (cr.as[k + 1] - cr.as[k]) / 32 + br.rs[k + 1] - br.rs[k]);
            for (int64_t i = 0, s0 = 0; i < n; i++) {
                Tagged x{};
                x.it.tree = (int32_t)ti;
                x.it.root = (int32_t)g;
                x.it.s0 = (int32_t)s0;
                x.it.ns = (int32_t)(S / n + (i < S % n ? 1 : 0));
                x.it.cost = std::max<int64_t>(nA, 1) * x.it.ns;
                x.chunks = chunks;
                x.smem = block_offsets(L, nA, nR, x.it.ns, kBlockMaxThreads / 32).end;
                if (x.smem > lim) return set_err(ctx, PASUR_EINVAL, "a block item exceeds a block's shared memory");
                x.per = per_sm(x.smem);
                all.push_back(x);
                s0 += x.it.ns;
            }
        }
    }
    std::stable_sort(all.begin(), all.end(), [](const Tagged &a, const Tagged &b) {
        if (a.per != b.per) return a.per < b.per;
        if (a.it.ns != b.it.ns) return a.it.ns > b.it.ns;
        return a.it.cost > b.it.cost;
    });
    // warps: what the registers allow among the blocks of one SM, no more than the widest level's chunks
    const bool few = (int64_t)all.size() <= ctx->num_sms;
    int chunks = 1;
    for (size_t i = 0; i < all.size(); i++) {
        const Tagged &x = all[i];
        if (i == 0 || x.per != all[i - 1].per || x.it.ns != all[i - 1].it.ns) {
            SweepLaunch l;
            l.W = x.it.ns;
            l.begin = (int64_t)i;
            plan.launches.push_back(l);
            chunks = 1;
        }
        SweepLaunch &l = plan.launches.back();
        l.end = (int64_t)i + 1;
        l.smem = std::max(l.smem, x.smem);
        chunks = std::max(chunks, x.chunks);
        l.threads = cfg->threads > 0 ? full : std::max(32, std::min(kBlockMaxThreads / (few ? 1 : x.per) / 32 * 32, 32 * chunks));
        plan.blk_h.push_back(x.it);
    }
    const size_t b = sizeof(BlockItem) * plan.blk_h.size();
    PASUR_TRY(dev_alloc(ctx, (void **)&plan.blk_d, b));
    owned.push_back({plan.blk_d, b});
    PASUR_CUDA(ctx, cudaMemcpyAsync(plan.blk_d, plan.blk_h.data(), b, cudaMemcpyHostToDevice, ctx->stream));
    return PASUR_OK;
}

int cfr_finalize_plan(pasur_ctx *ctx, CfrPlan &plan, std::vector<CfrItem> *cls_items, const std::vector<pasur_tree *> &trees,
                      const pasur_config *cfg, std::vector<std::pair<void *, size_t>> &owned,
                      const std::vector<ClusterItem> &clu) {
    if (cfg->threads < 0 || cfg->threads > 1024 || cfg->threads % 32)
        return set_err(ctx, PASUR_EINVAL, "cfg.threads must be 0 or a multiple of 32 <= 1024");
    if (cfg->split_bytes < 0) return set_err(ctx, PASUR_EINVAL, "cfg.split_bytes must be >= 0");
    if (cfg->stream_bytes < 0) return set_err(ctx, PASUR_EINVAL, "cfg.stream_bytes must be >= 0");
    plan.items_h.clear();
    // how the roots' state is stored: classes 0..4 of the roots solved in a block, 5 the
    // level-streaming sweep's items, 6 the roots split over clusters
    for (int c = 0; c <= kClsCluster; c++) {
        std::stable_sort(cls_items[c].begin(), cls_items[c].end(),
                         [](const CfrItem &a, const CfrItem &b) { return a.cost > b.cost; });
        plan.cls_begin[c] = (int64_t)plan.items_h.size();
        plan.items_h.insert(plan.items_h.end(), cls_items[c].begin(), cls_items[c].end());
        plan.cls_end[c] = (int64_t)plan.items_h.size();
    }
    plan.n_items = (int64_t)plan.items_h.size();
    if (plan.n_items) {
        size_t b = sizeof(CfrItem) * (size_t)plan.n_items;
        PASUR_TRY(dev_alloc(ctx, (void **)&plan.items_d, b));
        owned.push_back({plan.items_d, b});
        PASUR_CUDA(ctx, cudaMemcpyAsync(plan.items_d, plan.items_h.data(), b, cudaMemcpyHostToDevice, ctx->stream));
    }
    std::vector<TreeView> views;
    for (const pasur_tree *t : trees) views.push_back(t->view);
    if (!views.empty()) {
        size_t b = sizeof(TreeView) * views.size();
        PASUR_TRY(dev_alloc(ctx, (void **)&plan.views_d, b));
        owned.push_back({plan.views_d, b});
        PASUR_CUDA(ctx, cudaMemcpyAsync(plan.views_d, views.data(), b, cudaMemcpyHostToDevice, ctx->stream));
    }
    // class 5 runs as the level-streaming sweep: its prefixes, per-slot scales and sums
    plan.str_n = plan.cls_end[kClsGlobal] - plan.cls_begin[kClsGlobal];
    plan.str_nslots = 0;
    if (plan.str_n > 0) {
        const int64_t n = plan.str_n, b0 = plan.cls_begin[kClsGlobal];
        std::vector<int64_t> so((size_t)n + 1, 0);
        for (int64_t j = 0; j < n; j++) so[(size_t)j + 1] = so[(size_t)j] + plan.items_h[(size_t)(b0 + j)].ns;
        plan.str_nslots = so[(size_t)n];
        auto own = [&](void **p, size_t bytes) -> int {
            PASUR_TRY(dev_alloc(ctx, p, bytes));
            owned.push_back({*p, bytes});
            return PASUR_OK;
        };
        PASUR_TRY(own((void **)&plan.str_pairs, sizeof(int64_t) * 8 * (size_t)(n + 1)));
        PASUR_TRY(own((void **)&plan.str_locs, sizeof(int64_t) * (size_t)(n + 1)));
        PASUR_TRY(own((void **)&plan.str_slots, sizeof(int64_t) * (size_t)(n + 1)));
        PASUR_TRY(own((void **)&plan.str_tu, sizeof(uint32_t) * (size_t)plan.str_nslots));
        PASUR_TRY(own((void **)&plan.str_acc, sizeof(double) * (size_t)plan.str_nslots));
        PASUR_TRY(own((void **)&plan.str_desc, sizeof(StreamDesc) * (size_t)n));
        PASUR_CUDA(ctx, cudaMemcpyAsync(plan.str_slots, so.data(), sizeof(int64_t) * so.size(), cudaMemcpyHostToDevice,
                                        ctx->stream));
        k_stream_plan<<<1, 32, 0, ctx->stream>>>(plan.items_d + b0, n, plan.views_d, plan.str_pairs, plan.str_locs,
                                                 plan.str_slots, plan.str_desc);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    }
    PASUR_TRY(plan_sweeps(ctx, plan, trees, cfg, clu, owned));
    // the uploads read host vectors of this call
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return PASUR_OK;
}

int cfr_dcfr_factors(pasur_ctx *ctx, const pasur_config *cfg, int64_t t0, std::vector<float> &f, float **out, size_t *bytes) {
    *out = nullptr;
    *bytes = 0;
    if (cfg->variant != 1 || cfg->iters <= 0) return PASUR_OK;
    f.resize(3 * (size_t)cfg->iters);
    for (int i = 0; i < cfg->iters; i++) {
        double tt = (double)(t0 + i + 1), tp = tt - 1.0;
        double pa = std::pow(tp, (double)cfg->dcfr_alpha), pb = std::pow(tp, (double)cfg->dcfr_beta);
        f[3 * i] = (float)(pa / (pa + 1.0));
        f[3 * i + 1] = (float)(pb / (pb + 1.0));
        f[3 * i + 2] = (float)(tt > 1.0 ? std::pow(1.0 - 1.0 / tt, (double)cfg->dcfr_gamma) : 0.0);
    }
    *bytes = f.size() * sizeof(float);
    PASUR_TRY(dev_alloc(ctx, (void **)out, *bytes));
    PASUR_CUDA(ctx, cudaMemcpyAsync(*out, f.data(), *bytes, cudaMemcpyHostToDevice, ctx->stream));
    return PASUR_OK;
}

int ensure_aux(pasur_ctx *ctx) {
    if (ctx->fork) return PASUR_OK;
    PASUR_CUDA(ctx, cudaEventCreateWithFlags(&ctx->fork, cudaEventDisableTiming));
    int least = 0, greatest = 0;
    PASUR_CUDA(ctx, cudaDeviceGetStreamPriorityRange(&least, &greatest));
    for (int c = 0; c < kAuxStreams; c++) {
        // the level-streaming sweep is a chain of short dependent launches: its blocks go first
        // whenever an SM frees up, the block sweep and the clusters fill the rest
        PASUR_CUDA(ctx, cudaStreamCreateWithPriority(&ctx->aux[c], cudaStreamNonBlocking, c == kAuxStream ? greatest : least));
        PASUR_CUDA(ctx, cudaEventCreateWithFlags(&ctx->join[c], cudaEventDisableTiming));
        PASUR_CUDA(ctx, cudaEventCreate(&ctx->cls_t0[c]));
        PASUR_CUDA(ctx, cudaEventCreate(&ctx->cls_t1[c]));
    }
    return PASUR_OK;
}

// All iterations of the plan's class-5 items on stream st: set-up, 15 level launches per
// iteration, the root sums into the running utilities.
int stream_sweep(pasur_ctx *ctx, const CfrPlan &plan, CfrParams p, const pasur_config *cfg, cudaStream_t st) {
    p.items = plan.items_d + plan.cls_begin[kClsGlobal];
    StreamPlan sp{plan.str_pairs, plan.str_locs, plan.str_slots, plan.str_tu, plan.str_acc, plan.str_n, plan.str_desc};
    const unsigned grid = (unsigned)ctx->num_sms * 8;
    const unsigned lgrid = (unsigned)ctx->num_sms * 4;  // the level kernels: four (bottom-up: three) blocks per SM
    PASUR_CUDA(ctx, cudaMemsetAsync(plan.str_tu, 0, sizeof(uint32_t) * (size_t)plan.str_nslots, st));
    k_stream_setup<<<grid, 256, 0, st>>>(p, sp);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    for (int il = 0; il < cfg->iters; il++)
        for (int i = 0; i < 15; i++) {
            const int k = i < 7 ? i : 14 - i;
            if (cfg->variant == 1) {
                if (i < 7) k_stream_level<1, true><<<lgrid, kStreamThreads, 0, st>>>(p, sp, k, il);
                else k_stream_level<1, false><<<lgrid, kStreamThreads, 0, st>>>(p, sp, k, il);
            } else {
                if (i < 7) k_stream_level<0, true><<<lgrid, kStreamThreads, 0, st>>>(p, sp, k, il);
                else k_stream_level<0, false><<<lgrid, kStreamThreads, 0, st>>>(p, sp, k, il);
            }
            ctx->launches++;
            PASUR_CUDA(ctx, cudaGetLastError());
        }
    k_stream_finalize<<<grid, 256, 0, st>>>(p, sp);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    return PASUR_OK;
}

int cfr_launch_plan(pasur_ctx *ctx, CfrPlan &plan, const pasur_config *cfg, int64_t t0, const float *dcfr) {
    if (cfg->iters <= 0 || plan.n_items == 0) return PASUR_OK;
    PASUR_TRY(ensure_aux(ctx));
    CfrParams p{};
    p.items = plan.items_d;
    p.views = plan.views_d;
    p.dcfr = dcfr;
    p.iters = cfg->iters;
    p.t0 = t0;
    p.tau = cfg->rm_deadzone;
    p.err = ctx->errflag;
    // a call of few iterations feels every event (2 to 4 us of a launch of 20 to 60): the launches' times are taken for
    // PASUR_VERBOSE alone, and the first launch needs no other stream than the context's
    const bool timed = getenv("PASUR_VERBOSE") != nullptr;
    PASUR_CUDA(ctx, cudaEventRecord(ctx->fork, ctx->stream));
    auto stream = [&](int c) { return c == kAuxSweep ? ctx->stream : ctx->aux[c]; };
    auto fork = [&](int c) -> int {
        if (stream(c) != ctx->stream) PASUR_CUDA(ctx, cudaStreamWaitEvent(stream(c), ctx->fork, 0));
        if (timed) PASUR_CUDA(ctx, cudaEventRecord(ctx->cls_t0[c], stream(c)));
        return PASUR_OK;
    };
    auto join = [&](int c) -> int {
        if (timed) PASUR_CUDA(ctx, cudaEventRecord(ctx->cls_t1[c], stream(c)));
        if (stream(c) == ctx->stream) return PASUR_OK;
        PASUR_CUDA(ctx, cudaEventRecord(ctx->join[c], stream(c)));
        PASUR_CUDA(ctx, cudaStreamWaitEvent(ctx->stream, ctx->join[c], 0));
        return PASUR_OK;
    };
    // the launches are independent: each runs on its own stream (beyond their number,
    // several share one), clusters first, largest subtrees first; the level-streaming sweep (thousands
    // of short launches) is queued last, so that the host never waits on its queue before the others
    // start.  The joins come after it: streams share the device's few hardware queues, and an event
    // record holds its queue until the launch before it has ended.  With the joins first the streamed
    // sweep of a 1.9e9-node final round began after the clusters (1052 ms, 1012 with a thread to a
    // (node, slot) in the clusters); so both run together
    const int nb = (int)std::min<size_t>(plan.launches.size(), kAuxStreams - kAuxSweep);
    const bool streamed = plan.cls_end[kClsGlobal] != plan.cls_begin[kClsGlobal];
    auto launch = [&]() -> int {
        for (int x = 0; x < nb; x++) PASUR_TRY(fork(kAuxSweep + x));
        for (size_t i = 0; i < plan.launches.size(); i++) {
            const SweepLaunch &l = plan.launches[i];
            BlockParams bp{nullptr, plan.views_d, dcfr, cfg->iters, t0, cfg->rm_deadzone, ctx->errflag};
            const ClusterItem *ci = nullptr;
            void *args[] = {&bp, &ci};
            cudaLaunchConfig_t lc{};
            cudaLaunchAttribute at[1];
            sweep_launch_config(l, &lc, at);
            lc.stream = stream(kAuxSweep + (int)(i % (size_t)nb));
            if (l.ctas > 1) ci = plan.clu_d + l.begin;
            else bp.items = plan.blk_d + l.begin;
            PASUR_CUDA(ctx, cudaLaunchKernelExC(&lc, l.ctas > 1 ? cluster_kernel(cfg->variant, l.W) : block_kernel(cfg->variant, l.W), args));
            ctx->launches++;
        }
        if (streamed) {
            PASUR_TRY(fork(kAuxStream));
            PASUR_TRY(stream_sweep(ctx, plan, p, cfg, ctx->aux[kAuxStream]));
        }
        return PASUR_OK;
    };
    // joined whether or not all could be launched: the caller frees in the context's stream what the launches use
    int rc = launch();
    auto also = [&](int r) { rc = rc == PASUR_OK ? r : rc; };
    for (int x = 0; x < nb; x++) also(join(kAuxSweep + x));
    if (streamed) also(join(kAuxStream));
    return rc;
}

void cfr_plan_times(pasur_ctx *ctx, CfrPlan &plan) {
    const size_t nb = std::min<size_t>(plan.launches.size(), kAuxStreams - kAuxSweep);
    for (size_t i = 0; i < plan.launches.size(); i++) {
        plan.launches[i].ms = 0.f;
        if (i < nb) cudaEventElapsedTime(&plan.launches[i].ms, ctx->cls_t0[kAuxSweep + i], ctx->cls_t1[kAuxSweep + i]);
    }
    plan.str_ms = 0.f;
    if (plan.cls_end[kClsGlobal] != plan.cls_begin[kClsGlobal])
        cudaEventElapsedTime(&plan.str_ms, ctx->cls_t0[kAuxStream], ctx->cls_t1[kAuxStream]);
}

// one line per launch of a plan
void cfr_print_plan(const CfrPlan &plan) {
    for (const SweepLaunch &l : plan.launches) {
        int64_t cost = 0, maxcost = 0;
        for (int64_t i = l.begin; i < l.end; i++) {
            const int64_t x = l.ctas > 1 ? plan.clu_h[(size_t)i].cost : plan.blk_h[(size_t)i].cost;
            cost += x;
            maxcost = std::max(maxcost, x);
        }
        char ctas[32] = "";
        if (l.ctas > 1) snprintf(ctas, sizeof ctas, "%d CTAs x ", l.ctas);
        fprintf(stderr, "[pasur]   %s items: %lld of %d slots, %s%d threads, smem %zu B, active-node-slots %lld (largest item "
                        "%lld), %.3f ms\n",
                l.ctas > 1 ? "cluster" : "block", (long long)(l.end - l.begin), l.W, ctas, l.threads, l.smem, (long long)cost,
                (long long)maxcost, l.ms);
    }
    if (plan.str_n > 0)
        fprintf(stderr, "[pasur]   streamed items: %lld (slots %lld), %.3f ms\n", (long long)plan.str_n, (long long)plan.str_nslots,
                plan.str_ms);
}

static void print_plan(const pasur_tree *t, const CfrPlan &plan) {
    int64_t ne = 0;
    for (int k = 1; k < 9; k++) ne += t->Q[k];
    fprintf(stderr, "[pasur] round %d: GT roots %lld, FGT edges %lld, local %lld, active %lld, items %lld\n", t->round,
            (long long)t->n_roots, (long long)ne, (long long)t->n_local, (long long)t->n_active, (long long)plan.n_items);
    cfr_print_plan(plan);
}

int cfr_prepare(pasur_tree *t, const pasur_config *cfg) {
    pasur_ctx *ctx = t->ctx;
    std::vector<CfrItem> cls_items[8];
    std::vector<ClusterItem> clu;
    PASUR_TRY(cfr_setup_tree(t, cfg, 0, cls_items, &clu));
    std::vector<std::pair<void *, size_t>> owned;
    int rc = cfr_finalize_plan(ctx, t->plan, cls_items, {t}, cfg, owned, clu);
    for (auto &o : owned) {
        t->allocs.push_back(o.first);
        t->allocs.push_back((void *)(uintptr_t)o.second);
    }
    if (rc != PASUR_OK) return rc;
    if (getenv("PASUR_VERBOSE")) print_plan(t, t->plan);
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    t->cfr_ready = true;
    return PASUR_OK;
}

int cfr_run(pasur_tree *t, const pasur_config *cfg) {
    pasur_ctx *ctx = t->ctx;
    if (cfg->iters <= 0 || t->plan.n_items == 0) {
        t->last_ms = 0.f;
        t->last_launches = 0;
        return PASUR_OK;
    }
    // what the call holds on every way out: the factors (host and device) until the stream is done with them, its events
    struct Held {
        pasur_ctx *ctx;
        std::vector<float> factors;
        float *dcfr = nullptr;
        size_t bytes = 0;
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        ~Held() {
            dev_free(ctx, dcfr, bytes);
            if (e0) cudaEventDestroy(e0);
            if (e1) cudaEventDestroy(e1);
        }
    } held{ctx};
    cudaEvent_t &e0 = held.e0, &e1 = held.e1;
    PASUR_CUDA(ctx, cudaEventCreate(&e0));
    PASUR_CUDA(ctx, cudaEventCreate(&e1));
    int rc = cfr_dcfr_factors(ctx, cfg, t->iters_done, held.factors, &held.dcfr, &held.bytes);
    if (rc == PASUR_OK && cudaMemsetAsync(ctx->errflag, 0, sizeof(int32_t), ctx->stream) != cudaSuccess)
        rc = set_err(ctx, PASUR_ECUDA, "pasur_cfr_iterate: error word");
    if (rc == PASUR_OK && cudaEventRecord(e0, ctx->stream) != cudaSuccess) rc = set_err(ctx, PASUR_ECUDA, "pasur_cfr_iterate: event");
    const int64_t before = ctx->launches;
    if (rc == PASUR_OK) rc = cfr_launch_plan(ctx, t->plan, cfg, t->iters_done, held.dcfr);
    if (rc != PASUR_OK) {
        cudaStreamSynchronize(ctx->stream);
        return rc;
    }
    PASUR_CUDA(ctx, cudaEventRecord(e1, ctx->stream));
    int32_t ef = 0;
    PASUR_CUDA(ctx, cudaMemcpyAsync(&ef, ctx->errflag, sizeof ef, cudaMemcpyDeviceToHost, ctx->stream));
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    float ms = 0.f;
    PASUR_CUDA(ctx, cudaEventElapsedTime(&ms, e0, e1));
    t->last_ms = ms;
    t->last_launches = (int32_t)(ctx->launches - before);
    t->iters_done += cfg->iters;
    if (getenv("PASUR_VERBOSE")) {
        cfr_plan_times(ctx, t->plan);
        fprintf(stderr, "[pasur] round %d: %d iterations in %.3f ms\n", t->round, cfg->iters, ms);
        cfr_print_plan(t->plan);
    }
    if (ef) return set_err(ctx, PASUR_ENUMERIC, "non-finite root value in the CFR sweep");
    return PASUR_OK;
}

int sigma_sqdiff(const pasur_tree *t, const float *a_dev, const float *b_dev, double *acc_dev) {
    pasur_ctx *ctx = t->ctx;
    int64_t cb = 0;
    for (int k = 1; k < 9; k++) {
        if (t->M[k] > 0) {
            const unsigned grid = (unsigned)std::min<int64_t>((t->M[k] * 32 + 255) / 256, (int64_t)ctx->num_sms * 16);
            k_sigma_sqdiff<<<grid, 256, 0, ctx->stream>>>(t->root[k], t->M[k], t->cfgt_off[k], t->csoff_d, t->cmult_d,
                                                         a_dev + cb, b_dev + cb, acc_dev);
            ctx->launches++;
            PASUR_CUDA(ctx, cudaGetLastError());
        }
        cb += t->cQ[k];
    }
    return PASUR_OK;
}

// average strategies of the solved slots (levels 1..8 concatenated in solved FGT order)
int export_sigma_solved(const pasur_tree *t, float *out_dev) {
    pasur_ctx *ctx = t->ctx;
    LevelPtrs lp{};
    int64_t base = 0, ne = 0;
    for (int k = 0; k < 9; k++) {
        lp.fgt[k] = t->cfgt_off[k];
        lp.child[k] = k < 8 ? t->child_off[k] : nullptr;
        lp.base[k] = k >= 1 ? base : 0;
        if (k >= 1) base += t->cQ[k];
    }
    ne = base;
    if (ne > 0) {
        k_fill<<<grid_for(ne, 256), 256, 0, ctx->stream>>>(out_dev, ne, 1.0f);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
    }
    if (t->plan.n_items) {
        // few items are large ones: share each out over blocks until the GPU is full
        dim3 g((unsigned)std::min<int64_t>(t->plan.n_items, 65535));
        g.y = (unsigned)std::min<int64_t>(64, (8 * (int64_t)ctx->num_sms + g.x - 1) / g.x);
        k_export_sigma<<<g, 256, 0, ctx->stream>>>(t->plan.items_d, t->plan.n_items, t->croots_d, t->act_cs, t->act_d,
                                                   t->act_gt, t->S, lp, out_dev);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
    }
    return PASUR_OK;
}

int cfr_export_sigma(const pasur_tree *t, float *out_dev) {
    if (!t->merged) return export_sigma_solved(t, out_dev);
    pasur_ctx *ctx = t->ctx;
    int64_t ce = 0;
    for (int k = 1; k < 9; k++) ce += t->cQ[k];
    float *tmp = nullptr;
    const size_t tb = sizeof(float) * (size_t)(ce + 1);
    PASUR_TRY(dev_alloc(ctx, (void **)&tmp, tb));
    int rc = export_sigma_solved(t, tmp);
    ExpandLevels L{};
    int64_t fb = 0, cb = 0, nodes = 0;
    for (int k = 1; k < 9; k++) {
        L.root[k] = t->root[k];
        L.fgt[k] = t->fgt_off[k];
        L.cfgt[k] = t->cfgt_off[k];
        L.first[k] = nodes;
        L.out[k] = fb;
        L.in[k] = cb;
        nodes += t->M[k];
        fb += t->Q[k];
        cb += t->cQ[k];
    }
    L.first[9] = nodes;
    if (rc == PASUR_OK && nodes > 0) {
        k_expand_edges<<<grid_for(nodes * 8, 256), 256, 0, ctx->stream>>>(L, t->score_off_d, t->csoff_d, t->cidx0_d, tmp, out_dev);
        ctx->launches++;
        if (cudaGetLastError() != cudaSuccess) rc = set_err(ctx, PASUR_ECUDA, "k_expand_edges launch");
    }
    dev_free(ctx, tmp, tb);  // stream-ordered: freed after the expansion has read it
    return rc;
}

int cfr_export_utilities(const pasur_tree *t, float *out_dev) { return cfr_export_utilities_n(t, t->iters_done, out_dev); }

// average root utility of every full root slot, from its solved slot (no allocation: the batch
// captures this into its graph)
int cfr_export_utilities_n(const pasur_tree *t, int64_t iters, float *out_dev) {
    pasur_ctx *ctx = t->ctx;
    if (t->Q[0] == 0) return PASUR_OK;
    double inv = iters > 0 ? 1.0 / (double)iters : 0.0;
    k_export_util<<<grid_for(t->Q[0], 256), 256, 0, ctx->stream>>>(t->uacc, t->cidx0_d, t->Q[0], inv, out_dev);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    return PASUR_OK;
}

}  // namespace pasur
