// Game values of a round under fixed or optimal play, in fp64, level by level from the leaves:
// minimax, a best response of one player to the other's strategy, or both players on a given
// strategy.  Chained over the rounds (leaf = the round's difference + the next round's value at
// the linked root, eq. passuputil) they give the best-response values whose gap is the
// exploitability of a strategy profile (section "CFR Algorithm": the average strategy converges
// to an equilibrium; exploitability measures the distance).  Sums are taken child by child in
// canonical order with explicitly rounded multiply and add.
#include <algorithm>
#include <string>
#include <vector>

#include "pasur_internal.cuh"

namespace pasur {
namespace {

// Everything the value passes read, per level.
struct ValueArgs {
    const GTState *leaf_state;
    const int32_t *leaf_root;
    const int64_t *child_off[8], *fgt_off[9];
    const float *sigma[9];  // of the edges into level k
    const int64_t *score_off;
    const pasur_score *scores;
    const int64_t *lnk;
    const double *next;
    double *v[9];
    bool final_round;
    int lanes_log2;  // lanes to a node, over its slots
    int mode;        // 0 minimax, 1 Alex best response (Bob follows sigma), 2 Bob best response, 3 both sigma
};

// leaf values of level 8 in FGT order (fp64), leaves lo .. hi-1
__device__ __forceinline__ void leaf_values(const ValueArgs &A, int64_t lo, int64_t hi) {
    const int lanes = 1 << A.lanes_log2, lane = threadIdx.x & (lanes - 1), step = blockDim.x >> A.lanes_log2;
    for (int64_t j = lo + (threadIdx.x >> A.lanes_log2); j < hi; j += step) {
        const GTState s = A.leaf_state[j];
        const int64_t q0 = A.fgt_off[8][j], ns = A.fgt_off[8][j + 1] - q0;
        if (A.final_round) {
            const uint64_t r = cleanup_rus(s.rus, s.pool);
            const int d = rus_diff(r);
            const pasur_score *sc = A.scores + A.score_off[A.leaf_root[j]];
            for (int64_t x = lane; x < ns; x += lanes)
                A.v[8][q0 + x] = (double)(d + bonus_points(bonus_after(sc[x].a_clubs, sc[x].b_clubs, sc[x].bonus, r)));
        } else {
            const double d = (double)rus_diff(s.rus);
            for (int64_t x = lane; x < ns; x += lanes) A.v[8][q0 + x] = __dadd_rn(d, A.next[A.lnk[q0 + x]]);
        }
    }
}

// values of nodes lo .. hi-1 of level k from those of level k+1
__device__ __forceinline__ void level_values(const ValueArgs &A, int k, int64_t lo, int64_t hi) {
    const bool alex = (k & 1) == 0;
    const bool opt = A.mode == 0 || (A.mode == 1 && alex) || (A.mode == 2 && !alex);
    const int64_t *child_off = A.child_off[k], *fgt_off = A.fgt_off[k], *fgt_off_next = A.fgt_off[k + 1];
    const float *sigma = A.sigma[k + 1];
    const double *vnext = A.v[k + 1];
    double *vout = A.v[k];
    const int lanes = 1 << A.lanes_log2, lane = threadIdx.x & (lanes - 1), step = blockDim.x >> A.lanes_log2;
    for (int64_t j = lo + (threadIdx.x >> A.lanes_log2); j < hi; j += step) {
        const int64_t cb = child_off[j], ce = child_off[j + 1];
        const int64_t q0 = fgt_off[j], ns = fgt_off[j + 1] - q0;
        for (int64_t s = lane; s < ns; s += lanes) {
            double best = 0.0, ev = 0.0;
#pragma unroll 4
            for (int64_t c = cb; c < ce; c++) {
                const int64_t q = fgt_off_next[c] + s;
                const double v = vnext[q];
                if (c == cb || (alex ? v > best : v < best)) best = v;
                if (!opt) ev = __dadd_rn(ev, __dmul_rn((double)sigma[q], v));
            }
            vout[q0 + s] = opt ? best : ev;
        }
    }
}

// Values of levels top .. 8 (bottom = 8: from the leaves on) or top .. bottom, a block per range of level `top`'s m
// nodes: their descendants are a range of every level below, so that a block needs no other's values.  One launch
// from `split_level` down, one block for the levels above it.  Bound by launches and by the chains of dependent loads
// (child range, slot offset, value), hence several lanes to a node and four children in flight.  Both players' best
// responses through the last four rounds of a deal (with the strategies' exports): 1.4 ms with a launch per level and a
// thread to a node, 0.7 so.  For rounds that fill the GPU level by level see wide_round.
__global__ void __launch_bounds__(1024) k_values(const ValueArgs A, int top, int bottom, int64_t m) {
    __shared__ int64_t lo[9], hi[9];
    if (threadIdx.x < 2) {
        int64_t x = m * (int64_t)(blockIdx.x + threadIdx.x) / gridDim.x;
        int64_t *at = threadIdx.x ? hi : lo;
        at[top] = x;
        for (int k = top; k < bottom; k++) at[k + 1] = x = A.child_off[k][x];
    }
    __syncthreads();
    if (bottom == 8) leaf_values(A, lo[8], hi[8]);
    for (int k = bottom - 1; k >= top; k--) {
        __syncthreads();
        level_values(A, k, lo[k], hi[k]);
    }
}

// One level on its own (k = 8: the leaves), a block to as many nodes as it holds at once.  Bound by the loads of the
// children's values, slots over lanes: a final round of 1.05e9 leaves in 23 ms (43 in ranges, 111 with a thread to a node).
__global__ void __launch_bounds__(256) k_value_level(const ValueArgs A, int k, int64_t m) {
    const int64_t per = blockDim.x >> A.lanes_log2;
    for (int64_t lo = (int64_t)blockIdx.x * per; lo < m; lo += (int64_t)gridDim.x * per) {
        const int64_t hi = lo + per < m ? lo + per : m;
        if (k == 8) leaf_values(A, lo, hi);
        else level_values(A, k, lo, hi);
    }
}

// first level with two nodes to an SM: the tree below it splits over the GPU, and the levels above it, of fewer nodes
// each, are a few passes of one block
int split_level(const pasur_tree *t) {
    int k = 0;
    while (k < 7 && t->M[k] < 2 * t->ctx->num_sms) k++;
    return k;
}

// Rounds that take a launch per level instead of a block per range of subtrees.  The subtrees' sizes differ by up to a
// hundred, and a block's range is fixed, so that a wide round waits for its heaviest range; nine launches cost some 25 us
// more than two.  Ranges and levels (root values, one call, ms): 376 roots, 2.2e6 leaves, 1.2e7 with their slots 2.51 and
// 0.60; 255 roots, 8.3e5, 4.4e6 1.98 and 0.32; 79 roots, 7.5e6, 9.5e8 196 and 19; 49 roots, 3.8e4, 1.5e6 0.165 and 0.166; 24
// roots, 1.6e4, 2.2e6 0.29 and 0.33; 81 roots, 9.0e4, 3.4e5 0.100 and 0.104; 90 roots, 1.5e5, 5.9e5 0.145 and 0.125.
bool wide_round(const pasur_tree *t) { return t->M[8] >= 1 << 17 || t->Q[8] >= 5 << 19; }

unsigned grid_of(int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 1 << 20)); }

}  // namespace
}  // namespace pasur

using namespace pasur;

namespace {

// The shared part of the value and reach passes: the strategy on the device (copied, or the
// tree's own average strategy when sigma is NULL), the next-round values on the device, and the
// values of every FGT level under `mode` (v[0..8]; mode 3 = both players on sigma).  Device
// temporaries are appended to tmp.
int value_levels(pasur_tree *t, int mode, const float *sigma, const double *next_values,
                 std::vector<std::pair<void *, size_t>> &tmp, const float **sg_out, double *v[9]) {
    pasur_ctx *ctx = t->ctx;
    int rc = PASUR_OK;
    auto al = [&](void **p, size_t b) {
        if (rc != PASUR_OK) return;
        rc = dev_alloc(ctx, p, b);
        if (rc == PASUR_OK) tmp.push_back({*p, b});
    };
    int64_t ne = 0, base[9] = {0};
    for (int k = 1; k < 9; k++) {
        base[k] = ne;
        ne += t->Q[k];
    }
    const float *sg = nullptr;
    if (mode != 0) {
        if (sigma && is_device_ptr(sigma)) {
            sg = sigma;
        } else {
            float *d = nullptr;
            al((void **)&d, sizeof(float) * (size_t)(ne + 1));
            if (rc == PASUR_OK) {
                if (sigma) rc = cudaMemcpyAsync(d, sigma, sizeof(float) * (size_t)ne, cudaMemcpyHostToDevice, ctx->stream) == cudaSuccess ? PASUR_OK : set_err(ctx, PASUR_ECUDA, "copy sigma");
                else rc = cfr_export_sigma(t, d);
            }
            sg = d;
        }
    }
    const double *nx = nullptr;
    if (!t->final_round) {
        if (is_device_ptr(next_values)) {
            nx = next_values;
        } else {
            double *d = nullptr;
            al((void **)&d, sizeof(double) * (size_t)(t->n_next_roots + 1));
            if (rc == PASUR_OK)
                rc = cudaMemcpyAsync(d, next_values, sizeof(double) * (size_t)t->n_next_roots, cudaMemcpyHostToDevice, ctx->stream) ==
                             cudaSuccess
                         ? PASUR_OK
                         : set_err(ctx, PASUR_ECUDA, "copy next values");
            nx = d;
        }
    }
    int64_t nv = 0;
    for (int k = 0; k < 9; k++) nv += t->Q[k] + 1;
    double *values = nullptr;
    al((void **)&values, sizeof(double) * (size_t)nv);
    ValueArgs A{};
    for (int k = 0; k < 9; k++) {
        A.v[k] = v[k] = values;
        values += t->Q[k] + 1;
        A.fgt_off[k] = t->fgt_off[k];
        if (k < 8) A.child_off[k] = t->child_off[k];
        if (k > 0 && sg) A.sigma[k] = sg + base[k];
    }
    A.leaf_state = t->st[8];
    A.leaf_root = t->root[8];
    A.score_off = t->score_off_d;
    A.scores = t->scores_d;
    A.lnk = t->lnk_d;
    A.next = nx;
    A.final_round = t->final_round;
    A.mode = mode;
    while (A.lanes_log2 < 3 && t->Q[8] > t->M[8] << A.lanes_log2) A.lanes_log2++;  // the leaves' slots on average
    if (rc == PASUR_OK && t->M[0] > 0 && wide_round(t)) {
        for (int k = 8; k >= 0; k--) {
            k_value_level<<<grid_of(t->M[k] << A.lanes_log2), 256, 0, ctx->stream>>>(A, k, t->M[k]);
            ctx->launches++;
        }
        if (cudaGetLastError() != cudaSuccess) rc = set_err(ctx, PASUR_ECUDA, "k_value_level launch");
    } else if (rc == PASUR_OK && t->M[0] > 0) {
        const int top = split_level(t);
        const int64_t blocks = std::min<int64_t>(t->M[top], 8 * (int64_t)ctx->num_sms);
        k_values<<<(unsigned)blocks, 256, 0, ctx->stream>>>(A, top, 8, t->M[top]);
        ctx->launches++;
        if (top > 0) {
            k_values<<<1, 1024, 0, ctx->stream>>>(A, 0, top, t->M[0]);
            ctx->launches++;
        }
        if (cudaGetLastError() != cudaSuccess) rc = set_err(ctx, PASUR_ECUDA, "k_values launch");
    }
    *sg_out = sg;
    return rc;
}

}  // namespace

extern "C" int pasur_root_values(pasur_tree *t, int mode, const float *sigma, const double *next_values, double *out,
                                 int64_t cap) {
    if (!t) return PASUR_EINVAL;
    pasur_ctx *ctx = t->ctx;
    if (mode < 0 || mode > 3) return set_err(ctx, PASUR_EINVAL, "pasur_root_values: mode must be 0..3");
    if (!t->unfolded) return set_err(ctx, PASUR_EINVAL, "pasur_root_values: tree not unfolded");
    if (!t->final_round && (!next_values || !t->has_next))
        return set_err(ctx, PASUR_EINVAL, "pasur_root_values: a non-final round needs pasur_next_roots and next_values");
    if (mode != 0 && !sigma && !t->cfr_ready) return set_err(ctx, PASUR_EINVAL, "pasur_root_values: no strategy (no CFR run, sigma NULL)");
    if (!out || cap < t->Q[0]) return set_err(ctx, PASUR_EOVERFLOW, "pasur_root_values: need " + std::to_string(t->Q[0]) + " doubles");
    cudaSetDevice(ctx->device);
    std::vector<std::pair<void *, size_t>> tmp;
    const float *sg = nullptr;
    double *v[9] = {nullptr};
    int rc = value_levels(t, mode, sigma, next_values, tmp, &sg, v);
    if (rc == PASUR_OK && t->Q[0] > 0 &&
        cudaMemcpyAsync(out, v[0], sizeof(double) * (size_t)t->Q[0], is_device_ptr(out) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                        ctx->stream) != cudaSuccess)
        rc = set_err(ctx, PASUR_ECUDA, "copy root values");
    if (cudaStreamSynchronize(ctx->stream) != cudaSuccess && rc == PASUR_OK) rc = set_err(ctx, PASUR_ECUDA, "pasur_root_values: sync");
    for (auto &x : tmp) dev_free(ctx, x.first, x.second);
    return rc;
}

namespace pasur {
namespace {

// reach of the FGT nodes of level k+1 from those of level k: both players following sigma
__global__ void k_reach_level(int64_t m, const int64_t *__restrict__ child_off, const int64_t *__restrict__ fgt_off,
                              const int64_t *__restrict__ fgt_off_next, const float *__restrict__ sigma_next,
                              const double *__restrict__ rin, double *__restrict__ rout) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cb = child_off[j], ce = child_off[j + 1];
        const int64_t q0 = fgt_off[j], ns = fgt_off[j + 1] - q0;
        for (int64_t c = cb; c < ce; c++)
            for (int64_t s = 0; s < ns; s++) {
                const int64_t q = fgt_off_next[c] + s;
                rout[q] = __dmul_rn(rin[q0 + s], (double)sigma_next[q]);
            }
    }
}

// reach of level k+1 from level k when one player best-responds (mode 1: Alex, 2: Bob; values of
// level k+1 under that mode in vnext): at the responder's nodes the whole reach goes to the child
// its value pass chose (the first best child in canonical order), at the other player's nodes it
// follows sigma
__global__ void k_response_reach_level(int k, int64_t m, int mode, const int64_t *__restrict__ child_off,
                                       const int64_t *__restrict__ fgt_off, const int64_t *__restrict__ fgt_off_next,
                                       const float *__restrict__ sigma_next, const double *__restrict__ vnext,
                                       const double *__restrict__ rin, double *__restrict__ rout) {
    const bool alex = (k & 1) == 0;
    const bool responder = (mode == 1 && alex) || (mode == 2 && !alex);
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cb = child_off[j], ce = child_off[j + 1];
        const int64_t q0 = fgt_off[j], ns = fgt_off[j + 1] - q0;
        for (int64_t s = 0; s < ns; s++) {
            const double r = rin[q0 + s];
            if (responder) {
                int64_t arg = cb;
                double best = 0.0;
                for (int64_t c = cb; c < ce; c++) {
                    const double v = vnext[fgt_off_next[c] + s];
                    if (c == cb || (alex ? v > best : v < best)) {
                        best = v;
                        arg = c;
                    }
                }
                for (int64_t c = cb; c < ce; c++) rout[fgt_off_next[c] + s] = c == arg ? r : 0.0;
            } else {
                for (int64_t c = cb; c < ce; c++) {
                    const int64_t q = fgt_off_next[c] + s;
                    rout[q] = __dmul_rn(r, (double)sigma_next[q]);
                }
            }
        }
    }
}

// every FGT leaf's reach added to its next-round root
__global__ void k_reach_next(int64_t n, const int64_t *__restrict__ lnk, const double *__restrict__ r, double *next) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        if (r[q] != 0.0) atomicAdd(&next[lnk[q]], r[q]);
}

}  // namespace
}  // namespace pasur

extern "C" int pasur_round_reach(pasur_tree *t, const float *sigma, const double *root_reach, double *next_reach,
                                 int64_t cap) {
    if (!t) return PASUR_EINVAL;
    pasur_ctx *ctx = t->ctx;
    if (!t->unfolded || t->final_round || !t->has_next)
        return set_err(ctx, PASUR_EINVAL, "pasur_round_reach: needs an unfolded non-final tree after pasur_next_roots");
    if (!sigma && !t->cfr_ready) return set_err(ctx, PASUR_EINVAL, "pasur_round_reach: no strategy (no CFR run, sigma NULL)");
    if (!next_reach || cap < t->n_next_roots)
        return set_err(ctx, PASUR_EOVERFLOW, "pasur_round_reach: need " + std::to_string(t->n_next_roots) + " doubles");
    cudaSetDevice(ctx->device);
    std::vector<std::pair<void *, size_t>> tmp;
    int rc = PASUR_OK;
    auto al = [&](void **p, size_t b) {
        if (rc != PASUR_OK) return;
        rc = dev_alloc(ctx, p, b);
        if (rc == PASUR_OK) tmp.push_back({*p, b});
    };
    int64_t ne = 0, base[9] = {0};
    for (int k = 1; k < 9; k++) {
        base[k] = ne;
        ne += t->Q[k];
    }
    const float *sg = nullptr;
    if (sigma && is_device_ptr(sigma)) {
        sg = sigma;
    } else {
        float *d = nullptr;
        al((void **)&d, sizeof(float) * (size_t)(ne + 1));
        if (rc == PASUR_OK) {
            if (sigma) rc = cudaMemcpyAsync(d, sigma, sizeof(float) * (size_t)ne, cudaMemcpyHostToDevice, ctx->stream) == cudaSuccess ? PASUR_OK : set_err(ctx, PASUR_ECUDA, "copy sigma");
            else rc = cfr_export_sigma(t, d);
        }
        sg = d;
    }
    double *r[9] = {nullptr}, *nx = nullptr;
    for (int k = 0; k < 9; k++) al((void **)&r[k], sizeof(double) * (size_t)(t->Q[k] + 1));
    al((void **)&nx, sizeof(double) * (size_t)(t->n_next_roots + 1));
    if (rc == PASUR_OK) {
        std::vector<double> ones;
        const double *src = root_reach;
        if (!root_reach) {
            ones.assign((size_t)t->Q[0], 1.0);
            src = ones.data();
        }
        if (t->Q[0] > 0 && cudaMemcpyAsync(r[0], src, sizeof(double) * (size_t)t->Q[0],
                                           is_device_ptr(src) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                           ctx->stream) != cudaSuccess)
            rc = set_err(ctx, PASUR_ECUDA, "copy root reach");
        if (rc == PASUR_OK && cudaMemsetAsync(nx, 0, sizeof(double) * (size_t)(t->n_next_roots + 1), ctx->stream) != cudaSuccess)
            rc = set_err(ctx, PASUR_ECUDA, "memset");
        if (rc == PASUR_OK && !root_reach) rc = cudaStreamSynchronize(ctx->stream) == cudaSuccess ? PASUR_OK : set_err(ctx, PASUR_ECUDA, "sync");
    }
    for (int k = 0; k < 8 && rc == PASUR_OK; k++) {
        if (t->M[k] == 0) continue;
        k_reach_level<<<grid_of(t->M[k]), 256, 0, ctx->stream>>>(t->M[k], t->child_off[k], t->fgt_off[k], t->fgt_off[k + 1],
                                                                 sg + base[k + 1], r[k], r[k + 1]);
        ctx->launches++;
        if (cudaGetLastError() != cudaSuccess) rc = set_err(ctx, PASUR_ECUDA, "k_reach_level launch");
    }
    if (rc == PASUR_OK && t->Q[8] > 0) {
        k_reach_next<<<grid_of(t->Q[8]), 256, 0, ctx->stream>>>(t->Q[8], t->lnk_d, r[8], nx);
        ctx->launches++;
        if (cudaGetLastError() != cudaSuccess) rc = set_err(ctx, PASUR_ECUDA, "k_reach_next launch");
    }
    if (rc == PASUR_OK && t->n_next_roots > 0 &&
        cudaMemcpyAsync(next_reach, nx, sizeof(double) * (size_t)t->n_next_roots,
                        is_device_ptr(next_reach) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess)
        rc = set_err(ctx, PASUR_ECUDA, "copy next reach");
    if (cudaStreamSynchronize(ctx->stream) != cudaSuccess && rc == PASUR_OK) rc = set_err(ctx, PASUR_ECUDA, "pasur_round_reach: sync");
    for (auto &x : tmp) dev_free(ctx, x.first, x.second);
    return rc;
}

extern "C" int pasur_response_reach(pasur_tree *t, int mode, const float *sigma, const double *next_values,
                                    const double *root_reach, double *next_reach, int64_t cap) {
    if (!t) return PASUR_EINVAL;
    pasur_ctx *ctx = t->ctx;
    if (mode < 1 || mode > 3) return set_err(ctx, PASUR_EINVAL, "pasur_response_reach: mode must be 1..3");
    if (!t->unfolded || t->final_round || !t->has_next)
        return set_err(ctx, PASUR_EINVAL, "pasur_response_reach: needs an unfolded non-final tree after pasur_next_roots");
    if (!next_values) return set_err(ctx, PASUR_EINVAL, "pasur_response_reach: next_values is required");
    if (!sigma && !t->cfr_ready) return set_err(ctx, PASUR_EINVAL, "pasur_response_reach: no strategy (no CFR run, sigma NULL)");
    if (!next_reach || cap < t->n_next_roots)
        return set_err(ctx, PASUR_EOVERFLOW, "pasur_response_reach: need " + std::to_string(t->n_next_roots) + " doubles");
    cudaSetDevice(ctx->device);
    std::vector<std::pair<void *, size_t>> tmp;
    const float *sg = nullptr;
    double *v[9] = {nullptr};
    int rc = value_levels(t, mode, sigma, next_values, tmp, &sg, v);
    auto al = [&](void **p, size_t b) {
        if (rc != PASUR_OK) return;
        rc = dev_alloc(ctx, p, b);
        if (rc == PASUR_OK) tmp.push_back({*p, b});
    };
    double *r[9] = {nullptr}, *nx = nullptr;
    for (int k = 0; k < 9; k++) al((void **)&r[k], sizeof(double) * (size_t)(t->Q[k] + 1));
    al((void **)&nx, sizeof(double) * (size_t)(t->n_next_roots + 1));
    std::vector<double> ones;
    if (rc == PASUR_OK) {
        const double *src = root_reach;
        if (!root_reach) {
            ones.assign((size_t)t->Q[0], 1.0);
            src = ones.data();
        }
        if (t->Q[0] > 0 && cudaMemcpyAsync(r[0], src, sizeof(double) * (size_t)t->Q[0],
                                           is_device_ptr(src) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                           ctx->stream) != cudaSuccess)
            rc = set_err(ctx, PASUR_ECUDA, "copy root reach");
        if (rc == PASUR_OK && cudaMemsetAsync(nx, 0, sizeof(double) * (size_t)(t->n_next_roots + 1), ctx->stream) != cudaSuccess)
            rc = set_err(ctx, PASUR_ECUDA, "memset");
    }
    int64_t base[9] = {0}, ne = 0;
    for (int k = 1; k < 9; k++) {
        base[k] = ne;
        ne += t->Q[k];
    }
    for (int k = 0; k < 8 && rc == PASUR_OK; k++) {
        if (t->M[k] == 0) continue;
        k_response_reach_level<<<grid_of(t->M[k]), 256, 0, ctx->stream>>>(k, t->M[k], mode, t->child_off[k], t->fgt_off[k],
                                                                          t->fgt_off[k + 1], sg + base[k + 1], v[k + 1], r[k],
                                                                          r[k + 1]);
        ctx->launches++;
        if (cudaGetLastError() != cudaSuccess) rc = set_err(ctx, PASUR_ECUDA, "k_response_reach_level launch");
    }
    if (rc == PASUR_OK && t->Q[8] > 0) {
        k_reach_next<<<grid_of(t->Q[8]), 256, 0, ctx->stream>>>(t->Q[8], t->lnk_d, r[8], nx);
        ctx->launches++;
        if (cudaGetLastError() != cudaSuccess) rc = set_err(ctx, PASUR_ECUDA, "k_reach_next launch");
    }
    if (rc == PASUR_OK && t->n_next_roots > 0 &&
        cudaMemcpyAsync(next_reach, nx, sizeof(double) * (size_t)t->n_next_roots,
                        is_device_ptr(next_reach) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess)
        rc = set_err(ctx, PASUR_ECUDA, "copy next reach");
    if (cudaStreamSynchronize(ctx->stream) != cudaSuccess && rc == PASUR_OK) rc = set_err(ctx, PASUR_ECUDA, "pasur_response_reach: sync");
    for (auto &x : tmp) dev_free(ctx, x.first, x.second);
    return rc;
}
