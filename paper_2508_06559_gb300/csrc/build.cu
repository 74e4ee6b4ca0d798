// Round game-tree build (legal-move enumeration, level-by-level expansion), the Unfolding
// Process and the leaf values of a round.
//
// Expansion of a level (section "Actions"): a device-wide exclusive scan of the nodes' degrees gives
// the child offsets, one thread per node notes its children's parent, and one thread per child finds
// its move from its place among its siblings, writes its state and counts its own degree for the next
// level.  A numeric card captures any set of pool numerics completing its value to 11; the sets are
// counted by a generating polynomial over the pool's cards (the coefficient of x^s: sets of sum s) and
// the r-th set in ascending order is found by dividing the cards out of it, highest first.  A thread
// per child does about 300 instructions; a warp per node that tested the sets of a table (2764 over
// the 40 cards) with a ballot spent about 230 warp instructions on every node, twice.
#include <algorithm>
#include <cstring>

#include "pasur_internal.cuh"

namespace pasur {
namespace {

// ---- sets of pool numerics by their sum -------------------------------------------------------
// Coefficients of x^0 .. x^10 in 11 bits each (with all 40 numerics in the pool the largest is 1702);
// what overflows above them does not reach them (arithmetic modulo a power of two).
typedef unsigned __int128 Poly;
constexpr int kSumBits = 11;

__device__ __forceinline__ int sets_of(Poly p, int sum) { return (int)(p >> (kSumBits * sum)) & ((1 << kSumBits) - 1); }

__device__ __forceinline__ Poly pool_sets(uint64_t pool) {
    Poly p = 1;
    for (uint64_t x = pool & kNumeric; x; x &= x - 1) p += p << (kSumBits * ((__ffsll((long long)x) - 1) / 4 + 1));
    return p;
}

// p without a card of value v: p / (1 + x^v) = p (1 - x^v) (1 + x^2v) (1 + x^4v) ... below x^11
__device__ __forceinline__ Poly without_card(Poly p, int v) {
    p -= p << (kSumBits * v);
    for (int s = 2 * kSumBits * v; s < 11 * kSumBits; s *= 2) p += p << s;
    return p;
}

// moves of hand card c (numeric: sets = pool_sets(pool))
__device__ __forceinline__ int card_moves(int c, uint64_t pool, Poly sets) {
    if (c < 40) return max(sets_of(sets, 10 - c / 4), 1);
    if (c < 44) return 1;
    return max(__popcll(pool & (c < 48 ? kQueens : kKings)), 1);
}

__device__ __forceinline__ int degree_of(uint64_t hand, uint64_t pool) {
    const Poly sets = pool_sets(pool);
    int n = 0;
    for (; hand; hand &= hand - 1) n += card_moves(__ffsll((long long)hand) - 1, pool, sets);
    return n;
}

// the picked set of move r of card c, moves in ascending order of their sets
__device__ __forceinline__ uint64_t picked_set(int c, int r, uint64_t pool, Poly sets) {
    if (c < 40) {
        int sum = 10 - c / 4;
        uint64_t pick = 0, left = pool & kNumeric;
        if (sets_of(sets, sum) == 0) return 0;
        while (sum > 0) {
            // sets without the highest card come first
            const int b = 63 - __clzll((long long)left), v = b / 4 + 1;
            left &= ~(1ULL << b);
            sets = without_card(sets, v);
            const int w = sets_of(sets, sum);
            if (r >= w) {
                r -= w;
                sum -= v;
                pick |= 1ULL << b;
            }
        }
        return pick;
    }
    if (c < 44) return pool & (kNumeric | kJacks);
    uint64_t same = pool & (c < 48 ? kQueens : kKings);
    for (int i = 0; i < r; i++) same &= same - 1;
    return same & (~same + 1);
}

// ---- one move (CodeSnippet "ApplyActions" + the running-score update) -----------------------
__device__ __forceinline__ GTState apply_move(GTState s, int mover, int c, uint64_t pick, bool final_round) {
    uint64_t bit = 1ULL << c;
    s.hand[mover] &= ~bit;
    if (pick == 0) {
        s.pool |= bit;
    } else {
        s.pool &= ~pick;
        uint64_t cap = pick | bit;
        s.rus = rus_add(s.rus, mover, set_clubs(cap));
        s.rus = rus_add(s.rus, 3 + 2 * mover, set_points(cap));
        s.rus = rus_set(s.rus, 2, mover + 1);
        bool jack = c >= 40 && c < 44;
        if (s.pool == 0 && !jack && !final_round) s.rus = rus_add(s.rus, 4 + 2 * mover, 1);
    }
    return s;
}

struct EmitOut {
    GTState *st;
    int8_t *lay;
    uint64_t *pick;
    int32_t *root;
};

__global__ void k_degrees(const GTState *__restrict__ st, int64_t m, int mover, int32_t *__restrict__ deg) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x)
        deg[j] = degree_of(st[j].hand[mover], st[j].pool);
}

__global__ void k_parents(const int64_t *__restrict__ child_off, int64_t m, int64_t *__restrict__ parent) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = child_off[j + 1];
        for (int64_t c = child_off[j]; c < e; c++) parent[c] = j;
    }
}

// the children of a level: child i is move i - child_off[parent[i]] of its parent, moves ordered by
// (card, picked set); deg (NULL at the last level): the children's own degrees
__global__ void __launch_bounds__(256) k_children(const GTState *__restrict__ st, const int32_t *__restrict__ root_in,
                                                  const int64_t *__restrict__ child_off, const int64_t *__restrict__ parent,
                                                  int64_t m, int mover, bool final_round, EmitOut o, int32_t *__restrict__ deg) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = parent[i];
        int r = (int)(i - child_off[j]);
        GTState s = st[j];
        const Poly sets = pool_sets(s.pool);
        int c = 0;
        for (uint64_t hand = s.hand[mover]; hand; hand &= hand - 1) {
            c = __ffsll((long long)hand) - 1;
            const int n = card_moves(c, s.pool, sets);
            if (r < n) break;
            r -= n;
        }
        const uint64_t pick = picked_set(c, r, s.pool, sets);
        s = apply_move(s, mover, c, pick, final_round);
        o.st[i] = s;
        o.lay[i] = (int8_t)c;
        o.pick[i] = pick;
        o.root[i] = root_in[j];
        if (deg) deg[i] = degree_of(s.hand[mover ^ 1], s.pool);
    }
}

__global__ void k_init_roots(const uint64_t *__restrict__ pools, int64_t n, uint64_t ha, uint64_t hb,
                             GTState *__restrict__ st, int32_t *__restrict__ root) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        GTState s;
        s.hand[0] = ha;
        s.hand[1] = hb;
        s.pool = pools[i];
        s.rus = 0;
        st[i] = s;
        root[i] = (int32_t)i;
    }
}

// first GT node of every root at every level: begin(g, 0) = g, begin(g, k+1) = child_off_k[begin(g, k)]
struct OffPtrs {
    const int64_t *p[9];
};
__global__ void k_root_bounds(int64_t n_roots, OffPtrs co, int64_t *__restrict__ out) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g <= n_roots; g += (int64_t)gridDim.x * blockDim.x) {
        int64_t b = g;
        out[g * 9] = b;
        for (int k = 0; k < 8; k++) {
            b = co.p[k][b];
            out[g * 9 + k + 1] = b;
        }
    }
}

// First FGT node of every GT node of all levels (one launch; nine of them were a quarter of a small round's
// unfolding): a root's nodes are consecutive, each with the root's slots (base: per level the roots' first,
// bounds[9 g + k]: the root's first GT node); the element after a level's last = its total.
struct SlotLevels {
    const int32_t *root[9];
    int64_t *out[9];
    int64_t off[10];  // first element of the level, M + 1 each
};

__global__ void k_slot_offsets(const SlotLevels L, const int64_t *__restrict__ bounds, const int64_t *__restrict__ bases,
                               const int64_t *__restrict__ slot_off, int64_t n_roots) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < L.off[9]; i += (int64_t)gridDim.x * blockDim.x) {
        int k = 0;
        while (i >= L.off[k + 1]) k++;
        const int64_t j = i - L.off[k], *base = bases + k * (n_roots + 1);
        if (i == L.off[k + 1] - 1) {
            L.out[k][j] = base[n_roots];
            continue;
        }
        const int32_t g = L.root[k][j];
        L.out[k][j] = base[g] + (j - bounds[9 * g + k]) * (slot_off[g + 1] - slot_off[g]);
    }
}

// leaf values (eq. final_util and eq. passuputil) of the solved slots: solved slot x of leaf j
// (root g) takes the score and the next-round link of its representative full slot crep; out in
// solved FGT order (cfgt_off); umax receives max |value| as float bits
__global__ void k_leaf_values(const GTState *__restrict__ st, const int32_t *__restrict__ root, int64_t m,
                              const int64_t *__restrict__ fgt_off, const int64_t *__restrict__ cfgt_off,
                              const int64_t *__restrict__ csoff, const int32_t *__restrict__ crep,
                              const int64_t *__restrict__ score_off, const pasur_score *__restrict__ scores,
                              bool final_round, const int64_t *__restrict__ lnk, const float *__restrict__ next_util,
                              float *__restrict__ out, unsigned *__restrict__ umax_bits) {
    float local_max = 0.f;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        GTState s = st[j];
        int32_t g = root[j];
        const int64_t q0 = fgt_off[j], c0 = cfgt_off[j], ns = cfgt_off[j + 1] - c0;
        const int32_t *rep = crep + csoff[g];
        if (final_round) {
            uint64_t r = cleanup_rus(s.rus, s.pool);
            int d = rus_diff(r);
            for (int64_t x = 0; x < ns; x++) {
                pasur_score sc = scores[score_off[g] + rep[x]];
                float v = (float)(d + bonus_points(bonus_after(sc.a_clubs, sc.b_clubs, sc.bonus, r)));
                out[c0 + x] = v;
                local_max = fmaxf(local_max, fabsf(v));
            }
        } else {
            int d = rus_diff(s.rus);
            for (int64_t x = 0; x < ns; x++) {
                float v = (float)d + next_util[lnk[q0 + rep[x]]];
                out[c0 + x] = v;
                local_max = fmaxf(local_max, fabsf(v));
            }
        }
    }
    if (!(local_max <= 3.0e38f)) local_max = __int_as_float(0x7f800000);  // non-finite -> +inf
    if (umax_bits) atomicMax(umax_bits, __float_as_uint(local_max));
}

// Every full slot of a non-final round's leaves must see the same next-round utility as the
// representative of its solved slot; flag a leaf where it does not (bitwise comparison).
__global__ void k_check_merge(const int32_t *__restrict__ root, int64_t m, const int64_t *__restrict__ fgt_off,
                              const int64_t *__restrict__ score_off, const int64_t *__restrict__ csoff,
                              const int32_t *__restrict__ crep, const int64_t *__restrict__ cidx0,
                              const int64_t *__restrict__ lnk, const float *__restrict__ next_util, int32_t *bad) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t g = root[j];
        const int64_t q0 = fgt_off[j], ns = fgt_off[j + 1] - q0, s0 = score_off[g];
        for (int64_t s = 0; s < ns; s++) {
            const int32_t r = crep[cidx0[s0 + s]];
            if (r != s && __float_as_uint(next_util[lnk[q0 + s]]) != __float_as_uint(next_util[lnk[q0 + r]])) {
                atomicOr(bad, 1);
                break;
            }
        }
    }
}

// full leaf values from the solved ones: leaf (j, s) takes the value of its solved slot
__global__ void k_expand_leaves(const int32_t *__restrict__ root, int64_t m, const int64_t *__restrict__ fgt_off,
                                const int64_t *__restrict__ cfgt_off, const int64_t *__restrict__ score_off,
                                const int64_t *__restrict__ csoff, const int64_t *__restrict__ cidx0,
                                const float *__restrict__ in, float *__restrict__ out) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t g = root[j];
        const int64_t q0 = fgt_off[j], ns = fgt_off[j + 1] - q0, c0 = cfgt_off[j] - csoff[g];
        for (int64_t s = 0; s < ns; s++) out[q0 + s] = in[c0 + cidx0[score_off[g] + s]];
    }
}

unsigned grid_for(int64_t threads, int block) {
    int64_t b = (threads + block - 1) / block;
    if (b < 1) b = 1;
    if (b > (1 << 20)) b = 1 << 20;
    return (unsigned)b;
}

}  // namespace

int build_levels(pasur_tree *t, const uint64_t *root_pools_dev) {
    pasur_ctx *ctx = t->ctx;
    int64_t m0 = t->n_roots;
    t->M[0] = m0;
    PASUR_TRY(tree_alloc(t, (void **)&t->st[0], sizeof(GTState) * (size_t)(m0 + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->root[0], sizeof(int32_t) * (size_t)(m0 + 1)));
    if (m0 > 0) {
        k_init_roots<<<grid_for(m0, 256), 256, 0, ctx->stream>>>(root_pools_dev, m0, t->hand_a, t->hand_b, t->st[0], t->root[0]);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
    }
    // degrees of the level being expanded: counted where its nodes are written
    int32_t *deg = nullptr;
    size_t degb = sizeof(int32_t) * (size_t)(m0 + 1);
    PASUR_TRY(dev_alloc(ctx, (void **)&deg, degb));
    struct Deg {
        pasur_ctx *c;
        int32_t **p;
        size_t *b;
        ~Deg() { dev_free(c, *p, *b); }
    } guard{ctx, &deg, &degb};
    if (m0 > 0) {
        k_degrees<<<grid_for(m0, 256), 256, 0, ctx->stream>>>(t->st[0], m0, 0, deg);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
    }
    for (int k = 0; k < 8; k++) {
        int64_t m = t->M[k];
        PASUR_TRY(tree_alloc(t, (void **)&t->child_off[k], sizeof(int64_t) * (size_t)(m + 1)));
        PASUR_TRY(exclusive_scan_i32(ctx, deg, t->child_off[k], m));
        dev_free(ctx, deg, degb);  // stream-ordered, before the next level's arrays are taken
        deg = nullptr;
        int64_t m1 = 0;
        PASUR_TRY(read_i64(ctx, t->child_off[k] + m, &m1));
        t->M[k + 1] = m1;
        // the level's five arrays in one allocation, each piece 256-byte aligned
        const size_t cap = (size_t)m1 + 1;
        auto piece = [](size_t b) { return (b + 255) & ~(size_t)255; };
        const size_t b_st = piece(sizeof(GTState) * cap), b_par = piece(sizeof(int64_t) * cap),
                     b_lay = piece(sizeof(int8_t) * cap), b_pick = piece(sizeof(uint64_t) * cap);
        char *lv = nullptr;
        PASUR_TRY(tree_alloc(t, (void **)&lv, b_st + b_par + b_lay + b_pick + piece(sizeof(int32_t) * cap)));
        t->st[k + 1] = (GTState *)lv;
        t->parent[k + 1] = (int64_t *)(lv + b_st);
        t->lay[k + 1] = (int8_t *)(lv + b_st + b_par);
        t->pick[k + 1] = (uint64_t *)(lv + b_st + b_par + b_lay);
        t->root[k + 1] = (int32_t *)(lv + b_st + b_par + b_lay + b_pick);
        if (k < 7) {
            degb = sizeof(int32_t) * cap;
            PASUR_TRY(dev_alloc(ctx, (void **)&deg, degb));
        }
        if (m > 0) {
            EmitOut o{t->st[k + 1], t->lay[k + 1], t->pick[k + 1], t->root[k + 1]};
            k_parents<<<grid_for(m, 256), 256, 0, ctx->stream>>>(t->child_off[k], m, t->parent[k + 1]);
            ctx->launches++;
            PASUR_CUDA(ctx, cudaGetLastError());
            k_children<<<grid_for(m1, 256), 256, 0, ctx->stream>>>(t->st[k], t->root[k], t->child_off[k], t->parent[k + 1], m1,
                                                                  k & 1, t->final_round, o, deg);
            ctx->launches++;
            PASUR_CUDA(ctx, cudaGetLastError());
        }
    }
    // per-root level bounds -> RootInfo (host + device)
    int64_t nr = t->n_roots;
    size_t bb = sizeof(int64_t) * 9 * (size_t)(nr + 1);
    PASUR_TRY(tree_alloc(t, (void **)&t->bounds_d, bb));
    int64_t *bounds = t->bounds_d;
    OffPtrs co;
    for (int k = 0; k < 8; k++) co.p[k] = t->child_off[k];
    co.p[8] = nullptr;
    k_root_bounds<<<grid_for(nr + 1, 256), 256, 0, ctx->stream>>>(nr, co, bounds);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    std::vector<int64_t> hb(9 * (size_t)(nr + 1));
    PASUR_CUDA(ctx, cudaMemcpyAsync(hb.data(), bounds, bb, cudaMemcpyDeviceToHost, ctx->stream));
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    t->roots_h.assign((size_t)nr, RootInfo{});
    for (int64_t g = 0; g < nr; g++) {
        RootInfo &ri = t->roots_h[(size_t)g];
        int64_t local = 0;
        for (int k = 0; k < 9; k++) {
            int64_t cnt = hb[(size_t)(g + 1) * 9 + k] - hb[(size_t)g * 9 + k];
            if (local + cnt > INT32_MAX) return set_err(ctx, PASUR_EOVERFLOW, "a root subtree exceeds 2^31 nodes");
            ri.lvl_count[k] = (int32_t)cnt;
            local += cnt;
        }
    }
    return PASUR_OK;
}

// The FGT levels over given slots per root (slot_off: prefix over the roots, host and device): sizes
// from the roots' node counts on the host, then every level's offsets in one launch, without a scan or
// a synchronisation.
// base: filled here and read by the upload until the stream gets there, so it belongs to the tree.
static int slot_levels(pasur_tree *t, const std::vector<int64_t> &slot_off, const int64_t *slot_off_d, std::vector<int64_t> &base,
                       int64_t **off, int64_t *sizes) {
    pasur_ctx *ctx = t->ctx;
    const int64_t nr = t->n_roots;
    base.assign((size_t)(9 * (nr + 1)), 0);
    for (int k = 0; k < 9; k++) {
        int64_t *b = base.data() + (size_t)k * (size_t)(nr + 1), q = 0;
        for (int64_t g = 0; g < nr; g++) {
            b[g] = q;
            q += t->roots_h[(size_t)g].lvl_count[k] * (slot_off[(size_t)g + 1] - slot_off[(size_t)g]);
        }
        b[nr] = sizes[k] = q;
    }
    int64_t *base_d = nullptr;
    const size_t bytes = sizeof(int64_t) * base.size();
    PASUR_TRY(dev_alloc(ctx, (void **)&base_d, bytes));
    int rc = PASUR_OK;
    cudaError_t e = cudaMemcpyAsync(base_d, base.data(), bytes, cudaMemcpyHostToDevice, ctx->stream);
    if (e != cudaSuccess) rc = cuda_err(ctx, e, "slot_levels: upload");
    SlotLevels L{};
    for (int k = 0; k < 9 && rc == PASUR_OK; k++) {
        if (!off[k]) rc = tree_alloc(t, (void **)&off[k], sizeof(int64_t) * (size_t)(t->M[k] + 1));
        L.root[k] = t->root[k];
        L.out[k] = off[k];
        L.off[k + 1] = L.off[k] + t->M[k] + 1;
    }
    if (rc == PASUR_OK) {
        k_slot_offsets<<<grid_for(L.off[9], 256), 256, 0, ctx->stream>>>(L, t->bounds_d, base_d, slot_off_d, nr);
        ctx->launches++;
        e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_err(ctx, e, "k_slot_offsets");
    }
    dev_free(ctx, base_d, bytes);
    return rc;
}

int unfold_levels(pasur_tree *t) { return slot_levels(t, t->score_off_h, t->score_off_d, t->lvl_base_h, t->fgt_off, t->Q); }

// leaf values without any host synchronisation (the batch solver captures this in a CUDA graph);
// umax_bits (device, may be NULL) receives max |value| as float bits
int launch_leaf_values(pasur_tree *t, const float *next_util_dev, unsigned *umax_bits) {
    pasur_ctx *ctx = t->ctx;
    if (t->M[8] == 0) return PASUR_OK;
    k_leaf_values<<<grid_for(t->M[8], 256), 256, 0, ctx->stream>>>(t->st[8], t->root[8], t->M[8], t->fgt_off[8],
                                                                  t->cfgt_off[8], t->csoff_d, t->crep_d, t->score_off_d,
                                                                  t->scores_d, t->final_round, t->lnk_d, next_util_dev,
                                                                  t->leaf_v, umax_bits);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    return PASUR_OK;
}

int compute_leaf_values(pasur_tree *t, const float *next_util_dev) {
    pasur_ctx *ctx = t->ctx;
    int64_t q8 = t->cQ[8];
    if (!t->leaf_v) PASUR_TRY(tree_alloc(t, (void **)&t->leaf_v, sizeof(float) * (size_t)(q8 + 1)));
    unsigned *umax = nullptr;
    PASUR_TRY(dev_alloc(ctx, (void **)&umax, sizeof(unsigned)));
    PASUR_CUDA(ctx, cudaMemsetAsync(umax, 0, sizeof(unsigned), ctx->stream));
    if (t->M[8] > 0) {
        k_leaf_values<<<grid_for(t->M[8], 256), 256, 0, ctx->stream>>>(
            t->st[8], t->root[8], t->M[8], t->fgt_off[8], t->cfgt_off[8], t->csoff_d, t->crep_d, t->score_off_d,
            t->scores_d, t->final_round, t->lnk_d, next_util_dev, t->leaf_v, umax);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
    }
    unsigned hb = 0;
    PASUR_CUDA(ctx, cudaMemcpyAsync(&hb, umax, sizeof(unsigned), cudaMemcpyDeviceToHost, ctx->stream));
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    dev_free(ctx, umax, sizeof(unsigned));
    float u;
    memcpy(&u, &hb, sizeof u);
    if (!(u <= 3.0e38f)) return set_err(ctx, PASUR_ENUMERIC, "non-finite leaf value");
    t->umax = u;
    return PASUR_OK;
}

int plan_solve_slots(pasur_tree *t, bool merge, const float *next_util_dev) {
    pasur_ctx *ctx = t->ctx;
    if (t->csoff_d) return PASUR_OK;
    const int64_t nr = t->n_roots, q0 = t->Q[0];
    // group the slots of every root by (a_clubs, b_clubs, bonus), numbered by first appearance
    std::vector<int64_t> csoff((size_t)nr + 1, 0), cidx0((size_t)q0 + 1, 0);
    std::vector<int32_t> crep;
    crep.reserve((size_t)q0 + 1);
    bool any = false;
    for (int64_t g = 0; g < nr; g++) {
        const int64_t a = t->score_off_h[(size_t)g], b = t->score_off_h[(size_t)g + 1];
        const int64_t base = (int64_t)crep.size();
        std::vector<std::pair<uint32_t, int32_t>> seen;  // key -> solved slot within the root
        for (int64_t s = a; s < b; s++) {
            const pasur_score &x = t->scores_h[(size_t)s];
            const uint32_t key = merge ? ((uint32_t)x.a_clubs << 8) | ((uint32_t)x.b_clubs << 2) | (uint32_t)x.bonus
                                       : (uint32_t)(s - a);
            int32_t c = -1;
            for (const auto &k : seen)
                if (k.first == key) c = k.second;
            if (c < 0) {
                c = (int32_t)seen.size();
                seen.push_back({key, c});
                crep.push_back((int32_t)(s - a));
            } else {
                any = true;
            }
            cidx0[(size_t)s] = base + c;
        }
        csoff[(size_t)g + 1] = (int64_t)crep.size();
    }
    const int64_t cq0 = (int64_t)crep.size();
    PASUR_TRY(tree_alloc(t, (void **)&t->csoff_d, sizeof(int64_t) * (size_t)(nr + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->crep_d, sizeof(int32_t) * (size_t)(cq0 + 1)));
    PASUR_TRY(tree_alloc(t, (void **)&t->cidx0_d, sizeof(int64_t) * (size_t)(q0 + 1)));
    PASUR_CUDA(ctx, cudaMemcpyAsync(t->csoff_d, csoff.data(), sizeof(int64_t) * (size_t)(nr + 1), cudaMemcpyHostToDevice, ctx->stream));
    if (cq0) PASUR_CUDA(ctx, cudaMemcpyAsync(t->crep_d, crep.data(), sizeof(int32_t) * (size_t)cq0, cudaMemcpyHostToDevice, ctx->stream));
    if (q0) PASUR_CUDA(ctx, cudaMemcpyAsync(t->cidx0_d, cidx0.data(), sizeof(int64_t) * (size_t)q0, cudaMemcpyHostToDevice, ctx->stream));
    // a non-final round merges only slots whose leaves see the same next-round utilities
    if (any && !t->final_round && next_util_dev && t->M[8] > 0) {
        int32_t *bad = nullptr;
        PASUR_TRY(dev_alloc(ctx, (void **)&bad, sizeof(int32_t)));
        PASUR_CUDA(ctx, cudaMemsetAsync(bad, 0, sizeof(int32_t), ctx->stream));
        k_check_merge<<<grid_for(t->M[8], 256), 256, 0, ctx->stream>>>(t->root[8], t->M[8], t->fgt_off[8], t->score_off_d,
                                                                      t->csoff_d, t->crep_d, t->cidx0_d, t->lnk_d,
                                                                      next_util_dev, bad);
        ctx->launches++;
        int32_t hb = 0;
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&hb, bad, sizeof hb, cudaMemcpyDeviceToHost, ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
        dev_free(ctx, bad, sizeof(int32_t));
        if (e != cudaSuccess) return cuda_err(ctx, e, "k_check_merge");
        if (hb) {
            // the given utilities differ between slots that differ only in delta: solve every slot
            PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
            for (int64_t g = 0; g <= nr; g++) csoff[(size_t)g] = t->score_off_h[(size_t)g];
            crep.resize((size_t)q0);
            for (int64_t g = 0; g < nr; g++)
                for (int64_t s = t->score_off_h[(size_t)g]; s < t->score_off_h[(size_t)g + 1]; s++) {
                    crep[(size_t)s] = (int32_t)(s - t->score_off_h[(size_t)g]);
                    cidx0[(size_t)s] = s;
                }
            any = false;
            PASUR_TRY(tree_alloc(t, (void **)&t->crep_d, sizeof(int32_t) * (size_t)(q0 + 1)));
            PASUR_CUDA(ctx, cudaMemcpyAsync(t->csoff_d, csoff.data(), sizeof(int64_t) * (size_t)(nr + 1), cudaMemcpyHostToDevice, ctx->stream));
            if (q0) {
                PASUR_CUDA(ctx, cudaMemcpyAsync(t->crep_d, crep.data(), sizeof(int32_t) * (size_t)q0, cudaMemcpyHostToDevice, ctx->stream));
                PASUR_CUDA(ctx, cudaMemcpyAsync(t->cidx0_d, cidx0.data(), sizeof(int64_t) * (size_t)q0, cudaMemcpyHostToDevice, ctx->stream));
            }
        }
    }
    t->merged = any;
    t->csoff_h = csoff;
    {
        // full slots per solved slot (the weight of a solved slot in averages over the FGT)
        std::vector<int32_t> mult((size_t)csoff[(size_t)nr] + 1, 0);
        for (int64_t q = 0; q < q0; q++) mult[(size_t)cidx0[(size_t)q]]++;
        PASUR_TRY(tree_alloc(t, (void **)&t->cmult_d, sizeof(int32_t) * mult.size()));
        PASUR_CUDA(ctx, cudaMemcpyAsync(t->cmult_d, mult.data(), sizeof(int32_t) * mult.size(), cudaMemcpyHostToDevice,
                                        ctx->stream));
        PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    }
    if (!any) {
        for (int k = 0; k < 9; k++) {
            t->cfgt_off[k] = t->fgt_off[k];
            t->cQ[k] = t->Q[k];
        }
    } else {
        for (int k = 0; k < 9; k++) t->cfgt_off[k] = nullptr;
        PASUR_TRY(slot_levels(t, t->csoff_h, t->csoff_d, t->clvl_base_h, t->cfgt_off, t->cQ));
    }
    return PASUR_OK;
}

int expand_leaf_values(const pasur_tree *t, float *out_dev) {
    pasur_ctx *ctx = t->ctx;
    if (t->M[8] == 0) return PASUR_OK;
    if (!t->merged) {
        PASUR_CUDA(ctx, cudaMemcpyAsync(out_dev, t->leaf_v, sizeof(float) * (size_t)t->Q[8], cudaMemcpyDeviceToDevice, ctx->stream));
        return PASUR_OK;
    }
    k_expand_leaves<<<grid_for(t->M[8], 256), 256, 0, ctx->stream>>>(t->root[8], t->M[8], t->fgt_off[8], t->cfgt_off[8],
                                                                    t->score_off_d, t->csoff_d, t->cidx0_d, t->leaf_v, out_dev);
    ctx->launches++;
    PASUR_CUDA(ctx, cudaGetLastError());
    return PASUR_OK;
}

}  // namespace pasur
