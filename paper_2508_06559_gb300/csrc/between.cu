// Between-hand update (section "Between-Hand Updates", CodeSnippet "BetweenHands"): the next
// round's FGT roots and the link of every FGT leaf to its next root (t_lnk).
//
// The leaves of a round reach few distinct roots (3e8 FGT leaves, 1e5 roots on a wide deal), so the keys
// are made distinct by a hash table that stays in L2 and only the distinct ones are sorted: first the
// pools of the GT leaves, then (pool number, normalised next score) of the FGT leaves, which numbers the
// next FGT roots in canonical order (pool ascending, then score ascending).  Sorting every leaf's key by
// 8-bit digits instead moved 32 bytes per leaf and pass, 7 and 5 passes.
#include <algorithm>
#include <type_traits>

#include "pasur_internal.cuh"

namespace pasur {
namespace {

unsigned grid_for(int64_t threads, int block) {
    int64_t b = (threads + block - 1) / block;
    if (b < 1) b = 1;
    if (b > (1 << 20)) b = 1 << 20;
    return (unsigned)b;
}

// Open-addressing table of 64-bit keys (kEmpty: free), linear probing; its size is a power of two.
constexpr uint64_t kEmpty = ~0ULL;
constexpr int kMaxProbe = 128;

__device__ __forceinline__ uint32_t key_hash(uint64_t k) {  // the finaliser of SplitMix64
    k = (k ^ (k >> 30)) * 0xBF58476D1CE4E5B9ULL;
    k = (k ^ (k >> 27)) * 0x94D049BB133111EBULL;
    return (uint32_t)(k ^ (k >> 31));
}

// the slot of key, put in if it is new; *full set (and slot 0 returned) when no place is found near
__device__ __forceinline__ uint32_t table_slot(unsigned long long *__restrict__ tab, uint32_t mask, uint64_t key, int32_t *full) {
    uint32_t h = key_hash(key) & mask;
    for (int i = 0; i < kMaxProbe; i++) {
        unsigned long long x = tab[h];
        if (x == kEmpty) x = atomicCAS(&tab[h], (unsigned long long)kEmpty, (unsigned long long)key);
        if (x == kEmpty || x == key) return h;
        h = (h + 1) & mask;
    }
    atomicOr(full, 2);
    return 0;
}

__global__ void k_pool_slots(const GTState *__restrict__ st, int64_t m, unsigned long long *__restrict__ tab, uint32_t mask,
                             int64_t *__restrict__ slot, int32_t *__restrict__ flags) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x)
        slot[j] = table_slot(tab, mask, st[j].pool, flags);
}

// One FGT leaf per lane: LPL lanes share a GT leaf's slots.  Bound by the table's atomics and misses; keys found in
// the table only are sorted (with the counted moves of the tree build, a wide forward sweep went from 31.1 to 7.4 ms).
template <int LPL>
__global__ void k_root_slots(const GTState *__restrict__ st, const int32_t *__restrict__ root, int64_t m,
                             const int64_t *__restrict__ fgt_off, const int64_t *__restrict__ score_off,
                             const pasur_score *__restrict__ scores, const int64_t *__restrict__ pool_slot,
                             const int64_t *__restrict__ pool_rank, unsigned long long *__restrict__ tab, uint32_t mask,
                             int64_t *__restrict__ slot, int32_t *__restrict__ flags) {
    const int64_t step = (int64_t)gridDim.x * blockDim.x / LPL;
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / LPL; j < m; j += step) {
        const uint64_t rus = st[j].rus;
        const int32_t g = root[j];
        const int64_t q0 = fgt_off[j], ns = fgt_off[j + 1] - q0, s0 = score_off[g];
        const int d = rus_diff(rus);
        const uint64_t hi = (uint64_t)pool_rank[pool_slot[j]] << kScoreKeyBits;
        for (int64_t x = threadIdx.x % LPL; x < ns; x += LPL) {
            const pasur_score sc = scores[s0 + x];
            int ac = sc.a_clubs + rus_get(rus, 0), bc = sc.b_clubs + rus_get(rus, 1), bonus = sc.bonus;
            const int delta = sc.delta + d;
            normalize_score(ac, bc, bonus);
            if (delta < -32768 || delta > 32767 || ac > 15 || bc > 15) atomicOr(flags, 4);
            slot[q0 + x] = table_slot(tab, mask, hi | score_key(ac, bc, delta, bonus), flags);
        }
    }
}

// the table's keys and their slots, in any order; *n counts them
__global__ void k_table_keys(const unsigned long long *__restrict__ tab, int64_t size, uint64_t *__restrict__ keys,
                             int64_t *__restrict__ at, unsigned long long *__restrict__ n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < size; i += (int64_t)gridDim.x * blockDim.x) {
        if (tab[i] == kEmpty) continue;
        const unsigned long long x = atomicAdd(n, 1ULL);
        keys[x] = tab[i];
        at[x] = i;
    }
}

// rank[slot of the i-th key] = i
__global__ void k_slot_ranks(const int64_t *__restrict__ at, int64_t n, int64_t *__restrict__ rank) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) rank[at[i]] = i;
}

__global__ void k_ranks_of(int64_t *__restrict__ slot, int64_t n, const int64_t *__restrict__ rank) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) slot[i] = rank[slot[i]];
}

int bits_for(int64_t n) {
    int b = 0;
    while (((int64_t)1 << b) < n) b++;
    return b;
}

// A table filled by `insert` (which may find it too small), its distinct keys in ascending order (host)
// and the rank of every slot's key (device).
struct KeyTable {
    pasur_ctx *ctx;
    unsigned long long *tab = nullptr;
    int64_t size = 0, n = 0;
    uint64_t *keys = nullptr;
    int64_t *at = nullptr, *rank = nullptr;
    size_t cap = 0;
    std::vector<uint64_t> host;
    explicit KeyTable(pasur_ctx *c) : ctx(c) {}
    ~KeyTable() {
        release();
        dev_free(ctx, rank, sizeof(int64_t) * (size_t)size);
    }
    void release() {
        dev_free(ctx, tab, sizeof(unsigned long long) * (size_t)(size + 1));
        dev_free(ctx, keys, cap);
        dev_free(ctx, at, cap);
        tab = nullptr;
        keys = nullptr;
        at = nullptr;
    }
    // first: entries of the first attempt (a power of two); grown eightfold while too small for the
    // at most `most` keys
    template <typename Insert>
    int fill(int64_t first, int64_t most, int bits, const Insert &insert) {
        for (size = first;; size *= 8) {
            PASUR_TRY(dev_alloc(ctx, (void **)&tab, sizeof(unsigned long long) * (size_t)(size + 1)));
            PASUR_CUDA(ctx, cudaMemsetAsync(tab, 0xFF, sizeof(unsigned long long) * (size_t)size, ctx->stream));
            PASUR_CUDA(ctx, cudaMemsetAsync(tab + size, 0, sizeof(unsigned long long), ctx->stream));
            PASUR_CUDA(ctx, cudaMemsetAsync(ctx->errflag, 0, sizeof(int32_t), ctx->stream));
            PASUR_TRY(insert(tab, (uint32_t)(size - 1), ctx->errflag));
            cap = sizeof(uint64_t) * (size_t)(std::min(size, most) + 1);
            PASUR_TRY(dev_alloc(ctx, (void **)&keys, cap));
            PASUR_TRY(dev_alloc(ctx, (void **)&at, cap));
            k_table_keys<<<grid_for(size, 256), 256, 0, ctx->stream>>>(tab, size, keys, at, tab + size);
            ctx->launches++;
            PASUR_CUDA(ctx, cudaGetLastError());
            int32_t flags = 0;
            PASUR_CUDA(ctx, cudaMemcpyAsync(&flags, ctx->errflag, sizeof flags, cudaMemcpyDeviceToHost, ctx->stream));
            PASUR_TRY(read_i64(ctx, (const int64_t *)(tab + size), &n));
            if (flags & 4) return set_err(ctx, PASUR_EOVERFLOW, "a next-round score leaves the int16 range");
            if (!(flags & 2)) break;
            release();
            if (size >= (int64_t)1 << 31) return set_err(ctx, PASUR_EOVERFLOW, "too many next-round roots");
        }
        // the keys are read: the ranks take the table's place
        dev_free(ctx, tab, sizeof(unsigned long long) * (size_t)(size + 1));
        tab = nullptr;
        PASUR_TRY(radix_sort_pairs(ctx, keys, at, n, bits));
        PASUR_TRY(dev_alloc(ctx, (void **)&rank, sizeof(int64_t) * (size_t)size));
        host.resize((size_t)n);
        if (n > 0) {
            k_slot_ranks<<<grid_for(n, 256), 256, 0, ctx->stream>>>(at, n, rank);
            ctx->launches++;
            PASUR_CUDA(ctx, cudaGetLastError());
            PASUR_CUDA(ctx, cudaMemcpyAsync(host.data(), keys, sizeof(uint64_t) * (size_t)n, cudaMemcpyDeviceToHost, ctx->stream));
        }
        PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        release();
        return PASUR_OK;
    }
};

int64_t table_size(int64_t keys, int64_t largest) {
    int64_t n = 1 << 10;
    while (n < 2 * keys && n < largest) n *= 2;
    return n;
}

}  // namespace

int next_roots(pasur_tree *t, std::vector<uint64_t> &pools, std::vector<int64_t> &score_off,
               std::vector<pasur_score> &scores) {
    pasur_ctx *ctx = t->ctx;
    const int64_t m8 = t->M[8], q8 = t->Q[8];
    // 1. distinct pools of the GT leaves
    int64_t *pool_slot = nullptr;
    const size_t b8 = sizeof(int64_t) * (size_t)(m8 + 1);
    PASUR_TRY(dev_alloc(ctx, (void **)&pool_slot, b8));
    struct Guard {
        pasur_ctx *c;
        void *p;
        size_t b;
        ~Guard() { dev_free(c, p, b); }
    } guard{ctx, pool_slot, b8};
    KeyTable pt(ctx);
    PASUR_TRY(pt.fill(table_size(m8, 1 << 18), m8, 52, [&](unsigned long long *tab, uint32_t mask, int32_t *flags) -> int {
        if (m8 == 0) return PASUR_OK;
        k_pool_slots<<<grid_for(m8, 256), 256, 0, ctx->stream>>>(t->st[8], m8, tab, mask, pool_slot, flags);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        return PASUR_OK;
    }));
    const int64_t n_pools = pt.n;
    pools = pt.host;
    // 2. next FGT roots: the leaves' slots in the table, then their ranks, in the links
    if (!t->lnk_d) PASUR_TRY(tree_alloc(t, (void **)&t->lnk_d, sizeof(int64_t) * (size_t)(q8 + 1)));
    KeyTable rt(ctx);
    PASUR_TRY(rt.fill(table_size(q8, 1 << 20), q8, kScoreKeyBits + bits_for(n_pools + 1),
                      [&](unsigned long long *tab, uint32_t mask, int32_t *flags) -> int {
        if (m8 == 0) return PASUR_OK;
        // lanes per GT leaf: fewer than its slots, so that a lane's look-ups overlap: two from 2 slots on, eight from 64 (a wide
        // forward sweep: as many lanes as slots 7.4 ms, four throughout 7.06, two 6.85, one 7.14)
        const int64_t ns = q8 / m8;
        auto go = [&](auto lpl) {
            constexpr int LPL = decltype(lpl)::value;
            k_root_slots<LPL><<<grid_for(m8 * LPL, 256), 256, 0, ctx->stream>>>(t->st[8], t->root[8], m8, t->fgt_off[8], t->score_off_d,
                                                                             t->scores_d, pool_slot, pt.rank, tab, mask, t->lnk_d, flags);
        };
        if (ns >= 64) go(std::integral_constant<int, 8>());
        else if (ns >= 2) go(std::integral_constant<int, 2>());
        else go(std::integral_constant<int, 1>());
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
        return PASUR_OK;
    }));
    if (q8 > 0) {
        k_ranks_of<<<grid_for(q8, 256), 256, 0, ctx->stream>>>(t->lnk_d, q8, rt.rank);
        ctx->launches++;
        PASUR_CUDA(ctx, cudaGetLastError());
    }
    const int64_t n_roots = rt.n;
    const std::vector<uint64_t> &rk = rt.host;
    score_off.assign((size_t)n_pools + 1, 0);
    scores.resize((size_t)n_roots);
    for (int64_t r = 0; r < n_roots; r++) {
        int64_t p = (int64_t)(rk[(size_t)r] >> kScoreKeyBits);
        int ac, bc, delta, bonus;
        score_unkey((uint32_t)(rk[(size_t)r] & ((1ULL << kScoreKeyBits) - 1)), ac, bc, delta, bonus);
        scores[(size_t)r] = pasur_score{(int16_t)ac, (int16_t)bc, (int16_t)delta, (int16_t)bonus};
        score_off[(size_t)p + 1] = r + 1;
    }
    for (int64_t p = 1; p <= n_pools; p++) score_off[(size_t)p] = std::max(score_off[(size_t)p], score_off[(size_t)p - 1]);
    t->n_next_roots = n_roots;
    t->has_next = true;
    return PASUR_OK;
}

}  // namespace pasur
