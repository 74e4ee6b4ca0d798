// Checkpoint and resume of a round's CFR state.  The paper keeps every round's tensors in host
// memory between the rounds of a deal and stores the solved strategy profiles (section
// "Experimental Evaluation"); here a round can also stop and resume mid-run: its regrets R,
// strategy sums S, root-value sums and iteration count go to a host buffer and back.  A header of
// sizes and an order-independent hash of the round's leaf values make a checkpoint refuse a tree
// that was built, unfolded or given next-round utilities differently.
//
// R and S are written as they are stored.  A root split over a cluster is stored by its own nodes, slot by slot
// (mark PSRCKPT2); it used to be stored by its top and parts (mark PSRCKPT1, also written for a while with the
// present storage), and FormerStorage puts such checkpoints into the present places.
#include <cstring>
#include <memory>
#include <new>

#include "cfr_split.cuh"
#include "pasur_internal.cuh"

namespace pasur {
namespace {

constexpr uint64_t kCkptFormer = 0x3154504B43525350ull;  // "PSRCKPT1", little-endian
constexpr uint64_t kCkptMagic = 0x3254504B43525350ull;   // "PSRCKPT2"

struct CkptHeader {
    uint64_t magic;
    int32_t round, variant;
    int64_t n_roots, iters_done, data_size, n_uacc, n_leaves;
    int64_t cQ[9];
    int64_t swept_edges, swept_pairs;
    uint64_t leaf_hash;
};

// sum over i of (w[i] + 1) * (2 i + 1) mod 2^64: changes with any word or its position, and is
// independent of the order in which the terms are added
__global__ void k_word_hash(const uint32_t *__restrict__ w, int64_t n, unsigned long long *out) {
    unsigned long long acc = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        acc += ((unsigned long long)w[i] + 1ull) * (2ull * (unsigned long long)i + 1ull);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

int leaf_hash(const pasur_tree *t, uint64_t *h) {
    pasur_ctx *ctx = t->ctx;
    unsigned long long *d = nullptr;
    PASUR_TRY(dev_alloc(ctx, (void **)&d, sizeof(unsigned long long)));
    int rc = PASUR_OK;
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof(unsigned long long), ctx->stream);
    const int64_t n = t->cQ[8];
    if (e == cudaSuccess && n > 0) {
        const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)ctx->num_sms * 8);
        k_word_hash<<<(unsigned)blocks, 256, 0, ctx->stream>>>((const uint32_t *)t->leaf_v, n, d);
        ctx->launches++;
        e = cudaGetLastError();
    }
    unsigned long long v = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&v, d, sizeof v, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) rc = cuda_err(ctx, e, "checkpoint: leaf hash");
    dev_free(ctx, d, sizeof(unsigned long long));
    *h = v;
    return rc;
}

int make_header(const pasur_tree *t, CkptHeader *hd) {
    std::memset(hd, 0, sizeof *hd);
    hd->magic = kCkptMagic;
    hd->round = t->round;
    hd->variant = t->variant;
    hd->n_roots = t->n_roots;
    hd->iters_done = t->iters_done;
    hd->data_size = t->data_size;
    hd->n_uacc = t->cQ[0];
    hd->n_leaves = t->cQ[8];
    for (int k = 0; k < 9; k++) hd->cQ[k] = t->cQ[k];
    hd->swept_edges = t->swept_edges;
    hd->swept_pairs = t->swept_pairs;
    return leaf_hash(t, &hd->leaf_hash);
}

int tree_ok(const pasur_tree *t) { return t && t->ctx ? PASUR_OK : PASUR_EINVAL; }

size_t ckpt_bytes(const CkptHeader &hd) {
    return sizeof(CkptHeader) + 2 * sizeof(float) * (size_t)hd.data_size + sizeof(double) * (size_t)hd.n_uacc;
}

// How R and S were stored when split roots lay part by part: a root split then (16 bytes per (node, slot), one slot
// per cluster of up to 16 CTAs) holds for every slot its top (levels <= ell) and, part by part, the nodes below its
// active level-ell nodes level by level and a place for each of these nodes' parents' reach.  Other roots were stored
// as now, except that one split only now was stored in wider items.
struct FormerStorage {
    static constexpr size_t kReserve = 576;  // part of a block's shared memory its cluster kernels left free
    struct Root {
        int64_t base = 0;                    // its first word
        int64_t width = 1, words = 0;        // slots per item; words per slot of a split root
        std::vector<int32_t> at;             // split: place of every local node in a slot's words
    };
    std::vector<Root> roots;
    int64_t size = 0;
    bool as_now = true;                      // every word lies where it does now

    int plan(const pasur_tree *t) {
        pasur_ctx *ctx = t->ctx;
        const pasur_config &cfg = t->layout_cfg;
        const Storage storage(ctx->smem_optin, cfg.slots_per_item);
        const size_t limit = std::min(storage.most(), ctx->smem_optin > kReserve ? ctx->smem_optin - kReserve : 0);
        const size_t nr = (size_t)t->n_roots, NA = (size_t)t->n_active;
        roots.assign(nr, Root());
        std::vector<char> work(nr, 0), streamed(nr, 0), split(nr, 0);
        bool any = false;
        for (size_t g = 0; g < nr; g++) {
            const CfrRoot &cr = t->croots_h[g];
            const int64_t slots = t->csoff_h[g + 1] - t->csoff_h[g], L = cr.ls[9], nA = cr.as[9];
            if (slots == 0 || L == 0 || !t->in_range((int64_t)g)) continue;
            const size_t need = resident_bytes(L, nA, 1);
            work[g] = 1;
            streamed[g] = (cfg.stream_bytes > 0 && need > (size_t)cfg.stream_bytes) || (need > storage.most() && slots >= kStreamMinSlots);
            split[g] = nA >= 2 && !streamed[g] && (need > storage.most() || (cfg.split_bytes > 0 && need > (size_t)cfg.split_bytes));
            any |= split[g] != 0;
        }
        std::vector<int32_t> li, cs;
        std::vector<uint16_t> dd;
        if (any) {
            li.resize(NA);
            cs.resize(NA);
            dd.resize(NA);
            PASUR_CUDA(ctx, cudaMemcpy(li.data(), t->act_li, sizeof(int32_t) * NA, cudaMemcpyDeviceToHost));
            PASUR_CUDA(ctx, cudaMemcpy(cs.data(), t->act_cs, sizeof(int32_t) * NA, cudaMemcpyDeviceToHost));
            PASUR_CUDA(ctx, cudaMemcpy(dd.data(), t->act_d, sizeof(uint16_t) * NA, cudaMemcpyDeviceToHost));
        }
        const bool ok = on_threads(nr, [&](size_t g) {
            const CfrRoot &cr = t->croots_h[g];
            if (split[g]) split_root(cr, cfg, limit, li.data() + cr.act_off, cs.data() + cr.act_off, dd.data() + cr.act_off, roots[g]);
        });
        if (!ok) return set_err(ctx, PASUR_ENOMEM, "pasur_load_round: host allocation failed");
        for (size_t g = 0; g < nr; g++) {
            if (!work[g]) continue;
            const CfrRoot &cr = t->croots_h[g];
            const int64_t slots = t->csoff_h[g + 1] - t->csoff_h[g], L = cr.ls[9];
            Root &r = roots[g];
            r.base = size;
            int cls = 0;
            if (r.words == 0) r.width = storage.width(L, cr.as[9], slots, streamed[g], &cls);
            as_now &= r.words == 0 && (r.width == cr.W || slots == 1);
            size += slots * (r.words ? r.words : L);
        }
        return PASUR_OK;
    }

    // the root's split: the places of its nodes (left out where none was found)
    static void split_root(const CfrRoot &cr, const pasur_config &cfg, size_t limit, const int32_t *li, const int32_t *cs,
                           const uint16_t *dd, Root &out) {
        const int64_t L = cr.ls[9];
        const size_t target = cfg.split_bytes > 0 ? std::min<size_t>((size_t)cfg.split_bytes, limit) : limit;
        auto bytes = [](int64_t l, int64_t a) { return resident_bytes(l, a, 1); };
        for (int ell = 1; ell <= 6; ell++) {
            if (cr.as[ell + 1] - cr.as[ell] < 2) continue;
            const size_t top = bytes(cr.ls[ell + 1], cr.as[ell]);
            if (top >= limit) return;
            LevelCut cut;
            cut.make(cr, ell, li, cs, dd);
            const int q0 = (int)std::min<size_t>(cfg.split_bytes > 0 ? kMaxClusterCtas : 8,
                                                 std::max<size_t>(2, (bytes(L, cr.as[9]) + target - 1) / target));
            const PartPacking<decltype(bytes)> packing{cut, bytes, limit, top};
            const int fewest = packing.fewest();
            std::vector<int> first;
            for (int Q = std::max(q0, fewest); fewest > 0 && Q <= kMaxClusterCtas; Q++) {
                if (!packing.balanced(Q, first)) continue;
                out.at.assign((size_t)L, 0);
                for (int32_t x = 0; x < cr.ls[ell + 1]; x++) out.at[(size_t)x] = x;
                int64_t n = cr.ls[ell + 1];
                for (size_t q = 0; q < first.size(); q++) {
                    const int32_t h0 = first[q], h1 = q + 1 < first.size() ? first[q + 1] : (int32_t)cut.heads.size();
                    n += h1 - h0;  // the heads themselves: their regrets are the top's
                    for (int64_t x = cr.ls[ell + 1]; x < L; x++)
                        if (cut.sub[(size_t)x] >= h0 && cut.sub[(size_t)x] < h1) out.at[(size_t)x] = (int32_t)n++;
                    n += h1 - h0;  // the parents' reaches
                }
                out.words = n;
                return;
            }
        }
    }

    // the words in their present places
    bool convert(const pasur_tree *t, const float *from, float *to) const {
        return on_threads(roots.size(), [&](size_t g) {
            const CfrRoot &cr = t->croots_h[g];
            const int64_t slots = t->csoff_h[g + 1] - t->csoff_h[g], L = cr.ls[9];
            const Root &r = roots[g];
            if (cr.cls < 0) return;
            for (int64_t s0 = 0, ns = r.width; s0 < slots; s0 += ns) {
                while (ns > slots - s0) ns /= 2;
                for (int64_t s = s0; s < s0 + ns; s++) {
                    float *dst = to + t->slot_base_h[(size_t)(t->csoff_h[g] + s)];
                    const int64_t str = t->slot_str_h[(size_t)(t->csoff_h[g] + s)];
                    if (r.words)
                        for (int64_t x = 0; x < L; x++) dst[x * str] = from[r.base + s * r.words + r.at[(size_t)x]];
                    else
                        for (int64_t x = 0; x < L; x++) dst[x * str] = from[r.base + s0 * L + x * ns + (s - s0)];
                }
            }
        });
    }
};

}  // namespace
}  // namespace pasur

using namespace pasur;

int pasur_save_round(const pasur_tree *t, void *buf, size_t cap, size_t *bytes) {
    if (tree_ok(t)) return PASUR_EINVAL;
    pasur_ctx *ctx = t->ctx;
    cudaSetDevice(ctx->device);
    if (!t->cfr_ready) return set_err(ctx, PASUR_EINVAL, "pasur_save_round: no CFR run yet");
    if (!buf && !bytes) return set_err(ctx, PASUR_EINVAL, "pasur_save_round: buf and bytes are NULL");
    CkptHeader hd;
    PASUR_TRY(make_header(t, &hd));
    const size_t need = ckpt_bytes(hd);
    if (bytes) *bytes = need;
    if (!buf) return PASUR_OK;
    if (cap < need) return set_err(ctx, PASUR_EINVAL, "pasur_save_round: cap < " + std::to_string(need) + " bytes");
    char *p = (char *)buf;
    std::memcpy(p, &hd, sizeof hd);
    p += sizeof hd;
    const size_t fb = sizeof(float) * (size_t)hd.data_size;
    PASUR_CUDA(ctx, cudaMemcpyAsync(p, t->R, fb, cudaMemcpyDeviceToHost, ctx->stream));
    PASUR_CUDA(ctx, cudaMemcpyAsync(p + fb, t->S, fb, cudaMemcpyDeviceToHost, ctx->stream));
    PASUR_CUDA(ctx, cudaMemcpyAsync(p + 2 * fb, t->uacc, sizeof(double) * (size_t)hd.n_uacc, cudaMemcpyDeviceToHost,
                                    ctx->stream));
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return PASUR_OK;
}

int pasur_load_round(pasur_tree *t, const void *buf, size_t bytes) {
    if (tree_ok(t)) return PASUR_EINVAL;
    pasur_ctx *ctx = t->ctx;
    cudaSetDevice(ctx->device);
    if (!t->cfr_ready) return set_err(ctx, PASUR_EINVAL, "pasur_load_round: set the tree up first (pasur_cfr_iterate, iters 0)");
    if (!buf || bytes < sizeof(CkptHeader)) return set_err(ctx, PASUR_EINVAL, "pasur_load_round: no checkpoint header");
    CkptHeader in;
    std::memcpy(&in, buf, sizeof in);
    CkptHeader mine;
    PASUR_TRY(make_header(t, &mine));
    if (in.magic != kCkptMagic && in.magic != kCkptFormer) return set_err(ctx, PASUR_EINVAL, "pasur_load_round: not a round checkpoint");
    if (in.data_size < 0 || in.n_uacc < 0 || bytes < ckpt_bytes(in)) return set_err(ctx, PASUR_EINVAL, "pasur_load_round: checkpoint truncated");
    bool same = in.round == mine.round && in.variant == mine.variant && in.n_roots == mine.n_roots &&
                in.n_uacc == mine.n_uacc && in.n_leaves == mine.n_leaves && in.swept_edges == mine.swept_edges && in.swept_pairs == mine.swept_pairs && in.leaf_hash == mine.leaf_hash;
    for (int k = 0; k < 9; k++) same = same && in.cQ[k] == mine.cQ[k];
    // a checkpoint of the former mark is of the former storage or of the present one; their sizes tell them apart, but
    // where no root was split that is stored in other places now (then it could be either)
    FormerStorage former;
    bool convert = false;
    if (same && in.magic == kCkptFormer) {
        try {
            PASUR_TRY(former.plan(t));
        } catch (const std::bad_alloc &) {
            return set_err(ctx, PASUR_ENOMEM, "pasur_load_round: host allocation failed");
        }
        convert = in.data_size == former.size && !former.as_now;
        same = convert ? former.size != mine.data_size : in.data_size == mine.data_size;
    } else {
        same = same && in.data_size == mine.data_size;
    }
    if (!same)
        return set_err(ctx, PASUR_EINVAL, "pasur_load_round: the checkpoint is of another round, layout, variant or leaf values");
    if (in.iters_done < 0) return set_err(ctx, PASUR_EINVAL, "pasur_load_round: bad iteration count");
    const char *p = (const char *)buf + sizeof in;
    const size_t fb = sizeof(float) * (size_t)in.data_size;
    const char *R = p, *S = p + fb;
    std::unique_ptr<float[]> now;
    if (convert) {
        const size_t n = (size_t)mine.data_size, m = (size_t)in.data_size;
        now.reset(new (std::nothrow) float[2 * n]());
        std::unique_ptr<float[]> was(new (std::nothrow) float[2 * m]);  // the buffer's words, aligned
        if (!now || !was) return set_err(ctx, PASUR_ENOMEM, "pasur_load_round: host allocation failed");
        std::memcpy(was.get(), p, 2 * fb);
        if (!former.convert(t, was.get(), now.get()) || !former.convert(t, was.get() + m, now.get() + n))
            return set_err(ctx, PASUR_ENOMEM, "pasur_load_round: host allocation failed");
        R = (const char *)now.get();
        S = (const char *)(now.get() + n);
    }
    const size_t mb = sizeof(float) * (size_t)mine.data_size;
    PASUR_CUDA(ctx, cudaMemcpyAsync(t->R, R, mb, cudaMemcpyHostToDevice, ctx->stream));
    PASUR_CUDA(ctx, cudaMemcpyAsync(t->S, S, mb, cudaMemcpyHostToDevice, ctx->stream));
    PASUR_CUDA(ctx, cudaMemcpyAsync(t->uacc, p + 2 * fb, sizeof(double) * (size_t)in.n_uacc, cudaMemcpyHostToDevice,
                                    ctx->stream));
    PASUR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    t->iters_done = in.iters_done;
    return PASUR_OK;
}
