// Host side of how a root's CFR state is stored and split: the storage classes, the cut of a root at a
// level and the packing of the subtrees below it into parts.  Shared by the solver's set-up and the
// checkpoints.
#pragma once

#include <algorithm>
#include <atomic>
#include <thread>
#include <vector>

#include "pasur_internal.cuh"

namespace pasur {

// classes by which R and S are stored in device memory (slots per stored item): budget of a block's
// shared memory at 16 bytes per (node, slot), then the streamed items.  A checkpoint holds R and S as
// they are stored, so the classes stay as they are whatever the sweep's own layout is.
constexpr int kNumCls = 6;
constexpr size_t kStorageReserve = 352;  // part of a block's shared memory the storage classes leave free
constexpr size_t kClsBudget[kNumCls - 1] = {37536, 54 * 1024, 74 * 1024, 112 * 1024, 0 /* opt-in max */};
constexpr int kClsGlobal = kNumCls - 1;
constexpr int kClsCluster = 6;  // roots split over clusters
constexpr int kMaxSlots = 32;   // score slots per stored item
// a root too large for one block is streamed (class 5) rather than split over a cluster when it
// has at least this many score slots
constexpr int64_t kStreamMinSlots = 16;

inline size_t al16(size_t x) { return (x + 15) & ~(size_t)15; }

// shared memory of a resident item as the storage classes count it: packed active entries (8 B each) and R, S, V, X
// per (local node, slot); resident items must have fewer than 65535 local nodes
inline size_t resident_bytes(int64_t L, int64_t nA, int64_t W) {
    return L >= 65535 ? ~(size_t)0 >> 1 : 2 * al16((size_t)nA * 4) + 4 * al16((size_t)L * W * 4);
}

// Slots per stored item, a power of two (the streaming sweep indexes slots with shifts), and the class.
// Automatic: the smallest class the root fits with one slot, then the largest count that class holds.
// With slots_per_item: that many slots (at most the root's), in the smallest class that holds them, fewer
// where no class does.
struct Storage {
    size_t budget[kNumCls - 1];
    int slots_per_item, wcap;
    Storage(size_t smem_optin, int slots) : slots_per_item(slots), wcap(slots > 0 ? std::min(slots, kMaxSlots) : kMaxSlots) {
        const size_t most = smem_optin > kStorageReserve ? smem_optin - kStorageReserve : 0;
        for (int c = 0; c < kNumCls - 1; c++) budget[c] = kClsBudget[c] ? std::min<size_t>(kClsBudget[c], most) : most;
    }
    size_t most() const { return budget[kNumCls - 2]; }
    int64_t width(int64_t L, int64_t nA, int64_t slots, bool streamed, int *cls) const {
        int64_t want = 1, w = 1;
        int store = kClsGlobal;
        if (slots_per_item > 0)
            while (want * 2 <= std::min<int64_t>(slots, wcap)) want *= 2;
        for (; want >= 1 && store == kClsGlobal && !streamed; want /= 2)
            for (int c = 0; c < kNumCls - 1; c++)
                if (resident_bytes(L, nA, want) <= budget[c]) {
                    store = c;
                    break;
                }
        while (w * 2 <= std::min<int64_t>(slots, wcap) && (store == kClsGlobal || resident_bytes(L, nA, w * 2) <= budget[store])) w *= 2;
        *cls = store;
        return w;
    }
};

// fn(0) .. fn(n - 1) on up to 16 host threads (fewer where a thread does not start); false if one of them threw
template <typename Fn>
bool on_threads(size_t n, const Fn &fn) {
    std::atomic<size_t> next{0};
    std::atomic<bool> failed{false};
    auto worker = [&]() {
        try {
            for (size_t i = next++; i < n; i = next++) fn(i);
        } catch (...) {
            failed = true;
        }
    };
    const size_t most = std::min<size_t>({(size_t)std::max(1u, std::thread::hardware_concurrency()), (size_t)16, n});
    std::vector<std::thread> threads;
    try {
        for (size_t w = 1; w < most; w++) threads.emplace_back(worker);
    } catch (...) {
    }
    worker();
    for (std::thread &x : threads) x.join();
    return !failed;
}

// What the cut of a root at a level gives, whatever the slots: the active level-ell nodes (heads, by local index), the
// subtree of every local node below them (-1: none), and the subtrees' active entries and nodes.  Made once for all
// slot counts tried: 79 roots of 1.0e7 nodes are split in 13 ms (51 with a cut per count).
struct LevelCut {
    bool made = false;
    std::vector<int32_t> heads, sub;
    std::vector<int64_t> sa, sl;
    int64_t tot = 0, amax = 0;

    // li, cs, dd: the root's active entries (own and first child's local index, children)
    void make(const CfrRoot &cr, int ell, const int32_t *li, const int32_t *cs, const uint16_t *dd) {
        if (made) return;
        const int64_t L = cr.ls[9];
        for (int32_t e = cr.as[ell]; e < cr.as[ell + 1]; e++) heads.push_back(li[e]);
        std::sort(heads.begin(), heads.end());
        const size_t ns = heads.size();
        sub.assign((size_t)L, -1);
        for (size_t i = 0; i < ns; i++) sub[(size_t)heads[i]] = (int32_t)i;
        sa.assign(ns, 0);
        sl.assign(ns, 0);
        for (int k = ell; k < 8; k++)
            for (int32_t e = cr.as[k]; e < cr.as[k + 1]; e++) {
                const int32_t sid = sub[(size_t)li[e]];
                if (sid < 0) continue;
                sa[(size_t)sid]++;
                for (int a = 0; a < dd[e]; a++) sub[(size_t)(cs[e] + a)] = sid;
            }
        for (int64_t x = cr.ls[ell]; x < L; x++)
            if (sub[(size_t)x] >= 0) sl[(size_t)sub[(size_t)x]]++;
        for (int64_t n : sa) {
            tot += n;
            amax = std::max(amax, n);
        }
        made = true;
    }
};

// The subtrees of a cut in order, packed into parts of at most `limit` bytes (the first one beside the top's):
// bytes(nodes, entries) of a part.  first: the first subtree of every part.
template <typename Bytes>
struct PartPacking {
    const LevelCut &cut;
    const Bytes &bytes;
    size_t limit, top;

    // greedily, with at most `cap` entries to a part of several subtrees; false: a subtree fits no block
    bool fill(int64_t cap, std::vector<int> &first) const {
        first.assign(1, 0);
        int64_t pa = 0, plc = 0, pg = 0;
        for (int i = 0; i < (int)cut.heads.size(); i++) {
            const size_t lim = first.size() == 1 ? limit - top : limit;
            const bool fits = bytes(plc + cut.sl[(size_t)i] + pg + 1, pa + cut.sa[(size_t)i]) <= lim;
            if (pa > 0 && (!fits || pa + cut.sa[(size_t)i] > cap)) {
                first.push_back(i);
                pa = plc = pg = 0;
            }
            const size_t lim2 = first.size() == 1 ? limit - top : limit;
            pa += cut.sa[(size_t)i];
            plc += cut.sl[(size_t)i];
            pg += 1;
            if (bytes(plc + pg, pa) > lim2) return false;
        }
        return true;
    }
    // the fewest parts, without an entry cap; 0 where a subtree fits no block
    int fewest() const {
        std::vector<int> first;
        return fill(cut.tot, first) ? (int)first.size() : 0;
    }
    // at most Q parts with the smallest entry cap, by bisection
    bool balanced(int Q, std::vector<int> &first) const {
        int64_t lo = std::max<int64_t>(cut.amax, (cut.tot + Q - 1) / Q), hi = cut.tot;
        while (lo < hi) {
            const int64_t mid = lo + (hi - lo) / 2;
            if (fill(mid, first) && (int)first.size() <= Q) hi = mid;
            else lo = mid + 1;
        }
        return fill(lo, first) && (int)first.size() <= Q;
    }
};

}  // namespace pasur
