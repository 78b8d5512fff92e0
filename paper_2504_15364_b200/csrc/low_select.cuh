// Exact selection at the low end of a key table by 256 threads: only the E = n - N smallest keys go, so two passes over
// the table and the ranking of a short list are enough.
#pragma once
#include "fused_kernel.cuh"   // kBins
#include "sel_barrier.cuh"

namespace kd {

constexpr int kSelList = 1024;    // keys under the first bound that are listed
constexpr int kSelTies = 256;     // keys of the threshold bin ranked exactly
constexpr int kSelDirect = 128;   // units of so few keys are ranked whole (at 230 keys that takes 143 instead of 124 us a step on 4000 units)
constexpr int kMinBins = 1024;    // histogram of the classes' smallest keys

struct SelectorScratch {   // 128-byte aligned
    int hist[kBins], min_hist[kMinBins];
    uint32_t list_key[kSelList]; int list_idx[kSelList];
    uint32_t tie_key[kSelTies]; int tie_idx[kSelTies];
    int wtot[48];   // 0 .. 7 warp totals, 16 .. 31 warp minima and bounds
    int misc[8];    // 0 listed keys, 1 the caller's, 2 / 3 broadcast, 6 keys of the threshold bin
    // What lies between a word's last read and its next write.  misc[0]: written once per selection.  misc[2] / [3]: read behind the last
    // barrier of a radix round, written behind the first ones of the next.  misc[6]: read behind the barrier in front of the ranking, reset
    // behind the first barrier of select_evicted_any.  wtot[0 .. 7]: a scan begins with a barrier; between two crossings lies the pass
    // that marks or lists.  wtot[16 .. 31]: written once per selection.
};
struct Selector {
    int* hist; int* min_hist; uint32_t* list_key; int* list_idx; uint32_t* tie_key; int* tie_idx;
    uint32_t* bitmap; uint32_t* eq; int* misc; int* wtot;   // bitmap: evicted tokens; eq: as long, work space
    __device__ Selector(SelectorScratch& x, uint32_t* bits, uint32_t* work)
        : hist(x.hist), min_hist(x.min_hist), list_key(x.list_key), list_idx(x.list_idx), tie_key(x.tie_key), tie_idx(x.tie_idx),
          bitmap(bits), eq(work), misc(x.misc), wtot(x.wtot) {}
};

// Exclusive sum over the selector threads.
__device__ __forceinline__ int sel_exclusive_scan(int v, int st, int* wtot) {
    const int lane = st & 31, w = st >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += x; }
    sel_sync();   // the totals of an earlier scan have been read
    if (lane == 31) wtot[w] = incl;
    sel_sync();
    int base = 0;
#pragma unroll
    for (int q = 0; q < kSelWarps; ++q) base += q < w ? wtot[q] : 0;
    return base + incl - v;
}

// Bins in ascending order, 256 per warp of the first kNBins / 256: the bin in which the running count reaches E (kNBins if it
// never does) and the count in front of it.  One barrier.
template <int kNBins>
__device__ __forceinline__ int2 sel_find_crossing(const int* h, int E, int st, int* wtot) {
    constexpr int kW = kNBins / 256;
    const int lane = st & 31, w = st >> 5;
    const int4* h4 = reinterpret_cast<const int4*>(h);
    if (w < kW) {
        const int4 a = h4[64 * w + 2 * lane], b = h4[64 * w + 2 * lane + 1];
        const int s = __reduce_add_sync(0xffffffffu, (a.x + a.y) + (a.z + a.w) + (b.x + b.y) + (b.z + b.w));
        if (lane == 0) wtot[w] = s;
    }
    sel_sync();
    int before = 0, W = -1;
#pragma unroll
    for (int q = 0; q < kW; ++q)
        if (W < 0) { if (before + wtot[q] >= E) W = q; else before += wtot[q]; }
    if (W < 0) return make_int2(kNBins, before);
    const int4 a = h4[64 * W + 2 * lane], b = h4[64 * W + 2 * lane + 1];
    const int c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    int tot = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) tot += c[q];
    int incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += x; }
    const int J = __ffs(__ballot_sync(0xffffffffu, before + incl >= E)) - 1;
    int run = before + incl - tot, bin = 7, at = run;   // (lane J's answer counts)
    bool found = false;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if (!found && run + c[q] >= E) { found = true; bin = q; at = run; }
        run += c[q];
    }
    return make_int2(256 * W + 8 * J + __shfl_sync(0xffffffffu, bin, J), __shfl_sync(0xffffffffu, at, J));
}

// Linear bins over [lo, hi]: the right shift that leaves fewer than 2^bits values.
__device__ __forceinline__ uint32_t bin_shift(uint32_t lo, uint32_t hi, int bits) {
    const int have = 32 - __clz(hi - lo);
    return have > bits ? have - bits : 0;
}

// f(key, token) for this thread's share of the n keys of a table (its end is padded to 128-bit words).
template <typename F>
__device__ __forceinline__ void for_all_keys(const uint32_t* keys, int n, int st, const F& f) {
    const uint4* k4 = reinterpret_cast<const uint4*>(keys);
#pragma unroll 2
    for (int q = st; 4 * q < n; q += kSelThreads) {
        const uint4 k = k4[q];
        f(k.x, 4 * q);
        if (4 * q + 1 < n) f(k.y, 4 * q + 1);
        if (4 * q + 2 < n) f(k.z, 4 * q + 2);
        if (4 * q + 3 < n) f(k.w, 4 * q + 3);
    }
}
// Marks, among the keys that f's caller visits, those under the E-th smallest's bin and ranks the bin's own keys exactly; false
// if the bin is crowded.  lo .. hi: at least E of the visited keys lie in it, none below lo.  Histogram and ties zero on entry.
template <typename Visit>
__device__ __forceinline__ bool mark_smallest(const Visit& visit, uint32_t lo, uint32_t hi, int E, int st, const Selector& s) {
    const int lane = st & 31, w = st >> 5;
    const uint32_t shift = bin_shift(lo, hi, 11);
    visit([&](uint32_t k, int) { if (k <= hi) atomicAdd(&s.hist[(k - lo) >> shift], 1); });
    sel_sync();
    const int2 cross = sel_find_crossing<kBins>(s.hist, E, st, s.wtot);
    const uint32_t bstar = static_cast<uint32_t>(cross.x);
    const int need = E - cross.y;   // this many keys of the threshold bin go
    visit([&](uint32_t k, int i) {
        const uint32_t b = (k - lo) >> shift;
        if (k > hi || b > bstar) return;
        if (b < bstar) {
            atomicOr(&s.bitmap[i >> 5], 1u << (i & 31));
        } else {
            const int at = atomicAdd(&s.misc[6], 1);
            if (at < kSelTies) { s.tie_key[at] = k; s.tie_idx[at] = i; }
        }
    });
    sel_sync();
    const int ties = s.misc[6];
    if (ties > kSelTies) return false;
    for (int c = w; c < ties; c += kSelWarps) {
        const uint32_t mk = s.tie_key[c];
        const int mi = s.tie_idx[c];
        int rank = 0;
        for (int q = lane; q < ties; q += 32) {
            const uint32_t ok = s.tie_key[q];
            rank += (ok < mk) || (ok == mk && s.tie_idx[q] > mi);
        }
        rank = __reduce_add_sync(0xffffffffu, rank);
        if (lane == 0 && rank < need) atomicOr(&s.bitmap[mi >> 5], 1u << (mi & 31));
    }
    sel_sync();
    return true;
}
// The same over the whole table, and where that is crowded too (many equal keys) the radix route: the exact E-th key by four
// 8-bit digits, then the newest of its equals.
__device__ __noinline__ void select_evicted_any(const uint32_t* keys, int n, int E, uint32_t lo, uint32_t hi, int st, const Selector& s) {
    const int lane = st & 31, nwords = (n + 31) >> 5;
    sel_sync();   // every warp has read misc[6], and with it that the list is crowded, before it is reset
    for (int b = st; b < kBins; b += kSelThreads) s.hist[b] = 0;
    for (int q = st; q < nwords; q += kSelThreads) s.bitmap[q] = 0;
    if (st == 0) s.misc[6] = 0;
    sel_sync();
    auto visit = [&](const auto& f) { for_all_keys(keys, n, st, f); };
    if (mark_smallest(visit, lo, hi, E, st, s)) return;
    uint32_t prefix = 0, mask = 0;
    int want = E, equal = 0;
#pragma unroll 1
    for (int sh = 24; sh >= 0; sh -= 8) {
        sel_sync();
        s.hist[st] = 0;   // (256 threads, 256 digits)
        sel_sync();
        visit([&](uint32_t k, int) {
            if ((k & mask) == prefix) {   // one shared-memory atomic per digit and group of lanes: thousands of equal keys share a digit
                const int digit = (k >> sh) & 0xff;
                const unsigned act = __activemask(), peers = __match_any_sync(act, digit);
                if (lane == __ffs(peers) - 1) atomicAdd(&s.hist[digit], __popc(peers));
            }
        });
        sel_sync();
        const int mine = s.hist[st], excl = sel_exclusive_scan(mine, st, s.wtot);
        if (excl < want && want <= excl + mine) { s.misc[2] = st; s.misc[3] = excl; }
        sel_sync();
        prefix |= static_cast<uint32_t>(s.misc[2]) << sh;
        mask |= 0xffu << sh;
        want -= s.misc[3];
        equal = s.hist[s.misc[2]];
    }
    uint32_t* eq = s.eq;
    for (int q = st; q < nwords; q += kSelThreads) { s.bitmap[q] = 0; eq[q] = 0; }
    sel_sync();
    visit([&](uint32_t k, int i) {
        if (k < prefix) atomicOr(&s.bitmap[i >> 5], 1u << (i & 31));
        if (k == prefix) atomicOr(&eq[i >> 5], 1u << (i & 31));
    });
    sel_sync();
    const int per = (nwords + kSelThreads - 1) / kSelThreads;
    const int w0 = min(nwords, st * per), w1 = min(nwords, w0 + per);
    int cnt = 0;
    for (int q = w0; q < w1; ++q) cnt += __popc(eq[q]);
    int rank = sel_exclusive_scan(cnt, st, s.wtot);
    for (int q = w0; q < w1; ++q) {
        uint32_t go = 0;
        for (uint32_t m = eq[q]; m; m &= m - 1, ++rank) go |= rank >= equal - want ? m & (0u - m) : 0u;   // the newest `want` of the equals
        s.bitmap[q] |= go;
    }
    sel_sync();
}
// Ranks at most 256 keys against each other and sets the bits of the E smallest: a thread per key, two with half the
// comparisons each when there are at most 128.  token(c): the key's token.  Bits zero and keys visible on entry; ends with a barrier.
template <typename Token>
__device__ __forceinline__ void rank_all(const uint32_t* list, int count, int E, int st, const Selector& s, const Token& token) {
    const int parts = count <= kSelThreads / 2 ? 2 : 1, c = parts == 2 ? st >> 1 : st, quads = count >> 2;
    const uint32_t mk = c < count ? list[c] : 0u;
    const uint4* l4 = reinterpret_cast<const uint4*>(list);
    int rank = 0;
    if (c < count) {
#pragma unroll 4
        for (int q = parts == 2 ? st & 1 : 0; q < quads; q += parts) {
            const uint4 k = l4[q];
            rank += (k.x < mk) + (k.y < mk) + (k.z < mk) + (k.w < mk);
        }
        if (parts == 1 || (st & 1)) for (int q = 4 * quads; q < count; ++q) rank += list[q] < mk;
    }
    if (parts == 2) rank += __shfl_xor_sync(0xffffffffu, rank, 1);
    // equal keys share a rank: more than E keys with one under E means that equal ones lie across the threshold
    const bool counts = c < count && rank < E && (parts == 1 || !(st & 1));
    const int all = sel_count(counts);
    if (counts) {
        const int mi = token(c);
        bool go = true;
        if (all != E) {   // among equal keys the newer tokens go first
            int newer = 0;
            for (int q = 0; q < count; ++q) newer += list[q] == mk && token(q) > mi;
            go = rank + newer < E;
        }
        if (go) atomicOr(&s.bitmap[mi >> 5], 1u << (mi & 31));
    }
    sel_sync();
}

// Bits of the E tokens that go -- the E smallest keys of the table under (key ascending, token descending) -- in s.bitmap, all
// other bits zero; visible to the selectors when this returns.
// Two passes over the n keys.  The first finds the smallest key of each of 1024 classes (four per thread); where E of those
// fall (a histogram of the minima) bounds the E-th smallest key, since the minima are distinct keys, and tightly: about 140
// of 8320 keys lie under it at E = 128, 290 of 4352 at E = 256.  The second lists the keys under the bound.  A short list is
// ranked key against key, a longer one goes through a histogram, and
// a list that runs over takes the whole table instead.
__device__ __forceinline__ void select_evicted(const uint32_t* keys, int n, int E, int st, const Selector& s) {
    const int lane = st & 31, w = st >> 5, nwords = (n + 31) >> 5;
    const uint4* k4 = reinterpret_cast<const uint4*>(keys);
    if (n <= kSelDirect) {
        if (st < nwords) s.bitmap[st] = 0;
        sel_sync();
        rank_all(keys, n, E, st, s, [](int c) { return c; });
        return;
    }
    uint32_t* wkey = reinterpret_cast<uint32_t*>(s.wtot) + 16;
    reinterpret_cast<int4*>(s.min_hist)[st] = make_int4(0, 0, 0, 0);
    for (int q = st; q < nwords; q += kSelThreads) s.bitmap[q] = 0;
    if (st == 0) { s.misc[0] = 0; s.misc[6] = 0; }
    uint32_t lo[4] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu};
    {
        const int whole = n >> 2;   // quads without a gap
#pragma unroll 4
        for (int q = st; q < whole; q += kSelThreads) {
            const uint4 k = k4[q];
            lo[0] = min(lo[0], k.x); lo[1] = min(lo[1], k.y); lo[2] = min(lo[2], k.z); lo[3] = min(lo[3], k.w);
        }
        if ((n & 3) && st == whole % kSelThreads)   // (the thread whose next quad it is)
#pragma unroll
            for (int c = 0; c < 3; ++c) if (4 * whole + c < n) lo[c] = min(lo[c], keys[4 * whole + c]);
        // class c of thread st is empty only if 4 st + c >= n
        uint32_t tlo = min(min(lo[0], lo[1]), min(lo[2], lo[3])), thi = 0u;
#pragma unroll
        for (int c = 0; c < 4; ++c) if (4 * st + c < n) thi = max(thi, lo[c]);
        const uint32_t wlo = __reduce_min_sync(0xffffffffu, tlo), whi = __reduce_max_sync(0xffffffffu, thi);
        if (lane == 0) { wkey[w] = wlo; wkey[kSelWarps + w] = whi; }
    }
    sel_sync();
    uint32_t kmin = wkey[0], bound = wkey[kSelWarps];   // min(1024, n) keys, the classes' smallest, are not above `bound`
#pragma unroll
    for (int q = 1; q < kSelWarps; ++q) { kmin = min(kmin, wkey[q]); bound = max(bound, wkey[kSelWarps + q]); }
    if (E > min(4 * kSelThreads, n)) {   // fewer classes than keys to go
        select_evicted_any(keys, n, E, kmin, 0xffffffffu, st, s);
        return;
    }
    {
        const uint32_t shift = bin_shift(kmin, bound, 10);
#pragma unroll
        for (int c = 0; c < 4; ++c) if (4 * st + c < n) atomicAdd(&s.min_hist[(lo[c] - kmin) >> shift], 1);
        sel_sync();
        const int bin = sel_find_crossing<kMinBins>(s.min_hist, E, st, s.wtot).x;   // (all minima are counted: it is found)
        const uint32_t width = ((static_cast<uint32_t>(bin) + 1u) << shift) - 1u;
        bound = min(bound, width > 0xffffffffu - kmin ? 0xffffffffu : kmin + width);
    }
    for_all_keys(keys, n, st, [&](uint32_t k, int i) {
        if (k <= bound) {
            const int at = atomicAdd(&s.misc[0], 1);
            if (at < kSelList) { s.list_key[at] = k; s.list_idx[at] = i; }
        }
    });
    sel_sync();
    const int count = s.misc[0];
    if (count <= kSelThreads) {
        rank_all(s.list_key, count, E, st, s, [&](int c) { return s.list_idx[c]; });
        return;
    }
    if (count <= kSelList) {
        for (int b = st; b < kBins / 4; b += kSelThreads) reinterpret_cast<int4*>(s.hist)[b] = make_int4(0, 0, 0, 0);
        sel_sync();
        auto visit = [&](const auto& f) { for (int c = st; c < count; c += kSelThreads) f(s.list_key[c], s.list_idx[c]); };
        if (mark_smallest(visit, kmin, bound, E, st, s)) return;
    }
    select_evicted_any(keys, n, E, kmin, bound, st, s);
}

}  // namespace kd
