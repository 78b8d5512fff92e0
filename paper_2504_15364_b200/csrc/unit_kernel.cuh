// The whole step of a unit by ONE thread block of 256 threads, several blocks per SM, one launch: many small units.
// Nothing stays on chip but the keys: the block reads the unit's key rows once to score them, selects, and reads them again
// -- from L2, where the units that are being worked on fit -- to move them.  While one block of an SM waits for memory or
// works through its selection, which is a chain of barriers, the others keep the SM busy.  (The cluster kernels hold a unit on
// chip and fill an SM with one block, which for a unit of a few hundred rows is latency from end to end.)
//
// What bounds it: three blocks per SM (80 registers, by launch bounds; at 64 registers and four blocks most shapes lose 3-10 %)
// work through a chain of about 14 us for a unit of 300 rows: 1344 x 316 rows, 16 a step, in clusters of one
// and here, 169 -> 102 us in token order, 155 -> 53 with slot reuse.
// Long units: HBM, with slot reuse (2000 x 8224 rows, 32 a step, 690-730 us, 683 at the copy rate).
// The ring's 64 KB leave room for two blocks per SM: on 224 x 2176 rows the 224 blocks are all there at once, and the step is
// one chain (143 MB of traffic in 46 us, issue slots 43 % busy).
#pragma once
#include "evicted_list.cuh"
#include "row_terms.cuh"
#include "slot_kernel.cuh"      // issue_rows
#include "staged_kernels.cuh"   // concat_row

namespace kd {

constexpr int kUnitThreads = 256, kUnitWarps = 8;
constexpr int kUnitMaxDepth = 2;    // ring tiles per warp
constexpr int kUnitMoveRows = 64;   // rows of each tensor moved between two barriers
static_assert(kUnitThreads == kSelThreads, "the selector's 256 threads");

struct UnitLayout {
    int mbar, mu, sums, keys, ring, scratch, bitmap, lists, total;
};
__host__ __device__ inline UnitLayout unit_layout(int nmax, int max_block, int depth) {
    UnitLayout L;
    int off = 0;
    auto take = [&off](int bytes) { const int o = off; off += (bytes + 127) & ~127; return o; };
    L.mbar = take(kUnitWarps * kUnitMaxDepth * 8);
    L.mu = take(kHeadDim * 4);
    L.sums = take(kUnitWarps * kHeadDim * 8);
    L.keys = take(((nmax + 3) & ~3) * 4);        // the keys; then (ordered layout) the source row of every destination
    L.ring = off;                                // what follows is used when the last tile has been scored
    L.scratch = take(static_cast<int>(sizeof(SelectorScratch)));
    L.bitmap = take(2 * ((nmax + 31) / 32) * 4); // evicted-candidate bitmap, work space as long
    L.lists = take(3 * max_block * 4);           // evicted candidates; slot reuse: freed slots, kept block rows
    const int ring_end = L.ring + kUnitWarps * depth * kTileRows * kRowBytes;
    L.total = off > ring_end ? off : ring_end;
    return L;
}

struct UnitParams {
    uint4* k_cache; uint4* v_cache; const uint4* new_k; const uint4* new_v;
    int len, B, N, nmax, max_block;
    int depth;            // ring tiles per warp (kRing)
    float eps;
    float* scores; int32_t* kept_idx; int32_t* first_evicted;
    unsigned long long* moved_rows; int32_t* status;
    double* anchor_sum;   // [U][128] sum of the cached rows' terms, carried from step to step
    int rebuild;          // 1: that sum is not there, all rows are summed
    int raw_anchor, window;
    int32_t* pos; int next_pos;   // slot reuse
    int32_t* kept_mirror;
};

// Slot reuse, behind the selection: the block's 256 threads take the evicted rows' terms off the running sum (channel tid's sum over all n
// rows: `sum`) and place the kept block rows.  before: evicted candidates in front of every word of the bitmap; ev_of: their
// list, with room for two more behind it; sums: [8][128] doubles.
template <int kDeep>
__device__ __forceinline__ void place_block_rows(const UnitParams& p, int u, int tid, int n, int E, const uint32_t* bitmap, const int* before, int* ev_of,
                                                 int first_evicted, double sum, float inv_eps, bool raw, double* sums) {
    const int len = p.len, B = p.B, N = p.N, t = tid & 7;
    auto evicted = [&](int i) { return ((bitmap[i >> 5] >> (i & 31)) & 1u) != 0; };
    auto evicted_before = [&](int i) { return before[i >> 5] + __popc(bitmap[i >> 5] & ((1u << (i & 31)) - 1u)); };
    int32_t* kept = p.kept_idx + static_cast<size_t>(u) * N;
    int32_t* mirror = p.kept_mirror ? p.kept_mirror + static_cast<size_t>(u) * N : nullptr;
    int* slot_of = ev_of + p.max_block;   // freed slots, ascending
    int* blk_of = slot_of + p.max_block;  // kept block rows, ascending
    const int evicted_cache = evicted_before(len);   // evicted candidates among the len cache slots (len < n)
    const int kept_cache = len - evicted_cache;
    const int kb = N - kept_cache;                   // kept block rows = freed slots
    for (int e = tid; e < evicted_cache; e += kUnitThreads) slot_of[e] = ev_of[e];
    for (int e = len + tid; e < N; e += kUnitThreads)   // slots that were still empty
        if (KD_ROW_OK(evicted_cache + (e - len), p.max_block, p.status)) slot_of[evicted_cache + (e - len)] = e;
    for (int j = tid; j < B; j += kUnitThreads) {
        const int i = len + j, at = (i - evicted_before(i)) - kept_cache;
        if (!evicted(i) && KD_ROW_OK(at, p.max_block, p.status)) blk_of[at] = j;
    }
    // kept cache rows keep their slot.  Four entries at a time where they can be (an evicted row's entry is written again below, behind a barrier):
    // 1344 x 316 rows 51.6 -> 49.7 us a step
    if (((N | len) & 3) == 0 && !mirror) {
        int4* kept4 = reinterpret_cast<int4*>(kept);
#pragma unroll 4
        for (int i = tid; 4 * i < len; i += kUnitThreads) kept4[i] = make_int4(4 * i, 4 * i + 1, 4 * i + 2, 4 * i + 3);
    } else {
        for (int i = tid; i < len; i += kUnitThreads)
            if (!evicted(i)) { kept[i] = i; if (mirror) mirror[i] = i; }
    }
    if (tid == 0) {
        p.first_evicted[u] = first_evicted;
        atomicAdd(p.moved_rows, static_cast<unsigned long long>(kb));
    }
    // (the barrier inside makes the lists visible and lies behind every read of an evicted row)
    const double gone = block_sum_of_terms<kDeep>(E, [&](int r) { return concat_row(p.k_cache, p.new_k, u, min(max(ev_of[r], 0), n - 1), len, B, N); },
                                                 inv_eps, raw, sums, tid);
    if (tid < kHeadDim) p.anchor_sum[static_cast<size_t>(u) * kHeadDim + tid] = sum - gone;
#pragma unroll 2
    for (int r = tid >> 3; r < kb; r += kUnitThreads / kLanesPerRow) {   // kept block row r into freed slot r
        const int slot = slot_of[r], j = blk_of[r];
        if (!(KD_ROW_OK(slot, N, p.status) && KD_ROW_OK(j, B, p.status))) continue;
        const uint4* sk = p.new_k + (static_cast<size_t>(u) * B + j) * kRowVec;
        const uint4* sv = p.new_v + (static_cast<size_t>(u) * B + j) * kRowVec;
        uint4* dk = p.k_cache + (static_cast<size_t>(u) * N + slot) * kRowVec;
        uint4* dv = p.v_cache + (static_cast<size_t>(u) * N + slot) * kRowVec;
        const uint4 k0 = sk[t], k1 = sk[t + 8], v0 = sv[t], v1 = sv[t + 8];
        dk[t] = k0; dk[t + 8] = k1;
        dv[t] = v0; dv[t + 8] = v1;
        if (t == 0) {
            kept[slot] = len + j;
            if (mirror) mirror[slot] = len + j;
            p.pos[static_cast<size_t>(u) * N + slot] = p.next_pos + j;
        }
    }
}

template <bool kSlots, bool kRing>
__global__ void __launch_bounds__(kUnitThreads, 3) unit_evict_kernel(const UnitParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const UnitLayout L = unit_layout(p.nmax, p.max_block, p.depth);
    SelectorScratch& scratch = *reinterpret_cast<SelectorScratch*>(smem + L.scratch);
    double* sums = reinterpret_cast<double*>(smem + L.sums);
    const uint4* ring = reinterpret_cast<const uint4*>(smem + L.ring);
    const uint32_t ring_sa = smem_addr(ring), mbar_sa = smem_addr(smem + L.mbar);
    float* mu = reinterpret_cast<float*>(smem + L.mu);
    uint32_t* keys = reinterpret_cast<uint32_t*>(smem + L.keys);
    uint32_t* bitmap = reinterpret_cast<uint32_t*>(smem + L.bitmap);
    int* ev_of = reinterpret_cast<int*>(smem + L.lists);   // evicted candidates, ascending
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, t = tid & 7, sub = lane >> 3;
    const int len = p.len, B = p.B, N = p.N, n = len + B, E = n - N;
    const float inv_eps = 1.0f / p.eps;
    const bool raw = p.raw_anchor != 0;
    const int tiles = (n + kTileRows - 1) / kTileRows, D = p.depth;
    if (kRing && tid == 0) {
        for (int j = 0; j < kUnitWarps * D; ++j) mbar_init(mbar_sa + 8 * j, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    grid_dependency_wait();
    if (kRing) __syncthreads();
    // kRing: the key rows come through a ring of 16-row tiles: warp w takes tiles w, w + 8, ... through its own D slots
    auto issue = [&](int tile, int d) {   // one lane
        const int lo = tile * kTileRows, slot = warp * D + d;
        issue_rows(p.k_cache, p.new_k, u, len, B, N, lo, min(n, lo + kTileRows) - lo, ring_sa + slot * kTileRows * kRowBytes, mbar_sa + 8 * slot);
    };
    if (kRing && lane == 0)
        for (int d = 0; d < D && warp + kUnitWarps * d < tiles; ++d) issue(warp + kUnitWarps * d, d);

    // ------------------------------------------------------------ anchor: running sum + the block rows' terms
    double sum = 0.0;   // tid < 128: channel tid's sum over all n rows
    {
        if (tid < kHeadDim && !p.rebuild) sum = p.anchor_sum[static_cast<size_t>(u) * kHeadDim + tid];
        const int first = p.rebuild ? 0 : len;
        sum += block_sum_of_terms(n - first, [&](int r) { return concat_row(p.k_cache, p.new_k, u, first + r, len, B, N); }, inv_eps, raw, sums, tid);
        if (tid < kHeadDim) mu[tid] = static_cast<float>(sum / static_cast<double>(n));
        __syncthreads();
    }
    // ------------------------------------------------------------ scores
    bool in_time = true;
    {
        float2 w[8];
        load_anchor(mu, t, w);
        const float m = anchor_norm(mu, lane);
        float* sc = p.scores + static_cast<size_t>(u) * p.nmax;
        int d = 0;
        uint32_t par = 0;   // bit d: parity the next wait on slot d expects
#pragma unroll 1
        for (int tile = warp; tile < tiles; tile += kUnitWarps) {
            const int slot = warp * D + d, lo = tile * kTileRows;
            if (kRing) {
                in_time = mbar_wait(mbar_sa + 8 * slot, (par >> d) & 1u, p.status) && in_time;
                par ^= 1u << d;
            }
            const uint4* rows = ring + slot * kTileRows * kRowVec;
            uint4 a[4], b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = q * 4 + sub;
                a[q] = make_uint4(0, 0, 0, 0); b[q] = a[q];
                if (lo + r < n) {
                    const uint4* row = kRing ? rows + r * kRowVec : concat_row(p.k_cache, p.new_k, u, lo + r, len, B, N);
                    a[q] = row[t]; b[q] = row[t + 8];
                }
            }
            float vs[4];
            double vd[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) lane_sumsq_dot(a[q], b[q], w, vs[q], vd[q]);
            const uint32_t key = score4(vs, vd, t, m, p.eps);
            const int i = lo + (t >> 1) * 4 + sub;
            if (!(t & 1) && i < n) { keys[i] = key; sc[i] = key_score(key); }
            if (kRing) {
                __syncwarp();   // the tile's only readers are this warp's lanes: the copy engine may refill it
                if (lane == 0 && tile + kUnitWarps * D < tiles) issue(tile + kUnitWarps * D, d);
                if (++d == D) d = 0;
            }
        }
    }
    if (!__syncthreads_and(in_time)) return;   // (a tile never landed, the status word says so: nothing is moved or placed)
    if (p.window > 0) {
        // sliding window (Sec. 3.2): the tokens at the last `window` positions get the largest possible key
        if (kSlots) {
            const int first_recent = p.next_pos + B - p.window;
            for (int i = len + max(B - p.window, 0) + tid; i < n; i += kUnitThreads) keys[i] = 0xffffffffu;
            if (p.window > B) {
                const int32_t* ps = p.pos + static_cast<size_t>(u) * N;
                for (int i = tid; i < len; i += kUnitThreads) if (ps[i] >= first_recent) keys[i] = 0xffffffffu;
            }
        } else {
            for (int i = n - p.window + tid; i < n; i += kUnitThreads) keys[i] = 0xffffffffu;
        }
        __syncthreads();
    }
    // ------------------------------------------------------------ selection
    Selector s(scratch, bitmap, bitmap + ((p.nmax + 31) >> 5));
    select_evicted(keys, n, E, tid, s);
    auto evicted = [&](int i) { return ((bitmap[i >> 5] >> (i & 31)) & 1u) != 0; };
    int* before = reinterpret_cast<int*>(s.eq);   // evicted candidates in front of every word
    const int first_evicted = list_evicted(n, tid, s, before, ev_of, p.max_block, p.status);
    auto evicted_before = [&](int i) { return before[i >> 5] + __popc(bitmap[i >> 5] & ((1u << (i & 31)) - 1u)); };
    int32_t* kept = p.kept_idx + static_cast<size_t>(u) * N;
    int32_t* mirror = p.kept_mirror ? p.kept_mirror + static_cast<size_t>(u) * N : nullptr;
    if constexpr (!kSlots) {
        int* src_of = reinterpret_cast<int*>(keys);   // (the keys are dead)
        for (int i = tid; i < n; i += kUnitThreads)
            if (!evicted(i)) {
                const int d = i - evicted_before(i);
                src_of[d] = i;
                kept[d] = i;
                if (mirror) mirror[d] = i;
            }
        // (the barrier inside makes the list visible and lies behind every read of an evicted row)
        const double gone = block_sum_of_terms(E, [&](int r) { return concat_row(p.k_cache, p.new_k, u, min(max(ev_of[r], 0), n - 1), len, B, N); },
                                              inv_eps, raw, sums, tid);
        if (tid < kHeadDim) p.anchor_sum[static_cast<size_t>(u) * kHeadDim + tid] = sum - gone;
        const int first_moved = min(first_evicted, len);   // block rows always move into the cache
        if (tid == 0) {
            p.first_evicted[u] = first_evicted;
            atomicAdd(p.moved_rows, static_cast<unsigned long long>(N - first_moved));
        }
        // Rows move to lower places only: once all threads hold their part of a chunk of destinations, it may be written; the
        // sources of later chunks lie behind it.
        uint4* k_out = p.k_cache + static_cast<size_t>(u) * N * kRowVec;
        uint4* v_out = p.v_cache + static_cast<size_t>(u) * N * kRowVec;
        const int c = tid & 15;
#pragma unroll 1
        for (int base = first_moved; base < N; base += kUnitMoveRows) {
            constexpr int kPer = kUnitMoveRows * kRowVec / kUnitThreads;
            uint4 a[kPer], b[kPer];
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const int d = base + (tid >> 4) + q * (kUnitThreads / 16);
                if (d < N) {
                    const int src = src_of[d];
                    if (!KD_ROW_OK(src, n, p.status)) continue;
                    a[q] = concat_row(p.k_cache, p.new_k, u, src, len, B, N)[c];
                    b[q] = concat_row(p.v_cache, p.new_v, u, src, len, B, N)[c];
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const int d = base + (tid >> 4) + q * (kUnitThreads / 16);
                if (d < N) { k_out[d * kRowVec + c] = a[q]; v_out[d * kRowVec + c] = b[q]; }
            }
        }
    } else {
        place_block_rows<4>(p, u, tid, n, E, bitmap, before, ev_of, first_evicted, sum, inv_eps, raw, sums);
    }
}

}  // namespace kd
