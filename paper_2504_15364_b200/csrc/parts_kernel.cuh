// Slot reuse, more units than SMs: scores by several blocks per unit, and the rest of a unit's step in the same launch.  Whoever finishes a unit's
// last part selects and places the kept block rows, while the other blocks go on to score the units behind it.  The anchors have been
// formed by wide_anchor_kernel from the running sum.  No block waits for another one.
//
// A unit's rows are read once, and a unit is no longer tied to one block: the units need not fill the SMs in whole rounds, and of all
// selections only the last ones are not hidden behind the reading of keys.  What bounds it: HBM (1000 x 8256 rows 365 us a step, 5.8 TB/s),
// and at the ends about 5 us for the anchors and a chain of 13 us (units of 2000 rows) to 19 us (8000) for the last unit: keys 2, selection 6,
// lists 3, evicted rows 4, placement 3.  Against a block per unit, or per unit and round, us a step: 300 x 8256 rows 172 -> 125, 180 x 8256 119 -> 84,
// 512 x 4160 140 -> 115, 896 x 4352 246 -> 220 (256 a step: 263 -> 240), 1000 x 8256 388 -> 365, 160 x 16448 182 -> 145.
#pragma once
#include "unit_kernel.cuh"
#include "wide_kernels.cuh"

namespace kd {

struct PartsLayout { int keys, bitmap, scratch, total; };
__host__ __device__ inline PartsLayout parts_layout(int n, int max_block) {
    PartsLayout L;
    int off = 0;
    auto take = [&off](int bytes) { const int o = off; off += (bytes + 127) & ~127; return o; };
    // The keys; behind the selection the lists of evicted candidates, freed slots and kept block rows.  Beside the keys, 6 KB for blocks of 512 rows, they
    // cost three blocks per SM at 8192 rows their L1: 400 x 8704 rows, 512 a step, 261 us against 227.
    const int keys = (n + 3) & ~3;
    L.keys = take((keys > 3 * max_block ? keys : 3 * max_block) * 4);
    L.bitmap = take(2 * ((n + 31) / 32) * 4);
    L.scratch = take(static_cast<int>(sizeof(SelectorScratch)));
    L.total = off;
    return L;
}

struct PartsParams {
    UnitParams unit;        // (depth and rebuild are not used)
    const float* mu;        // [U][kMuStride]
    unsigned* parts_done;   // [U] zero between steps
    int parts, rows_per_part;
};

// Scores of rows [r0, r1) of unit u by 256 threads, 16 rows of a warp together; the next ones are requested as soon as a lane has its shares
// of the ones before.
__device__ __forceinline__ void score_rows(const UnitParams& p, const float* mu, int u, int r0, int r1, int tid) {
    const int lane = tid & 31, warp = tid >> 5, t = tid & 7, sub = lane >> 3;
    uint4 a[4], b[4];
    auto load = [&](int i0) {   // rows i0 + 4q + sub
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + 4 * q + sub;
            a[q] = make_uint4(0, 0, 0, 0); b[q] = a[q];
            if (i < r1) {
                const uint4* row = concat_row(p.k_cache, p.new_k, u, i, p.len, p.B, p.N);
                a[q] = __ldcg(row + t); b[q] = __ldcg(row + t + 8);
            }
        }
    };
    const int first = r0 + 16 * warp;
    load(first);              // (in front of the wait: the kernel that forms the anchors lets this one in when everything before it is complete)
    grid_dependency_wait();   // the anchors
    mu += static_cast<size_t>(u) * kMuStride;
    float2 w[8];
    load_anchor(mu, t, w);
    const float m = mu[kHeadDim];
    float* out = p.scores + static_cast<size_t>(u) * p.nmax;
#pragma unroll 1
    for (int base = first; base < r1; base += 16 * kUnitWarps) {
        float ss[4];
        double dot[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) lane_sumsq_dot(a[q], b[q], w, ss[q], dot[q]);
        load(base + 16 * kUnitWarps);
        const float e = key_score(score4(ss, dot, t, m, p.eps));
        const int i = base + (t >> 1) * 4 + sub;
        if (!(t & 1) && i < r1) out[i] = e;
    }
}

// grid = (parts, U): parts of a unit are started together, unit after unit.
__global__ void __launch_bounds__(kUnitThreads, 3) parts_kernel(const PartsParams q) {
    extern __shared__ __align__(128) unsigned char smem[];
    const UnitParams& p = q.unit;
    const int u = blockIdx.y, tid = threadIdx.x, len = p.len, B = p.B, N = p.N, n = len + B, E = n - N;
    const int r0 = blockIdx.x * q.rows_per_part;
    score_rows(p, q.mu, u, r0, min(n, r0 + q.rows_per_part), tid);
    __syncthreads();
    bool last = false;
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(q.parts_done + u, 1u) == static_cast<unsigned>(q.parts - 1);
        if (last) { __threadfence(); q.parts_done[u] = 0u; }
    }
    if (!__syncthreads_or(last)) return;   // (no shared memory beside what parts_layout says: its sum decides which step comes here)
    // ------------------------------------------------------------ the unit's last part: all scores are there
    const PartsLayout L = parts_layout(n, p.max_block);
    uint32_t* keys = reinterpret_cast<uint32_t*>(smem + L.keys);
    uint32_t* bitmap = reinterpret_cast<uint32_t*>(smem + L.bitmap);
    SelectorScratch& scratch = *reinterpret_cast<SelectorScratch*>(smem + L.scratch);
    Selector s(scratch, bitmap, bitmap + ((n + 31) >> 5));
    int* before = reinterpret_cast<int*>(s.eq);
    double* sums = reinterpret_cast<double*>(scratch.hist);   // (behind the selection the histograms are dead)
    static_assert(sizeof(scratch.hist) >= kTermWarps * kHeadDim * 8, "the terms' table");
    load_keys(p.scores + static_cast<size_t>(u) * p.nmax, n, n, (p.nmax & 3) == 0, keys, tid);
    __syncthreads();
    if (p.window > 0) {
        // sliding window (Sec. 3.2): the tokens at the last `window` positions get the largest possible key
        for (int i = len + max(B - p.window, 0) + tid; i < n; i += kUnitThreads) keys[i] = 0xffffffffu;
        if (p.window > B) {
            const int first_recent = p.next_pos + B - p.window;
            const int32_t* ps = p.pos + static_cast<size_t>(u) * N;
            for (int i = tid; i < len; i += kUnitThreads) if (ps[i] >= first_recent) keys[i] = 0xffffffffu;
        }
        __syncthreads();
    }
    select_evicted(keys, n, E, tid, s);
    int* ev_of = reinterpret_cast<int*>(keys);
    const int first = list_evicted(n, tid, s, before, ev_of, p.max_block, p.status);
    const double sum = tid < kHeadDim ? p.anchor_sum[static_cast<size_t>(u) * kHeadDim + tid] : 0.0;
    place_block_rows<kWideTermsDeep>(p, u, tid, n, E, bitmap, before, ev_of, first, sum, 1.0f / p.eps, p.raw_anchor != 0, sums);
}

}  // namespace kd
