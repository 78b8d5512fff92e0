// Ordered layout for units that no cluster can hold on chip (budgets beyond about 12000 tokens), for many of those that only
// clusters of ten or more hold, and for steps of many long units that evict one row: four launches per step, as in the staged
// path, but with the anchor's sum carried from step to step, so that the keys are read twice and not three times.
//
//   wide_anchor   running sum of the cached rows + the block rows' terms = this step's anchor (App. B.1, first expression)
//   wide_score    norm, dot product and score of every key in one pass (second expression)
//   wide_select   exact top-N, kept-index list; the evicted rows' terms leave the running sum
//   compact_kernel (staged_kernels.cuh), or for few units wide_move, which gives a unit several blocks per tensor
//
// The running sum cannot drift: a row's terms are the fixed bit pattern that the other kernels add and take out as well
// (row_terms.cuh), added and subtracted in double.
//
// What bounds it: HBM.  256 units of 16512 keys, 5.4 GB of traffic a step: 886 us; in the staged kernels 1280 us (anchor and
// score pass 308 + 229, selection 66, compaction 684).  The score pass takes 172 us (6.3 TB/s), the selection 25, the
// compaction 679 (6.3 TB/s, and the last units' keys from L2).
#pragma once
#include "evicted_list.cuh"
#include "row_terms.cuh"
#include "staged_kernels.cuh"

namespace kd {

constexpr int kWideThreads = 256, kWideGroups = kWideThreads / kLanesPerRow;
constexpr int kWideDeep = 4;             // rows a row group requests together
constexpr int kWideTermsDeep = 8;        // 128 block rows or evicted rows requested together
constexpr int kMuStride = kHeadDim + 4;  // a unit's anchor and its norm
static_assert(kWideDeep == 4, "group_sum_of4");
static_assert(kWideThreads == kSelThreads, "wide_select runs the selector's 256 threads");

// grid = U.  Also clears wide_move's counter and flags (2 * kMaxSegments per unit), if that is to follow.
__global__ void __launch_bounds__(kWideThreads)
wide_anchor_kernel(const uint4* __restrict__ new_k, int B, int n, float eps, int raw_anchor,
                   const double* sum_in, double* sum_out /* may be the same */, double* __restrict__ deltas, int ndeltas, float* __restrict__ mu,
                   unsigned* __restrict__ move_sync /* or nullptr */, bool let_in) {
    __shared__ __align__(16) double table[kTermWarps * kHeadDim];
    __shared__ float mu_sh[kHeadDim];
    grid_dependency_wait();
    // parts_kernel requests keys and block rows before it waits for the anchors: let in behind the wait above, never in front of it, and nothing here
    // writes either tensor (common.cuh)
    if (let_in) grid_dependency_trigger();
    const int u = blockIdx.x, tid = threadIdx.x;
    const uint4* blk = new_k + static_cast<size_t>(u) * B * kRowVec;
    if (move_sync && tid < 2 * kMaxSegments) move_sync[1 + u * 2 * kMaxSegments + tid] = 0u;
    if (move_sync && u == 0 && tid == 2 * kMaxSegments) move_sync[0] = 0u;
    // the sum, and what the CTAs of the cluster kernel left beside it, all requested at once
    double run = 0.0, left[kMaxCluster];
    double* delta = deltas + (static_cast<size_t>(u) * ndeltas) * kHeadDim + tid;
    if (tid < kHeadDim) {
        run = sum_in[static_cast<size_t>(u) * kHeadDim + tid];
#pragma unroll
        for (int c = 0; c < kMaxCluster; ++c) left[c] = c < ndeltas ? delta[c * kHeadDim] : 0.0;
#pragma unroll
        for (int c = 0; c < kMaxCluster; ++c) {
            run += left[c];   // (in the order in which that kernel adds it)
            if (left[c] != 0.0) delta[c * kHeadDim] = 0.0;
        }
    }
    const double sum = run + block_sum_of_terms<kWideTermsDeep>(B, [&](int r) { return blk + static_cast<size_t>(r) * kRowVec; }, 1.0f / eps,
                                                                raw_anchor != 0, table, tid);
    if (tid < kHeadDim) {
        sum_out[static_cast<size_t>(u) * kHeadDim + tid] = sum;
        mu_sh[tid] = static_cast<float>(sum / static_cast<double>(n));
        mu[static_cast<size_t>(u) * kMuStride + tid] = mu_sh[tid];
    }
    __syncthreads();
    if (tid < 32) {
        float v = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) { const float w = mu_sh[tid * 4 + j]; v = fmaf(w, w, v); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (tid == 0) mu[static_cast<size_t>(u) * kMuStride + kHeadDim] = sqrtf(v);
    }
}

// One pass over the keys.  grid = (parts, U), rows_per_part a multiple of 128.  Four rows of a row group are requested
// together: 32 KB in flight per block, three blocks per SM, which HBM's latency needs (with one row at a time, 8 KB per
// block, and every lane finishing its row by itself the pass over 1.08 GB took 229 us; now 172).
__global__ void __launch_bounds__(kWideThreads, 3)
wide_score_kernel(const uint4* __restrict__ k_cache, const uint4* __restrict__ new_k, int len, int B, int N, float eps,
                  int rows_per_part, int nmax, const float* __restrict__ mu, float* __restrict__ scores) {
    grid_dependency_wait();
    const int u = blockIdx.y, n = len + B;
    const int g = threadIdx.x >> 3, t = threadIdx.x & 7;
    const int r0 = blockIdx.x * rows_per_part, r1 = min(n, r0 + rows_per_part);
    const float* m4 = mu + static_cast<size_t>(u) * kMuStride;
    float2 w[8];   // w[j] = channels j and 4 + j of the lane's first eight, w[4 + j] of its last eight: the chains of lane_dot16 in pairs
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float4 x = *reinterpret_cast<const float4*>(m4 + lane_channel(t, 8 * h)), y = *reinterpret_cast<const float4*>(m4 + lane_channel(t, 8 * h + 4));
        w[4 * h] = make_float2(x.x, y.x); w[4 * h + 1] = make_float2(x.y, y.y);
        w[4 * h + 2] = make_float2(x.z, y.z); w[4 * h + 3] = make_float2(x.w, y.w);
    }
    const float m = m4[kHeadDim];
    float* out = scores + static_cast<size_t>(u) * nmax;
#pragma unroll 1
    for (int base = r0; base < r1; base += kWideGroups * kWideDeep) {
        uint4 a[kWideDeep], b[kWideDeep];
#pragma unroll
        for (int k = 0; k < kWideDeep; ++k) {
            const int i = base + k * kWideGroups + g;
            a[k] = make_uint4(0, 0, 0, 0); b[k] = a[k];
            if (i < r1) {
                const uint4* row = concat_row(k_cache, new_k, u, i, len, B, N);
                a[k] = row[t]; b[k] = row[t + 8];
            }
        }
        float ss[kWideDeep];
        double dot[kWideDeep];
#pragma unroll
        for (int k = 0; k < kWideDeep; ++k) {   // lane_sumsq and lane_dot16 in packed pairs
            float x[16];
            unpack_row(a[k], b[k], x);
            float2 q = make_float2(0.f, 0.f), c0 = q, c1 = q;
#pragma unroll
            for (int j = 0; j < 8; ++j) { const float2 v = make_float2(x[j], x[8 + j]); q = __ffma2_rn(v, v, q); }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                c0 = __ffma2_rn(make_float2(x[j], x[4 + j]), w[j], c0);
                c1 = __ffma2_rn(make_float2(x[8 + j], x[12 + j]), w[4 + j], c1);
            }
            ss[k] = q.x + q.y;
            dot[k] = (static_cast<double>(c0.x) + static_cast<double>(c0.y)) + (static_cast<double>(c1.x) + static_cast<double>(c1.y));
        }
        const float r = sqrtf(group_sum_of4(ss, t));
        const float e = eviction_score(static_cast<float>(group_sum_of4(dot, t)), m, r, eps);
        const int i = base + (2 * (t & 1) + ((t >> 1) & 1)) * kWideGroups + g;
        if (t < 4 && i < r1) out[i] = e;
    }
}

// The keys of a unit's scores into shared memory, by 256 threads; tokens from `scored` on get the largest possible key (sliding window, Sec. 3.2).
// Four at a time where the rows of the scratch begin on 16 bytes: with the list below made by the same threads 256 x 16512 rows 900 -> 895 us a
// step, 200 x 12064 533 -> 528.
// The scores may have been written in the same launch, by other SMs: they are read past L1.
__device__ __forceinline__ void load_keys(const float* sc, int n, int scored, bool quads, uint32_t* keys, int tid) {
    if (quads) {   // the row begins on 16 bytes, and so does the next: the last quad's end is padding
        const float4* sc4 = reinterpret_cast<const float4*>(sc);
        uint4* k4 = reinterpret_cast<uint4*>(keys);
#pragma unroll 4
        for (int q = tid; 4 * q < n; q += kSelThreads) {
            const float4 e = __ldcg(&sc4[q]);
            const int i = 4 * q;
            k4[q] = make_uint4(i < scored ? order_key(e.x) : 0xffffffffu, i + 1 < scored ? order_key(e.y) : 0xffffffffu,
                               i + 2 < scored ? order_key(e.z) : 0xffffffffu, i + 3 < scored ? order_key(e.w) : 0xffffffffu);
        }
    } else {
#pragma unroll 8
        for (int i = tid; i < n; i += kSelThreads) keys[i] = i < scored ? order_key(__ldcg(&sc[i])) : 0xffffffffu;
    }
}
// Exact top-N of a unit (ties keep the older token), its kept-index list, and the evicted rows' terms off the running sum.
// grid = U; dynamic shared memory: n keys (padded to four), two bitmaps.
__global__ void __launch_bounds__(kSelThreads)
wide_select_kernel(const uint4* __restrict__ k_cache, const uint4* __restrict__ new_k, const float* __restrict__ scores,
                   int len, int B, int N, float eps, int raw_anchor, int nmax, int window, double* __restrict__ anchor_sum,
                   int32_t* __restrict__ kept_idx, int32_t* __restrict__ first_evicted, unsigned long long* __restrict__ moved_rows,
                   int32_t* status) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(128) SelectorScratch scratch;
    __shared__ __align__(16) double table[kTermWarps * kHeadDim];
    grid_dependency_wait();
    const int u = blockIdx.x, tid = threadIdx.x, n = len + B, nwords = (n + 31) >> 5;
    uint32_t* keys = reinterpret_cast<uint32_t*>(smem);
    uint32_t* bitmap = keys + ((n + 3) & ~3);
    Selector s(scratch, bitmap, bitmap + nwords);
    load_keys(scores + static_cast<size_t>(u) * nmax, n, n - window, (nmax & 3) == 0, keys, tid);
    __syncthreads();
    select_evicted(keys, n, n - N, tid, s);
    int* before = reinterpret_cast<int*>(s.eq);
    int* gone = reinterpret_cast<int*>(keys);   // (the keys are dead)
    const int first = list_evicted(n, tid, s, before, gone, n - N, status);
    double sum = 0.0;   // (requested in front of the rows)
    if (anchor_sum && tid < kHeadDim) sum = __ldcg(&anchor_sum[static_cast<size_t>(u) * kHeadDim + tid]);
    if (tid == 0) {
        first_evicted[u] = first;
        // block rows always move into the cache, cache rows only from the first evicted one on
        atomicAdd(moved_rows, static_cast<unsigned long long>(N - min(len, first)));
    }
    int32_t* out = kept_idx + static_cast<size_t>(u) * N;
#pragma unroll 4
    for (int i = tid; i < n; i += kSelThreads) {
        const uint32_t wd = bitmap[i >> 5], bit = 1u << (i & 31);
        if (!(wd & bit)) out[i - before[i >> 5] - __popc(wd & (bit - 1u))] = i;
    }
    if (!anchor_sum) return;   // (the staged path keeps no sum)
    const double terms = block_sum_of_terms<kWideTermsDeep>(n - N, [&](int r) { return concat_row(k_cache, new_k, u, gone[r], len, B, N); },
                                                            1.0f / eps, raw_anchor != 0, table, tid);
    if (tid < kHeadDim) anchor_sum[static_cast<size_t>(u) * kHeadDim + tid] = sum - terms;
}

// Step a4 in place by `segments` blocks per (unit, tensor): compact_kernel gives a tensor of a unit one block, which for fewer
// than 150 units leaves the SMs short of bytes in flight (a step on 100 x 10600 rows 318 -> 287 us, 60 x 10600 246 -> 193,
// 16 x 8600 below 60; the gather of 16 x 20100 rows was most of the 405 us that a step took, now 124).
// A segment owns a range [d0, d1) of destinations.  Rows move to lower places only, by at most m = (source of row d1 - 1) - (d1 -
// 1), so the sources of its first d1 - m - d0 rows lie under d1, and nobody but itself writes there.  The last m rows may come
// from where the next segment writes, and not from further on (segments.h: m <= kHaloRows <= kMinSegmentRows): the segment
// reads them into shared memory first and says so (flag, release); the next one waits for that flag before its first store.
// Segments are claimed from a counter in ascending order, so a block waits only for one that is already running, and that one
// waits for nothing before it sets its flag.  The host picks several segments only when at most kHaloRows rows are evicted per
// unit.  Waits are bounded: one that runs out sets the status word, and the block stores nothing.
__global__ void __launch_bounds__(kCompactThreads)
wide_move_kernel(uint4* k_cache, uint4* v_cache, const uint4* __restrict__ new_k, const uint4* __restrict__ new_v,
                 int len, int B, int N, int segments, const int32_t* __restrict__ kept_idx, const int32_t* __restrict__ first_evicted,
                 unsigned* __restrict__ move_sync, int32_t* status) {
    extern __shared__ __align__(128) uint4 smem_rows[];   // [kCompactRows] rows being moved, [kHaloRows] rows read ahead
    __shared__ int job_sh, go_sh;
    uint4* stage = smem_rows;
    uint4* halo = smem_rows + kCompactRows * kRowVec;
    grid_dependency_wait();
    const int tid = threadIdx.x;
    if (tid == 0) job_sh = static_cast<int>(atomicAdd(&move_sync[0], 1u));
    __syncthreads();
    const int job = job_sh, s = job % segments, tensor = (job / segments) & 1, u = job / (2 * segments);
    uint4* cache = tensor == 0 ? k_cache : v_cache;
    const uint4* block = tensor == 0 ? new_k : new_v;
    const int32_t* src_of = kept_idx + static_cast<size_t>(u) * N;
    unsigned* flag = move_sync + 1 + (u * 2 + tensor) * kMaxSegments;
    // cache rows in front of the first evicted row stay; block rows (index >= len) always move
    const int first = min(first_evicted[u], len);
    const Segment seg = segment_of(first, N, segments, s);
    const int d0 = seg.d0, d1 = seg.d1;
    const int m = rows_read_ahead(seg, N, d1 > d0 ? src_of[d1 - 1] : 0);
    auto load_row = [&](int d, int c) {
        const int src = src_of[d];
        return KD_ROW_OK(src, len + B, status) ? concat_row(cache, block, u, src, len, B, N)[c] : make_uint4(0, 0, 0, 0);
    };
    uint4* out = cache + static_cast<size_t>(u) * N * kRowVec;
    const bool fits = m <= kHaloRows;
    if (fits) for (int q = tid; q < m * kRowVec; q += kCompactThreads) halo[q] = load_row(d1 - m + (q >> 4), q & 15);
    __syncthreads();
    if (tid == 0) {
        bool ok = fits;
        if (!fits) atomicExch(status, kErrInternal);   // (cannot occur: at most kHaloRows rows are evicted)
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flag + s), "r"(1u) : "memory");
        if (s > 0) {
            unsigned seen = 0;
            for (uint32_t spin = 0; spin < (1u << 22) && ok; ++spin) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(flag + s - 1) : "memory");
                if (seen) break;
                __nanosleep(100);
                if ((spin & 255u) == 255u && *reinterpret_cast<volatile int32_t*>(status) != 0) ok = false;
            }
            if (!seen) { if (ok) atomicExch(status, kErrTimeout); ok = false; }
        }
        go_sh = ok;
    }
    // (the first chunk is requested while thread 0 waits)
    for (int base = d0; base < d1 - m; base += kCompactRows) {
        const int cnt = min(kCompactRows, d1 - m - base) * kRowVec;
        for (int q = tid; q < cnt; q += kCompactThreads) stage[q] = load_row(base + (q >> 4), q & 15);
        __syncthreads();
        if (!go_sh) return;
        for (int q = tid; q < cnt; q += kCompactThreads) out[base * kRowVec + q] = stage[q];
        __syncthreads();
    }
    __syncthreads();
    if (!go_sh) return;
    for (int q = tid; q < m * kRowVec; q += kCompactThreads) out[(d1 - m) * kRowVec + q] = halo[q];
}

}  // namespace kd
