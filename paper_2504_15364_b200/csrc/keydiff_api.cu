// Host side of the KeyDiff eviction-step library: context, argument validation, launch
// configuration and the extern "C" entry points declared in include/keydiff.h.
#include "../../include/keydiff.h"

#include <algorithm>
#include <cfloat>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <new>
#include <vector>

#include "common.cuh"
#include "staged_kernels.cuh"
#include "fused_kernel.cuh"
#include "slot_kernel.cuh"
#include "unit_kernel.cuh"
#include "wide_kernels.cuh"
#include "parts_kernel.cuh"

namespace {

thread_local int g_last_cuda_error = 0;

inline bool cuda_ok(cudaError_t e) {
    if (e == cudaSuccess) return true;
    g_last_cuda_error = static_cast<int>(e);
    return false;
}
#define KD_CUDA(call) do { if (!cuda_ok(call)) return KEYDIFF_ERR_CUDA; } while (0)

constexpr float kDefaultEps = 1e-8f;
// The eps that the kernels get.  Not below the smallest normal number: 1/eps must be finite (a key of zeros, or a row that is not there and
// counts as one, adds its zeros times min(1/||k||, 1/eps) to the anchor), and the kernels' products of norms are flushed to
// zero below it anyway.
inline float effective_eps(float eps) { return eps > 0.f ? std::max(eps, FLT_MIN) : kDefaultEps; }

// Launch-tuning aids (named in include/keydiff.h): read from the environment ONCE, by keydiff_create; a step
// never looks at the environment.  A value < 0 means "not set".
int env_int(const char* name) {
    const char* v = std::getenv(name);
    return (v && *v) ? std::atoi(v) : -1;
}

// Test hook (keydiff_debug_fail_alloc): the n-th device allocation from now on fails once.
int g_fail_alloc_countdown = 0;
cudaError_t kd_malloc(void** p, size_t bytes) {
    if (g_fail_alloc_countdown > 0 && --g_fail_alloc_countdown == 0) { *p = nullptr; return cudaErrorMemoryAllocation; }
    return cudaMalloc(p, bytes);
}
template <typename T> cudaError_t kd_malloc(T** p, size_t bytes) { return kd_malloc(reinterpret_cast<void**>(p), bytes); }
#ifdef KEYDIFF_DEBUG_CHECKS
// Test hook of the debug-checks build (keydiff_debug_fail_launch): the n-th kernel launch from now on is not made and returns an error.
int g_fail_launch_countdown = 0;
#endif
constexpr int kMaxSelectSmem = 200 * 1024;   // score keys of one unit must fit one CTA

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

struct keydiff_ctx {
    keydiff_config cfg;
    int U = 0;            // independent units = n_layers * batch * n_kv_heads
    int nmax = 0;         // N + max_block
    int len = 0;          // tokens currently cached (same for every unit)
    int splits = 1;       // row slices per unit in the staged anchor/score kernels
    int path = KEYDIFF_PATH_STAGED;
    int cluster = 1;            // fused path: CTAs per cluster
    int fused_smem_rows = 0;    // fused path: slice rows resident in shared memory
    int fused_nkeys = 0;        // fused path: key-table capacity
    int fused_smem_bytes = 0;
    int fused_max_clusters = 0; // co-resident clusters (grid = min(U, this) * cluster)
    int fused_reg_rows = 0;     // kernel instance: rows per row group kept in registers
    int unit_depth = 0;
    bool unit_blocks = false;   // one block per unit serves the step (either layout, on anchor_sum[0])
    bool slot_stream = false;   // slot reuse: the streaming kernel serves the step (cluster, fused_nkeys,
    int slot_ring_tiles = 0;    //   fused_smem_bytes, fused_max_clusters describe it)
    int slot_nwords = 0;
    int sm_count = 0;           // SMs of the ctx's device
    int tune_cluster = -1, tune_stagger_ns = -1, tune_late_ns = -1, tune_max_clusters = -1;   // KEYDIFF_* tuning aids as keydiff_create read them
    // running anchor of the fused path: sum of k/||k|| over the cached rows, per unit
    bool incremental = true;    // use it (one-pass kernel) when it is valid
    bool anchor_valid = false;  // the buffers describe the cache as the last evicting step left it
    int anchor_par = 0;         // which of the two sum buffers the next step reads
    int steps_since_full = 0;   // one-pass steps since the anchor was last recomputed from all rows
    double* anchor_sum[2] = {nullptr, nullptr};   // [U][128]
    double* anchor_delta = nullptr;               // [U][cluster][128]
    bool wide = false;                            // ordered layout, no cluster holds a unit: wide_kernels.cuh on anchor_sum[0]
    bool wide_single = false;                     // ordered layout, cluster kernel: steps that evict one row go to wide_kernels.cuh
    bool parts = false;                           // slot reuse: several blocks per unit serve a step (parts_kernel.cuh, on anchor_sum[0])
    unsigned* parts_done = nullptr;               // [U] zero between steps
    float* mu = nullptr;                          // [U][kMuStride], the running step's anchors
    unsigned* move_sync = nullptr;                // [1 + U * 2 * kMaxSegments] counter and flags of wide_move_kernel
    float eps = kDefaultEps;
    // device scratch
    double* partial = nullptr;        // [U][splits][128]
    float* norms = nullptr;           // [U][nmax]
    float* scores = nullptr;          // [U][nmax]
    int32_t* kept_idx = nullptr;      // [U][N]
    int32_t* first_evicted = nullptr; // [U]
    int32_t* status = nullptr;        // [1]
    unsigned long long* moved_rows = nullptr;   // [1] cumulative count of rows that changed position
    // unordered slot reuse: token position held by every slot, and the position of the next new token
    int32_t* pos = nullptr;           // [U][N]
    long long next_pos = 0;
    bool pos_stale = true;            // pos must be reset to the identity before the next step uses it
    // keydiff_evict_host only: two sets of staging buffers [U][max_block][128] bf16 filled on a copy stream
    // of the ctx, so that the block of step i+1 crosses the bus while the kernels of step i run
    void* stage_k[2] = {nullptr, nullptr};
    void* stage_v[2] = {nullptr, nullptr};
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_copied[2] = {nullptr, nullptr};   // the set's block has arrived
    cudaEvent_t ev_consumed[2] = {nullptr, nullptr}; // the step that read the set has finished
    bool consumed_recorded[2] = {false, false};
    int stage_next = 0;
    int32_t* kept_mirror = nullptr;   // set by keydiff_evict_host around its step: the fused kernels also write the
                                      // kept-index list there (the caller's pinned buffer), so no copy follows
};

namespace {

void free_scratch(keydiff_ctx* c) {
    cudaFree(c->partial); cudaFree(c->norms); cudaFree(c->scores); cudaFree(c->kept_idx);
    cudaFree(c->first_evicted); cudaFree(c->status); cudaFree(c->moved_rows);
    for (int b = 0; b < 2; ++b) {
        cudaFree(c->stage_k[b]); cudaFree(c->stage_v[b]);
        if (c->ev_copied[b]) cudaEventDestroy(c->ev_copied[b]);
        if (c->ev_consumed[b]) cudaEventDestroy(c->ev_consumed[b]);
    }
    if (c->copy_stream) cudaStreamDestroy(c->copy_stream);
    cudaFree(c->anchor_sum[0]); cudaFree(c->anchor_sum[1]); cudaFree(c->anchor_delta); cudaFree(c->pos);
    cudaFree(c->mu); cudaFree(c->move_sync); cudaFree(c->parts_done);
}

int check_step_args(const keydiff_ctx* ctx, const void* k_cache, const void* v_cache,
                    const void* new_k, const void* new_v, int32_t N, int32_t B, int32_t H, int32_t d) {
    if (!ctx || !k_cache || !v_cache || !new_k || !new_v) return KEYDIFF_ERR_INVALID_ARG;
    if (N != ctx->cfg.budget || H != ctx->cfg.n_kv_heads || d != ctx->cfg.head_dim) return KEYDIFF_ERR_INVALID_ARG;
    if (B < 1 || B > ctx->cfg.max_block) return KEYDIFF_ERR_INVALID_ARG;
    if (!aligned16(k_cache) || !aligned16(v_cache) || !aligned16(new_k) || !aligned16(new_v)) return KEYDIFF_ERR_INVALID_ARG;
    if (k_cache == v_cache || k_cache == new_k || v_cache == new_v) return KEYDIFF_ERR_INVALID_ARG;
    int dev = -1;
    KD_CUDA(cudaGetDevice(&dev));
    if (dev != ctx->cfg.device) return KEYDIFF_ERR_STATE;   // the ctx's device must be current
    return KEYDIFF_OK;
}

inline int prop_sm_count(const keydiff_ctx* c) { return c->sm_count > 0 ? c->sm_count : 148; }
inline bool slot_reuse(const keydiff_ctx* c) { return c->cfg.compaction == KEYDIFF_COMPACT_SLOT_REUSE; }
// The next step may go on from the running sum.
inline bool sum_valid(const keydiff_ctx* c) { return c->incremental && c->anchor_valid && c->steps_since_full < 1024; }

// Every kernel of a step goes through here: launched with programmatic stream serialization (it waits for the kernels in
// front of it by itself, see grid_dependency_wait), as clusters of `cluster` blocks when that is not 0.  early = false: an
// ordinary launch, for clusters that are to fill the device: placed while the kernel in front drains, SM by SM, they can
// be left without room for all of them at once (896 units of 4352 rows in clusters of five: +6 % of the step).
template <typename... P, typename... A>
cudaError_t launch(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, int cluster, bool early, A... args) {
#ifdef KEYDIFF_DEBUG_CHECKS
    if (g_fail_launch_countdown > 0 && --g_fail_launch_countdown == 0) return cudaErrorLaunchOutOfResources;
#endif
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int attrs = 0;
    if (early) {
        attr[attrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[attrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 0) {
        attr[attrs].id = cudaLaunchAttributeClusterDimension;
        attr[attrs].val.clusterDim.x = cluster; attr[attrs].val.clusterDim.y = 1; attr[attrs++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr; cfg.numAttrs = attrs;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

cudaError_t launch_append(uint4* kc, uint4* vc, const uint4* nk, const uint4* nv, int len, int B, int N, int U,
                          int32_t* pos, int next_pos, int pos_rows, cudaStream_t st) {
    using namespace kd;
    const int per_block = kAppendThreads * kAppendWords;
    return launch(append_kernel, dim3((B * kRowVec + per_block - 1) / per_block, U, 2), kAppendThreads, 0, st, 0, true,
                  kc, vc, nk, nv, len, B, N, pos, next_pos, pos_rows);
}

using FusedKernel = void (*)(kd::FusedParams);

// Kernel instance for `reg_rows` register-resident rows per row group (rounded up to one that is
// built); one_pass = the variant that takes the anchor from the running sum; few_pre = the variant that holds one
// block row per warp and kind across the K stores instead of four (one-pass kernels only).
template <bool kOnePass, int kPre>
FusedKernel fused_instance_of(int reg_rows, int* built) {
    using namespace kd;
    if (reg_rows <= 0) { *built = 0; return fused_evict_kernel<0, kOnePass, kPre>; }
    if (reg_rows <= 2) { *built = 2; return fused_evict_kernel<2, kOnePass, kPre>; }
    if (reg_rows <= 4) { *built = 4; return fused_evict_kernel<4, kOnePass, kPre>; }
    if (reg_rows <= 5) { *built = 5; return fused_evict_kernel<5, kOnePass, kPre>; }
    *built = 6; return fused_evict_kernel<6, kOnePass, kPre>;
}
FusedKernel fused_instance(int reg_rows, int* built, bool one_pass = false, bool few_pre = false) {
    if (!one_pass) return fused_instance_of<false, 4>(reg_rows, built);
    return few_pre ? fused_instance_of<true, 1>(reg_rows, built) : fused_instance_of<true, 4>(reg_rows, built);
}

// Lets a kernel be launched with as much shared memory as a block may have, its static part included.  The limit belongs to the
// kernel on the device, not to a context: it is always the same, so that a context created later for smaller units does not lower it
// under an earlier one.
template <typename Kernel>
bool allow_shared_memory(Kernel kern) {
    cudaFuncAttributes attr;
    return cuda_ok(cudaFuncGetAttributes(&attr, kern)) &&
           cuda_ok(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kd::kSmemLimit - static_cast<int>(attr.sharedSizeBytes)));
}

// Co-resident clusters of `C` CTAs of the kernel `kern` with `smem` bytes each.
template <typename Kernel>
int max_active_clusters(Kernel kern, int C, int smem, int sm_count) {
    using namespace kd;
    if (!allow_shared_memory(kern)) return 0;
    if (C > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C * sm_count);
    cfg.blockDim = dim3(kFusedThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    return n;
}

// Choose the cluster size and shared-memory split of the fused kernel for units of up to nmax
// rows; returns false if no cluster can hold a unit on chip.  Every cluster size from 1 to 16 is
// tried: how many clusters the device holds at once depends on how the SMs are grouped (on a B200
// 15 clusters fit both at 8 and at 9 CTAs, i.e. 120 or 135 SMs), and the estimated step time
//   ceil(U / clusters) * (fixed cost per unit + cost per slice row * slice rows)
// picks the winner (constants from per-phase timings of the kernel on a B200).
bool plan_fused(keydiff_ctx* c, int sm_count) {
    using namespace kd;
    constexpr double kUnitFixedUs = 10.0, kRowUs = 0.0165, kManyRegRowsUs = 4.5;   // (more than 4 register rows: spills)
    const int forced = c->tune_cluster;
    double best = 0.0;
    bool found = false;
    for (int C = 1; C <= kMaxCluster; ++C) {
        if (forced > 0 && C != forced) continue;
        const int per_cta = ((c->nmax + C - 1) / C + 3) & ~3;        // slices are multiples of 4 rows
        const int nkeys = C * per_cta;
        int sr = std::min(kMaxTiles * kTileRows, (per_cta + kTileRows - 1) / kTileRows * kTileRows);
        while (sr > 0 && fused_layout(sr, nkeys, C).total > kSmemLimit) sr -= kTileRows;
        if (sr <= 0) break;                                          // the key table alone does not fit
        if (sr + kMaxRegRows * kGroups < per_cta) continue;          // slice too long for this cluster size
        const int smem = fused_layout(sr, nkeys, C).total;
        int reg_rows = 0;
        const FusedKernel kern = fused_instance((std::max(0, per_cta - sr) + kGroups - 1) / kGroups, &reg_rows);
        const int clusters = max_active_clusters(kern, C, smem, sm_count);
        if (clusters < 1) continue;
        const int used = std::min(c->U, clusters);
        const double est = static_cast<double>((c->U + used - 1) / used) *
                           (kUnitFixedUs + kRowUs * per_cta + (reg_rows > 4 ? kManyRegRowsUs : 0.0));
        if (!found || est < 0.95 * best) {   // a larger cluster has to pay for its extra barrier traffic
            found = true; best = est;
            c->cluster = C; c->fused_smem_rows = sr; c->fused_nkeys = nkeys; c->fused_smem_bytes = smem;
            c->fused_max_clusters = clusters; c->fused_reg_rows = reg_rows;
        }
    }
    if (!found) return false;
    // the attributes of the three kernels of the chosen instance (the loop has set those of the two-pass kernel alone)
    int built = 0;
    return max_active_clusters(fused_instance(c->fused_reg_rows, &built, false), c->cluster, c->fused_smem_bytes, sm_count) >= 1 &&
           max_active_clusters(fused_instance(c->fused_reg_rows, &built, true, false), c->cluster, c->fused_smem_bytes, sm_count) >= 1 &&
           max_active_clusters(fused_instance(c->fused_reg_rows, &built, true, true), c->cluster, c->fused_smem_bytes, sm_count) >= 1;
}

// Slot reuse: cluster size and ring of the streaming kernel for units of up to nmax rows; false if it
// cannot serve the configuration (then the resident kernel or the staged path does).  Nothing has to
// stay on chip, so small clusters are possible and many units are in flight; the estimate
//   ceil(U / clusters) * (fixed cost per unit + cost per slice row * slice rows)
// picks the size (constants from per-phase timings on a B200: anchor, selection, lists and barriers are
// a fixed cost, the stream runs at the pace of one SM's share of the HBM bandwidth).
bool plan_slot_stream(keydiff_ctx* c, int sm_count) {
    using namespace kd;
    if (c->cfg.max_block > kSlotMaxBlock) return false;
    const int forced = c->tune_cluster;
    const int nwords = (c->nmax + 31) / 32;
    double best = 0.0;
    bool found = false;
    for (int C = 1; C <= kMaxCluster; ++C) {
        if (forced > 0 && C != forced) continue;
        const int per_cta = ((c->nmax + C - 1) / C + kTileRows - 1) / kTileRows * kTileRows;
        const int nkeys = C * per_cta;
        int ring = 3 * kFusedWarps;   // up to three tiles per warp in flight
        while (ring > 0 && slot_layout(ring, nkeys, nwords, c->cfg.max_block).total > kSmemLimit) ring -= kFusedWarps;
        if (ring <= 0) continue;
        const int smem = slot_layout(ring, nkeys, nwords, c->cfg.max_block).total;
        const int clusters = max_active_clusters(slot_evict_kernel, C, smem, sm_count);
        if (clusters < 1) continue;
        const int used = std::min(c->U, clusters);
        const double row_us = 256.0 / (6.0e6 / std::min(sm_count, used * C));   // one SM's share of ~6 TB/s, in bytes per us
        const double est = static_cast<double>((c->U + used - 1) / used) * ((C > 1 ? 11.0 : 9.0) + std::max(row_us, 0.0045) * per_cta);
        if (!found || est < best) {
            found = true; best = est;
            c->cluster = C; c->fused_nkeys = nkeys; c->fused_smem_bytes = smem; c->fused_max_clusters = clusters;
            c->slot_ring_tiles = ring; c->slot_nwords = nwords;
        }
    }
    if (!found) return false;
    return max_active_clusters(slot_evict_kernel, c->cluster, c->fused_smem_bytes, sm_count) >= 1;
}

int launch_slot_stream(keydiff_ctx* c, uint4* kc, uint4* vc, const uint4* nk, const uint4* nv, int B, cudaStream_t st) {
    using namespace kd;
    const int N = c->cfg.budget, n = c->len + B;
    if (!sum_valid(c)) {
        // the running sum of the cached rows, rebuilt from all of them: first evicting step, after appends,
        // set_len / reset, periodically against rounding drift, and every step when the caller asked for it
        const int rows_per_split = (c->len + c->splits - 1) / c->splits;
        KD_CUDA(launch(anchor_partial_kernel, dim3(c->splits, c->U), kStagedThreads, 0, st, 0, true, kc, nk, c->len, 0, N, c->eps, rows_per_split,
                       c->nmax, c->partial, static_cast<float*>(nullptr), c->cfg.anchor_mode == KEYDIFF_ANCHOR_RAW_MEAN));
        KD_CUDA(launch(anchor_fold_kernel, dim3(c->U), kHeadDim, 0, st, 0, true, c->partial, c->splits, c->anchor_sum[c->anchor_par],
                       c->anchor_delta, c->cluster));
        c->steps_since_full = 0;
    } else {
        ++c->steps_since_full;
    }
    SlotParams p;
    p.k_cache = kc; p.v_cache = vc; p.new_k = nk; p.new_v = nv;
    p.len = c->len; p.B = B; p.N = N; p.U = c->U; p.eps = c->eps;
    p.cluster = c->cluster;
    p.rows_per_cta = ((n + c->cluster - 1) / c->cluster + kTileRows - 1) / kTileRows * kTileRows;
    p.ring_tiles = c->slot_ring_tiles; p.nkeys = c->fused_nkeys; p.nwords = c->slot_nwords; p.nmax = c->nmax;
    p.max_block = c->cfg.max_block;
    p.scores = c->scores; p.kept_idx = c->kept_idx; p.first_evicted = c->first_evicted;
    p.moved_rows = c->moved_rows; p.status = c->status;
    p.anchor_in = c->anchor_sum[c->anchor_par];
    p.anchor_out = c->anchor_sum[c->anchor_par ^ 1];
    p.anchor_delta = c->anchor_delta;
    p.raw_anchor = c->cfg.anchor_mode == KEYDIFF_ANCHOR_RAW_MEAN;
    p.window = c->cfg.recent_window;
    p.pos = c->pos; p.next_pos = static_cast<int>(c->next_pos);
    p.kept_mirror = c->kept_mirror;
    const int nclusters = std::min(c->U, c->fused_max_clusters);
    // Start-up stagger: clusters launched together stream together and then select together, leaving HBM
    // idle in between.  When every cluster serves at least three units, starting cluster c a little later
    // than cluster c-1 (about half a unit's duration over all of them) spreads the phases; with fewer
    // units per cluster the delay would only postpone the end (sweep on a B200, by this kernel whichever serves
    // the shape now: 896 units of 4352 rows gain 12 %, 256 units of 8320 rows lose 3 %).
    p.stagger_ns = 0;
    p.late_ns = 0;
    {
        const double share = 6500.0 / std::min(prop_sm_count(c), nclusters * c->cluster);   // bytes per ns for one SM
        const double unit_ns = 9000.0 + static_cast<double>(p.rows_per_cta) * kRowBytes / share;
        if (nclusters > 1 && c->U >= 3 * nclusters) {
            p.stagger_ns = static_cast<unsigned>(0.55 * unit_ns / nclusters);
        } else if (c->U > nclusters && c->U % nclusters != 0) {
            // Two rounds, the second one partial: the clusters with a single unit start half a unit late, so that
            // they stream while the others are between their two streams (sweep on a B200: best at 0.4-0.6 of a
            // unit's duration; 256 units of 8320 rows gain 5 %, 224 units of 2176 rows 6 %)
            p.late_ns = static_cast<unsigned>(0.5 * unit_ns);
        }
    }
    if (c->tune_stagger_ns >= 0) p.stagger_ns = static_cast<unsigned>(c->tune_stagger_ns);
    if (c->tune_late_ns >= 0) p.late_ns = static_cast<unsigned>(c->tune_late_ns);
    KD_CUDA(launch(slot_evict_kernel, dim3(nclusters * c->cluster), kFusedThreads, c->fused_smem_bytes, st, c->cluster,
                   c->cluster == 1 || nclusters < c->fused_max_clusters, p));
    c->anchor_par ^= 1;
    c->anchor_valid = true;
    return KEYDIFF_OK;
}

// Many small units: one block per unit (unit_kernel.cuh).
constexpr int kSmemPerSm = 228 * 1024;   // shared memory of an SM; a block takes 1 KB beside its own
using UnitKernel = void (*)(kd::UnitParams);
UnitKernel unit_instance(const keydiff_ctx* c) {   // unit_depth 0, and the ordered layout: rows straight from global memory
    using namespace kd;
    if (!slot_reuse(c)) return unit_evict_kernel<false, false>;
    return c->unit_depth > 0 ? unit_evict_kernel<true, true> : unit_evict_kernel<true, false>;
}
// Where the block per unit is the faster kernel (us a step on a B200, unit kernel against cluster kernel):
//   ordered layout   short units: 300 x 364 rows 26 / 46, 3000 x 364 225 / 310, 1000 x 564 137 / 137; while two blocks per SM serve
//                    all units, longer ones: 150 x 764 33 / 43, 300 x 964 77 / 76, 450 x 764 99 / 82 (the second read of the
//                    keys then misses L2).  Fewer than 80 units leave SMs idle: 40 x 764 23 / 16; not at 220 rows, 13 / 13.
//   slot reuse       nothing but the block rows is read twice: 400 x 2112 54 / 69, 1000 x 4160 226 / 237, 800 x 1764 131 / 160.
//                    148 units or fewer: up to 1100 rows, 100 x 1064 17.8 / 18.5, 100 x 2112 25 / 23; a few units up to 600
//                    rows, 8 x 564 14 / 15, 8 x 1064 18 / 15.  Beyond 4500 rows only with many rounds
//                    of units: 600 x 8224 268 / 263, 1000 x 8224 377 / 388, 4096 x 8224 1381 / 1460.  (These are the two kernels alone;
//                    where several blocks per unit are faster than either, parts_are_faster says so: 1000 x 4160, 600 and 1000 x 8224.)
// The ring (rows through shared memory by the copy engine) needs shared memory that short units' blocks put to better use: 800 x
// 1764 142 with it, 131 without; with at most two blocks per SM, or long units, it is what keeps HBM busy: 224 x 2176 44 / 45,
// 200 x 4160 59 / 64, 1000 x 8224 376 / 437, 2000 x 8224 697 / 826.
bool plan_unit(keydiff_ctx* c) {
    using namespace kd;
    if (c->tune_cluster > 0 || c->cfg.max_block > kSlotMaxBlock) return false;
    const int n = c->nmax, U = c->U, sms = c->sm_count;
    bool use, ring = false;
    if (slot_reuse(c)) {
        use = n <= 600 || (n <= 1100 && U >= 60) || (n <= 4500 && U > sms) || U >= 6 * sms;
        ring = n > 4500 || (n > 1500 && U <= 2 * sms);
    } else {
        use = n <= 260 || (U >= 80 && (n <= 520 || (n <= 1000 && U <= 2 * sms)));
    }
    if (!use) return false;
    // two tiles per warp: 64 KB in flight per block, of which two have to fit an SM
    const int depth = ring ? 2 : 0, smem = unit_layout(n, c->cfg.max_block, depth).total;
    if (smem > kSmemLimit || (ring && 2 * (smem + 1024) > kSmemPerSm)) return false;
    c->cluster = 1;
    c->unit_depth = depth;
    c->fused_smem_bytes = smem;
    return allow_shared_memory(unit_instance(c));
}

int launch_unit(keydiff_ctx* c, uint4* kc, uint4* vc, const uint4* nk, const uint4* nv, int B, cudaStream_t st) {
    using namespace kd;
    UnitParams p;
    p.k_cache = kc; p.v_cache = vc; p.new_k = nk; p.new_v = nv;
    p.len = c->len; p.B = B; p.N = c->cfg.budget; p.nmax = c->nmax; p.max_block = c->cfg.max_block; p.eps = c->eps;
    p.depth = c->unit_depth;
    p.scores = c->scores; p.kept_idx = c->kept_idx; p.first_evicted = c->first_evicted;
    p.moved_rows = c->moved_rows; p.status = c->status;
    p.anchor_sum = c->anchor_sum[0];
    p.rebuild = !sum_valid(c);
    p.raw_anchor = c->cfg.anchor_mode == KEYDIFF_ANCHOR_RAW_MEAN;
    p.window = c->cfg.recent_window;
    p.pos = c->pos; p.next_pos = static_cast<int>(c->next_pos);
    p.kept_mirror = c->kept_mirror;
    KD_CUDA(launch(unit_instance(c), dim3(c->U), kUnitThreads, c->fused_smem_bytes, st, 0, true, p));
    c->anchor_valid = true;
    c->steps_since_full = p.rebuild ? 0 : c->steps_since_full + 1;
    return KEYDIFF_OK;
}

int launch_fused(keydiff_ctx* c, uint4* kc, uint4* vc, const uint4* nk, const uint4* nv, int B, cudaStream_t st) {
    if (c->unit_blocks) return launch_unit(c, kc, vc, nk, nv, B, st);
    if (c->slot_stream) return launch_slot_stream(c, kc, vc, nk, nv, B, st);
    using namespace kd;
    FusedParams p;
    p.k_cache = kc; p.v_cache = vc; p.new_k = nk; p.new_v = nv;
    p.len = c->len; p.B = B; p.N = c->cfg.budget; p.U = c->U; p.eps = c->eps;
    p.cluster = c->cluster;
    p.rows_per_cta = ((c->len + B + c->cluster - 1) / c->cluster + 3) & ~3;
    p.smem_rows = c->fused_smem_rows; p.nkeys = c->fused_nkeys; p.nmax = c->nmax;
    p.scores = c->scores; p.kept_idx = c->kept_idx; p.first_evicted = c->first_evicted;
    p.moved_rows = c->moved_rows; p.status = c->status;
    // The one-pass kernel needs the running anchor of the cache as it stands; every 1024 steps the
    // anchor is recomputed from all rows anyway, which sheds whatever rounding drift has built up.
    const bool one_pass = sum_valid(c);
    p.anchor_in = c->anchor_sum[c->anchor_par];
    p.anchor_out = c->anchor_sum[c->anchor_par ^ 1];
    p.anchor_delta = c->anchor_delta;
    p.raw_anchor = c->cfg.anchor_mode == KEYDIFF_ANCHOR_RAW_MEAN;
    p.window = c->cfg.recent_window;
    p.kept_mirror = c->kept_mirror;
    int nclusters = std::min(c->U, c->fused_max_clusters);
    if (c->tune_max_clusters > 0) nclusters = std::min(nclusters, c->tune_max_clusters);
    // Start-up stagger: somewhat less than one unit's duration spread evenly over the co-resident
    // clusters.  A unit moves 4 slices (K in, K out, V in, V out) per SM at roughly 60 GB/s per SM when
    // the other SMs are busy too, plus a few microseconds of arithmetic and barriers (a sweep of the
    // delay on a B200 put the best value at 0.7-0.95 of unit time / clusters for the large workloads).
    p.stagger_ns = 0;
    if (nclusters > 1 && c->U > nclusters) {
        const double unit_ns = 4.0 * p.rows_per_cta * kRowBytes / 60.0 + 6000.0;
        p.stagger_ns = static_cast<unsigned>(unit_ns / nclusters);
    }
    if (c->tune_stagger_ns >= 0) p.stagger_ns = static_cast<unsigned>(c->tune_stagger_ns);
    int built = 0;
    const bool few_pre = B <= 16 * c->cluster;   // a CTA's share of the block: at most one row per warp
    KD_CUDA(launch(fused_instance(c->fused_reg_rows, &built, one_pass, few_pre), dim3(nclusters * c->cluster), kFusedThreads,
                   c->fused_smem_bytes, st, c->cluster, c->cluster == 1 || nclusters < c->fused_max_clusters, p));
    c->anchor_par ^= 1;
    c->anchor_valid = true;
    c->steps_since_full = one_pass ? c->steps_since_full + 1 : 0;
    return KEYDIFF_OK;
}

// Ordered layout, units beyond a cluster: four launches on the running anchor (wide_kernels.cuh).
constexpr int kWideSelectSmem = 196 * 1024;   // beside the kernel's 31 KB of static shared memory
constexpr int kMoveSmem = (kd::kCompactRows + kd::kHaloRows) * kd::kRowBytes;
size_t wide_select_smem(int n) { return 4u * ((n + 3) & ~3) + 8u * ((n + 31) / 32); }

// Units that only clusters of ten or more hold leave the device room for seven to eleven of those (a B200: 105 to 112 SMs), and
// four launches that read the keys twice are the faster way (us a step, wide against cluster): 250 x 9500 rows 521 / 629, 500 x
// 11800 1244 / 1698, 60 x 10600 193 / 200, 16 x 8600 55 / 58; 200 x 8600, which clusters of nine hold, 387 / 384.  Few units need
// the gather in several blocks per unit, which wants at most kHaloRows evicted rows; without it 150 x 10600 408 / 469,
// 100 x 10600 318 / 321.
bool wide_is_faster(const keydiff_ctx* c) {
    return c->cfg.path == KEYDIFF_PATH_AUTO && c->tune_cluster <= 0 && c->cluster >= 10 && c->nmax > 8000 &&
           c->U >= (c->cfg.max_block <= kd::kHaloRows ? 16 : 120) && wide_select_smem(c->nmax) <= kWideSelectSmem;
}

// Token by token: a step that evicts one row moves only what lies behind it, half of the cache on average, and the cluster
// kernel's time hardly falls with the rows that move.  One evicted row, wide against cluster (us a step): 1024 x 8192 rows
// 1130 / 1477, 896 x 4096 539 / 658, 300 x 4096 212 / 240, 256 x 8192 347 / 391, 224 x 2048 92 / 104; but 400 x 1500 119 / 118,
// 160 x 8192 266 / 254 and 64 x 8192 124 / 119 (too few blocks in the gather).  Two evicted rows leave 1.04-1.1x at best where
// evictions are spread evenly and less where they are not; from four on the cluster kernel is the faster one.
bool wide_serves_single(const keydiff_ctx* c) {
    return c->cfg.path == KEYDIFF_PATH_AUTO && c->tune_cluster <= 0 && !c->unit_blocks && !slot_reuse(c) && 4 * c->U >= 5 * c->sm_count &&
           c->nmax >= 2000 && wide_select_smem(c->nmax) <= kWideSelectSmem;
}

bool single_evicted(const keydiff_ctx* c, int B) {
    return c->wide_single && c->len + B == c->cfg.budget + 1 && sum_valid(c);
}

bool capturing(cudaStream_t st) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &status) != cudaSuccess) { cudaGetLastError(); return false; }   // (the launch will say what is wrong)
    return status != cudaStreamCaptureStatusNone;
}

int launch_wide(keydiff_ctx* c, uint4* kc, uint4* vc, const uint4* nk, const uint4* nv, int B, cudaStream_t st) {
    using namespace kd;
    const int N = c->cfg.budget, n = c->len + B, U = c->U;
    const int raw = c->cfg.anchor_mode == KEYDIFF_ANCHOR_RAW_MEAN;
    // A step of single_evicted takes the sum from one buffer, and the deltas that the cluster kernel left beside it, and leaves it in the
    // other, as that kernel does: steps captured in a graph go on from replay to replay whichever kernels serve them.
    double* sum = c->anchor_sum[c->anchor_par];
    double* sum_out = c->wide_single ? c->anchor_sum[c->anchor_par ^ 1] : sum;
    // A captured step of a context that always runs here rebuilds the sum each time it is replayed: a graph replayed on a cache that was refilled
    // meanwhile (keydiff_reset and appends, keydiff_set_len) cannot see that the carried sum is another cache's, and such
    // contexts could always be replayed like that with the staged kernels.  It costs 240 of 1140 us on 256 units of 16512 rows.
    if (!sum_valid(c) || (c->wide && capturing(st))) {   // (never a step of single_evicted)
        const int rows_per_split = (c->len + c->splits - 1) / c->splits;
        KD_CUDA(launch(anchor_partial_kernel, dim3(c->splits, U), kStagedThreads, 0, st, 0, true, kc, nk, c->len, 0, N, c->eps, rows_per_split,
                       c->nmax, c->partial, static_cast<float*>(nullptr), raw));
        KD_CUDA(launch(anchor_fold_kernel, dim3(U), kHeadDim, 0, st, 0, true, c->partial, c->splits, sum,
                       static_cast<double*>(nullptr), 0));
        c->steps_since_full = 0;
    } else {
        ++c->steps_since_full;
    }
    c->anchor_valid = false;   // until all launches of the step are made: one that fails leaves the sum, or the deltas, of a step half done
    KD_CUDA(launch(wide_anchor_kernel, dim3(U), kWideThreads, 0, st, 0, true, nk, B, n, c->eps, raw, sum, sum_out,
                   c->anchor_delta, c->anchor_delta ? c->cluster : 0, c->mu, c->move_sync, false));
    // parts of at least 256 rows, enough of them for several rounds of three blocks per SM
    const long long rows = 1LL * U * n;
    const int want = static_cast<int>(rows / (12LL * c->sm_count));
    const int rows_per_part = std::min(2048, std::max(256, want)) / 128 * 128;
    KD_CUDA(launch(wide_score_kernel, dim3((n + rows_per_part - 1) / rows_per_part, U), kWideThreads, 0, st, 0, true, kc, nk, c->len, B, N,
                   c->eps, rows_per_part, c->nmax, c->mu, c->scores));
    KD_CUDA(launch(wide_select_kernel, dim3(U), kSelThreads, wide_select_smem(n), st, 0, true, kc, nk, c->scores, c->len, B, N, c->eps, raw,
                   c->nmax, c->cfg.recent_window, sum_out, c->kept_idx, c->first_evicted, c->moved_rows, c->status));
    // as many blocks as run at once, three per SM, of at least 512 rows each (150 x 10600 rows: 408 us with 300 blocks, 474
    // with 600; 100 x 10600: 318 with 200, 287 with 400, 328 with 600); one per unit and tensor when the rows that a
    // block reads ahead do not fit its shared memory
    const int segments = n - N > kHaloRows ? 1 : std::max(1, std::min({3 * c->sm_count / (2 * U), N / 512, kMaxSegments}));
    if (segments > 1)
        KD_CUDA(launch(wide_move_kernel, dim3(2 * U * segments), kCompactThreads, kMoveSmem, st, 0, true, kc, vc, nk, nv, c->len, B, N,
                       segments, c->kept_idx, c->first_evicted, c->move_sync, c->status));
    else
        KD_CUDA(launch(compact_kernel, dim3(2, U), kCompactThreads, 0, st, 0, true, kc, vc, nk, nv, c->len, B, N, c->kept_idx, c->first_evicted,
                       c->status));
    if (c->wide_single) c->anchor_par ^= 1;
    c->anchor_valid = true;
    return KEYDIFF_OK;
}

// Slot reuse: where several blocks per unit are the faster way for a step of B rows.  Us a step, the kernel that serves otherwise / parts; rows a step in
// brackets.  The lines are drawn so that of some 4700 shapes none loses more than 3 %, with blocks from one row to the largest that the context
// takes.
//   up to 4500 rows   otherwise a block per unit, at its best when its last round of units is full (fill: the share of the places of all rounds, three
//                     per SM, that have a unit): 512 x 2112 (64) 84 / 75, 1000 x 2112 (64) 144 / 138, 900 x 4160 (64) 212 / 187; 700 x 2112 (64),
//                     fill 0.79, 96 / 97.  Hardly more units than SMs: 160 x 2112 (64) 39 / 34, 177 x 2028 (128) 42 / 42; 224 x 2112 (64) 38 / 42.
//                     Large blocks make one chain longer, which shows on short units: 160 x 2812 (512) 68 / 66, 177 x 2412 (512) 64 / 66, 149 x 2964
//                     (1024) 97 / 102; 683 x 2284 (384), fill 0.77, 147 / 149, 600 x 2304 (256), 0.68, 126 / 122; 640 x 3828 (128) 160 /
//                     148.  Budgets under 1940: 160 x 2006 (256) up 5 %.
//   about 10000 rows  as long as three blocks of parts leave an SM its L1 (launch_parts): everywhere (150 x 8256 (64) 109 / 73, 236 x 8256 (64) 108 / 102, 512 x
//                     8256 (64) 223 / 196, 400 x 8704 (512) 231 / 227, 1025 x 9216 (1024) 736 / 653) but with nearly two units per SM
//                     (250 x 8448 (256) 127 / 132; the clusters are at their best with middling blocks, 236 x 4850 (200) 86 / 89, 400 x 6300 (200)
//                     151 / 155), up to ten per SM (1480 x 8256 (64) 561 / 533; many more, and HBM bounds both).
//   beyond            two blocks of parts per SM: hardly more units than one, two or three per SM: 160 x 16448 (64) 181 / 143, 183 x 12128 (128) 139 / 135, 345
//                     x 16640 (256) 332 / 321, 460 x 14256 (256) 392 / 369; 207 x 12128 (128) 143 / 149, 560 x 10428 (128) 299 / 320; from 17700 rows
//                     on earlier: 310 x 18128 (128) 353 / 325, 183 x 18128 (128) 195 / 203, 345 x 18128 (128) 335 / 359.
//   blocks of > 512   take the clusters longer (400 x 10412 (512) 261, 400 x 10540 (640) 322), so that the lines lie further out: 190 x 12640 (640) 240 /
//                     189, and there with 16 rows a step 132 / 125; 400 x 9916 (16) 188 / 179, but 400 x 11016 (16) 206 / 223.
//   up to an SM's worth of units a step is one chain, and this one is longer: 130 x 8256 59 / 67, 64 x 4160 26 / 28.
constexpr int kSmemBesideL1 = 196 * 1024;   // shared memory of an SM that leaves its L1 60 KB (the next larger split: 28)
bool parts_are_faster(const keydiff_ctx* c, int B) {
    const int U = c->U, sms = c->sm_count, n = c->nmax, N = c->cfg.budget, max_block = c->cfg.max_block;
    if (c->cfg.path != KEYDIFF_PATH_AUTO || !slot_reuse(c) || c->tune_cluster > 0 || max_block > kd::kSlotMaxBlock || U <= sms || n < 2000 || N < 1940 ||
        2 * (kd::parts_layout(n, max_block).total + 1024) > kSmemPerSm)
        return false;
    const auto within = [&](int from, int to) { return 100 * U > from * sms && 100 * U <= to * sms; };   // hundredths of a unit per SM
    if (n <= 4500) {
        const bool longer = N >= (B <= 512 ? 2600 : 3100);
        if (U <= 2 * sms) return (B <= 512 || longer) && within(100, B <= 160 || longer ? 120 : 110);
        const int rounds = (U + 3 * sms - 1) / (3 * sms);
        const double fill = static_cast<double>(U) / (static_cast<double>(rounds) * 3 * sms);
        return rounds > 1 && fill <= (B <= 64 || rounds > 2 || longer ? 0.77 : 0.70);
    }
    const bool large = max_block > 512, mid = max_block > 128 && max_block < 256;
    if (3 * (kd::parts_layout(large && !c->unit_blocks ? N + 64 : n, max_block).total + 1024) <= kSmemBesideL1)
        return within(100, mid && n <= 8000 ? 150 : 160) || (within(200, 1000) && !(mid && within(260, 296)));
    if (n > 17700) return within(100, large ? 130 : 122) || within(200, large ? 233 : 210);
    return within(100, large ? 135 : 124) || within(200, 233) || within(300, 311);
}

// The facts reported are those of a step of max_block rows as the context stands: on the running sum, or without it for good
// (keydiff_set_incremental), which a block per unit serves where it can.
bool parts_named(const keydiff_ctx* c) {
    return c->parts && (!c->unit_blocks || (c->incremental && parts_are_faster(c, c->cfg.max_block)));
}

// A block per unit rebuilds the sum by itself where that is needed, and goes on from the same sum.
bool parts_serve(const keydiff_ctx* c, int B) { return c->parts && (!c->unit_blocks || (sum_valid(c) && parts_are_faster(c, B))); }

int launch_parts(keydiff_ctx* c, uint4* kc, uint4* vc, const uint4* nk, const uint4* nv, int B, cudaStream_t st) {
    using namespace kd;
    const int N = c->cfg.budget, n = c->len + B, U = c->U;
    const bool raw = c->cfg.anchor_mode == KEYDIFF_ANCHOR_RAW_MEAN;
    double* sum = c->anchor_sum[0];
    if (!sum_valid(c)) {
        const int rows_per_split = (c->len + c->splits - 1) / c->splits;
        KD_CUDA(launch(anchor_partial_kernel, dim3(c->splits, U), kStagedThreads, 0, st, 0, true, kc, nk, c->len, 0, N, c->eps, rows_per_split,
                       c->nmax, c->partial, static_cast<float*>(nullptr), raw));
        KD_CUDA(launch(anchor_fold_kernel, dim3(U), kHeadDim, 0, st, 0, true, c->partial, c->splits, sum, static_cast<double*>(nullptr), 0));
        c->steps_since_full = 0;
    } else {
        ++c->steps_since_full;
    }
    c->anchor_valid = false;   // (as in launch_wide)
    KD_CUDA(launch(wide_anchor_kernel, dim3(U), kWideThreads, 0, st, 0, true, nk, B, n, c->eps, raw, sum, sum, static_cast<double*>(nullptr), 0, c->mu,
                   static_cast<unsigned*>(nullptr), true));
    PartsParams q;
    UnitParams& p = q.unit;
    p.k_cache = kc; p.v_cache = vc; p.new_k = nk; p.new_v = nv;
    p.len = c->len; p.B = B; p.N = N; p.nmax = c->nmax; p.max_block = c->cfg.max_block; p.eps = c->eps;
    p.depth = 0; p.rebuild = 0;
    p.scores = c->scores; p.kept_idx = c->kept_idx; p.first_evicted = c->first_evicted;
    p.moved_rows = c->moved_rows; p.status = c->status;
    p.anchor_sum = sum; p.raw_anchor = raw; p.window = c->cfg.recent_window;
    p.pos = c->pos; p.next_pos = static_cast<int>(c->next_pos);
    p.kept_mirror = c->kept_mirror;
    q.mu = c->mu; q.parts_done = c->parts_done;
    // a dozen parts per SM or more: 896 x 4352 rows 220 us a step, 227 with 512 rows a part; with fewer smaller ones: 224 x 2176 47 us, 50 with 1024
    q.rows_per_part = 1LL * U * n >= 1024LL * 12 * c->sm_count ? 1024 : 512;
    q.parts = (n + q.rows_per_part - 1) / q.rows_per_part;
    // Three blocks per SM have 98 KB of loads in flight, which L1 holds on their way: beyond kSmemBesideL1 it is down to 28 KB, and two blocks are faster than
    // three (400 x 10156 rows, 256 a step, 251 us against 262; 177 x 12128, 128 a step, 132 against 139).  They are given more than they use.
    int smem = parts_layout(n, c->cfg.max_block).total;
    if (3 * (smem + 1024) > kSmemBesideL1) smem = std::max(smem, kSmemPerSm / 3);
    KD_CUDA(launch(parts_kernel, dim3(q.parts, U), kUnitThreads, smem, st, 0, true, q));
    c->anchor_valid = true;
    return KEYDIFF_OK;
}

int launch_staged(keydiff_ctx* c, uint4* kc, uint4* vc, const uint4* nk, const uint4* nv, int B, cudaStream_t st) {
    using namespace kd;
    const int N = c->cfg.budget, n = c->len + B, U = c->U;
    const int rows_per_split = (n + c->splits - 1) / c->splits;
    const dim3 grid(c->splits, U);
    KD_CUDA(launch(anchor_partial_kernel, grid, kStagedThreads, 0, st, 0, true, kc, nk, c->len, B, N, c->eps, rows_per_split, c->nmax,
                   c->partial, c->norms, c->cfg.anchor_mode == KEYDIFF_ANCHOR_RAW_MEAN));
    KD_CUDA(launch(score_kernel, grid, kStagedThreads, 0, st, 0, true, kc, nk, c->len, B, N, c->eps, rows_per_split, c->nmax,
                   c->partial, c->norms, c->scores));
    if (!slot_reuse(c) && wide_select_smem(n) <= kWideSelectSmem)
        KD_CUDA(launch(wide_select_kernel, dim3(U), kSelThreads, wide_select_smem(n), st, 0, true, kc, nk, c->scores, c->len, B, N, c->eps, 0,
                       c->nmax, c->cfg.recent_window, static_cast<double*>(nullptr), c->kept_idx, c->first_evicted, c->moved_rows, c->status));
    else
        KD_CUDA(launch(select_kernel, dim3(U), kSelectThreads, static_cast<size_t>(n) * 4, st, 0, true, c->scores, n, N, c->nmax, c->len, c->kept_idx,
                       c->first_evicted, c->moved_rows, c->cfg.recent_window, slot_reuse(c) ? c->pos : nullptr,
                       static_cast<int>(c->next_pos)));
    if (slot_reuse(c))
        KD_CUDA(launch(slot_place_kernel, dim3(U), kCompactThreads, static_cast<size_t>(B) * 8, st, 0, true, kc, vc, nk, nv, c->len, B, N,
                       c->kept_idx, c->pos, static_cast<int>(c->next_pos), c->moved_rows));
    else
        KD_CUDA(launch(compact_kernel, dim3(2, U), kCompactThreads, 0, st, 0, true, kc, vc, nk, nv, c->len, B, N, c->kept_idx, c->first_evicted,
                       c->status));
    return KEYDIFF_OK;
}

bool alloc_wide(keydiff_ctx* c) {
    return kd_malloc(&c->mu, sizeof(float) * c->U * kd::kMuStride) == cudaSuccess &&
           kd_malloc(&c->move_sync, sizeof(unsigned) * (1 + c->U * 2 * kd::kMaxSegments)) == cudaSuccess &&
           allow_shared_memory(kd::wide_move_kernel);
}

int create_impl(const keydiff_config* cfg, keydiff_ctx** out) {
    if (!cfg || !out) return KEYDIFF_ERR_INVALID_ARG;
    if (cfg->n_layers < 1 || cfg->batch < 1 || cfg->n_kv_heads < 1 || cfg->budget < 1 || cfg->max_block < 1 ||
        cfg->device < 0 || cfg->eps < 0.f)
        return KEYDIFF_ERR_INVALID_ARG;
    if (cfg->path != KEYDIFF_PATH_AUTO && cfg->path != KEYDIFF_PATH_STAGED && cfg->path != KEYDIFF_PATH_FUSED)
        return KEYDIFF_ERR_INVALID_ARG;
    if (cfg->anchor_mode != KEYDIFF_ANCHOR_NORMALISED && cfg->anchor_mode != KEYDIFF_ANCHOR_RAW_MEAN) return KEYDIFF_ERR_INVALID_ARG;
    if (cfg->recent_window < 0 || cfg->recent_window > cfg->budget) return KEYDIFF_ERR_INVALID_ARG;
    if (cfg->compaction != KEYDIFF_COMPACT_ORDERED && cfg->compaction != KEYDIFF_COMPACT_SLOT_REUSE) return KEYDIFF_ERR_INVALID_ARG;
    if (cfg->dtype != KEYDIFF_BF16 || cfg->head_dim != kd::kHeadDim) return KEYDIFF_ERR_UNSUPPORTED;
    const long long U = 1LL * cfg->n_layers * cfg->batch * cfg->n_kv_heads;
    const long long nmax = 1LL * cfg->budget + cfg->max_block;
    if (U > 65535 || nmax > (1 << 30)) return KEYDIFF_ERR_UNSUPPORTED;   // gridDim.y limit of the staged kernels
    if (nmax * 4 > kMaxSelectSmem) return KEYDIFF_ERR_UNSUPPORTED;
    if (cfg->compaction == KEYDIFF_COMPACT_SLOT_REUSE && 8LL * cfg->max_block > kMaxSelectSmem) return KEYDIFF_ERR_UNSUPPORTED;

    int count = 0;
    KD_CUDA(cudaGetDeviceCount(&count));
    if (cfg->device >= count) return KEYDIFF_ERR_INVALID_ARG;
    cudaDeviceProp prop;
    KD_CUDA(cudaGetDeviceProperties(&prop, cfg->device));
    if (prop.major != 10) return KEYDIFF_ERR_UNSUPPORTED;   // built for sm_100a only; no fallback

    int prev = -1;
    KD_CUDA(cudaGetDevice(&prev));
    KD_CUDA(cudaSetDevice(cfg->device));

    keydiff_ctx* c = new (std::nothrow) keydiff_ctx();
    if (!c) { cudaSetDevice(prev); return KEYDIFF_ERR_ALLOC; }
    c->cfg = *cfg;
    c->U = static_cast<int>(U);
    c->nmax = static_cast<int>(nmax);
    c->eps = effective_eps(cfg->eps);
    c->sm_count = prop.multiProcessorCount;
    c->tune_cluster = env_int("KEYDIFF_CLUSTER_SIZE");
    c->tune_stagger_ns = env_int("KEYDIFF_STAGGER_NS");
    c->tune_late_ns = env_int("KEYDIFF_LATE_NS");
    c->tune_max_clusters = env_int("KEYDIFF_MAX_CLUSTERS");
    c->path = KEYDIFF_PATH_STAGED;
    // enough CTAs to fill 148 SMs a few times over, but at least 64 rows per slice
    const int want = (4 * prop.multiProcessorCount + c->U - 1) / c->U;
    c->splits = std::max(1, std::min({want, (c->nmax + 63) / 64, 64}));

    bool ok = true;
    ok = ok && kd_malloc(&c->partial, sizeof(double) * c->U * c->splits * kd::kHeadDim) == cudaSuccess;
    ok = ok && kd_malloc(&c->norms, sizeof(float) * U * nmax) == cudaSuccess;
    ok = ok && kd_malloc(&c->scores, sizeof(float) * U * nmax) == cudaSuccess;
    ok = ok && kd_malloc(&c->kept_idx, sizeof(int32_t) * U * cfg->budget) == cudaSuccess;
    ok = ok && kd_malloc(&c->first_evicted, sizeof(int32_t) * U) == cudaSuccess;
    ok = ok && kd_malloc(&c->status, sizeof(int32_t)) == cudaSuccess;
    ok = ok && kd_malloc(&c->moved_rows, sizeof(unsigned long long)) == cudaSuccess;
    if (ok) {
        ok = cudaMemset(c->scores, 0, sizeof(float) * U * nmax) == cudaSuccess &&
             cudaMemset(c->kept_idx, 0, sizeof(int32_t) * U * cfg->budget) == cudaSuccess &&
             cudaMemset(c->first_evicted, 0, sizeof(int32_t) * U) == cudaSuccess &&
             cudaMemset(c->status, 0, sizeof(int32_t)) == cudaSuccess &&
             cudaMemset(c->moved_rows, 0, sizeof(unsigned long long)) == cudaSuccess;
    }
    if (ok) {
        ok = allow_shared_memory(kd::select_kernel) && allow_shared_memory(kd::wide_select_kernel);
    }
    if (ok && cfg->compaction == KEYDIFF_COMPACT_SLOT_REUSE) {
        ok = kd_malloc(&c->pos, sizeof(int32_t) * U * cfg->budget) == cudaSuccess &&
             cudaMemset(c->pos, 0, sizeof(int32_t) * U * cfg->budget) == cudaSuccess &&
             allow_shared_memory(kd::slot_place_kernel);
    }
    if (ok) ok = cudaDeviceSynchronize() == cudaSuccess;
    if (ok && cfg->path != KEYDIFF_PATH_STAGED) {
        // slot reuse is served by the streaming kernel (or, where that cannot hold a unit's keys, by the staged path)
        c->unit_blocks = plan_unit(c);
        c->parts = parts_are_faster(c, c->unit_blocks ? 1 : cfg->max_block);   // (a block per unit takes the steps that it is faster at)
        c->slot_stream = slot_reuse(c) && !c->unit_blocks && !c->parts && plan_slot_stream(c, prop.multiProcessorCount);
        if (c->unit_blocks || c->parts || c->slot_stream || (!slot_reuse(c) && plan_fused(c, prop.multiProcessorCount) && !wide_is_faster(c))) {
            c->path = KEYDIFF_PATH_FUSED;
            const size_t sum_bytes = sizeof(double) * U * kd::kHeadDim;
            ok = kd_malloc(&c->anchor_sum[0], sum_bytes) == cudaSuccess && cudaMemset(c->anchor_sum[0], 0, sum_bytes) == cudaSuccess;
            if (c->parts)
                ok = ok && kd_malloc(&c->mu, sizeof(float) * U * kd::kMuStride) == cudaSuccess && kd_malloc(&c->parts_done, sizeof(unsigned) * U) == cudaSuccess &&
                     cudaMemset(c->parts_done, 0, sizeof(unsigned) * U) == cudaSuccess && allow_shared_memory(kd::parts_kernel);
            else if (!c->unit_blocks)   // (a unit's block, or its last part, keeps its sum in place)
                ok = ok && kd_malloc(&c->anchor_sum[1], sum_bytes) == cudaSuccess &&
                     kd_malloc(&c->anchor_delta, sum_bytes * c->cluster) == cudaSuccess &&
                     cudaMemset(c->anchor_sum[1], 0, sum_bytes) == cudaSuccess && cudaMemset(c->anchor_delta, 0, sum_bytes * c->cluster) == cudaSuccess;
            ok = ok && cudaDeviceSynchronize() == cudaSuccess;
            c->wide_single = wide_serves_single(c);
            if (c->wide_single) ok = ok && alloc_wide(c);
        } else if (cfg->path == KEYDIFF_PATH_AUTO && !slot_reuse(c) && wide_select_smem(c->nmax) <= kWideSelectSmem) {
            c->wide = true;
            c->cluster = 1;   // (a plan for clusters may have been made and found slower)
            const size_t sum_bytes = sizeof(double) * U * kd::kHeadDim;
            ok = kd_malloc(&c->anchor_sum[0], sum_bytes) == cudaSuccess &&
                 alloc_wide(c) && cudaMemset(c->anchor_sum[0], 0, sum_bytes) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
        } else if (cfg->path == KEYDIFF_PATH_FUSED) {
            free_scratch(c);
            delete c;
            cudaSetDevice(prev);
            return KEYDIFF_ERR_UNSUPPORTED;
        }
    }
    if (!ok) {
        g_last_cuda_error = static_cast<int>(cudaGetLastError());
        free_scratch(c);
        delete c;
        cudaSetDevice(prev);
        return KEYDIFF_ERR_ALLOC;
    }
    cudaSetDevice(prev);
    *out = c;
    return KEYDIFF_OK;
}
}  // namespace

extern "C" {

int keydiff_create(const keydiff_config* cfg, keydiff_ctx** out) {
    const int rc = create_impl(cfg, out);
    g_fail_alloc_countdown = 0;   // the test hook serves one keydiff_create
    return rc;
}

int keydiff_evict(keydiff_ctx* ctx, void* k_cache, void* v_cache, const void* new_k, const void* new_v,
                  int32_t budget_N, int32_t block_B, int32_t n_kv_heads, int32_t head_dim, void* stream) {
    const int rc = check_step_args(ctx, k_cache, v_cache, new_k, new_v, budget_N, block_B, n_kv_heads, head_dim);
    if (rc != KEYDIFF_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint4* kc = static_cast<uint4*>(k_cache);
    uint4* vc = static_cast<uint4*>(v_cache);
    const uint4* nk = static_cast<const uint4*>(new_k);
    const uint4* nv = static_cast<const uint4*>(new_v);
    const int N = ctx->cfg.budget, n = ctx->len + block_B;
    if (slot_reuse(ctx)) {
        if (ctx->next_pos + block_B > 0x7fffffffLL) return KEYDIFF_ERR_STATE;   // positions are int32
        if (ctx->pos_stale && ctx->len > 0) {
            // the cache as the caller declared it: slot s holds token s (for an empty cache the append writes it, and an
            // evicting step fills every slot)
            const int total = ctx->U * N;
            KD_CUDA(launch(kd::pos_iota_kernel, dim3((total + 255) / 256), 256, 0, st, 0, true, ctx->pos, N, total));
        }
    }
    if (n <= N) {
        // Sec. 2.3: the budget is not exceeded, nothing is evicted
        KD_CUDA(launch_append(kc, vc, nk, nv, ctx->len, block_B, N, ctx->U, ctx->pos, static_cast<int>(ctx->next_pos),
                              ctx->pos_stale && ctx->len == 0 ? N : block_B, st));
        ctx->pos_stale = false;
        ctx->len = n;
        ctx->next_pos += block_B;
        ctx->anchor_valid = false;   // the appended rows are not in the running anchor
        return KEYDIFF_OK;
    }
    const bool single = single_evicted(ctx, block_B);
    const int lrc = parts_serve(ctx, block_B) ? launch_parts(ctx, kc, vc, nk, nv, block_B, st) : ctx->path == KEYDIFF_PATH_FUSED && !single ? launch_fused(ctx, kc, vc, nk, nv, block_B, st)
                     : ctx->wide || single              ? launch_wide(ctx, kc, vc, nk, nv, block_B, st)
                                                        : launch_staged(ctx, kc, vc, nk, nv, block_B, st);
    if (lrc != KEYDIFF_OK) return lrc;
    ctx->pos_stale = false;
    ctx->len = N;
    ctx->next_pos += block_B;
    return KEYDIFF_OK;
}

int keydiff_evict_host(keydiff_ctx* ctx, void* k_cache, void* v_cache, const void* new_k_host, const void* new_v_host,
                       int32_t budget_N, int32_t block_B, int32_t n_kv_heads, int32_t head_dim,
                       int32_t* kept_idx_host, int32_t* status_host, void* stream) {
    if (!ctx || !new_k_host || !new_v_host) return KEYDIFF_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!ctx->copy_stream) {
        const size_t bytes = static_cast<size_t>(ctx->U) * ctx->cfg.max_block * kd::kRowBytes;
        bool ok = cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking) == cudaSuccess;
        for (int b = 0; b < 2 && ok; ++b)
            ok = cudaMalloc(&ctx->stage_k[b], bytes) == cudaSuccess && cudaMalloc(&ctx->stage_v[b], bytes) == cudaSuccess &&
                 cudaEventCreateWithFlags(&ctx->ev_copied[b], cudaEventDisableTiming) == cudaSuccess &&
                 cudaEventCreateWithFlags(&ctx->ev_consumed[b], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) {
            g_last_cuda_error = static_cast<int>(cudaGetLastError());
            for (int b = 0; b < 2; ++b) {
                cudaFree(ctx->stage_k[b]); cudaFree(ctx->stage_v[b]); ctx->stage_k[b] = ctx->stage_v[b] = nullptr;
                if (ctx->ev_copied[b]) { cudaEventDestroy(ctx->ev_copied[b]); ctx->ev_copied[b] = nullptr; }
                if (ctx->ev_consumed[b]) { cudaEventDestroy(ctx->ev_consumed[b]); ctx->ev_consumed[b] = nullptr; }
            }
            if (ctx->copy_stream) { cudaStreamDestroy(ctx->copy_stream); ctx->copy_stream = nullptr; }
            return KEYDIFF_ERR_ALLOC;
        }
    }
    const int b = ctx->stage_next;
    const int rc = check_step_args(ctx, k_cache, v_cache, ctx->stage_k[b], ctx->stage_v[b], budget_N, block_B, n_kv_heads, head_dim);
    if (rc != KEYDIFF_OK) return rc;
    const size_t bytes = static_cast<size_t>(ctx->U) * block_B * kd::kRowBytes;
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    KD_CUDA(cudaStreamIsCapturing(st, &capturing));
    if (capturing == cudaStreamCaptureStatusNone) {
        // the copy does not wait for what is queued on `st`: only for the step that last read this set
        if (ctx->consumed_recorded[b]) KD_CUDA(cudaStreamWaitEvent(ctx->copy_stream, ctx->ev_consumed[b], 0));
        KD_CUDA(cudaMemcpyAsync(ctx->stage_k[b], new_k_host, bytes, cudaMemcpyHostToDevice, ctx->copy_stream));
        KD_CUDA(cudaMemcpyAsync(ctx->stage_v[b], new_v_host, bytes, cudaMemcpyHostToDevice, ctx->copy_stream));
        KD_CUDA(cudaEventRecord(ctx->ev_copied[b], ctx->copy_stream));
        KD_CUDA(cudaStreamWaitEvent(st, ctx->ev_copied[b], 0));
    } else {
        // inside a stream capture everything stays on the captured stream
        KD_CUDA(cudaMemcpyAsync(ctx->stage_k[b], new_k_host, bytes, cudaMemcpyHostToDevice, st));
        KD_CUDA(cudaMemcpyAsync(ctx->stage_v[b], new_v_host, bytes, cudaMemcpyHostToDevice, st));
    }
    // Pinned host memory has a device alias: on the fused path an evicting step writes the kept-index list
    // there itself, as it writes it to scratch, so the list crosses the bus during the step
    bool mirrored = false;
    if (kept_idx_host && ctx->path == KEYDIFF_PATH_FUSED && ctx->len + block_B > ctx->cfg.budget && !single_evicted(ctx, block_B)) {
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, kept_idx_host) == cudaSuccess && attr.type == cudaMemoryTypeHost && attr.devicePointer) {
            ctx->kept_mirror = static_cast<int32_t*>(attr.devicePointer);
            mirrored = true;
        } else {
            cudaGetLastError();
        }
    }
    const int erc = keydiff_evict(ctx, k_cache, v_cache, ctx->stage_k[b], ctx->stage_v[b], budget_N, block_B, n_kv_heads,
                                  head_dim, stream);
    ctx->kept_mirror = nullptr;
    if (erc != KEYDIFF_OK) return erc;
    if (capturing == cudaStreamCaptureStatusNone) {
        KD_CUDA(cudaEventRecord(ctx->ev_consumed[b], st));
        ctx->consumed_recorded[b] = true;
    }
    ctx->stage_next = b ^ 1;
    if (kept_idx_host && !mirrored)
        KD_CUDA(cudaMemcpyAsync(kept_idx_host, ctx->kept_idx, sizeof(int32_t) * ctx->U * ctx->cfg.budget,
                                cudaMemcpyDeviceToHost, st));
    if (status_host)
        KD_CUDA(cudaMemcpyAsync(status_host, ctx->status, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    return KEYDIFF_OK;
}

int keydiff_destroy(keydiff_ctx* ctx) {
    if (!ctx) return KEYDIFF_OK;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(ctx->cfg.device);
    cudaDeviceSynchronize();
    free_scratch(ctx);
    if (prev >= 0) cudaSetDevice(prev);
    delete ctx;
    return KEYDIFF_OK;
}

int keydiff_reset(keydiff_ctx* ctx) {
    if (!ctx) return KEYDIFF_ERR_INVALID_ARG;
    ctx->len = 0;
    ctx->anchor_valid = false;
    ctx->next_pos = 0;
    ctx->pos_stale = true;
    return KEYDIFF_OK;
}

int keydiff_set_incremental(keydiff_ctx* ctx, int32_t on) {
    if (!ctx) return KEYDIFF_ERR_INVALID_ARG;
    ctx->incremental = on != 0;
    return KEYDIFF_OK;
}

int keydiff_get_len(const keydiff_ctx* ctx, int32_t* len_out) {
    if (!ctx || !len_out) return KEYDIFF_ERR_INVALID_ARG;
    *len_out = ctx->len;
    return KEYDIFF_OK;
}

int keydiff_set_len(keydiff_ctx* ctx, int32_t len) {
    if (!ctx || len < 0 || len > ctx->cfg.budget) return KEYDIFF_ERR_INVALID_ARG;
    ctx->len = len;
    ctx->anchor_valid = false;   // the caller brought its own cache contents
    ctx->next_pos = len;         // ... which are tokens 0 .. len-1 in token order
    ctx->pos_stale = true;
    return KEYDIFF_OK;
}

int keydiff_get_scratch(const keydiff_ctx* ctx, const float** scores, const int32_t** kept_idx,
                        const int32_t** first_evicted, const int32_t** status) {
    if (!ctx) return KEYDIFF_ERR_INVALID_ARG;
    if (scores) *scores = ctx->scores;
    if (kept_idx) *kept_idx = ctx->kept_idx;
    if (first_evicted) *first_evicted = ctx->first_evicted;
    if (status) *status = ctx->status;
    return KEYDIFF_OK;
}

int keydiff_get_positions(const keydiff_ctx* ctx, const int32_t** pos, long long* next_pos) {
    if (!ctx) return KEYDIFF_ERR_INVALID_ARG;
    if (!slot_reuse(ctx)) return KEYDIFF_ERR_STATE;
    if (pos) *pos = ctx->pos;
    if (next_pos) *next_pos = ctx->next_pos;
    return KEYDIFF_OK;
}

int keydiff_set_positions(keydiff_ctx* ctx, const int32_t* pos_device, int32_t len, long long next_pos, void* stream) {
    if (!ctx || len < 0 || len > ctx->cfg.budget || next_pos < len || next_pos > 0x7fffffffLL) return KEYDIFF_ERR_INVALID_ARG;
    if (!slot_reuse(ctx)) return KEYDIFF_ERR_STATE;
    int dev = -1;
    KD_CUDA(cudaGetDevice(&dev));
    if (dev != ctx->cfg.device) return KEYDIFF_ERR_STATE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int total = ctx->U * ctx->cfg.budget;
    if (pos_device) {
        KD_CUDA(cudaMemcpyAsync(ctx->pos, pos_device, sizeof(int32_t) * total, cudaMemcpyDeviceToDevice, st));
    } else {
        KD_CUDA(launch(kd::pos_iota_kernel, dim3((total + 255) / 256), 256, 0, st, 0, true, ctx->pos, ctx->cfg.budget, total));
    }
    ctx->len = len;
    ctx->next_pos = next_pos;
    ctx->pos_stale = false;
    ctx->anchor_valid = false;   // the caller brought its own cache contents
    return KEYDIFF_OK;
}

int keydiff_get_moved_rows(const keydiff_ctx* ctx, const unsigned long long** counter) {
    if (!ctx || !counter) return KEYDIFF_ERR_INVALID_ARG;
    *counter = ctx->moved_rows;
    return KEYDIFF_OK;
}

int keydiff_get_launch_info(const keydiff_ctx* ctx, int32_t* path, int32_t* launches_per_step, int32_t* cluster_size) {
    if (!ctx) return KEYDIFF_ERR_INVALID_ARG;
    if (path) *path = ctx->path;
    if (launches_per_step) *launches_per_step = parts_named(ctx) ? 2 : ctx->path == KEYDIFF_PATH_FUSED ? 1 : 4;
    if (cluster_size) *cluster_size = ctx->cluster;
    return KEYDIFF_OK;
}

const char* keydiff_get_kernel_name(const keydiff_ctx* ctx) {
    if (!ctx) return "";
    if (parts_named(ctx)) return "parts_kernel";
    if (ctx->unit_blocks) return "unit_evict_kernel";
    if (ctx->slot_stream) return "slot_evict_kernel";
    if (ctx->path == KEYDIFF_PATH_FUSED) return "fused_evict_kernel";
    return ctx->wide ? "wide kernels (4 launches)" : "staged kernels (4 launches)";
}

const char* keydiff_strerror(int code) {
    switch (code) {
        case KEYDIFF_OK: return "ok";
        case KEYDIFF_ERR_INVALID_ARG: return "invalid argument";
        case KEYDIFF_ERR_UNSUPPORTED: return "unsupported configuration or device";
        case KEYDIFF_ERR_ALLOC: return "device memory allocation failed";
        case KEYDIFF_ERR_CUDA: return "CUDA runtime error";
        case KEYDIFF_ERR_STATE: return "call not valid in the current state (is the ctx's device current?)";
        case KEYDIFF_ERR_TIMEOUT: return "bounded device-side wait expired";
        case KEYDIFF_ERR_TOO_LARGE: return "request needs more scratch than the built-in static scratch array holds";
        case KEYDIFF_ERR_INTERNAL: return "a kernel computed a row index outside its tensor (debug-checks build)";
        default: return "unknown keydiff status";
    }
}

int keydiff_last_cuda_error(void) { return g_last_cuda_error; }

int keydiff_selftest_bounded_wait(int32_t* status_device, int32_t polls, void* stream) {
    if (!status_device || polls < 1 || polls > 4096) return KEYDIFF_ERR_INVALID_ARG;
    kd::bounded_wait_selftest_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream)>>>(status_device, static_cast<uint32_t>(polls));
    KD_CUDA(cudaGetLastError());
    return KEYDIFF_OK;
}

#ifdef KEYDIFF_DEBUG_CHECKS
__attribute__((visibility("default"))) int keydiff_debug_fail_launch(int32_t nth) {
    if (nth < 0) return KEYDIFF_ERR_INVALID_ARG;
    g_fail_launch_countdown = nth;
    return KEYDIFF_OK;
}

// Debug-checks build only: the running sum of the cached rows' anchor terms as the latest step left it, [U][128] doubles, to out_host.
// KEYDIFF_ERR_STATE when the next step would rebuild it.  Synchronises the device.
__attribute__((visibility("default"))) int keydiff_debug_anchor_sum(const keydiff_ctx* ctx, double* out_host) {
    if (!ctx || !out_host) return KEYDIFF_ERR_INVALID_ARG;
    if (!ctx->anchor_valid) return KEYDIFF_ERR_STATE;
    const size_t units = ctx->U, ranks = ctx->anchor_delta ? ctx->cluster : 0;
    std::vector<double> deltas(units * ranks * kd::kHeadDim);
    KD_CUDA(cudaDeviceSynchronize());
    KD_CUDA(cudaMemcpy(out_host, ctx->anchor_sum[ctx->anchor_par], sizeof(double) * units * kd::kHeadDim, cudaMemcpyDeviceToHost));
    if (ranks > 0) KD_CUDA(cudaMemcpy(deltas.data(), ctx->anchor_delta, sizeof(double) * deltas.size(), cudaMemcpyDeviceToHost));
    for (size_t i = 0; i < deltas.size(); ++i) out_host[i / kd::kHeadDim / ranks * kd::kHeadDim + i % kd::kHeadDim] += deltas[i];
    return KEYDIFF_OK;
}
#endif

#ifdef KEYDIFF_PHASE_STAMPS
// Phase-stamp build only: copies the per-CTA, per-phase nanosecond totals of the fused kernel to out_host
// ([ctas][16] unsigned 64-bit, ctas <= 2368) and optionally clears them.  Synchronises the device.
__attribute__((visibility("default"))) int keydiff_debug_phase_ns(unsigned long long* out_host, int32_t ctas, int32_t reset) {
    if (!out_host || ctas < 1 || ctas > kd::kMaxStampCtas) return KEYDIFF_ERR_INVALID_ARG;
    KD_CUDA(cudaDeviceSynchronize());
    KD_CUDA(cudaMemcpyFromSymbol(out_host, kd::g_phase_ns, sizeof(unsigned long long) * ctas * kd::kMaxPhases));
    if (reset) {
        void* addr = nullptr;
        KD_CUDA(cudaGetSymbolAddress(&addr, kd::g_phase_ns));
        KD_CUDA(cudaMemset(addr, 0, sizeof(unsigned long long) * kd::kMaxStampCtas * kd::kMaxPhases));
    }
    return KEYDIFF_OK;
}
#endif

int keydiff_debug_fail_alloc(int32_t nth) {
    if (nth < 0) return KEYDIFF_ERR_INVALID_ARG;
    g_fail_alloc_countdown = nth;
    return KEYDIFF_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// Allocation-free entry point.
//
// Some callers cannot allocate device memory at all: code running inside a serving process whose
// memory pool already owns the whole GPU (any cudaMalloc would fail or fragment the pool), plugin
// code that is only handed tensors, and set-ups where allocation is forbidden after start-up
// because it synchronises the device.  keydiff_create needs cudaMalloc for its scratch, so such
// callers get keydiff_evict_static instead: the same staged kernels, with their scratch carved
// out of one array that is part of the library image.
//
// The array's name below is, in host code, only a handle for the runtime -- it is NOT a device
// address, and a kernel handed it directly would read the wrong memory.  The device address is
// looked up once per device with cudaGetSymbolAddress (with that device current) and cached.
namespace {

constexpr size_t kStaticScratchBytes = 16u << 20;   // 16 MiB, resident on every GPU that loads the library
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

constexpr int kMaxStaticDevices = 64;
unsigned char* g_static_scratch_addr[kMaxStaticDevices] = {};   // device address per device ordinal
std::mutex g_static_mutex;

// Resolve (once per device) the device address of the scratch array for the CURRENT device and
// raise the select kernel's dynamic shared-memory limit there.
int static_scratch_for_current_device(unsigned char** out) {
    int dev = -1;
    KD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxStaticDevices) return KEYDIFF_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_scratch_addr[dev]) {
        int major = 0;
        KD_CUDA(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
        if (major != 10) return KEYDIFF_ERR_UNSUPPORTED;
        void* addr = nullptr;
        KD_CUDA(cudaGetSymbolAddress(&addr, g_static_scratch));
        if (!allow_shared_memory(kd::select_kernel) || !allow_shared_memory(kd::wide_select_kernel)) return KEYDIFF_ERR_CUDA;
        g_static_scratch_addr[dev] = static_cast<unsigned char*>(addr);
    }
    *out = g_static_scratch_addr[dev];
    return KEYDIFF_OK;
}

inline size_t round256(size_t b) { return (b + 255) & ~static_cast<size_t>(255); }

}  // namespace

extern "C" int keydiff_evict_static(void* k_cache, void* v_cache, const void* new_k, const void* new_v,
                                    int32_t len, int32_t budget_N, int32_t block_B, int32_t n_units,
                                    int32_t head_dim, float eps, void* stream) {
    using namespace kd;
    if (!k_cache || !v_cache || !new_k || !new_v) return KEYDIFF_ERR_INVALID_ARG;
    if (!aligned16(k_cache) || !aligned16(v_cache) || !aligned16(new_k) || !aligned16(new_v)) return KEYDIFF_ERR_INVALID_ARG;
    if (k_cache == v_cache || k_cache == new_k || v_cache == new_v) return KEYDIFF_ERR_INVALID_ARG;
    if (budget_N < 1 || block_B < 1 || n_units < 1 || len < 0 || len > budget_N || eps < 0.f) return KEYDIFF_ERR_INVALID_ARG;
    if (head_dim != kHeadDim) return KEYDIFF_ERR_UNSUPPORTED;
    if (n_units > 65535) return KEYDIFF_ERR_TOO_LARGE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint4* kc = static_cast<uint4*>(k_cache);
    uint4* vc = static_cast<uint4*>(v_cache);
    const uint4* nk = static_cast<const uint4*>(new_k);
    const uint4* nv = static_cast<const uint4*>(new_v);
    const long long n = static_cast<long long>(len) + block_B;
    const int N = budget_N, U = n_units;
    // set-up (first call on a device only) comes before anything is enqueued, whatever kind of step this is
    unsigned char* base = nullptr;
    const int src = static_scratch_for_current_device(&base);
    if (src != KEYDIFF_OK) return src;
    {
        // the tensors must live on the current device: the scratch address was looked up for it
        int dev = -1;
        KD_CUDA(cudaGetDevice(&dev));
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, k_cache) != cudaSuccess) { cudaGetLastError(); return KEYDIFF_ERR_INVALID_ARG; }
        if (attr.type == cudaMemoryTypeDevice && attr.device != dev) return KEYDIFF_ERR_STATE;
    }
    if (n <= N) {   // budget not exceeded: plain append, no scratch involved
        KD_CUDA(launch_append(kc, vc, nk, nv, len, block_B, N, U, nullptr, 0, 0, st));
        return KEYDIFF_OK;
    }
    if (n * 4 > kMaxSelectSmem) return KEYDIFF_ERR_TOO_LARGE;
    const int splits = static_cast<int>(std::max(1LL, std::min({(592LL + U - 1) / U, (n + 63) / 64, 64LL})));
    // carve the static array: [moved counter][partials][norms][scores][kept_idx][first_evicted]
    size_t off = 0;
    auto take = [&off](size_t bytes) { const size_t o = off; off += round256(bytes); return o; };
    const size_t o_moved = take(sizeof(unsigned long long));
    const size_t o_partial = take(sizeof(double) * U * splits * kHeadDim);
    const size_t o_norms = take(sizeof(float) * U * n);
    const size_t o_scores = take(sizeof(float) * U * n);
    const size_t o_kept = take(sizeof(int32_t) * static_cast<size_t>(U) * N);
    const size_t o_first = take(sizeof(int32_t) * U);
    if (off > kStaticScratchBytes) return KEYDIFF_ERR_TOO_LARGE;
    unsigned long long* moved = reinterpret_cast<unsigned long long*>(base + o_moved);
    double* partial = reinterpret_cast<double*>(base + o_partial);
    float* norms = reinterpret_cast<float*>(base + o_norms);
    float* scores = reinterpret_cast<float*>(base + o_scores);
    int32_t* kept = reinterpret_cast<int32_t*>(base + o_kept);
    int32_t* first = reinterpret_cast<int32_t*>(base + o_first);
    // the array still holds the previous call's contents; the counter accumulates, so it is the
    // one part that must start from zero (everything else is fully overwritten before it is read)
    KD_CUDA(cudaMemsetAsync(moved, 0, sizeof(unsigned long long), st));
    const float e = effective_eps(eps);
    const int nn = static_cast<int>(n);
    const int rows_per_split = (nn + splits - 1) / splits;
    const dim3 grid(splits, U);
    KD_CUDA(launch(anchor_partial_kernel, grid, kStagedThreads, 0, st, 0, true, kc, nk, len, block_B, N, e, rows_per_split, nn, partial, norms, 0));
    KD_CUDA(launch(score_kernel, grid, kStagedThreads, 0, st, 0, true, kc, nk, len, block_B, N, e, rows_per_split, nn, partial, norms, scores));
    if (wide_select_smem(nn) <= kWideSelectSmem)
        KD_CUDA(launch(wide_select_kernel, dim3(U), kSelThreads, wide_select_smem(nn), st, 0, true, kc, nk, scores, len, block_B, N, e, 0, nn, 0,
                       static_cast<double*>(nullptr), kept, first, moved, static_cast<int32_t*>(nullptr)));
    else
        KD_CUDA(launch(select_kernel, dim3(U), kSelectThreads, static_cast<size_t>(nn) * 4, st, 0, true, scores, nn, N, nn, len, kept, first, moved, 0,
                       nullptr, 0));
    KD_CUDA(launch(compact_kernel, dim3(2, U), kCompactThreads, 0, st, 0, true, kc, vc, nk, nv, len, block_B, N, kept, first, nullptr));
    return KEYDIFF_OK;
}
