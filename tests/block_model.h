// One thread block of 256 threads on the host, for device code whose only ties between threads are block barriers and warp
// exchanges: every thread is a fiber and runs until it waits.  One warp can be held back: it then runs only when
// no other warp can.  Between two barriers that is the order in which a missing barrier shows.
#pragma once
#include <ucontext.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <functional>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
using std::max;
using std::min;
struct int2 { int x, y; };
struct alignas(16) int4 { int x, y, z, w; };
struct alignas(16) uint4 { uint32_t x, y, z, w; };
inline int2 make_int2(int x, int y) { return {x, y}; }
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
inline int __popc(uint32_t v) { return __builtin_popcount(v); }
inline int __ffs(uint32_t v) { return __builtin_ffs(static_cast<int>(v)); }
inline int __clz(uint32_t v) { return v ? __builtin_clz(v) : 32; }
inline int atomicAdd(int* p, int v) { const int o = *p; *p += v; return o; }
inline uint32_t atomicOr(uint32_t* p, uint32_t v) { const uint32_t o = *p; *p |= v; return o; }

namespace model {

constexpr int kThreads = 256, kLanes = 32;
enum State { kReady, kAtBarrier, kAtWarp, kDone };
struct Fiber { ucontext_t ctx; std::vector<char> stack; State state; uint32_t value; bool pred; };
struct Block {
    Fiber f[kThreads];
    ucontext_t main;
    int self = 0, count = 0;
    uint32_t lanes[kThreads / kLanes][kLanes];   // what the lanes brought to the warp's latest exchange
    std::function<void(int)> body;
};
inline Block* block = nullptr;

inline void wait(State s) {
    Fiber& me = block->f[block->self];
    me.state = s;
    swapcontext(&me.ctx, &block->main);
}
inline const uint32_t* exchange(uint32_t v) {
    block->f[block->self].value = v;
    wait(kAtWarp);
    return block->lanes[block->self / kLanes];
}
inline void entry() {
    const int id = block->self;
    block->body(id);
    block->f[id].state = kDone;
    swapcontext(&block->f[id].ctx, &block->main);
}

// Runs body(thread) in all threads; false if some of them wait for good.
inline bool run(const std::function<void(int)>& body, int held_warp) {
    static Block storage;
    block = &storage;
    block->body = body;
    for (Fiber& f : block->f) {
        f.stack.resize(128 * 1024);
        getcontext(&f.ctx);
        f.ctx.uc_stack.ss_sp = f.stack.data();
        f.ctx.uc_stack.ss_size = f.stack.size();
        f.ctx.uc_link = nullptr;
        makecontext(&f.ctx, entry, 0);
        f.state = kReady;
    }
    auto run_warp = [&](int w) {   // until none of its lanes can go on; whether any went on
        bool went = false;
        for (bool more = true; more;) {
            more = false;
            for (int l = 0; l < kLanes; ++l)
                if (Fiber& f = block->f[kLanes * w + l]; f.state == kReady) {
                    block->self = kLanes * w + l;
                    swapcontext(&block->main, &f.ctx);
                    went = more = true;
                }
            bool all = true;
            for (int l = 0; l < kLanes; ++l) all = all && block->f[kLanes * w + l].state == kAtWarp;
            if (all) {
                for (int l = 0; l < kLanes; ++l) { block->lanes[w][l] = block->f[kLanes * w + l].value; block->f[kLanes * w + l].state = kReady; }
                more = true;
            }
        }
        return went;
    };
    for (;;) {
        bool went = false;
        for (int w = 0; w < kThreads / kLanes; ++w) if (w != held_warp) went = run_warp(w) || went;
        // a barrier opens for everyone, the held warp included, once all threads have come to it
        const auto in = [&](State s) { return std::count_if(block->f, block->f + kThreads, [&](const Fiber& f) { return f.state == s; }); };
        if (in(kDone) == kThreads) return true;
        if (in(kAtBarrier) == kThreads) {
            block->count = static_cast<int>(std::count_if(block->f, block->f + kThreads, [](const Fiber& f) { return f.pred; }));
            for (Fiber& f : block->f) f.state = kReady;
            went = true;
        }
        if (!went && !(held_warp >= 0 && run_warp(held_warp))) return false;
    }
}

}  // namespace model

template <typename T> T __shfl_sync(unsigned, T v, int src) { return static_cast<T>(model::exchange(static_cast<uint32_t>(v))[src & 31]); }
template <typename T> T __shfl_up_sync(unsigned, T v, int by) {
    const int lane = model::block->self & 31;
    const uint32_t* a = model::exchange(static_cast<uint32_t>(v));
    return static_cast<T>(a[lane >= by ? lane - by : lane]);
}
template <typename T> T __shfl_xor_sync(unsigned, T v, int by) {
    const int lane = model::block->self & 31;
    return static_cast<T>(model::exchange(static_cast<uint32_t>(v))[lane ^ by]);
}
inline uint32_t __ballot_sync(unsigned, bool p) {
    const uint32_t* a = model::exchange(p);
    uint32_t r = 0;
    for (int l = 0; l < 32; ++l) r |= (a[l] & 1u) << l;
    return r;
}
template <typename T> T __reduce_add_sync(unsigned, T v) {
    const uint32_t* a = model::exchange(static_cast<uint32_t>(v));
    uint32_t r = 0;
    for (int l = 0; l < 32; ++l) r += a[l];
    return static_cast<T>(r);
}
inline uint32_t __reduce_min_sync(unsigned, uint32_t v) { const uint32_t* a = model::exchange(v); return *std::min_element(a, a + 32); }
inline uint32_t __reduce_max_sync(unsigned, uint32_t v) { const uint32_t* a = model::exchange(v); return *std::max_element(a, a + 32); }
// lanes that reach a branch are taken one by one
inline uint32_t __activemask() { return 1u << (model::block->self & 31); }
inline uint32_t __match_any_sync(uint32_t mask, int) { return mask; }
