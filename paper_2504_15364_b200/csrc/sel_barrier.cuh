// The selector's threads and their barrier (a barrier of its own, 1: the selectors may be a part of a block).
#pragma once
#include <cstdint>

namespace kd {

constexpr int kSelWarps = 8, kSelThreads = 32 * kSelWarps;

__device__ __forceinline__ void sel_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kSelThreads) : "memory"); }

// Number of selector threads with `p` (a barrier, too).
__device__ __forceinline__ int sel_count(bool p) {
    int r;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\tbarrier.cta.red.popc.u32 %0, 1, %2, q;\n\t}" : "=r"(r) : "r"(static_cast<uint32_t>(p)), "n"(kSelThreads) : "memory");
    return r;
}

}  // namespace kd
