// The list of a unit's evicted tokens, from the bitmap that the selection leaves.
#pragma once
#include "common.cuh"       // KD_ROW_OK
#include "low_select.cuh"

namespace kd {

// Behind the selection: tokens evicted in front of every word of the bitmap (of n tokens), and their list, ascending, of at most `limit`; it may
// lie where the keys were.  Returns the first evicted token (E >= 1).
__device__ __forceinline__ int list_evicted(int n, int st, const Selector& s, int* before, int* list, int limit, int32_t* status) {
    const int nwords = (n + 31) >> 5;
    const int per = (nwords + kSelThreads - 1) / kSelThreads, w0 = min(nwords, st * per), w1 = min(nwords, w0 + per);
    int cnt = 0;
    for (int q = w0; q < w1; ++q) cnt += __popc(s.bitmap[q]);
    int run = sel_exclusive_scan(cnt, st, s.wtot);
    for (int q = w0; q < w1; ++q) {
        before[q] = run;
        for (uint32_t wd = s.bitmap[q]; wd; wd &= wd - 1) {
            if (!KD_ROW_OK(run, limit, status)) break;
            list[run++] = 32 * q + __ffs(wd) - 1;
        }
    }
    sel_sync();
    return list[0];
}

}  // namespace kd
