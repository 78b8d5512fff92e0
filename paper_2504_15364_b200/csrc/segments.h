// Which rows the blocks of wide_move_kernel own and how far they read past their own: plain arithmetic, for the device and for
// a compiler without CUDA.
#pragma once
#ifdef __CUDACC__
#define KD_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define KD_HOST_DEVICE inline
#endif

namespace kd {

constexpr int kCompactRows = 128;   // rows staged per iteration of the gathers (32 KB)
constexpr int kMaxSegments = 8;     // blocks per unit and tensor, at most
constexpr int kHaloRows = 144;      // rows of a segment that are read ahead, at most (36 KB)
// A segment waits only for the one in front of it, so that one must not read past the rows of its direct successor: no segment with
// a successor has fewer rows than are read ahead.  (With 128 rows and 144 read ahead, the rows a segment reads could be those of
// the next but one, which does not wait for it.)
constexpr int kMinSegmentRows = (kHaloRows + kCompactRows - 1) / kCompactRows * kCompactRows;
static_assert(kMinSegmentRows >= kHaloRows, "a segment's read-ahead ends in its direct successor");

struct Segment { int d0, d1; };     // destination rows [d0, d1)

// Segment s of the rows [first, N) that move: all segments have the same number of rows but the last that has any.
KD_HOST_DEVICE Segment segment_of(int first, int N, int segments, int s) {
    int per = ((N - first + segments - 1) / segments + kCompactRows - 1) / kCompactRows * kCompactRows;
    per = per > kMinSegmentRows ? per : kMinSegmentRows;
    const long long at = static_cast<long long>(first) + static_cast<long long>(s) * per;
    const int d0 = at < N ? static_cast<int>(at) : N;
    return Segment{d0, N - d0 < per ? N : d0 + per};
}

// Rows at the segment's end that it reads ahead: those whose sources may lie behind its end.  last_source: source of row d1 - 1.  The
// last segment that has rows has no successor.  At most kHaloRows when no more rows than that are evicted, hence no more than it has.
KD_HOST_DEVICE int rows_read_ahead(Segment g, int N, int last_source) {
    return g.d1 > g.d0 && g.d1 < N ? last_source - (g.d1 - 1) : 0;
}

}  // namespace kd
