// A row's anchor terms (warp_row_terms, fused_kernel.cuh) summed over rows by a block of 256 threads.  Every kernel that adds a row to
// a running sum or takes one out forms the terms this way, so that a row takes away what it brought, whichever kernels
// served the two steps.
#pragma once
#include "fused_kernel.cuh"

namespace kd {

constexpr int kTermWarps = 8;

// block_sum_of_terms: the terms of rows r0, r0 + 16, ... r0 + 16 (kDeep - 1) of a half warp, requested together; a row that is not there counts
// as zeros, which add nothing but take as long as one that is.
template <int kDeep, typename RowAt>
__device__ __forceinline__ void add_row_terms(int r0, int rows, const RowAt& row_at, float inv_eps, bool raw, int j, double (&acc)[8]) {
    uint2 a[kDeep], b[kDeep];
#pragma unroll
    for (int k = 0; k < kDeep; ++k) {
        const int r = r0 + 2 * kTermWarps * k;
        a[k] = make_uint2(0, 0); b[k] = a[k];
        if (r < rows) { const uint2* row = reinterpret_cast<const uint2*>(row_at(r)); a[k] = row[j]; b[k] = row[j + 16]; }
    }
    float ss[kDeep];
#pragma unroll
    for (int k = 0; k < kDeep; ++k) {
        const float x0 = bf16_lo(a[k].x), x1 = bf16_hi(a[k].x), x2 = bf16_lo(a[k].y), x3 = bf16_hi(a[k].y);
        const float y0 = bf16_lo(b[k].x), y1 = bf16_hi(b[k].x), y2 = bf16_lo(b[k].y), y3 = bf16_hi(b[k].y);
        ss[k] = fmaf(x3, x3, fmaf(x2, x2, fmaf(x1, x1, x0 * x0))) + fmaf(y3, y3, fmaf(y2, y2, fmaf(y1, y1, y0 * y0)));
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < kDeep; ++k) ss[k] += __shfl_xor_sync(0xffffffffu, ss[k], o);
#pragma unroll
    for (int k = 0; k < kDeep; ++k) {
        const float inv = raw ? 1.0f : fminf(approx_rsqrt(ss[k]), inv_eps);
        acc[0] += static_cast<double>(__fmul_rn(bf16_lo(a[k].x), inv)); acc[1] += static_cast<double>(__fmul_rn(bf16_hi(a[k].x), inv));
        acc[2] += static_cast<double>(__fmul_rn(bf16_lo(a[k].y), inv)); acc[3] += static_cast<double>(__fmul_rn(bf16_hi(a[k].y), inv));
        acc[4] += static_cast<double>(__fmul_rn(bf16_lo(b[k].x), inv)); acc[5] += static_cast<double>(__fmul_rn(bf16_hi(b[k].x), inv));
        acc[6] += static_cast<double>(__fmul_rn(bf16_lo(b[k].y), inv)); acc[7] += static_cast<double>(__fmul_rn(bf16_hi(b[k].y), inv));
    }
}

// Sum of the anchor terms of `rows` rows over a block of 256 threads, row r at row_at(r): channel st's total in threads st < 128.
// The terms are those of warp_row_terms, bit for bit: lane j of a half warp holds channels 4j .. 4j+3 and 64+4j .. 64+4j+3, so
// its sum of the two four-term chains is what the butterfly's first exchange would give; the rest of the butterfly
// follows.  Two rows per warp and step, up to 2 kDeep requested together, but no more than are left: what bounds this is the
// conversion of a row's 128 terms to double, also of rows that are not there.  1344 units of 316 rows, us a step, always four deep / by
// what is left: 16 new rows with slot reuse 54.0 / 51.6, one 46.9 / 45.2; 16 in token order 83.3 / 80.9, 100 103.4 / 101.8.
// The depth is chosen again only for what the full steps leave: with the choice inside the loop a sum over all rows of 1000 x 8224 took 995 us a step,
// now 973.
// A thread adds its rows in the same order at any depth.  table: [8][128] doubles, 16-byte aligned; one barrier inside, behind
// which every row has been read.
template <int kDeep = 4, typename RowAt>
__device__ __forceinline__ double block_sum_of_terms(int rows, const RowAt& row_at, float inv_eps, bool raw, double* table, int st) {
    const int wid = st >> 5, lane = st & 31, half = lane >> 4, j = lane & 15;
    constexpr int kStep = 2 * kTermWarps;   // rows of the block at depth 1
    double acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = 0.0;
    int r = 2 * wid;   // (warp-uniform)
#pragma unroll 1
    for (; r + kStep * (kDeep / 2) < rows; r += kStep * kDeep) add_row_terms<kDeep>(r + half, rows, row_at, inv_eps, raw, j, acc);
    if (r + kStep * (kDeep / 4) < rows) add_row_terms<kDeep / 2>(r + half, rows, row_at, inv_eps, raw, j, acc);
    else if (r < rows) add_row_terms<kDeep / 4>(r + half, rows, row_at, inv_eps, raw, j, acc);
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 16);
    if (half == 0) {
        double2* row = reinterpret_cast<double2*>(table + wid * kHeadDim + 4 * j);
        row[0] = make_double2(acc[0], acc[1]); row[1] = make_double2(acc[2], acc[3]);
        row[32] = make_double2(acc[4], acc[5]); row[33] = make_double2(acc[6], acc[7]);
    }
    __syncthreads();
    double sum = 0.0;
    if (st < kHeadDim) {
#pragma unroll
        for (int q = 0; q < kTermWarps; ++q) sum += table[q * kHeadDim + st];
    }
    return sum;
}

}  // namespace kd
