// A graph without the entries that the iterations of a run have no use for, made on the device: the rows of its batch alone, or the columns
// that are training rows alone.
#pragma once
#include "common.cuh"

namespace retexo {

constexpr int kKeptRowWarps = 8;
constexpr uint8_t kMarkTrain = 1, kMarkBatch = 2;      // marks of a node: a training row; a training or validation row
static __global__ void mark_nodes_kernel(const int32_t* __restrict__ idx, int64_t n, uint8_t value, uint8_t* __restrict__ marks) {
    const int64_t i = blockIdx.x * 256ll + threadIdx.x;
    if (i < n) marks[idx[i]] = value;
}
// Entries of row v that are kept: all of a batch row's (columns == 0), or those whose column is a training row.
__device__ __forceinline__ bool row_kept(const uint8_t* marks, int64_t v, int columns) { return columns || (marks[v] & kMarkBatch); }
// The rows' kept entries: a warp a row, 128 entries a trip.
static __global__ void __launch_bounds__(32 * kKeptRowWarps) count_kept_kernel(int64_t n, const int64_t* __restrict__ rowptr,
                                                                                  const int32_t* __restrict__ colidx, const uint8_t* __restrict__ marks,
                                                                                  int columns, int64_t* __restrict__ count) {
    const int64_t v = blockIdx.x * (int64_t)kKeptRowWarps + (threadIdx.x >> 5);
    if (v >= n) return;
    const int lane = threadIdx.x & 31;
    const int64_t beg = rowptr[v], end = rowptr[v + 1];
    int kept = 0;
    if (columns) {
#pragma unroll 4
        for (int64_t e = beg + lane; e < end; e += 32) kept += __ldg(marks + __ldcs(colidx + e)) & kMarkTrain;
        kept = __reduce_add_sync(0xffffffffu, kept);
    }
    if (lane == 0) count[v] = columns ? (int64_t)kept : row_kept(marks, v, columns) ? end - beg : 0;
}
// count[v] = sum of count[0, v), in place, and the total behind them, in two launches: every block its own kScanRows rows and their total,
// then every block what lies before it.
constexpr int kScanPer = 8, kScanRows = 256 * kScanPer;
static __global__ void __launch_bounds__(256) scan_kernel(int64_t n, int64_t* __restrict__ count, int64_t* __restrict__ totals) {
    __shared__ int64_t warp_total[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * kScanRows + threadIdx.x * kScanPer;
    int64_t c[kScanPer], mine = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        c[k] = i + k < n ? count[i + k] : 0;
        mine += c[k];
    }
    int64_t at = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += y;
    }
    if (lane == 31) warp_total[warp] = at;
    at -= mine;
    __syncthreads();
    for (int w = 0; w < warp; ++w) at += warp_total[w];
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        if (i + k < n) count[i + k] = at;
        at += c[k];
    }
    if (threadIdx.x == 255) totals[blockIdx.x] = at;
}
static __global__ void __launch_bounds__(256) scan_add_kernel(int64_t n, int64_t* __restrict__ count, const int64_t* __restrict__ totals) {
    __shared__ unsigned long long before_s;
    if (threadIdx.x == 0) before_s = 0ull;
    __syncthreads();
    unsigned long long part = 0;
    for (unsigned b = threadIdx.x; b < blockIdx.x; b += 256) part += (unsigned long long)totals[b];
    if (part) atomicAdd(&before_s, part);
    __syncthreads();
    const int64_t before = (int64_t)before_s;
    for (int64_t i = (int64_t)blockIdx.x * kScanRows + threadIdx.x; i < n && i < ((int64_t)blockIdx.x + 1) * kScanRows; i += 256) count[i] += before;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) count[n] = before + totals[blockIdx.x];
}
static __global__ void __launch_bounds__(32 * kKeptRowWarps) copy_kept_kernel(int64_t n, const int64_t* __restrict__ rowptr,
                                                                                 const int32_t* __restrict__ colidx, const uint8_t* __restrict__ marks,
                                                                                 int columns, const int64_t* __restrict__ first,
                                                                                 int32_t* __restrict__ kept) {
    const int64_t v = blockIdx.x * (int64_t)kKeptRowWarps + (threadIdx.x >> 5);
    if (v >= n || !row_kept(marks, v, columns)) return;
    const int lane = threadIdx.x & 31;
    const int64_t beg = rowptr[v], end = rowptr[v + 1];
    int32_t* dst = kept + first[v];
    for (int64_t e0 = beg; e0 < end; e0 += 32) {
        const int64_t e = e0 + lane;
        const int32_t u = e < end ? __ldcs(colidx + e) : -1;
        const bool keep = u >= 0 && (!columns || (__ldg(marks + u) & kMarkTrain));
        const unsigned all = __ballot_sync(0xffffffffu, keep);
        if (keep) dst[__popc(all & ((1u << lane) - 1u))] = u;
        dst += __popc(all);
    }
}

inline int64_t kept_scan_words(int64_t n) { return (n + kScanRows - 1) / kScanRows; }
// columns: 1 keeps the entries whose column is marked kMarkTrain, 0 the rows marked kMarkBatch.  rowptr [n + 1], colidx as long as the
// graph's; totals: kept_scan_words(n).
inline int keep_entries_launch(const retexo_csr& g, const uint8_t* marks, int columns, int64_t* rowptr, int32_t* colidx, int64_t* totals, cudaStream_t st) {
    const int64_t n = g.n_nodes;
    const unsigned blocks = (unsigned)((n + kKeptRowWarps - 1) / kKeptRowWarps), threads = 32 * kKeptRowWarps, scan_blocks = (unsigned)kept_scan_words(n);
    count_kept_kernel<<<blocks, threads, 0, st>>>(n, g.rowptr, g.colidx, marks, columns, rowptr);
    scan_kernel<<<scan_blocks, 256, 0, st>>>(n, rowptr, totals);
    scan_add_kernel<<<scan_blocks, 256, 0, st>>>(n, rowptr, totals);
    copy_kept_kernel<<<blocks, threads, 0, st>>>(n, g.rowptr, g.colidx, marks, columns, rowptr, colidx);
    return launch_status();
}

}  // namespace retexo
