// Full-graph neighbour aggregation of one message-passing round (Eq. 1) over a CSR graph:
// GCN symmetric-normalised sum, GraphSAGE mean and max (+ self concat); the GAT pass is in gat.cu.
//
// The work is a gather-reduce bound by the memory system, not a dense contraction: neighbour rows are streamed with the
// widest aligned vector loads, several rows in flight per lane, sums kept in registers.  Rows go to lanes by a fixed
// rule (no work counter: a draw per row from one address is 2 ns each, more than a row of ten entries takes the chip),
// rows of heavy_degree() entries or more are cut into segments that are taken first, each segment's partial sum goes to
// scratch, and a second kernel adds a row's segments in order.  Nothing depends on which warp ran what when, so results
// are the same bits on every call.
#include "common.cuh"
#include "aggregate.h"
#include "gat.h"
#include "gat_lanes.cuh"

namespace retexo {

constexpr int kAggThreads = 128, kAggBlocksPerSm = 9;      // (56 registers a thread)
constexpr int kAggWarps = kAggThreads / kWarp;

// Rows of heavy_degree entries or more are cut into segments of half as many: 2048 entries, fewer on graphs so small that
// one warp on a long row would keep the grid waiting.
static inline int32_t seg_len(int64_t n_edges) {
    int32_t len = 64;
    while (len < 2048 && (int64_t)len * 148 * 128 < n_edges) len *= 2;
    return len;
}
static inline int32_t heavy_degree(int64_t n_edges) { return 2 * seg_len(n_edges); }

// Upper bounds on the number of heavy rows and of segments of a graph with n_edges entries.
static inline int64_t max_heavy(int64_t n_edges) { return n_edges / heavy_degree(n_edges) + 1; }
static inline int64_t max_segments(int64_t n_edges) { return n_edges / seg_len(n_edges) + max_heavy(n_edges); }

// ---------------------------------------------------------------- pre-pass
struct HeavyRows {
    int32_t seg_entries;             // entries per segment; rows of twice as many are heavy
    int32_t* list;                   // [heavy rows] node id
    int32_t* seg_base;               // [heavy rows] first segment of the row
    int32_t* seg_slot;               // [segments] index into list
    int32_t* counters;               // [0] heavy rows, [1] segments
};

// Lists row v and its segments if it is heavy (list order is arbitrary; no result depends on it).
__device__ __forceinline__ void list_if_heavy(const HeavyRows& h, int64_t v, int64_t deg) {
    if (deg < 2 * h.seg_entries) return;
    const int32_t slot = atomicAdd(h.counters + 0, 1);
    const int32_t nseg = (int32_t)((deg + h.seg_entries - 1) / h.seg_entries);
    const int32_t base = atomicAdd(h.counters + 1, nseg);
    h.list[slot] = (int32_t)v;
    h.seg_base[slot] = base;
    for (int32_t i = 0; i < nseg; ++i) h.seg_slot[base + i] = slot;
}

__device__ __forceinline__ float gcn_coef(int64_t deg) { return 1.0f / sqrtf((float)deg + 1.0f); }

// Heavy rows, and (GCN, coef != nullptr) the normalisation (deg + 1)^-1/2.
__global__ void prep_rows_kernel(int64_t n, const int64_t* __restrict__ rowptr, HeavyRows h, float* __restrict__ coef) {
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v >= n) return;
    const int64_t deg = rowptr[v + 1] - rowptr[v];
    if (coef) coef[v] = gcn_coef(deg);
    list_if_heavy(h, v, deg);
}

// The same for a GCN round whose rows are laid out ahead in rows of ld_qs floats (a multiple of 8): scaled, qs[u] = n_u q[u], so that the
// gather needs no coefficient per entry, or as they are (coef != nullptr: the coefficients go there).  1 << lanes_log2 lanes a row,
// 8 columns each; a stream over q.
__global__ void __launch_bounds__(256) gcn_lay_out_rows_kernel(int64_t n, const int64_t* __restrict__ rowptr, HeavyRows h,
                                                               const float* __restrict__ q, int64_t ldq, int32_t dim, int vec4,
                                                               float* __restrict__ qs, int64_t ld_qs, int lanes_log2, float* __restrict__ coef) {
    const int64_t t = blockIdx.x * 256ll + threadIdx.x, v = t >> lanes_log2;
    if (v >= n) return;
    const int lanes = 1 << lanes_log2, lane = (int)t & (lanes - 1);
    const int64_t deg = rowptr[v + 1] - rowptr[v];
    if (lane == 0) list_if_heavy(h, v, deg);
    float c = gcn_coef(deg);
    if (coef) {
        if (lane == 0) coef[v] = c;
        c = 1.f;
    }
    const float* src = q + v * ldq;
    float* dst = qs + v * ld_qs;
    for (int col = 8 * lane; col < ld_qs; col += 8 * lanes) {
        float x[8];
        if (vec4 && col + 8 <= dim) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(src + col)), b = __ldg(reinterpret_cast<const float4*>(src + col + 4));
            x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = col + i < dim ? __ldg(src + col + i) : 0.f;
        }
        *reinterpret_cast<float4*>(dst + col) = make_float4(c * x[0], c * x[1], c * x[2], c * x[3]);
        *reinterpret_cast<float4*>(dst + col + 4) = make_float4(c * x[4], c * x[5], c * x[6], c * x[7]);
    }
}

// What a row's accumulator does with a neighbour row: plain sum (SAGE mean; GCN of rows scaled ahead), element-wise maximum (SAGE
// max-pooling), sum weighted by coef[u] (GCN of rows as they are), or compensated sum (GCN of narrow rows scaled ahead).
constexpr int kOpSum = 0, kOpGcn = 1, kOpMax = 2, kOpGcnWeighted = 3, kOpGcnNarrow = 4;

struct AggArgs {
    int64_t n;
    const int64_t* rowptr;
    const int32_t* colidx;
    const float* q;         // the rows that are gathered (GCN through agg_lanes_kernel: scaled by n_u)
    int64_t ldq;
    int32_t dim;
    const float* coef;      // GCN weighted
    float* out;             // may be null
    int64_t ldout;
    __nv_bfloat16* out16;   // may be null
    int64_t ldout16;
    int32_t concat_self;    // SAGE
    int32_t vec_out, vec_out16;      // 16-byte stores of 4 floats / 8-byte stores of 4 bf16 values are aligned
    HeavyRows heavy;
    float* seg_partial;              // [segments x round_up(dim, 4)] raw sums
    int64_t ld_partial;
    GatRowOrder order;               // agg_lanes_kernel: rows by falling length (null: as they come)
    int32_t* next_item;              // agg_rows_kernel: work counter
    float hub_coef;                  // agg_rows_kernel: rows of nodes with coef <= hub_coef (hubs) are loaded "evict last", all
                                     // others "evict first"
};

__device__ __forceinline__ void store_elem(const AggArgs& a, int64_t v, int col, float val) {
    if (a.out) a.out[v * a.ldout + col] = val;
    if (a.out16) a.out16[v * a.ldout16 + col] = f32_to_bf16(val);
}

// E floats from read-only memory, aligned to as much.
template <int E>
__device__ __forceinline__ void load_vec(const float* p, float (&v)[E]) {
    if constexpr (E == 8) {
        asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(p));
    } else if constexpr (E == 4) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(p));
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else if constexpr (E == 2) {
        const float2 x = __ldg(reinterpret_cast<const float2*>(p));
        v[0] = x.x; v[1] = x.y;
    } else {
        v[0] = __ldg(p);
    }
}
// ---------------------------------------------------------------- rows to lanes
// A slab of up to LPG x E x NV columns is aggregated at a time.  LPG lanes (a power of two) take one CSR entry: lane `li` of group
// `g` owns the NV vectors of E columns at E (li + LPG k) of the slab, so a warp reads G = 32 / LPG neighbour rows per load
// instruction in whole runs.  A row of up to kGroupEntries entries is summed by one group in CSR order (a warp works on G rows
// at once), a longer one by the whole warp: group g adds the entries g, g + G, ... and the groups' sums are added in a fixed tree.
constexpr int kGroupEntries = 32;

template <int LPG, int E, int NV, int OP>
struct AggLanes {
    static constexpr int G = kWarp / LPG, kCols = LPG * E * NV;
    static constexpr bool kGcn = OP == kOpGcn || OP == kOpGcnWeighted || OP == kOpGcnNarrow, kCompensated = OP == kOpGcnNarrow;
    static constexpr int U = kCompensated ? 2 : E >= 4 || E * NV > 2 ? 4 : 8;      // entries in flight per lane
    static constexpr int kBlocks = E < 4 && E * NV > 4 ? 8 : E == 4 && LPG == 32 ? 12 : kAggBlocksPerSm;      // (64, 40 and 56 registers)
    const AggArgs& a;
    int g, li, c0;                      // c0: the lane's first column; vector k starts at c0 + E LPG k
    bool on[NV];                        // the vector exists
    float acc[NV][E], self[NV][E];
    float lost[NV][kCompensated ? E : 1];      // what rounding has added to acc beyond its terms

    __device__ __forceinline__ AggLanes(const AggArgs& a_, int lane, int col0) : a(a_) {
        g = lane / LPG;
        li = lane % LPG;
        c0 = col0 + E * li;
#pragma unroll
        for (int k = 0; k < NV; ++k) on[k] = c0 + E * LPG * k < a.dim;
        if (NV == 1 && !on[0]) c0 = col0;      // (reads the group's first vector and drops it: no predicate on the load)
    }
    // This lane's vectors of row u.
    __device__ __forceinline__ void load_row(int64_t u, float (&x)[NV][E]) {
        const float* p = a.q + u * a.ldq + c0;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            if (NV == 1 || on[k]) {
                load_vec<E>(p + E * LPG * k, x[k]);
            } else {
#pragma unroll
                for (int i = 0; i < E; ++i) x[k][i] = 0.f;
            }
        }
    }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int k = 0; k < NV; ++k)
#pragma unroll
            for (int i = 0; i < E; ++i) {
                acc[k][i] = OP == kOpMax ? -INFINITY : 0.f;
                if constexpr (kCompensated) lost[k][i] = 0.f;
            }
    }
    // What the end of row v needs.
    __device__ __forceinline__ void load_self(int64_t v) {
        if (kGcn || a.concat_self) {
            load_row(v, self);
        }
    }
    // Adds the rows u[t] (GCN weighted: times w[t]) where ok[t]; where it is not, u[t] is some node whose row is loaded and dropped.
    template <int N>
    __device__ __forceinline__ void batch(const int32_t (&u)[N], const bool (&ok)[N], const float (&w)[N]) {
        float x[N][NV][E];
#pragma unroll
        for (int t = 0; t < N; ++t)
            load_row(u[t], x[t]);
#pragma unroll
        for (int t = 0; t < N; ++t) {
            if (!ok[t]) continue;
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    if constexpr (kCompensated) {
                        const float more = __fsub_rn(x[t][k][i], lost[k][i]), sum = __fadd_rn(acc[k][i], more);
                        lost[k][i] = __fsub_rn(__fsub_rn(sum, acc[k][i]), more);
                        acc[k][i] = sum;
                    } else {
                        acc[k][i] = OP == kOpMax ? fmaxf(acc[k][i], x[t][k][i])
                                  : OP == kOpGcnWeighted ? fmaf(w[t], x[t][k][i], acc[k][i]) : acc[k][i] + x[t][k][i];
                    }
                }
        }
    }
    __device__ __forceinline__ float weight(int32_t u) const { return OP == kOpGcnWeighted ? __ldg(a.coef + u) : 1.f; }
    // Entries [first, last) of the CSR by the whole warp, 32 columns at a time, fetched two trips ahead.
    __device__ __forceinline__ void walk_by_warp(int64_t first, int64_t last, int lane) {
        auto column = [&](int64_t e0) -> int32_t { return __ldcs(a.colidx + (e0 + lane < last ? e0 + lane : first)); };
        if (first >= last) return;
        int32_t next_u = column(first), after_u = first + kWarp < last ? column(first + kWarp) : 0;
        for (int64_t e0 = first; e0 < last; e0 += kWarp) {
            const int cnt = (int)min((int64_t)kWarp, last - e0);
            const int32_t my_u = next_u;
            next_u = after_u;
            if (e0 + 2 * kWarp < last) after_u = column(e0 + 2 * kWarp);
            const float my_w = weight(my_u);
            constexpr int N = G * U > kWarp ? kWarp / G : U;
#pragma unroll 1
            for (int j = 0; j < cnt; j += G * N) {
                int32_t u[N];
                bool ok[N];
                float w[N];
#pragma unroll
                for (int t = 0; t < N; ++t) {
                    const int at = j + t * G + g;
                    u[t] = __shfl_sync(0xffffffffu, my_u, at & 31);
                    w[t] = OP == kOpGcnWeighted ? __shfl_sync(0xffffffffu, my_w, at & 31) : 1.f;
                    ok[t] = at < cnt;
                }
                batch<N>(u, ok, w);
            }
        }
#pragma unroll
        for (int o = LPG; o < kWarp; o <<= 1) {
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    const float y = __shfl_xor_sync(0xffffffffu, acc[k][i], o);
                    acc[k][i] = OP == kOpMax ? fmaxf(acc[k][i], y) : acc[k][i] + y;
                }
        }
    }
    // Every group its own row of `total` entries from beg on (0: none); longest = the largest total of the warp.
    __device__ __forceinline__ void walk_by_group(int64_t beg, int total, int longest, int32_t some_node) {
        constexpr int N = U < LPG ? U : LPG;
        auto column = [&](int e) -> int32_t { return total > 0 ? __ldg(a.colidx + beg + (e < total ? e : 0)) : some_node; };
        int32_t next_u = column(li);
        for (int e0 = 0; e0 < longest; e0 += LPG) {
            const int32_t my_u = next_u;
            if (e0 + LPG < longest) next_u = column(e0 + LPG + li);
            const int cnt = min(LPG, longest - e0);
            const float my_w = weight(my_u);
#pragma unroll 1
            for (int j = 0; j < cnt; j += N) {
                int32_t u[N];
                bool ok[N];
                float w[N];
#pragma unroll
                for (int t = 0; t < N; ++t) {
                    u[t] = __shfl_sync(0xffffffffu, my_u, g * LPG + j + t);
                    w[t] = OP == kOpGcnWeighted ? __shfl_sync(0xffffffffu, my_w, g * LPG + j + t) : 1.f;
                    ok[t] = e0 + j + t < total;
                }
                batch<N>(u, ok, w);
            }
        }
    }
    __device__ __forceinline__ void store(int64_t v, int col, const float (&x)[E]) {
        if (a.out) {
            float* o = a.out + v * a.ldout + col;
            if (E >= 4 && a.vec_out) {
#pragma unroll
                for (int i = 0; i < E; i += 4) *reinterpret_cast<float4*>(o + i) = make_float4(x[i], x[(i + 1) % E], x[(i + 2) % E], x[(i + 3) % E]);
            } else {
#pragma unroll
                for (int i = 0; i < E; ++i) o[i] = x[i];
            }
        }
        if (a.out16) {
            __nv_bfloat16* o = a.out16 + v * a.ldout16 + col;
            if (E >= 4 && a.vec_out16) {
#pragma unroll
                for (int i = 0; i < E; i += 4) {
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(x[i], x[(i + 1) % E]), hi = __floats2bfloat162_rn(x[(i + 2) % E], x[(i + 3) % E]);
                    *reinterpret_cast<uint2*>(o + i) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                }
            } else {
#pragma unroll
                for (int i = 0; i < E; ++i) o[i] = f32_to_bf16(x[i]);
            }
        }
    }
    // GCN adds the (scaled) self row and scales, SAGE divides by the degree and (optionally) copies the self row.
    __device__ __forceinline__ void finish(int64_t v, int64_t deg) {
        const float cv = kGcn ? gcn_coef(deg) : 0.f;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            if (!on[k]) continue;
#pragma unroll
            for (int i = 0; i < E; ++i) {
                if (OP == kOpGcn) acc[k][i] = cv * (self[k][i] + acc[k][i]);
                else if constexpr (kCompensated) acc[k][i] = cv * __fadd_rn(acc[k][i], __fsub_rn(self[k][i], lost[k][i]));
                else if (OP == kOpGcnWeighted) acc[k][i] = cv * fmaf(cv, self[k][i], acc[k][i]);
                else acc[k][i] = deg <= 0 ? 0.f : OP == kOpMax ? acc[k][i] : acc[k][i] / (float)deg;
            }
            const bool concat = !kGcn && a.concat_self;
            const int col = c0 + E * LPG * k, n_cols = a.dim - col;
            if (E == 1 || n_cols >= E) {
                if (concat) store(v, col, self[k]);
                store(v, col + (concat ? a.dim : 0), acc[k]);
            } else {                    // the ragged last vector
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    if (i >= n_cols) break;
                    if (concat) store_elem(a, v, col + i, self[k][i]);
                    store_elem(a, v, col + (concat ? a.dim : 0) + i, acc[k][i]);
                }
            }
        }
    }
};

// One block's share of a slab: the first seg_blocks blocks take the segments of the heavy rows (their raw sums go to scratch), the
// others a fixed set of rows each, rows_per_warp (up to G) per warp.
template <int LPG, int E, int NV, int OP>
__device__ __forceinline__ void agg_block(const AggArgs& a, int col0, unsigned b, unsigned seg_blocks, int rows_per_warp, const GatGrid& by_length) {
    constexpr int G = kWarp / LPG;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    AggLanes<LPG, E, NV, OP> L(a, lane, col0);
    const int32_t seg_entries = a.heavy.seg_entries;
    if (b < seg_blocks) {
        const int n_seg = a.heavy.counters[1];
        for (int item = (int)b * kAggWarps + warp; item < n_seg; item += (int)seg_blocks * kAggWarps) {
            const int32_t slot = a.heavy.seg_slot[item];
            const int64_t v = a.heavy.list[slot];
            const int64_t beg = a.rowptr[v] + (int64_t)(item - a.heavy.seg_base[slot]) * seg_entries;
            L.clear();
            L.walk_by_warp(beg, min(a.rowptr[v + 1], beg + seg_entries), lane);
            float* dst = a.seg_partial + (int64_t)item * a.ld_partial;
            if (L.g == 0) {
#pragma unroll
                for (int k = 0; k < NV; ++k)
#pragma unroll
                    for (int i = 0; i < E; ++i) {
                        const int col = L.c0 + E * LPG * k + i;
                        if (L.on[k] && col < a.dim) dst[col] = L.acc[k][i];
                    }
            }
        }
        return;
    }
    int64_t v, beg;
    int32_t total;
    if (a.order.rows) {
        int rows;
        const int64_t i0 = gat_first_row<LPG>(a.order, by_length, (int64_t)(b - seg_blocks) * kAggWarps + warp, rows);
        if (rows == 0) return;
        const GatRow row = load_row_entry(a.order.rows + i0 + min(L.g, rows - 1));
        v = row.v;
        beg = row.beg;
        total = L.g < rows ? row.deg : INT32_MAX;      // (nobody's row)
    } else {
        const int64_t v0 = ((int64_t)(b - seg_blocks) * kAggWarps + warp) * rows_per_warp;
        if (v0 >= a.n) return;
        v = min(v0 + L.g, a.n - 1);
        beg = __ldg(a.rowptr + v);
        const bool some = L.g < rows_per_warp && v0 + L.g < a.n;
        total = some ? (int32_t)(__ldg(a.rowptr + v + 1) - beg) : INT32_MAX;
    }
    const bool mine = G > 1 && total <= kGroupEntries;
    if constexpr (G > 1) {
        if (__any_sync(0xffffffffu, mine)) {
            const int longest = __reduce_max_sync(0xffffffffu, mine ? total : 0);
            L.clear();
            L.load_self(v);                 // (ahead of time: short rows are bound by latencies)
            L.walk_by_group(beg, mine ? total : 0, longest, (int32_t)v);
            if (mine) L.finish(v, total);
        }
    }
    unsigned longer = __ballot_sync(0xffffffffu, L.li == 0 && !mine && total < 2 * seg_entries);
    while (longer) {
        const int src = __ffs(longer) - 1;
        longer &= longer - 1;
        const int64_t w = __shfl_sync(0xffffffffu, v, src), w_beg = __shfl_sync(0xffffffffu, beg, src);
        const int32_t w_total = __shfl_sync(0xffffffffu, total, src);
        L.clear();
        L.walk_by_warp(w_beg, w_beg + w_total, lane);
        L.load_self(w);
        if (L.g == 0) L.finish(w, w_total);
    }
}

struct AggGrid {
    unsigned slabs, blocks_per_slab, seg_blocks;      // whole slabs first, then the columns that are left
    int rows_per_warp, tail_rows_per_warp;
    GatGrid by_length, tail_by_length;                // (rows by length)
};

// Blocks are ordered slab by slab, so that at any time the whole grid gathers from the same few columns of the matrix: a slab of
// 64 columns stays in L2 where the whole matrix does not.  The columns left over are taken by groups of TLPG lanes, as many as they
// need: a second slab for 8 columns of 72 with the lanes of a whole one costs as much as the first.
// Bound by the L2 -> SM path (64 bytes a cycle and SM) on dense graphs, by row pointer -> column -> row latencies on sparse ones;
// measured against a persistent kernel that drew its rows from one counter, a warp each (SAGE, bf16 out, with concatenation):
//   233 k nodes, 113 M entries, 256 columns: 6.95 -> 6.3 ms (18.5 TB/s of neighbour rows); GCN 9.5 -> 6.6 ms
//   58 k nodes, 7 M entries, 256 columns: 820 -> 492 us (14.4 TB/s); GCN 1036 -> 498 us
//   600 k nodes, 30 M entries, 256 columns: 4.05 -> 3.2 ms;  20 k nodes, 88 k entries, 500 columns: 142 -> 62 us
// Slabs of 32 or 128 columns instead of 64 take 1.4 and 1.2 times as long on the first of these; 4 entries in flight, since
// with 56 registers 36 warps fit an SM (64: 32 warps, level; 48: 5 % slower; 80 and more: 1.4 times as long).  At 8 columns a lane the compiler
// spills 4 to 64 bytes a thread of these.
template <int LPG, int E, int NV, int TLPG, int TNV, int OP>
__global__ void __launch_bounds__(kAggThreads, AggLanes<LPG, E, NV, OP>::kBlocks) agg_lanes_kernel(AggArgs a, AggGrid grid) {
    constexpr int kCols = LPG * E * NV;
    const unsigned whole = grid.slabs * grid.blocks_per_slab;
    if ((LPG == TLPG && NV == TNV) || blockIdx.x < whole) {
        const unsigned slab = blockIdx.x / grid.blocks_per_slab;
        agg_block<LPG, E, NV, OP>(a, (int)slab * kCols, blockIdx.x - slab * grid.blocks_per_slab, grid.seg_blocks, grid.rows_per_warp,
                                   grid.by_length);
    } else {
        agg_block<TLPG, E, TNV, OP>(a, (int)grid.slabs * kCols, blockIdx.x - whole, grid.seg_blocks, grid.tail_rows_per_warp,
                                     grid.tail_by_length);
    }
}

// Adds the heavy rows' segment sums in segment order and finishes the rows; a block per row, a thread per column.  self_scaled: q
// holds rows scaled by n_u (GCN).
template <int OP>
__global__ void __launch_bounds__(kAggThreads) agg_combine_kernel(AggArgs a, int self_scaled) {
    const int n_heavy = a.heavy.counters[0];
    for (int h = blockIdx.x; h < n_heavy; h += gridDim.x) {
        const int64_t v = a.heavy.list[h];
        const int64_t deg = a.rowptr[v + 1] - a.rowptr[v];
        const int nseg = (int)((deg + a.heavy.seg_entries - 1) / a.heavy.seg_entries);
        const float* src = a.seg_partial + (int64_t)a.heavy.seg_base[h] * a.ld_partial;
        const float cv = OP == kOpGcn ? gcn_coef(deg) : 0.f;
        for (int col = threadIdx.x; col < a.dim; col += kAggThreads) {
            float acc = OP == kOpMax ? -INFINITY : 0.f;
#pragma unroll 4
            for (int i = 0; i < nseg; ++i) {
                const float x = src[(int64_t)i * a.ld_partial + col];
                acc = OP == kOpMax ? fmaxf(acc, x) : acc + x;
            }
            const float self = a.q[v * a.ldq + col];
            if (OP == kOpGcn) {
                store_elem(a, v, col, cv * (self_scaled ? self + acc : fmaf(cv, self, acc)));
            } else {
                const float mean = OP == kOpMax ? acc : acc / (float)deg;
                if (a.concat_self) store_elem(a, v, col, self);
                store_elem(a, v, col + (a.concat_self ? a.dim : 0), mean);
            }
        }
    }
}

static int launch_combine(int op, const AggArgs& a, int64_t n_edges, int self_scaled, int n_sm, cudaStream_t st) {
    if (n_edges < heavy_degree(n_edges)) return launch_status();      // no row can be heavy
    const int64_t most = max_heavy(n_edges);
    const unsigned grid = (unsigned)(most < 8ll * n_sm ? most : 8ll * n_sm);      // (a row is a chain of latencies: as many at once as fit; a block an SM: 8.8 and 15.3 us where this takes 5.6 and 6.9)
    if (op == kOpGcn) agg_combine_kernel<kOpGcn><<<grid, kAggThreads, 0, st>>>(a, self_scaled);
    else if (op == kOpMax) agg_combine_kernel<kOpMax><<<grid, kAggThreads, 0, st>>>(a, 0);
    else agg_combine_kernel<kOpSum><<<grid, kAggThreads, 0, st>>>(a, 0);
    return launch_status();
}

// Rows a warp takes side by side: as many as it has groups where rows are short.  Rows above kGroupEntries entries it takes one after
// the other, so there should be few enough of them a warp to keep every SM busy (2 k nodes, 200 k entries, 8 columns: 65 us with
// 32 rows a warp, 16 blocks in all).
static int rows_per_warp(int groups, int64_t n, int64_t n_edges, int n_sm) {
    int rows = groups;
    if (n_edges > n * kGroupEntries)
        while (rows > 1 && n < (int64_t)rows * kAggWarps * n_sm * kAggBlocksPerSm) rows /= 2;
    return rows;
}

template <int LPG, int E, int NV, int TLPG, int TNV>
static int launch_lanes(int op, const AggArgs& a, int64_t n_edges, int n_sm, cudaStream_t st) {
    constexpr int kCols = LPG * E * NV;
    AggGrid g;
    g.slabs = (unsigned)(a.dim / kCols);
    int left = a.dim % kCols;
    if (left && LPG == TLPG && NV == TNV) {      // the last slab is like the others
        g.slabs += 1;
        left = 0;
    }
    g.rows_per_warp = rows_per_warp(kWarp / LPG, a.n, n_edges, n_sm);
    g.tail_rows_per_warp = rows_per_warp(kWarp / TLPG, a.n, n_edges, n_sm);
    const int64_t segs = n_edges >= heavy_degree(n_edges) ? (max_segments(n_edges) + kAggWarps - 1) / kAggWarps : 0;
    g.seg_blocks = (unsigned)(segs < 4ll * n_sm ? segs : 4ll * n_sm);
    static_assert(kAggWarps == kGatWarps && kGroupEntries == kGatGroupEntries, "one order serves both");
    g.by_length = gat_grid<LPG>(a.n, n_edges, n_sm, 0);
    g.tail_by_length = gat_grid<TLPG>(a.n, n_edges, n_sm, 0);
    auto blocks = [&](int64_t rows, const GatGrid& by_length) {
        return (a.order.rows ? (int64_t)by_length.blocks : (a.n + kAggWarps * rows - 1) / (kAggWarps * rows)) + g.seg_blocks;
    };
    const int64_t total = g.slabs * blocks(g.rows_per_warp, g.by_length) + (left ? blocks(g.tail_rows_per_warp, g.tail_by_length) : 0);
    if (total > INT32_MAX) return RETEXO_ERR_UNSUPPORTED;
    g.blocks_per_slab = (unsigned)blocks(g.rows_per_warp, g.by_length);
    const unsigned grid = (unsigned)total;
    if constexpr (E == 8) {
        if (op == kOpGcn) agg_lanes_kernel<LPG, E, NV, TLPG, TNV, kOpGcn><<<grid, kAggThreads, 0, st>>>(a, g);
    }
    if constexpr (E == 8 && kCols <= 16) {
        if (op == kOpGcnNarrow) agg_lanes_kernel<LPG, E, NV, TLPG, TNV, kOpGcnNarrow><<<grid, kAggThreads, 0, st>>>(a, g);
    }
    if (op == kOpGcnWeighted) agg_lanes_kernel<LPG, E, NV, TLPG, TNV, kOpGcnWeighted><<<grid, kAggThreads, 0, st>>>(a, g);
    else if (op == kOpMax) agg_lanes_kernel<LPG, E, NV, TLPG, TNV, kOpMax><<<grid, kAggThreads, 0, st>>>(a, g);
    else if (op == kOpSum) agg_lanes_kernel<LPG, E, NV, TLPG, TNV, kOpSum><<<grid, kAggThreads, 0, st>>>(a, g);
    const bool gcn = op == kOpGcn || op == kOpGcnWeighted || op == kOpGcnNarrow;
    return launch_combine(gcn ? kOpGcn : op, a, n_edges, op != kOpGcnWeighted, n_sm, st);
}

constexpr size_t kSlabBytes = (size_t)64 << 20;      // a slab of all rows may take this much of L2
// The matrix does not fit L2, and its rows are read often enough for a slab that does to pay.
static bool beyond_l2(int64_t n, int64_t n_edges, int32_t dim) { return (size_t)n * dim * 4 > ((size_t)100 << 20) && n_edges >= 16 * n; }

// Rows in whole 32-byte pieces.
static int launch_lanes8(int op, const AggArgs& a, int64_t n_edges, int n_sm, cudaStream_t st) {
    if (a.dim <= 8) return launch_lanes<1, 8, 1, 1, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 16) return launch_lanes<2, 8, 1, 2, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 32) return launch_lanes<4, 8, 1, 4, 1>(op, a, n_edges, n_sm, st);
    if (a.dim > 96 && a.dim < 128 && (size_t)a.n * a.dim * 4 <= kSlabBytes) return launch_lanes<16, 8, 1, 16, 1>(op, a, n_edges, n_sm, st);
    const int left = a.dim % 64;
    if (left == 0 || left > 32 || a.dim > 320) return launch_lanes<8, 8, 1, 8, 1>(op, a, n_edges, n_sm, st);
    if (left <= 8) return launch_lanes<8, 8, 1, 1, 1>(op, a, n_edges, n_sm, st);
    if (left <= 16) return launch_lanes<8, 8, 1, 2, 1>(op, a, n_edges, n_sm, st);
    return launch_lanes<8, 8, 1, 4, 1>(op, a, n_edges, n_sm, st);
}
// ... in 16-byte pieces.
static int launch_lanes4(int op, const AggArgs& a, int64_t n_edges, int n_sm, cudaStream_t st) {
    if (a.dim <= 8) return launch_lanes<2, 4, 1, 2, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 16) return launch_lanes<4, 4, 1, 4, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 32) return launch_lanes<8, 4, 1, 8, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 64) return launch_lanes<16, 4, 1, 16, 1>(op, a, n_edges, n_sm, st);
    if (a.dim > 256 && beyond_l2(a.n, n_edges, a.dim) && (size_t)a.n * 256 <= kSlabBytes) return launch_lanes<16, 4, 1, 16, 1>(op, a, n_edges, n_sm, st);
    const int left = a.dim % 128;
    if (left == 0 || left > 64) return launch_lanes<32, 4, 1, 32, 1>(op, a, n_edges, n_sm, st);
    if (left <= 16) return launch_lanes<32, 4, 1, 4, 1>(op, a, n_edges, n_sm, st);
    if (left <= 32) return launch_lanes<32, 4, 1, 8, 1>(op, a, n_edges, n_sm, st);
    return launch_lanes<32, 4, 1, 16, 1>(op, a, n_edges, n_sm, st);
}
// How many vectors of 32 lanes a slab of rows in narrow pieces takes, at most `most`: all of them where that is one pass, else about
// equal slabs, of 64 MB where the matrix is beyond L2, such slabs fit it and rows are read often enough to come back to them.  (An
// entry costs a warp as much in shuffles and addresses as in loads, so a second pass for a few columns costs almost what the first
// does: 20 k nodes, 2 M entries, 96 / 97 columns in slabs of 96: 90 / 162 us, in one pass 77 / 79.)
static int slab_vectors(int64_t n, int64_t n_edges, int32_t dim, int cols, int most) {
    const int vecs = (dim + cols - 1) / cols;
    if (beyond_l2(n, n_edges, dim)) {
        const int64_t fit = (int64_t)kSlabBytes / (n * cols * 4);
        if (fit * cols >= 64 && fit < most) most = (int)fit;
    }
    const int slabs = (vecs + most - 1) / most;
    return (vecs + slabs - 1) / slabs;
}
// ... in 8-byte pieces.
static int launch_lanes2(int op, const AggArgs& a, int64_t n_edges, int n_sm, cudaStream_t st) {
    if (a.dim <= 8) return launch_lanes<4, 2, 1, 4, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 16) return launch_lanes<8, 2, 1, 8, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 32) return launch_lanes<16, 2, 1, 16, 1>(op, a, n_edges, n_sm, st);
    switch (slab_vectors(a.n, n_edges, a.dim, 64, 3)) {
        case 1: return launch_lanes<32, 2, 1, 32, 1>(op, a, n_edges, n_sm, st);
        case 2: return launch_lanes<32, 2, 2, 32, 2>(op, a, n_edges, n_sm, st);
        default: return launch_lanes<32, 2, 3, 32, 3>(op, a, n_edges, n_sm, st);
    }
}
// ... float by float.
static int launch_lanes1(int op, const AggArgs& a, int64_t n_edges, int n_sm, cudaStream_t st) {
    if (a.dim <= 4) return launch_lanes<4, 1, 1, 4, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 8) return launch_lanes<8, 1, 1, 8, 1>(op, a, n_edges, n_sm, st);
    if (a.dim <= 16) return launch_lanes<16, 1, 1, 16, 1>(op, a, n_edges, n_sm, st);
    switch (slab_vectors(a.n, n_edges, a.dim, 32, 6)) {
        case 1: return launch_lanes<32, 1, 1, 32, 1>(op, a, n_edges, n_sm, st);
        case 2: return launch_lanes<32, 1, 2, 32, 2>(op, a, n_edges, n_sm, st);
        case 3: return launch_lanes<32, 1, 3, 32, 3>(op, a, n_edges, n_sm, st);
        case 4: return launch_lanes<32, 1, 4, 32, 4>(op, a, n_edges, n_sm, st);
        case 5: return launch_lanes<32, 1, 5, 32, 5>(op, a, n_edges, n_sm, st);
        default: return launch_lanes<32, 1, 6, 32, 6>(op, a, n_edges, n_sm, st);
    }
}

// ---------------------------------------------------------------- GCN on dense graphs far larger than L2
// Bound by HBM, so what counts is which rows stay in L2: a power-law graph reads its hubs' rows again and again, every other
// row a few times, and left to itself the cache keeps neither.  Rows of hubs (coef <= hub_coef) are loaded "evict last",
// all others "evict first"; the coefficient, gathered per entry anyway, tells which.  (2.45 M x 256 floats, 124 M entries:
// 15.8 ms, 18.1 ms without the priorities; 2.45 M x 100: 7.9 ms.)  A whole row per load instruction, one warp per row or
// segment; the items come from one counter.
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ float4 ldg_hinted(const float4* ptr, uint64_t policy) {
    float4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(ptr), "l"(policy));
    return v;
}
__device__ __forceinline__ void fma4(float4& a, float w, const float4& x) {
    a.x = fmaf(w, x.x, a.x); a.y = fmaf(w, x.y, a.y); a.z = fmaf(w, x.z, a.z); a.w = fmaf(w, x.w, a.w);
}

constexpr int kRowThreads = 256;
constexpr int kUnroll = 4;             // neighbour rows in flight per lane and column chunk

// Adds the weighted rows of CSR entries [beg, end), in order, for the float4 vectors vec0 + 32 c + lane of this lane.
template <int CH>
__device__ __forceinline__ void accumulate_range(const AggArgs& a, int64_t beg, int64_t end, int lane, int vec0, int nvec,
                                                 float4 (&acc)[CH]) {
    const int64_t ldv = a.ldq / 4;
    const float4* __restrict__ qv = reinterpret_cast<const float4*>(a.q);
    const bool hinting = a.hub_coef > 0.f;      // (always here; the test keeps the loads' registers apart: 256 columns 16.1 ms, without it 17.3)
    uint64_t keep = 0, pass = 0;
    if (hinting) { keep = l2_policy_evict_last(); pass = l2_policy_evict_first(); }
    for (int64_t e0 = beg; e0 < end; e0 += kWarp) {
        const int cnt = (int)min((int64_t)kWarp, end - e0);
        int my_u = 0;
        float my_w = 0.f;
        if (lane < cnt) {
            my_u = __ldg(a.colidx + e0 + lane);
            my_w = __ldg(a.coef + my_u);
        }
        int j = 0;
        for (; j + kUnroll <= cnt; j += kUnroll) {
            float4 x[kUnroll][CH];
            float w[kUnroll];
#pragma unroll
            for (int t = 0; t < kUnroll; ++t) {
                const int u = __shfl_sync(0xffffffffu, my_u, j + t);
                w[t] = __shfl_sync(0xffffffffu, my_w, j + t);
                const float4* row = qv + (int64_t)u * ldv;
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    const int vi = vec0 + c * kWarp + lane;
                    x[t][c] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (vi < nvec) {
                        if (hinting) x[t][c] = ldg_hinted(row + vi, w[t] <= a.hub_coef ? keep : pass);
                        else x[t][c] = __ldg(row + vi);
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < kUnroll; ++t)
#pragma unroll
                for (int c = 0; c < CH; ++c) fma4(acc[c], w[t], x[t][c]);
        }
        for (; j < cnt; ++j) {
            const int u = __shfl_sync(0xffffffffu, my_u, j);
            const float w = __shfl_sync(0xffffffffu, my_w, j);
            const float4* row = qv + (int64_t)u * ldv;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int vi = vec0 + c * kWarp + lane;
                if (vi < nvec) fma4(acc[c], w, __ldg(row + vi));
            }
        }
    }
}

// Persistent: items [0, n_seg) are segments of heavy rows, [n_seg, n_seg + n) whole rows (heavy ones are skipped).
template <int CH>
__global__ void __launch_bounds__(kRowThreads) agg_rows_kernel(AggArgs a) {
    const int lane = threadIdx.x & 31;
    const int nvec = (a.dim + 3) / 4;
    const int64_t n_seg = a.heavy.counters[1];
    const int64_t total = n_seg + a.n;
    for (;;) {
        int64_t item = 0;
        if (lane == 0) item = atomicAdd(reinterpret_cast<unsigned int*>(a.next_item), 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= total) break;
        if (item < n_seg) {
            const int32_t slot = a.heavy.seg_slot[item];
            const int64_t v = a.heavy.list[slot];
            const int64_t beg = a.rowptr[v] + (item - a.heavy.seg_base[slot]) * a.heavy.seg_entries;
            const int64_t end = min(a.rowptr[v + 1], beg + a.heavy.seg_entries);
            for (int vec0 = 0; vec0 < nvec; vec0 += CH * kWarp) {
                float4 acc[CH];
#pragma unroll
                for (int c = 0; c < CH; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
                accumulate_range<CH>(a, beg, end, lane, vec0, nvec, acc);
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    const int vi = vec0 + c * kWarp + lane;
                    if (vi < nvec) *reinterpret_cast<float4*>(a.seg_partial + item * a.ld_partial + 4 * vi) = acc[c];
                }
            }
            continue;
        }
        const int64_t v = item - n_seg;
        const int64_t beg = a.rowptr[v], end = a.rowptr[v + 1];
        if (end - beg >= 2 * a.heavy.seg_entries) continue;
        for (int vec0 = 0; vec0 < nvec; vec0 += CH * kWarp) {
            float4 acc[CH];
#pragma unroll
            for (int c = 0; c < CH; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
            accumulate_range<CH>(a, beg, end, lane, vec0, nvec, acc);
            const float cv = a.coef[v];
            const float4* self = reinterpret_cast<const float4*>(a.q) + v * (a.ldq / 4);
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int vi = vec0 + c * kWarp + lane;
                if (vi >= nvec) continue;
                const float4 s = self[vi];
                const float z[4] = {cv * fmaf(cv, s.x, acc[c].x), cv * fmaf(cv, s.y, acc[c].y), cv * fmaf(cv, s.z, acc[c].z),
                                    cv * fmaf(cv, s.w, acc[c].w)};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (4 * vi + i < a.dim) store_elem(a, v, 4 * vi + i, z[i]);
            }
        }
    }
}

// The same for rows in 8- or 4-byte pieces, without priorities.
// Adds the weighted rows of CSR entries [beg, end), in order, for the pieces vec0 + 32 c + lane of this lane.
template <int E, int CH>
__device__ __forceinline__ void accumulate_pieces(const AggArgs& a, int64_t beg, int64_t end, int lane, int vec0, int nvec,
                                                 float (&acc)[CH][E]) {
    for (int64_t e0 = beg; e0 < end; e0 += kWarp) {
        const int cnt = (int)min((int64_t)kWarp, end - e0);
        int my_u = 0;
        float my_w = 0.f;
        if (lane < cnt) {
            my_u = __ldg(a.colidx + e0 + lane);
            my_w = __ldg(a.coef + my_u);
        }
        int j = 0;
        for (; j + kUnroll <= cnt; j += kUnroll) {
            float x[kUnroll][CH][E], w[kUnroll];
#pragma unroll
            for (int t = 0; t < kUnroll; ++t) {
                const int u = __shfl_sync(0xffffffffu, my_u, j + t);
                w[t] = __shfl_sync(0xffffffffu, my_w, j + t);
                const float* row = a.q + (int64_t)u * a.ldq;
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    const int vi = vec0 + c * kWarp + lane;
#pragma unroll
                    for (int i = 0; i < E; ++i) x[t][c][i] = 0.f;
                    if (vi < nvec) load_vec<E>(row + E * vi, x[t][c]);
                }
            }
#pragma unroll
            for (int t = 0; t < kUnroll; ++t)
#pragma unroll
                for (int c = 0; c < CH; ++c)
#pragma unroll
                    for (int i = 0; i < E; ++i) acc[c][i] = fmaf(w[t], x[t][c][i], acc[c][i]);
        }
        for (; j < cnt; ++j) {
            const int u = __shfl_sync(0xffffffffu, my_u, j);
            const float w = __shfl_sync(0xffffffffu, my_w, j);
            const float* row = a.q + (int64_t)u * a.ldq;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int vi = vec0 + c * kWarp + lane;
                if (vi >= nvec) continue;
                float x[E];
                load_vec<E>(row + E * vi, x);
#pragma unroll
                for (int i = 0; i < E; ++i) acc[c][i] = fmaf(w, x[i], acc[c][i]);
            }
        }
    }
}

// Persistent: items [0, n_seg) are segments of heavy rows, [n_seg, n_seg + n) whole rows (heavy ones are skipped).
template <int E, int CH>
__global__ void __launch_bounds__(kRowThreads) agg_pieces_kernel(AggArgs a) {
    const int lane = threadIdx.x & 31;
    const int nvec = (a.dim + E - 1) / E;
    const int64_t n_seg = a.heavy.counters[1];
    const int64_t total = n_seg + a.n;
    for (;;) {
        int64_t item = 0;
        if (lane == 0) item = atomicAdd(reinterpret_cast<unsigned int*>(a.next_item), 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= total) break;
        if (item < n_seg) {
            const int32_t slot = a.heavy.seg_slot[item];
            const int64_t v = a.heavy.list[slot];
            const int64_t beg = a.rowptr[v] + (item - a.heavy.seg_base[slot]) * a.heavy.seg_entries;
            const int64_t end = min(a.rowptr[v + 1], beg + a.heavy.seg_entries);
            for (int vec0 = 0; vec0 < nvec; vec0 += CH * kWarp) {
                float acc[CH][E];
#pragma unroll
                for (int c = 0; c < CH; ++c)
#pragma unroll
                    for (int i = 0; i < E; ++i) acc[c][i] = 0.f;
                accumulate_pieces<E, CH>(a, beg, end, lane, vec0, nvec, acc);
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    const int vi = vec0 + c * kWarp + lane;
                    if (vi >= nvec) continue;
#pragma unroll
                    for (int i = 0; i < E; ++i) if (E * vi + i < a.dim) a.seg_partial[item * a.ld_partial + E * vi + i] = acc[c][i];
                }
            }
            continue;
        }
        const int64_t v = item - n_seg;
        const int64_t beg = a.rowptr[v], end = a.rowptr[v + 1];
        if (end - beg >= 2 * a.heavy.seg_entries) continue;
        for (int vec0 = 0; vec0 < nvec; vec0 += CH * kWarp) {
            float acc[CH][E];
#pragma unroll
            for (int c = 0; c < CH; ++c)
#pragma unroll
                for (int i = 0; i < E; ++i) acc[c][i] = 0.f;
            accumulate_pieces<E, CH>(a, beg, end, lane, vec0, nvec, acc);
            const float cv = a.coef[v];
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int vi = vec0 + c * kWarp + lane;
                if (vi >= nvec) continue;
                float self[E];
                load_vec<E>(a.q + v * a.ldq + E * vi, self);
#pragma unroll
                for (int i = 0; i < E; ++i)
                    if (E * vi + i < a.dim) store_elem(a, v, E * vi + i, cv * fmaf(cv, self[i], acc[c][i]));
            }
        }
    }
}

template <int E, int CH>
static int launch_rows(const AggArgs& a, int64_t n_edges, int n_sm, cudaStream_t st) {
    auto go = [&](auto kernel) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kRowThreads, 0) != cudaSuccess || per_sm < 1) {
            (void)cudaGetLastError();
            per_sm = 1;
        }
        kernel<<<n_sm * per_sm, kRowThreads, 0, st>>>(a);
    };
    if constexpr (E == 4) go(agg_rows_kernel<CH>);
    else go(agg_pieces_kernel<E, CH>);
    return launch_combine(kOpGcn, a, n_edges, 0, n_sm, st);
}

// Rows in pieces of E floats, as many chunks of 32 pieces as they need in one pass, up to 6.
template <int E>
static int launch_rows(const AggArgs& a, int64_t n_edges, int n_sm, cudaStream_t st) {
    const int chunks = (a.dim + 32 * E - 1) / (32 * E);
    if (chunks <= 1) return launch_rows<E, 1>(a, n_edges, n_sm, st);
    if (chunks <= 2) return launch_rows<E, 2>(a, n_edges, n_sm, st);
    if (chunks <= 3) return launch_rows<E, 3>(a, n_edges, n_sm, st);
    if (chunks <= 4) return launch_rows<E, 4>(a, n_edges, n_sm, st);
    if (chunks <= 5) return launch_rows<E, 5>(a, n_edges, n_sm, st);
    return launch_rows<E, 6>(a, n_edges, n_sm, st);
}

// ---------------------------------------------------------------- rows laid out for wide loads
// dst[i] = [src[i] | zeros], rows of ld_dst (a multiple of 4) floats from densely packed or strided rows of dim floats: the re-lay
// of features whose rows do not start on 16-byte boundaries.  A warp a row, whole 16-byte stores; a stream (561 MB in, 566 MB
// out: 193 us; a pitched device-to-device copy and the clearing of its padding took 420 us).
__global__ void __launch_bounds__(256) relay_rows_kernel(const float* __restrict__ src, int64_t ld_src, int32_t dim, int64_t n,
                                                         float* __restrict__ dst, int64_t ld_dst) {
    const int lane = threadIdx.x & 31;
    const int64_t i = blockIdx.x * 8ll + (threadIdx.x >> 5);
    if (i >= n) return;
    const float* s = src + i * ld_src;
    float4* d = reinterpret_cast<float4*>(dst + i * ld_dst);
#pragma unroll 4
    for (int p = lane; p < (int)(ld_dst >> 2); p += 32) {
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = 4 * p + k < dim ? __ldcs(s + 4 * p + k) : 0.f;
        d[p] = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// ---------------------------------------------------------------- which way a GCN round goes (by its sizes alone)
// Dense: rows of 32 entries or more on average.
static bool gcn_dense(int64_t n, int64_t n_edges) { return n_edges >= 32 * n; }

// agg_rows_kernel pays where the gather is bound by HBM whatever is done about locality: slabs of 64 columns far beyond L2, and rows
// read often enough for L2 to keep the hubs'.  Milliseconds, agg_rows_kernel / agg_lanes_kernel, graphs without hubs / with the
// largest degree 60 / 6000 times the mean: 2.45 M nodes, 50 entries a row, 100 columns 10.0 / 7.9 / 7.8 against 11.2 / 10.6 / 10.1,
// 256 columns 18.6 / 16.6 / 16.0 against 18.1 / 17.6 / 17.2; 25 entries a row, 100 columns 8.0 / 7.8 / 7.9 against 6.3 / 5.9 / 5.8,
// 256 columns 10.1 / 9.9 / 8.9 against 10.8 / 10.5 / 10.5; 1 M nodes, 50 entries, 256 columns 7.3 / 6.4 / 6.3 against 6.2 / 6.1 / 6.0;
// 200 k nodes, 40 entries, 1024 columns 6.6 against 3.3.
static bool gcn_hbm_bound(int64_t n, int64_t n_edges, int32_t dim) {
    return n_edges >= (dim >= 192 ? 16 : 32) * n && (size_t)n * (size_t)dim * 4 >= ((size_t)768 << 20) &&
           (size_t)n * 256 >= ((size_t)512 << 20);
}

// Stride of the copy of a GCN matrix: whole 32-byte pieces; whole 128-byte lines where a row is read often enough to pay for
// writing them.
static int64_t gcn_copy_stride(int32_t dim, int64_t n, int64_t n_edges) {
    const int64_t unit = dim > 64 && gcn_dense(n, n_edges) ? 32 : 8;
    return (dim + unit - 1) / unit * unit;
}

// What a GCN round adds up.  Scaling the rows ahead saves a gathered coefficient per entry but rounds every row once more: on dense
// graphs the longer rows' sums, in several parts, more than make up for it, on others the error against 64 bits would be 4 to 9 % up
// (uniform graphs of 2, 8, 16, 24 entries a row: 4.75, 8.1, 9.7, 10.9e-8, weighted 4.38, 7.5, 9.1, 10.3, 32 entries: 10.6 / 10.1 / 11.7
// before rows were scaled).  There the rows are weighted as they come, or, where a coefficient is as much to gather as a row, scaled and
// added with compensation (4.5, 6.5, 6.6, 6.8e-8; 1 M nodes, 8 M entries, 8 columns 84 us, weighted 128; 32 columns 268 / 211).
enum class GcnWay { kHbm, kScaled, kNarrow, kWeighted };
static GcnWay gcn_way(int64_t n, int64_t n_edges, int32_t dim) {
    if (gcn_hbm_bound(n, n_edges, dim)) return GcnWay::kHbm;
    if (n * gcn_copy_stride(dim, n, n_edges) > ((int64_t)2 << 30) / 4) return GcnWay::kWeighted;
    return gcn_dense(n, n_edges) ? GcnWay::kScaled : dim <= 16 ? GcnWay::kNarrow : GcnWay::kWeighted;
}

// Floats of the copy, 0 where there is none: scaled rows, and (lay_out) rows to be weighted that do not come in 16-byte pieces, up to
// 2 GB (beyond that a round gathers the caller's rows as they are, a few per cent slower when dense, up to half when narrow pieces are
// all there is; the largest graphs are where memory is short).
static int64_t gcn_copy_floats(int64_t n, int64_t n_edges, int32_t dim, bool lay_out) {
    const GcnWay way = gcn_way(n, n_edges, dim);
    if (way == GcnWay::kHbm || (way == GcnWay::kWeighted && !lay_out)) return 0;
    const int64_t floats = n * gcn_copy_stride(dim, n, n_edges);
    return floats <= ((int64_t)2 << 30) / 4 ? floats : 0;
}

// Rows that share warps are taken by falling length (gat_lanes.cuh) on sparse graphs: on a power-law graph the longest of four rows is twice
// the mean, and the lanes of the others wait for it.  The order takes two passes over the row pointers, about 10 us, and rows of a few
// entries gain nothing.  In node order / by length: 1 M nodes, 20 M entries, 128 columns, concatenated bf16 1612 / 1187 us; 2 M nodes, 80 M
// entries, 100 columns, GCN 6.2 / 5.2 ms; 1 M nodes, 16 M entries, 64 columns, GCN 711 / 590 us; 2 M nodes, 16 M entries, 8 columns 281 / 250.
// (In node order stay: a warp per row, 89 k nodes, 0.9 M entries of 77 floats 102 / 107 us; uniform rows of 6 entries, 35 columns 609 / 678.)
static bool rows_by_length(int64_t n, int64_t n_edges, int32_t dim) {
    return n_edges >= 8 * n && n_edges <= 48 * n && n_edges * dim >= ((int64_t)32 << 20);
}

}  // namespace retexo

using namespace retexo;

size_t retexo::aggregate_rows_workspace_size(int64_t n_nodes, int64_t n_edges, int32_t type, int32_t dim, int32_t heads, bool lay_out) {
    Sizer s;
    if (n_nodes < 0) return 0;
    if (type == RETEXO_GAT) {
        gat_forward_workspace(n_nodes, heads > 0 ? heads : 1, s);
    } else {
        s.take<int32_t>((size_t)max_heavy(n_edges));                      // heavy rows
        s.take<int32_t>((size_t)max_heavy(n_edges));                      // their first segment
        s.take<int32_t>((size_t)max_segments(n_edges));                   // segment -> heavy row
        s.take<int32_t>(64);                                              // counters
        s.take<float>((size_t)max_segments(n_edges) * (size_t)((dim + 3) / 4 * 4));   // segment sums
        if (type == RETEXO_GCN) {
            s.take<float>((size_t)n_nodes);                               // coef
            s.take<float>((size_t)gcn_copy_floats(n_nodes, n_edges, dim, lay_out));
        }
        if (rows_by_length(n_nodes, n_edges, dim)) {
            s.take<GatRow>((size_t)n_nodes);
            s.take<int32_t>(kGatOrderInts);
        }
    }
    return s.off + kAlign;
}

// (the caller's alignment is not known here)
extern "C" size_t retexo_aggregate_workspace_size(int64_t n_nodes, int64_t n_edges, int32_t type, int32_t dim, int32_t heads) {
    return aggregate_rows_workspace_size(n_nodes, n_edges, type, dim, heads, true);
}

static int aggregate(const retexo_csr* g, int32_t type, const float* q, int64_t ldq, int32_t dim, bool whole_rows, bool lay_out,
                     const retexo_gat_params* gat, float* out, int64_t ldout, int32_t concat_self, void* out_bf16,
                     int64_t ldout_bf16, void* workspace, size_t workspace_bytes, void* stream) {
    if (!g || g->n_nodes < 0 || g->n_edges < 0 || g->n_nodes > INT32_MAX) return RETEXO_ERR_INVALID_ARG;
    if (type != RETEXO_GCN && type != RETEXO_SAGE_MEAN && type != RETEXO_GAT && type != RETEXO_SAGE_MAX)
        return RETEXO_ERR_INVALID_ARG;
    if (dim <= 0 || ldq < dim) return RETEXO_ERR_INVALID_ARG;
    if (g->n_nodes == 0) return RETEXO_OK;                      // nothing to aggregate
    if (!out && !out_bf16) return RETEXO_ERR_INVALID_ARG;
    if (!g->rowptr || !q || (g->n_edges > 0 && !g->colidx)) return RETEXO_ERR_INVALID_ARG;
    const bool sage = type == RETEXO_SAGE_MEAN || type == RETEXO_SAGE_MAX;
    const int64_t width = (sage && concat_self) ? 2 * (int64_t)dim : dim;
    if (out && ldout < width) return RETEXO_ERR_INVALID_ARG;
    if (out_bf16 && ldout_bf16 < width) return RETEXO_ERR_INVALID_ARG;
    if (dim > 4096) return RETEXO_ERR_UNSUPPORTED;
    if (type == RETEXO_GAT) {
        if (!gat || gat->heads <= 0 || gat->head_dim <= 0 || !gat->a_src || !gat->a_dst) return RETEXO_ERR_INVALID_ARG;
        if ((int64_t)gat->heads * gat->head_dim != dim) return RETEXO_ERR_INVALID_ARG;
        if (gat->heads > kGatMaxHeads || dim > 256) return RETEXO_ERR_UNSUPPORTED;
    }
    const size_t need = aggregate_rows_workspace_size(g->n_nodes, g->n_edges, type, dim, gat ? gat->heads : 0, lay_out);
    if (!workspace || !aligned_to(workspace, kAlign) || workspace_bytes < need) return RETEXO_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int n_sm = sm_count();
    if (n_sm <= 0) return RETEXO_ERR_CUDA;
    Arena ws(workspace, workspace_bytes);
    const int64_t n = g->n_nodes;

    if (type == RETEXO_GAT) {
        GatForward f{};
        f.g = *g; f.p = q; f.ldp = ldq; f.gat = *gat; f.out = out; f.ldout = ldout;
        f.out16 = static_cast<__nv_bfloat16*>(out_bf16); f.ldout16 = ldout_bf16;
        return gat_forward_launch(f, ws, n_sm, st);
    }

    const int64_t e = g->n_edges;
    AggArgs a{};
    a.n = n; a.rowptr = g->rowptr; a.colidx = g->colidx; a.q = q; a.ldq = ldq; a.dim = dim;
    a.heavy.seg_entries = seg_len(e);
    a.heavy.list = ws.take<int32_t>((size_t)max_heavy(e));
    a.heavy.seg_base = ws.take<int32_t>((size_t)max_heavy(e));
    a.heavy.seg_slot = ws.take<int32_t>((size_t)max_segments(e));
    a.heavy.counters = ws.take<int32_t>(64);
    a.next_item = a.heavy.counters + 2;
    a.ld_partial = (dim + 3) / 4 * 4;
    a.seg_partial = ws.take<float>((size_t)max_segments(e) * (size_t)a.ld_partial);
    a.out = out; a.ldout = ldout;
    a.out16 = static_cast<__nv_bfloat16*>(out_bf16); a.ldout16 = ldout_bf16;
    a.concat_self = sage && concat_self ? 1 : 0;
    const bool cols4 = !a.concat_self || dim % 4 == 0;      // where the second half of a concatenated row starts
    a.vec_out = out && aligned_to(out, 16) && ldout % 4 == 0 && cols4;
    a.vec_out16 = out_bf16 && aligned_to(out_bf16, 8) && ldout_bf16 % 4 == 0 && cols4;
    RETEXO_CUDA_TRY(cudaMemsetAsync(a.heavy.counters, 0, 64 * sizeof(int32_t), st));

    // the widest pieces the rows come in (a last piece of 8 that holds 4 columns or fewer could reach beyond the last row's memory)
    const bool v8 = aligned_to(q, 32) && ldq % 8 == 0 && ldq >= (dim + 7) / 8 * 8 && (whole_rows || (dim + 7) / 8 * 8 - dim <= 3);
    const bool v4 = aligned_to(q, 16) && ldq % 4 == 0 && ldq >= (dim + 3) / 4 * 4;
    const bool v2 = aligned_to(q, 8) && ldq % 2 == 0 && ldq >= (dim + 1) / 2 * 2;
    const unsigned prep_blocks = (unsigned)((n + 255) / 256);
    float* coef = type == RETEXO_GCN ? ws.take<float>((size_t)n) : nullptr;
    const GcnWay way = gcn_way(n, e, dim);      // (GCN)
    const int64_t copy = type == RETEXO_GCN ? gcn_copy_floats(n, e, dim, lay_out) : 0;
    float* qs = ws.take<float>((size_t)copy);
    const bool copies = copy > 0 && (way != GcnWay::kWeighted || !v4);      // (rows that come in whole pieces are weighted as they are)
    if (rows_by_length(n, e, dim) && (v8 || copies) && !(type == RETEXO_GCN && way == GcnWay::kHbm)) {      // (heavy rows are the order's hubs)
        GatRow* rows = ws.take<GatRow>((size_t)n);
        int32_t* bins = ws.take<int32_t>(kGatOrderInts);
        const int32_t* all = nullptr;
        RETEXO_TRY(gat_order_launch(*g, 0, &all, &n, 1, rows, nullptr, bins, 2 * a.heavy.seg_entries, st));
        a.order = {rows, bins + kGatOrderCounts, nullptr, n};
    }
    auto lanes = [&](int op) {
        return v8 ? launch_lanes8(op, a, e, n_sm, st) : v4 ? launch_lanes4(op, a, e, n_sm, st)
             : v2 ? launch_lanes2(op, a, e, n_sm, st) : launch_lanes1(op, a, e, n_sm, st);
    };
    if (type == RETEXO_GCN) {
        if (!copies) {
            prep_rows_kernel<<<prep_blocks, 256, 0, st>>>(n, g->rowptr, a.heavy, coef);
            a.coef = coef;
            if (way != GcnWay::kHbm) return lanes(kOpGcnWeighted);
            a.hub_coef = (float)(1.0 / sqrt(4.0 * (double)e / (double)n + 1.0));      // hubs: at least four times the mean degree
            return v4 ? launch_rows<4>(a, e, n_sm, st) : v2 ? launch_rows<2>(a, e, n_sm, st) : launch_rows<1>(a, e, n_sm, st);
        }
        const int64_t ld_qs = gcn_copy_stride(dim, n, e);
        int lanes_log2 = 0;
        while (lanes_log2 < 5 && (8 << lanes_log2) < ld_qs) ++lanes_log2;
        const bool weighted = way == GcnWay::kWeighted;
        gcn_lay_out_rows_kernel<<<(unsigned)(((n << lanes_log2) + 255) / 256), 256, 0, st>>>(n, g->rowptr, a.heavy, q, ldq, dim, v4 ? 1 : 0,
                                                                                             qs, ld_qs, lanes_log2, weighted ? coef : nullptr);
        a.q = qs;
        a.ldq = ld_qs;
        a.coef = coef;
        return launch_lanes8(weighted ? kOpGcnWeighted : way == GcnWay::kNarrow ? kOpGcnNarrow : kOpGcn, a, e, n_sm, st);
    }
    if (e >= heavy_degree(e)) prep_rows_kernel<<<prep_blocks, 256, 0, st>>>(n, g->rowptr, a.heavy, nullptr);
    return lanes(type == RETEXO_SAGE_MAX ? kOpMax : kOpSum);
}

bool retexo::aggregate_copies_rows(int64_t n_nodes, int64_t n_edges, int32_t type, int32_t dim) {
    return type == RETEXO_GCN && gcn_copy_floats(n_nodes, n_edges, dim, false) > 0;
}

int retexo::relay_rows_launch(const float* src, int64_t ld_src, int32_t dim, int64_t n, float* dst, int64_t ld_dst, cudaStream_t st) {
    relay_rows_kernel<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(src, ld_src, dim, n, dst, ld_dst);
    return launch_status();
}

extern "C" int retexo_aggregate(const retexo_csr* g, int32_t type, const float* q, int64_t ldq, int32_t dim,
                                const retexo_gat_params* gat, float* out, int64_t ldout,
                                int32_t concat_self, void* out_bf16, int64_t ldout_bf16,
                                void* workspace, size_t workspace_bytes, void* stream) {
    return aggregate(g, type, q, ldq, dim, false, true, gat, out, ldout, concat_self, out_bf16, ldout_bf16, workspace, workspace_bytes,
                     stream);
}

int retexo::aggregate_rows(const retexo_csr* g, int32_t type, const float* q, int64_t ldq, int32_t dim, bool whole_rows, float* out,
                           int64_t ldout, int32_t concat_self, void* out_bf16, int64_t ldout_bf16, void* workspace,
                           size_t workspace_bytes, void* stream) {
    return aggregate(g, type, q, ldq, dim, whole_rows, false, nullptr, out, ldout, concat_self, out_bf16, ldout_bf16, workspace,
                     workspace_bytes, stream);
}
