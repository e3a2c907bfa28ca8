// Lane layout of the GAT kernels for head widths 4, 8, 16, ... 256 on aligned rows.  A lane owns W contiguous columns of one
// head (8, or 4 where the heads are 4 wide or rows come in 16-byte pieces only) and LPG lanes (a power of two) one CSR entry, so
// a warp reads G = 32 / LPG whole neighbour rows per load instruction and every lane scores its entry for its own head.  Sums
// over a head's columns are linear, so they are reduced once per row, not once per entry, wherever they are not a difference.
#pragma once
#include "common.cuh"
#include "gat.h"

namespace retexo {

constexpr int kGatThreads = 128, kGatWarps = kGatThreads / kWarp;      // (256: a block's slots idle until its longest row is done)
constexpr int kGatBlocksPerSm = 9;      // 56 registers a thread: 36 warps an SM.  (At 8 columns a lane the backward kernels spill 4 to 20 bytes; 10 blocks spill
                                        // more, 7 at 69 registers wait longer.)
// A row of up to kGatGroupEntries entries is taken by one group of lanes (so a warp works on G rows at once), a longer one
// by a whole warp, and one of `hub_entries` or more by a whole block.
constexpr int kGatGroupEntries = 32;
// A block costs more per entry (a barrier a row, four states to merge), so only rows go to blocks that would keep a warp
// busy for a good part of what the whole grid takes: a quarter of the entries a resident warp sees, but never below 64.
inline int gat_hub_entries(int64_t n_edges, int n_sm) {
    const int64_t share = n_edges / ((int64_t)n_sm * 128);
    return (int)(share < 64 ? 64 : share > 65536 ? 65536 : share);
}

// The rows a kernel takes, in order of falling length, so that the rows that share a warp (and the warps that share a block) take
// about the same time and the longest start first: hubs (hub_entries or more), then the others.  On a power-law graph of 20 entries a row
// the longest of four rows is 2.3 times the mean, and the lanes of the other three wait for it (717 k nodes, 14 M entries, 4 x 16, in node
// order / in this order: forward 617 / 440 to 470 us, destinations 763 / 520 to 550, sources 988 / 690).  Order inside a class of lengths
// is arbitrary; no result depends on it.  Slabs of 32 columns, which halve what L2 has to hold, take 1.5 times as long.
struct __align__(16) GatRow { int64_t beg; int32_t deg, v; };      // first entry, entries, node
__device__ __forceinline__ GatRow load_row_entry(const GatRow* p) {
    const int4 x = __ldg(reinterpret_cast<const int4*>(p));
    return GatRow{(int64_t)((uint64_t)(uint32_t)x.x | ((uint64_t)(uint32_t)x.y << 32)), x.z, x.w};
}
// Classes of lengths: hubs, eight per octave above kGatGroupEntries, one per length below.
constexpr int kGatOctave = 5, kGatLongBins = 1 + 8 * (16 - kGatOctave);      // (hubs start at 65536 entries at the latest)
constexpr int kGatBins = 128;
static_assert(kGatGroupEntries == 1 << kGatOctave && kGatLongBins + kGatGroupEntries < kGatBins, "classes of lengths");
__device__ __forceinline__ int gat_bin(int32_t total, int32_t hub_entries) {
    if (total >= hub_entries) return 0;
    if (total <= kGatGroupEntries) return kGatLongBins + kGatGroupEntries - total;
    const int octave = 31 - __clz(total);
    return kGatLongBins - 1 - ((octave - kGatOctave) * 8 + ((total >> (octave - 3)) & 7));
}
static_assert(kGatOrderCounts == 2 * kGatBins, "rows counted per class, rows placed so far (all cleared before the count)");

// Counts the rows idx[0, n) (null: all rows 0 .. n - 1) per class; see gat_order_kernel.
__global__ void __launch_bounds__(256) gat_order_count_kernel(int64_t n, const int32_t* __restrict__ idx, const int64_t* __restrict__ rowptr,
                                                              int32_t self_loop, int32_t hub_entries, int32_t* __restrict__ bins);
// Places them behind one another once all are counted; slots[i] (optional) receives slot0 + the row's position in the list.
__global__ void __launch_bounds__(256) gat_order_kernel(int64_t n, const int32_t* __restrict__ idx, const int64_t* __restrict__ rowptr,
                                                        int32_t self_loop, int32_t hub_entries, int32_t* __restrict__ bins,
                                                        GatRow* __restrict__ rows, int32_t* __restrict__ slots, int32_t slot0);
constexpr int kGatOrderRows = 1024;      // rows a block of either takes
inline unsigned gat_order_blocks(int64_t n) { return (unsigned)((n + kGatOrderRows - 1) / kGatOrderRows); }

// Blocks of a pass over an order: hub_blocks take the hubs, a block a row; then warps for the long rows, one each as far as the grid has
// some (long_warps), the rest of the order G rows a warp.  (22 k nodes, 365 k entries, long rows G to a warp one after the other instead: forward 22.3
// against 11.8 us, sources 26.0 against 19.7.  Groups taking rows of up to 64 entries: 14.4 and 24.5 us there, 2 % less on 717 k nodes;
// of up to 16: 12.6 and 20.2, 6 % more.)  How many long rows there are only the device knows, so the grid has as many
// warps for them as the entries allow, up to four times what is resident (a block without a row leaves at once).
struct GatGrid {
    int hub_blocks, long_warps;
    unsigned blocks;
};
template <int LPG>
inline GatGrid gat_grid(int64_t n, int64_t n_entries, int n_sm, int hub_blocks) {
    constexpr int64_t G = kWarp / LPG;
    GatGrid g;
    g.hub_blocks = hub_blocks;
    const int64_t most = (int64_t)n_sm * 4 * kGatBlocksPerSm * kGatWarps;
    int64_t want = n_entries / (kGatGroupEntries + 1) + 1;
    if (want > n) want = n;
    if (want > most) want = most;
    g.long_warps = G > 1 ? (int)((want + kGatWarps - 1) / kGatWarps * kGatWarps) : 0;
    g.blocks = (unsigned)(g.hub_blocks + (g.long_warps + (n + G - 1) / G + kGatWarps - 1) / kGatWarps);
    return g;
}
// The first entry of the order that warp w (counted behind the hubs' blocks) takes, and how many (0: none).
template <int LPG>
__device__ __forceinline__ int64_t gat_first_row(const GatRowOrder& order, const GatGrid& grid, int64_t w, int& count) {
    constexpr int G = kWarp / LPG;
    const int n_hubs = __ldg(order.counts), n_long = __ldg(order.counts + 1);
    const int64_t single = G > 1 ? min(n_long - n_hubs, grid.long_warps) : 0;      // rows with a warp of their own
    int64_t first;
    if (w < grid.long_warps) {
        count = w < single ? 1 : 0;
        first = n_hubs + w;
    } else {
        first = n_hubs + single + (w - grid.long_warps) * G;
        count = (int)max((int64_t)0, min((int64_t)G, order.n - first));
    }
    return first;
}

template <int LPG, int W>
struct GatLanes {
    static constexpr int G = kWarp / LPG;                                  // entries per step
    static constexpr int kMaxU = 2;                                        // neighbour rows in flight per lane (4: fewer warps fit)
    static constexpr int U = G * kMaxU > kWarp ? kWarp / G : kMaxU;        // ... of a warp on one row: at most one trip of 32 entries
    int g, li;
    bool on;                   // the lane owns columns (dim need not fill the lanes); if not, it reads column 0 and drops it
    int col, head;
    __device__ __forceinline__ GatLanes(int lane, int dim, int head_dim) {
        g = lane / LPG;
        li = lane % LPG;
        on = W * li < dim;
        col = on ? W * li : 0;
        head = col / head_dim;
    }
};

// Whether the lane layout covers a shape (p and, where given, q hold its rows), and with how many lanes / columns per lane: 8 columns
// where rows come in whole 32-byte pieces, else 4 where they come in 16-byte pieces and are no wider than 64 columns.  (A gradient of
// 100 k nodes, 2 M entries, 4 x 16 at a stride of 68 floats: 296 us, on the general kernels 7380; at a stride of 64 220.)
inline bool gat_lanes_cover(int32_t dim, int32_t head_dim, const float* p, int64_t ldp, const float* q, int64_t ldq, int* lpg, int* w) {
    if (head_dim < 4 || (head_dim & (head_dim - 1)) != 0 || dim > 256) return false;
    auto pieces_of = [&](int columns) {
        return ldp % columns == 0 && aligned_to(p, 4 * columns) && (!q || (ldq % columns == 0 && aligned_to(q, 4 * columns)));
    };
    if (head_dim >= 8 && pieces_of(8)) *w = 8;
    else if (dim <= 64 && pieces_of(4)) *w = 4;
    else return false;
    *lpg = 1;
    while (*lpg * *w < dim) *lpg <<= 1;
    return true;
}

// Calls go.template operator()<LPG, W>() for the layout gat_lanes_cover chose.
template <typename F>
inline int gat_lanes_dispatch(int lpg, int w, F&& go) {
    if (w == 4) {
        switch (lpg) {
            case 16: return go.template operator()<16, 4>();
            case 8: return go.template operator()<8, 4>();
            case 4: return go.template operator()<4, 4>();
            case 2: return go.template operator()<2, 4>();
            default: return go.template operator()<1, 4>();
        }
    }
    switch (lpg) {
        case 32: return go.template operator()<32, 8>();
        case 16: return go.template operator()<16, 8>();
        case 8: return go.template operator()<8, 8>();
        case 4: return go.template operator()<4, 8>();
        case 2: return go.template operator()<2, 8>();
        default: return go.template operator()<1, 8>();
    }
}

// A lane's W columns of a row.
template <int W>
struct Cols {
    float v[W];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < W; ++i) v[i] = 0.f;
    }
    // one 16- or 32-byte load of read-only memory (aligned to as much)
    __device__ __forceinline__ void load(const float* p) {
        if constexpr (W == 4) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(p));
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        } else {
            asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(p));
        }
    }
    __device__ __forceinline__ void load_unaligned(const float* p) {
#pragma unroll
        for (int i = 0; i < W; ++i) v[i] = __ldg(p + i);
    }
    __device__ __forceinline__ void scale(float f) {
#pragma unroll
        for (int i = 0; i < W; ++i) v[i] *= f;
    }
    __device__ __forceinline__ void fma(float w, const Cols& x) {
#pragma unroll
        for (int i = 0; i < W; ++i) v[i] = fmaf(w, x.v[i], v[i]);
    }
    __device__ __forceinline__ float dot(const Cols& x) const {
        float a = v[0] * x.v[0], b = v[1] * x.v[1];
#pragma unroll
        for (int i = 2; i < W; i += 2) { a = fmaf(v[i], x.v[i], a); b = fmaf(v[i + 1], x.v[i + 1], b); }
        return a + b;
    }
    __device__ __forceinline__ void add_xor(int o) {
#pragma unroll
        for (int i = 0; i < W; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    }
    __device__ __forceinline__ void store(float* p, bool vec) const {      // vec: p and its row stride are 16-byte aligned
        if (vec) {
#pragma unroll
            for (int i = 0; i < W; i += 4) *reinterpret_cast<float4*>(p + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        } else {
#pragma unroll
            for (int i = 0; i < W; ++i) p[i] = v[i];
        }
    }
    __device__ __forceinline__ void store(__nv_bfloat16* p, bool vec) const {      // vec: 8-byte aligned
        uint32_t b[W / 2];
#pragma unroll
        for (int i = 0; i < W / 2; ++i) {
            const __nv_bfloat162 x = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            b[i] = *reinterpret_cast<const uint32_t*>(&x);
        }
        if (vec) {
#pragma unroll
            for (int i = 0; i < W / 2; i += 2) *reinterpret_cast<uint2*>(p + 2 * i) = make_uint2(b[i], b[i + 1]);
        } else {
#pragma unroll
            for (int i = 0; i < W; ++i) p[i] = f32_to_bf16(v[i]);
        }
    }
};

__device__ __forceinline__ float leaky(float z, float slope) { return z * (z > 0.f ? 1.f : slope); }
// e^(x - ref) for x <= ref (0 for x = -inf, ref finite), by the hardware's base-2 exponential.  The subtraction comes first and the
// change of base second, so the error depends on how far x is below the row's maximum and not on how large scores are: at a
// gap g, two units in the last place of the exponential and g / 2 of the product, where the weight itself is e^-g.  (The product
// first, one operation less, put half a unit in the last place of 1.44 |x| on the exponent: 4e-5 of a weight at |x| = 1000.)
constexpr float kLog2E = 1.4426950408889634f;
__device__ __forceinline__ float exp_below(float x, float ref) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"((x - ref) * kLog2E));
    return y;
}
// The same where ref may be -inf too (a state without entries yet): 0 for x = -inf whatever ref is.
__device__ __forceinline__ float exp_rel(float x, float ref) { return x == -INFINITY ? 0.f : exp_below(x, ref); }

// sum += more, with what rounding adds beyond that in `lost`; the next `more` starts from -lost (Kahan's compensated sum: a row's
// sums run entry after entry in one lane, and without it lose up to a third more than a tree over the entries).
__device__ __forceinline__ void add_compensated(float& sum, float& lost, float more) {
    const float s = __fadd_rn(sum, more);
    lost = __fsub_rn(__fsub_rn(s, sum), more);
    sum = s;
}

// Hands the entries of a CSR row to pass.batch<U>(u, ok), U neighbours per lane at a time; entry `deg`, if any, is the row's
// own node `self`.  Where ok is false u is an entry of the row all the same (or `self`), so a pass may load its data
// without a predicate and give it weight zero.
// By a warp: trips of 32 entries from `first` on, `step` apart, dealt to the groups one by one.
template <int LPG, int W, class P>
__device__ __forceinline__ void gat_walk_by_warp(P& pass, const GatLanes<LPG, W>& L, const int32_t* __restrict__ colidx, int32_t self,
                                                 int64_t beg, int32_t deg, int32_t total, int32_t first, int32_t step, int lane) {
    constexpr int G = GatLanes<LPG, W>::G, U = GatLanes<LPG, W>::U;
    for (int32_t e0 = first; e0 < total; e0 += step) {
        const int cnt = min(kWarp, total - e0);
        const int32_t e = e0 + (lane < cnt ? lane : 0);
        const int32_t my_u = e < deg ? __ldg(colidx + beg + e) : self;
#pragma unroll 1
        for (int j = 0; j < cnt; j += G * U) {
            int32_t u[U];
            bool ok[U];
#pragma unroll
            for (int t = 0; t < U; ++t) {
                const int at = j + t * G + L.g;
                u[t] = __shfl_sync(0xffffffffu, my_u, at & 31);
                ok[t] = at < cnt;
            }
            pass.template batch<U>(u, ok);
        }
    }
}
// By a group: every group of the warp its own row (total = 0: none); longest = the largest total of the warp.
template <int LPG, int W, class P>
__device__ __forceinline__ void gat_walk_by_group(P& pass, const GatLanes<LPG, W>& L, const int32_t* __restrict__ colidx, int32_t self,
                                                  int64_t beg, int32_t deg, int32_t total, int32_t longest) {
    constexpr int U = GatLanes<LPG, W>::kMaxU < LPG ? GatLanes<LPG, W>::kMaxU : LPG;
    const int32_t stored = min(deg, total);
    auto entry = [&](int32_t e) -> int32_t {
        if (e >= total) e = 0;
        return e < stored ? __ldg(colidx + beg + e) : self;
    };
    int32_t next_u = entry(L.li);
    for (int32_t e0 = 0; e0 < longest; e0 += LPG) {
        const int32_t my_u = next_u;
        if (e0 + LPG < longest) next_u = entry(e0 + LPG + L.li);
        const int cnt = min(LPG, longest - e0);
#pragma unroll 1
        for (int j = 0; j < cnt; j += U) {
            int32_t u[U];
            bool ok[U];
#pragma unroll
            for (int t = 0; t < U; ++t) {
                u[t] = __shfl_sync(0xffffffffu, my_u, L.g * LPG + j + t);
                ok[t] = e0 + j + t < total;
            }
            pass.template batch<U>(u, ok);
        }
    }
}

// <a, x> over a head's columns, whose W-column pieces lie in hw neighbouring lanes (hw a power of two): the sum is taken in the
// order of a warp that owns the columns l, l + 32, ... in lane l and folds its lanes in halves, so that every kernel of the
// library gives a node the same score, bit for bit.  (Scores are not only values: where s_u + t_v is within rounding of zero,
// another order gives an edge the other slope of the LeakyReLU, and its gradient jumps.)
// The sum is complete in the head's last lane group (see head_last_block).
template <int W>
__device__ __forceinline__ float head_dot(const Cols<W>& a, const Cols<W>& x, int hw, int lane_of_head) {
    float q[W];
#pragma unroll
    for (int i = 0; i < W; ++i) q[i] = __fmul_rn(a.v[i], x.v[i]);
    constexpr int kBlock = 32 / W;                 // lanes that hold 32 columns
    for (int k = 1; k * kBlock < hw; ++k) {        // more than 32 columns: the chain l, l + 32, ... runs through the lane groups
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const float before = __shfl_up_sync(0xffffffffu, q[i], kBlock);
            if (lane_of_head / kBlock == k) q[i] = fmaf(a.v[i], x.v[i], before);
        }
    }
    for (int o = (hw < kBlock ? hw : kBlock) >> 1; o > 0; o >>= 1) {
#pragma unroll
        for (int i = 0; i < W; ++i) q[i] = __fadd_rn(q[i], __shfl_xor_sync(0xffffffffu, q[i], o));
    }
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) {
#pragma unroll
        for (int i = 0; i < o; ++i) q[i] = __fadd_rn(q[i], q[i + o]);
    }
    return q[0];
}
// First lane (counted inside the head) of the group that ends up with head_dot's sum.
template <int W>
__device__ __forceinline__ int head_last_block(int hw) { return hw > 32 / W ? hw - 32 / W : 0; }

// s_u = <a_src, p_u>, t_u = <a_dst, p_u> per head, and (bins != nullptr) how many rows there are of each class of lengths.
// A stream over p: LPG lanes a node, kNodes nodes in flight per group.
// (717 k nodes, 4 x 16: 39 us; a warp per node with 4-byte loads and two shuffle trees per head took 366 us.)
template <int LPG, int W>
__global__ void __launch_bounds__(256) gat_lane_scores_kernel(int64_t n, const int64_t* __restrict__ rowptr,
                                                              const float* __restrict__ p, int64_t ldp, int32_t heads,
                                                              int32_t head_dim, const float* __restrict__ a_src,
                                                              const float* __restrict__ a_dst, int32_t self_loop, int32_t hub_entries,
                                                              float* __restrict__ s, float* __restrict__ t, int32_t* __restrict__ bins) {
    constexpr int kNodes = 2, G = GatLanes<LPG, W>::G;
    __shared__ int32_t count[kGatBins];
    if (bins) {
        if (threadIdx.x < kGatBins) count[threadIdx.x] = 0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const GatLanes<LPG, W> L(lane, heads * head_dim, head_dim);
    const int hw = head_dim / W;                  // lanes a head spans
    const int of_head = L.li & (hw - 1);
    const bool writes = L.on && of_head == head_last_block<W>(hw);
    Cols<W> as, ad;
    as.zero(); ad.zero();
    if (L.on) { as.load_unaligned(a_src + L.col); ad.load_unaligned(a_dst + L.col); }
    const int64_t step = (int64_t)gridDim.x * 8 * G * kNodes;
    for (int64_t u0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * G * kNodes; u0 < n; u0 += step) {
        Cols<W> x[kNodes];
#pragma unroll
        for (int i = 0; i < kNodes; ++i) x[i].load(p + min(u0 + i * G + L.g, n - 1) * ldp + L.col);
        if (bins) {
            for (int64_t u = u0 + lane; u < min(n, u0 + G * kNodes); u += kWarp)
                atomicAdd(count + gat_bin((int32_t)(rowptr[u + 1] - rowptr[u]) + self_loop, hub_entries), 1);
        }
#pragma unroll
        for (int i = 0; i < kNodes; ++i) {
            const int64_t u = u0 + i * G + L.g;
            const float ss = head_dot(as, x[i], hw, of_head), tt = head_dot(ad, x[i], hw, of_head);
            if (u < n && writes) {
                s[u * heads + L.head] = ss;
                t[u * heads + L.head] = tt;
            }
        }
    }
    if (bins) {
        __syncthreads();
        if (threadIdx.x < kGatBins && count[threadIdx.x]) atomicAdd(bins + threadIdx.x, count[threadIdx.x]);
    }
}

template <int LPG, int W>
inline unsigned gat_lane_scores_grid(int64_t n, int n_sm) {
    const int64_t per_block = (int64_t)8 * GatLanes<LPG, W>::G * 2;
    const int64_t want = (n + per_block - 1) / per_block, most = (int64_t)n_sm * 16;
    return (unsigned)(want < most ? want : most);
}

}  // namespace retexo
