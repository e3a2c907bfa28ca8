// The GAT aggregation (Section 2.2): edge scores, segment soft-max and weighted sum of one message-passing round in one
// pass over the CSR rows.  Head widths that are powers of two from 4 on, on aligned rows, take the lane layout of
// gat_lanes.cuh; every other shape takes the general kernels at the end of the file.
#include "gat.h"
#include "gat_lanes.cuh"

namespace retexo {

constexpr int kGatRowThreads = 256, kGatRowWarps = kGatRowThreads / kWarp;      // general kernels
constexpr int kGatHubEntries = 128;      // general kernels: rows with at least this many entries are taken by a whole block

struct GatArgs {
    int64_t n;
    const int64_t* rowptr;
    const int32_t* colidx;
    const float* p;
    int64_t ldp;
    int32_t heads, head_dim, dim;
    const float* a_src;
    const float* a_dst;
    float slope;
    int32_t self_loop;
    float* s;               // [n x heads] scratch
    float* t;
    float* out;
    int64_t ldout;
    __nv_bfloat16* out16;
    int64_t ldout16;
    int32_t* hub_list;      // general kernels: rows a whole block takes, listed by gat_scores_kernel (order arbitrary; no result
    int32_t* hub_count;     // depends on it)
};

// ---------------------------------------------------------------- rows in order of their lengths (gat_lanes.cuh)
__global__ void __launch_bounds__(256) gat_order_count_kernel(int64_t n, const int32_t* __restrict__ idx, const int64_t* __restrict__ rowptr,
                                                              int32_t self_loop, int32_t hub_entries, int32_t* __restrict__ bins) {
    __shared__ int32_t count[kGatBins];
    if (threadIdx.x < kGatBins) count[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kGatOrderRows / 256; ++k) {
        const int64_t i = (int64_t)blockIdx.x * kGatOrderRows + k * 256 + threadIdx.x;
        if (i >= n) break;
        const int64_t v = idx ? idx[i] : i;
        atomicAdd(count + gat_bin((int32_t)(rowptr[v + 1] - rowptr[v]) + self_loop, hub_entries), 1);
    }
    __syncthreads();
    if (threadIdx.x < kGatBins && count[threadIdx.x]) atomicAdd(bins + threadIdx.x, count[threadIdx.x]);
}

// A stream over the row pointers: a block finds its rows' ranks per class in shared memory and reserves a run of each class with one
// addition (717 k rows: 8 us).
__global__ void __launch_bounds__(256) gat_order_kernel(int64_t n, const int32_t* __restrict__ idx, const int64_t* __restrict__ rowptr,
                                                        int32_t self_loop, int32_t hub_entries, int32_t* __restrict__ bins,
                                                        GatRow* __restrict__ rows, int32_t* __restrict__ slots, int32_t slot0) {
    constexpr int kRows = kGatOrderRows / 256;
    __shared__ int32_t count[kGatBins], base[kGatBins], warp_total[kGatBins / kWarp];
    const int t = threadIdx.x, lane = t & 31;
    int32_t mine = 0, before = 0;      // rows of class t; of the classes up to it
    if (t < kGatBins) {
        count[t] = 0;
        mine = before = bins[t];
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, before, o);
            if (lane >= o) before += y;
        }
        if (lane == kWarp - 1) warp_total[t / kWarp] = before;
    }
    __syncthreads();
    GatRow row[kRows];
    int bin[kRows], rank[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        const int64_t i = (int64_t)blockIdx.x * kGatOrderRows + k * 256 + t;
        bin[k] = -1;
        if (i >= n) continue;
        const int64_t v = idx ? idx[i] : i;
        row[k].beg = rowptr[v];
        row[k].deg = (int32_t)(rowptr[v + 1] - row[k].beg);
        row[k].v = (int32_t)v;
        bin[k] = gat_bin(row[k].deg + self_loop, hub_entries);
        rank[k] = atomicAdd(count + bin[k], 1);
    }
    __syncthreads();
    if (t < kGatBins) {
        for (int w = 0; w < t / kWarp; ++w) before += warp_total[w];
        if (blockIdx.x == 0 && t == 0) bins[kGatOrderCounts] = mine;
        if (blockIdx.x == 0 && t == kGatLongBins - 1) bins[kGatOrderCounts + 1] = before;
        base[t] = before - mine + (count[t] ? atomicAdd(bins + kGatBins + t, count[t]) : 0);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        if (bin[k] < 0) continue;
        const int32_t at = base[bin[k]] + rank[k];
        rows[at] = row[k];
        if (slots) slots[at] = slot0 + (int32_t)((int64_t)blockIdx.x * kGatOrderRows + k * 256 + t);
    }
}

// ---------------------------------------------------------------- lane layout
// Running soft-max state and weighted sum of one lane over the entries its group takes.
template <int W>
struct GatState {
    float m, l, lost;            // lost: what rounding has added to l beyond its terms
    Cols<W> acc;
    __device__ __forceinline__ void clear() { m = -INFINITY; l = lost = 0.f; acc.zero(); }
    // Adds the states of the warp's groups in a fixed tree; every lane ends up with the total of its columns.
    template <int LPG>
    __device__ __forceinline__ void merge_groups() {
        l -= lost;
        lost = 0.f;
#pragma unroll
        for (int o = LPG; o < kWarp; o <<= 1) {
            const float big = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            const float f = exp_rel(m, big);
            l *= f;
            acc.scale(f);
            l += __shfl_xor_sync(0xffffffffu, l, o);
            acc.add_xor(o);
            m = big;
        }
    }
};

// Scores the entries of a batch and adds their weighted rows to the state.  The rows are asked for before their scores are
// known: the two loads do not depend on each other.
template <int LPG, int W>
struct GatForwardPass {
    const GatArgs& a;
    const float* p;            // this lane's columns of row 0
    const float* s;            // this lane's head of node 0
    int head;
    float tv;
    GatState<W> st;
    __device__ __forceinline__ GatForwardPass(const GatArgs& a_, const GatLanes<LPG, W>& L)
        : a(a_), p(a_.p + L.col), s(a_.s + L.head), head(L.head) {}
    __device__ __forceinline__ void begin(int64_t v) {
        tv = __ldg(a.t + v * a.heads + head);
        st.clear();
    }
    template <int U>
    __device__ __forceinline__ void batch(const int32_t (&u)[U], const bool (&ok)[U]) {
        Cols<W> x[U];
        float e[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
            e[t] = __ldg(s + (int64_t)u[t] * a.heads);
            x[t].load(p + (int64_t)u[t] * a.ldp);
        }
        float big = st.m;
#pragma unroll
        for (int t = 0; t < U; ++t) {
            e[t] = ok[t] ? leaky(e[t] + tv, a.slope) : -INFINITY;
            big = fmaxf(big, e[t]);
        }
        const float f = exp_rel(st.m, big);
        const float ref = big == -INFINITY ? 0.f : big;         // (a group without entries yet)
        st.m = big;
        st.l *= f;
        st.lost *= f;
        st.acc.scale(f);
        float more = -st.lost;
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const float w = exp_below(e[t], ref);
            more += w;
            st.acc.fma(w, x[t]);
        }
        if (ok[0]) add_compensated(st.l, st.lost, more);      // (beyond the row's end nothing may change, not even what is lost)
    }
};

// Blocks [0, hub_blocks): one block per hub row at a time; warp w takes the trips w, w + 4, ... and the warps' states are
// merged in warp order, so the result does not depend on scheduling.  Blocks from hub_blocks on: G rows a warp in the order of
// lengths, the short ones at once, a group each, the longer ones one after the other.
// Bound by the gather of the neighbour rows (4 dim + 4 heads bytes an entry, out of L2 where p fits it) and, below that, by
// the chain row -> column -> neighbour row and the instructions an entry takes: hence a row per group, 32-byte loads and no
// shuffles per entry.  Measured with the score kernel (a warp per row, 4-byte loads, a soft-max reduction over the warp every
// 32 entries before): 717 k nodes, 14 M entries, 4 x 16: 2667 -> 684 us, in order of lengths 510 (8.2 TB/s of neighbour rows, 45 % of them out of L2); 60 k
// nodes, 12 M entries: 847 -> 266 us (12.1 TB/s); 100 k nodes, 3 M entries, 8 x 32: 1392 -> 335 us; 200 k nodes, 4 M entries,
// 1 x 8: 409 -> 84 us.
template <int LPG, int W>
__global__ void __launch_bounds__(kGatThreads, kGatBlocksPerSm) gat_lane_rows_kernel(GatArgs a, GatRowOrder order, GatGrid grid,
                                                                                     int vec_out, int vec_out16) {
    __shared__ Cols<W> sm_acc[2][kGatWarps][LPG];      // (used in turn: one barrier a hub row)
    __shared__ float2 sm_ml[2][kGatWarps][LPG];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const GatLanes<LPG, W> L(lane, a.dim, a.head_dim);
    GatForwardPass<LPG, W> pass(a, L);
    auto store_cols = [&](int64_t i, int64_t v, Cols<W> z, float den) {      // (entry i of the order)
#pragma unroll
        for (int k = 0; k < W; ++k) z.v[k] /= den;
        if (a.out) z.store(a.out + v * a.ldout + L.col, vec_out != 0);
        if (a.out16) z.store(a.out16 + (order.slots ? (int64_t)order.slots[i] : v) * a.ldout16 + L.col, vec_out16 != 0);
    };
    auto store_row = [&](int64_t i, int64_t v, int32_t total) {
        if (!L.on) return;
        if (total == 0) pass.st.acc.zero();                     // an empty row leaves zeros
        store_cols(i, v, pass.st.acc, total > 0 ? pass.st.l - pass.st.lost : 1.f);
    };
    if ((int)blockIdx.x >= grid.hub_blocks) {
        int rows;
        const int64_t i0 = gat_first_row<LPG>(order, grid, (int64_t)((int)blockIdx.x - grid.hub_blocks) * kGatWarps + warp, rows);
        if (rows == 0) return;
        const GatRow row = load_row_entry(order.rows + i0 + min(L.g, rows - 1));
        const int64_t v = row.v, beg = row.beg;
        const int32_t deg = row.deg;
        const int32_t total = L.g < rows ? deg + a.self_loop : INT32_MAX;      // (beyond the last row: nobody's)
        const bool mine = total <= kGatGroupEntries;
        const int32_t longest = __reduce_max_sync(0xffffffffu, mine ? total : 0);
        pass.begin(v);
        gat_walk_by_group<LPG, W>(pass, L, a.colidx, (int32_t)v, beg, deg, mine ? total : 0, longest);
        if (mine) store_row(i0 + L.g, v, total);
        unsigned longer = __ballot_sync(0xffffffffu, L.li == 0 && !mine && L.g < rows);
        while (longer) {
            const int src = __ffs(longer) - 1;
            longer &= longer - 1;
            const int64_t w = __shfl_sync(0xffffffffu, v, src), w_beg = __shfl_sync(0xffffffffu, beg, src);
            const int32_t w_deg = __shfl_sync(0xffffffffu, deg, src);
            pass.begin(w);
            gat_walk_by_warp<LPG, W>(pass, L, a.colidx, (int32_t)w, w_beg, w_deg, w_deg + a.self_loop, 0, kWarp, lane);
            pass.st.template merge_groups<LPG>();
            if (L.g == 0) store_row(i0 + src / LPG, w, w_deg + a.self_loop);
        }
        return;
    }
    const int n_hubs = *order.counts;
    int turn = 0;
    for (int hub = blockIdx.x; hub < n_hubs; hub += grid.hub_blocks, turn ^= 1) {
        const GatRow row = order.rows[hub];
        const int64_t v = row.v, beg = row.beg;
        const int32_t deg = row.deg;
        pass.begin(v);
        gat_walk_by_warp<LPG, W>(pass, L, a.colidx, (int32_t)v, beg, deg, deg + a.self_loop, warp * kWarp, kGatWarps * kWarp, lane);
        pass.st.template merge_groups<LPG>();
        if (L.g == 0) {
            sm_acc[turn][warp][L.li] = pass.st.acc;
            sm_ml[turn][warp][L.li] = make_float2(pass.st.m, pass.st.l);
        }
        __syncthreads();
        if (warp == 0 && L.g == 0 && L.on) {
            float big = -INFINITY, den = 0.f;
            for (int w = 0; w < kGatWarps; ++w) big = fmaxf(big, sm_ml[turn][w][L.li].x);
            Cols<W> z;
            z.zero();
            for (int w = 0; w < kGatWarps; ++w) {
                const float f = exp_rel(sm_ml[turn][w][L.li].x, big);                 // (0 for a warp without trips)
                den = fmaf(sm_ml[turn][w][L.li].y, f, den);
                z.fma(f, sm_acc[turn][w][L.li]);
            }
            store_cols(hub, v, z, den);
        }
    }
}

// ---------------------------------------------------------------- any other shape
// s_u = <a_src, p_u>, t_u = <a_dst, p_u> per head; one warp per node.  The warp also lists its node
// if the node's row is long enough for a whole block.
__global__ void __launch_bounds__(kGatRowThreads) gat_scores_kernel(GatArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t u = blockIdx.x * (int64_t)kGatRowWarps + (threadIdx.x >> 5);
    if (u >= a.n) return;
    if (lane == 0 && a.rowptr[u + 1] - a.rowptr[u] + (a.self_loop ? 1 : 0) >= kGatHubEntries)
        a.hub_list[atomicAdd(a.hub_count, 1)] = (int32_t)u;
    const float* row = a.p + u * a.ldp;
    for (int h = 0; h < a.heads; ++h) {
        float ss = 0.f, tt = 0.f;
        for (int j = lane; j < a.head_dim; j += kWarp) {
            const float x = row[h * a.head_dim + j];
            ss = fmaf(a.a_src[h * a.head_dim + j], x, ss);
            tt = fmaf(a.a_dst[h * a.head_dim + j], x, tt);
        }
        ss = warp_sum(ss);
        tt = warp_sum(tt);
        if (lane == 0) {
            a.s[u * a.heads + h] = ss;
            a.t[u * a.heads + h] = tt;
        }
    }
}

// The running soft-max state and weighted sum of one warp over the entries [e0, e0 + 32) of row v, for
// e0 = e_first, e_first + e_step, ...  (entry `deg`, if any, is the self loop).  Entries are taken 32 at
// a time: lane j scores entry j for every head, the chunk maximum and the rescale of the running
// soft-max state are warp reductions (one exp per entry and head in total), then all lanes add the
// weighted neighbour rows for the columns they own.
template <int NC>
__device__ __forceinline__ void gat_accumulate(const GatArgs& a, int64_t v, int64_t beg, int64_t deg, int64_t total,
                                               int64_t e_first, int64_t e_step, int lane, int warp,
                                               float (*p_s)[kWarp][kGatMaxHeads], const float (&tv)[kGatMaxHeads],
                                               const int (&head_of)[NC], float (&m)[kGatMaxHeads],
                                               float (&l)[kGatMaxHeads], float (&acc)[NC]) {
    for (int64_t e0 = e_first; e0 < total; e0 += e_step) {
        const int cnt = (int)min((int64_t)kWarp, total - e0);
        int my_u = 0;
        float e[kGatMaxHeads];
        const bool valid = lane < cnt;
        if (valid) my_u = (e0 + lane < deg) ? __ldg(a.colidx + beg + e0 + lane) : (int)v;
#pragma unroll
        for (int h = 0; h < kGatMaxHeads; ++h) {
            e[h] = -INFINITY;
            if (valid && h < a.heads) {
                const float z = a.s[(int64_t)my_u * a.heads + h] + tv[h];
                e[h] = z > 0.f ? z : a.slope * z;
            }
        }
        float scale[kGatMaxHeads];
#pragma unroll
        for (int h = 0; h < kGatMaxHeads; ++h) {
            scale[h] = 1.f;
            if (h < a.heads) {
                const float mn = fmaxf(m[h], warp_max(e[h]));     // finite: cnt >= 1
                scale[h] = expf(m[h] - mn);                       // exp(-inf) = 0 on the first chunk
                const float pj = valid ? expf(e[h] - mn) : 0.f;
                l[h] = l[h] * scale[h] + warp_sum(pj);
                m[h] = mn;
                p_s[warp][lane][h] = pj;
            }
        }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            float sc = 1.f;
#pragma unroll
            for (int h = 0; h < kGatMaxHeads; ++h) if (h == head_of[c]) sc = scale[h];
            acc[c] *= sc;
        }
        // several neighbour rows in flight per lane (a hub's row is otherwise one dependent load after
        // another); the products are still added in entry order
        constexpr int U = NC <= 2 ? 8 : (NC <= 4 ? 4 : 2);
        int j = 0;
        for (; j + U <= cnt; j += U) {
            float x[U][NC];
#pragma unroll
            for (int t = 0; t < U; ++t) {
                const int u = __shfl_sync(0xffffffffu, my_u, j + t);
                const float* row = a.p + (int64_t)u * a.ldp;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const int col = c * kWarp + lane;
                    x[t][c] = col < a.dim ? __ldg(row + col) : 0.f;
                }
            }
#pragma unroll
            for (int t = 0; t < U; ++t)
#pragma unroll
                for (int c = 0; c < NC; ++c) acc[c] = fmaf(p_s[warp][j + t][head_of[c]], x[t][c], acc[c]);
        }
        for (; j < cnt; ++j) {
            const int u = __shfl_sync(0xffffffffu, my_u, j);
            const float* row = a.p + (int64_t)u * a.ldp;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int col = c * kWarp + lane;
                if (col < a.dim) acc[c] = fmaf(p_s[warp][j][head_of[c]], __ldg(row + col), acc[c]);
            }
        }
        __syncwarp();
    }
}

// Blocks [0, hub_blocks): one block per listed hub row at a time.  Warp w takes the trips w, w + 8, ...
// of the row with a soft-max state of its own; the eight states are then merged in warp order
//   M = max m_w,  L = sum l_w e^(m_w - M),  Z = sum acc_w e^(m_w - M) / L,
// so the result does not depend on scheduling (it differs from the one-warp order only in rounding).
// Blocks from hub_blocks on: one warp per destination v, rows of fewer than kGatHubEntries entries.
// The hub blocks come first in launch order, so the longest rows start ahead of the short ones.
template <int NC>
__global__ void __launch_bounds__(kGatRowThreads) gat_rows_kernel(GatArgs a, int hub_blocks) {
    __shared__ float p_s[kGatRowWarps][kWarp][kGatMaxHeads];
    __shared__ float sm_m[kGatRowWarps][kGatMaxHeads], sm_l[kGatRowWarps][kGatMaxHeads];
    __shared__ float sm_acc[kGatRowWarps][NC * kWarp];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool hub_block = (int)blockIdx.x < hub_blocks;
    const int n_hubs = hub_block ? *a.hub_count : 0;
    int hub = blockIdx.x;
    int64_t v = hub_block ? -1 : (int64_t)(blockIdx.x - hub_blocks) * kGatRowWarps + warp;
    if (!hub_block && v >= a.n) return;

    float m[kGatMaxHeads], l[kGatMaxHeads], tv[kGatMaxHeads];
    float acc[NC];
    int head_of[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int col = c * kWarp + lane;
        head_of[c] = col < a.dim ? col / a.head_dim : 0;
    }

    if (!hub_block) {
        const int64_t beg = a.rowptr[v];
        const int64_t deg = a.rowptr[v + 1] - beg;
        const int64_t total = deg + (a.self_loop ? 1 : 0);
        if (total >= kGatHubEntries) return;                 // a hub block takes this row
#pragma unroll
        for (int h = 0; h < kGatMaxHeads; ++h) {
            m[h] = -INFINITY;
            l[h] = 0.f;
            tv[h] = h < a.heads ? a.t[v * a.heads + h] : 0.f;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = 0.f;
        gat_accumulate<NC>(a, v, beg, deg, total, 0, kWarp, lane, warp, p_s, tv, head_of, m, l, acc);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int col = c * kWarp + lane;
            if (col < a.dim) {
                float val = 0.f;
                if (total > 0) {
                    float lh = 1.f;
#pragma unroll
                    for (int h = 0; h < kGatMaxHeads; ++h) if (h == head_of[c]) lh = l[h];
                    val = acc[c] / lh;
                }
                if (a.out) a.out[v * a.ldout + col] = val;
                if (a.out16) a.out16[v * a.ldout16 + col] = f32_to_bf16(val);
            }
        }
        return;
    }

    for (; hub < n_hubs; hub += hub_blocks) {
        v = a.hub_list[hub];
        const int64_t beg = a.rowptr[v];
        const int64_t deg = a.rowptr[v + 1] - beg;
        const int64_t total = deg + (a.self_loop ? 1 : 0);
#pragma unroll
        for (int h = 0; h < kGatMaxHeads; ++h) {
            m[h] = -INFINITY;
            l[h] = 0.f;
            tv[h] = h < a.heads ? a.t[v * a.heads + h] : 0.f;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = 0.f;
        gat_accumulate<NC>(a, v, beg, deg, total, (int64_t)warp * kWarp, (int64_t)kGatRowWarps * kWarp, lane, warp, p_s, tv,
                           head_of, m, l, acc);
        if (lane < kGatMaxHeads) {
            float mm = -INFINITY, ll = 0.f;
#pragma unroll
            for (int h = 0; h < kGatMaxHeads; ++h) if (h == lane) { mm = m[h]; ll = l[h]; }
            sm_m[warp][lane] = mm;
            sm_l[warp][lane] = ll;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) sm_acc[warp][c * kWarp + lane] = acc[c];
        __syncthreads();
        for (int col = threadIdx.x; col < a.dim; col += kGatRowThreads) {
            const int h = col / a.head_dim;
            float big = -INFINITY;
            for (int w = 0; w < kGatRowWarps; ++w) big = fmaxf(big, sm_m[w][h]);
            float den = 0.f, num = 0.f;
            for (int w = 0; w < kGatRowWarps; ++w) {
                const float f = sm_m[w][h] == -INFINITY ? 0.f : expf(sm_m[w][h] - big);     // (a warp without trips)
                den = fmaf(sm_l[w][h], f, den);
                num = fmaf(sm_acc[w][col], f, num);
            }
            const float val = num / den;
            if (a.out) a.out[v * a.ldout + col] = val;
            if (a.out16) a.out16[v * a.ldout16 + col] = f32_to_bf16(val);
        }
        __syncthreads();
    }
}

void gat_forward_workspace(int64_t n_nodes, int32_t heads, Sizer& s) {
    s.take<float>((size_t)n_nodes * (size_t)heads);                   // s
    s.take<float>((size_t)n_nodes * (size_t)heads);                   // t
    s.take<GatRow>((size_t)n_nodes);                                  // rows in order (general kernels: hub rows)
    s.take<int32_t>(kGatOrderInts);                                   // rows per class of lengths (general kernels: hub rows)
}

bool gat_lanes_usable(int32_t heads, int32_t head_dim, const float* p, int64_t ldp, const float* q, int64_t ldq) {
    int lpg, w;
    return heads > 0 && heads <= kGatMaxHeads && head_dim > 0 && gat_lanes_cover(heads * head_dim, head_dim, p, ldp, q, ldq, &lpg, &w);
}

int gat_order_launch(const retexo_csr& g, int32_t self_loop, const int32_t* const* idx, const int64_t* n_idx, int lists, GatRow* rows,
                     int32_t* slots, int32_t* bins, int hub_entries, cudaStream_t st) {
    RETEXO_CUDA_TRY(cudaMemsetAsync(bins, 0, kGatOrderInts * sizeof(int32_t), st));
    for (int i = 0; i < lists; ++i)
        if (n_idx[i]) gat_order_count_kernel<<<gat_order_blocks(n_idx[i]), 256, 0, st>>>(n_idx[i], idx[i], g.rowptr, self_loop, hub_entries, bins);
    int32_t slot0 = 0;
    for (int i = 0; i < lists; slot0 += (int32_t)n_idx[i++])
        if (n_idx[i])
            gat_order_kernel<<<gat_order_blocks(n_idx[i]), 256, 0, st>>>(n_idx[i], idx[i], g.rowptr, self_loop, hub_entries, bins, rows, slots, slot0);
    return launch_status();
}

int gat_forward_launch(const GatForward& f, Arena& ws, int n_sm, cudaStream_t st) {
    const int64_t n = f.g.n_nodes;
    GatArgs a;
    a.n = n; a.rowptr = f.g.rowptr; a.colidx = f.g.colidx; a.p = f.p; a.ldp = f.ldp;
    a.heads = f.gat.heads; a.head_dim = f.gat.head_dim; a.dim = f.gat.heads * f.gat.head_dim;
    a.a_src = f.gat.a_src; a.a_dst = f.gat.a_dst; a.slope = f.gat.negative_slope;
    a.self_loop = f.gat.add_self_loop ? 1 : 0;
    a.s = ws.take<float>((size_t)n * a.heads);
    a.t = ws.take<float>((size_t)n * a.heads);
    GatRow* rows = ws.take<GatRow>((size_t)n);
    int32_t* bins = ws.take<int32_t>(kGatOrderInts);
    a.hub_list = reinterpret_cast<int32_t*>(rows);
    a.hub_count = bins;
    a.out = f.out; a.ldout = f.ldout; a.out16 = f.out16; a.ldout16 = f.ldout16;
    int lpg, w;
    if (gat_lanes_cover(a.dim, a.head_dim, a.p, a.ldp, nullptr, 0, &lpg, &w)) {
        const int vec_out = f.out && f.ldout % 4 == 0 && aligned_to(f.out, 16);
        const int vec_out16 = f.out16 && f.ldout16 % 4 == 0 && aligned_to(f.out16, 8);
        const int hub_entries = gat_hub_entries(f.g.n_edges, n_sm);
        const bool own = !f.order.rows;
        const GatRowOrder order = own ? GatRowOrder{rows, bins + kGatOrderCounts, nullptr, n} : f.order;
        if (own) RETEXO_CUDA_TRY(cudaMemsetAsync(bins, 0, kGatOrderInts * sizeof(int32_t), st));
        const int rc = gat_lanes_dispatch(lpg, w, [&]<int LPG, int W>() {
            gat_lane_scores_kernel<LPG, W><<<gat_lane_scores_grid<LPG, W>(n, n_sm), 256, 0, st>>>(
                n, a.rowptr, a.p, a.ldp, a.heads, a.head_dim, a.a_src, a.a_dst, a.self_loop, hub_entries, a.s, a.t, own ? bins : nullptr);
            return launch_status();
        });
        RETEXO_TRY(rc);
        if (own) gat_order_kernel<<<gat_order_blocks(n), 256, 0, st>>>(n, nullptr, a.rowptr, a.self_loop, hub_entries, bins, rows, nullptr, 0);
        return gat_lanes_dispatch(lpg, w, [&]<int LPG, int W>() {
            const GatGrid grid = gat_grid<LPG>(order.n, f.g.n_edges + n, n_sm, 6 * n_sm);
            gat_lane_rows_kernel<LPG, W><<<grid.blocks, kGatThreads, 0, st>>>(a, order, grid, vec_out, vec_out16);
            return launch_status();
        });
    }
    RETEXO_CUDA_TRY(cudaMemsetAsync(a.hub_count, 0, sizeof(int32_t), st));
    const unsigned blocks = (unsigned)((n + kGatRowWarps - 1) / kGatRowWarps);
    const int hub_blocks = 3 * n_sm;       // as many as are resident at once; those without a row leave at once
    const unsigned grid = blocks + (unsigned)hub_blocks;
    gat_scores_kernel<<<blocks, kGatRowThreads, 0, st>>>(a);
    const int nc = (a.dim + kWarp - 1) / kWarp;
    if (nc <= 1) gat_rows_kernel<1><<<grid, kGatRowThreads, 0, st>>>(a, hub_blocks);
    else if (nc <= 2) gat_rows_kernel<2><<<grid, kGatRowThreads, 0, st>>>(a, hub_blocks);
    else if (nc <= 4) gat_rows_kernel<4><<<grid, kGatRowThreads, 0, st>>>(a, hub_blocks);
    else gat_rows_kernel<8><<<grid, kGatRowThreads, 0, st>>>(a, hub_blocks);
    return launch_status();
}

}  // namespace retexo
