// Backward of the GAT aggregation (Section 2.2: AGGR may have trainable parameters; Section 3.1: a round
// trains the whole layer).  With z_uv = s_u + t_v, e = LeakyReLU(z), alpha = softmax over u in N(v) (+ v),
// Z_v = sum_u alpha_uv p_u and dz = dLoss/dZ:
//   dalpha_uv = <dz_v, p_u>             de_uv = alpha_uv (dalpha_uv - c_v),  c_v = sum_w alpha_wv dalpha_wv
//   dzz_uv    = de_uv (z_uv > 0 ? 1 : slope)
//   dt_v = sum_u dzz_uv                 ds_u = sum_v dzz_uv
//   dp_u = sum_v alpha_uv dz_v + ds_u a_src + dt_u a_dst
//   da_src = sum_u ds_u p_u             da_dst = sum_v dt_v p_v
// Two passes over the same CSR (the graph is symmetric, so the rows that attend over u are u's own row):
// the destinations first (soft-max statistics, c_v and dt_v), then the sources u, which walk the destinations v that attend
// over them and accumulate ds_u and dp_u.  No floating-point atomics: the parameter gradients are summed per block and the
// block sums in block order.  Shapes the lane layout of gat_lanes.cuh covers take its kernels, every other shape the general
// ones (one warp per row, shuffles per entry).
#include <algorithm>

#include "common.cuh"
#include "gat_lanes.cuh"

namespace retexo {

constexpr int kGbThreads = 256, kGbWarps = kGbThreads / kWarp, kGbMaxHeads = 8;

struct GatBwdArgs {
    int64_t n;
    const int64_t* rowptr;
    const int32_t* colidx;
    const float* p; int64_t ldp;
    int32_t heads, head_dim, dim;
    const float* a_src; const float* a_dst;
    float slope; int32_t self_loop;
    const float* dz; int64_t lddz;
    float* s; float* t;              // [n x heads]
    float4* stats;                   // [n x heads]: (row maximum, 1 / soft-max sum (0 = dz_v is zero), c_v, dt_v; lane layout: t_v)
    float* dp; int64_t lddp;
    __nv_bfloat16* dp16; int64_t lddp16;
    float* partial;                  // [blocks x 2 x dim]: per-block sums of ds_u p_u and dt_u p_u
    // lane layout only
    float* ds; float* dt;                       // [n x heads]
    int32_t* done;                              // blocks of the parameters' kernel that are done
};

__global__ void __launch_bounds__(kGbThreads) gat_bwd_scores_kernel(GatBwdArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t u = blockIdx.x * (int64_t)kGbWarps + (threadIdx.x >> 5);
    if (u >= a.n) return;
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
        if (lane == 0) { a.s[u * a.heads + h] = ss; a.t[u * a.heads + h] = tt; }
    }
}

// <x, y> restricted to each head's columns, summed over the warp: every lane ends up with all heads' values.
template <int NC>
__device__ __forceinline__ void head_dots(const float (&x)[NC], const float (&y)[NC], const int (&head_of)[NC], int heads,
                                          float (&out)[kGbMaxHeads]) {
#pragma unroll
    for (int h = 0; h < kGbMaxHeads; ++h) {
        out[h] = 0.f;
        if (h < heads) {
            float part = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) part = head_of[c] == h ? fmaf(x[c], y[c], part) : part;
            out[h] = warp_sum(part);
        }
    }
}

// Pass over destinations: one warp per v.  Lane L owns the columns L, L + 32, ...
template <int NC>
__global__ void __launch_bounds__(kGbThreads) gat_bwd_dst_kernel(GatBwdArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t v = blockIdx.x * (int64_t)kGbWarps + (threadIdx.x >> 5);
    if (v >= a.n) return;
    int head_of[NC];
    float g[NC];
    bool any = false;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int col = c * kWarp + lane;
        head_of[c] = col < a.dim ? col / a.head_dim : -1;
        g[c] = col < a.dim ? a.dz[v * a.lddz + col] : 0.f;
        any = any || g[c] != 0.f;
    }
    const int64_t beg = a.rowptr[v];
    const int64_t deg = a.rowptr[v + 1] - beg;
    const int64_t total = deg + (a.self_loop ? 1 : 0);
    if (!__any_sync(0xffffffffu, any) || total == 0) {       // outside the loss: nothing flows back through this row
        if (lane < a.heads) a.stats[v * a.heads + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    float tv[kGbMaxHeads], m[kGbMaxHeads], den[kGbMaxHeads];
#pragma unroll
    for (int h = 0; h < kGbMaxHeads; ++h) {
        tv[h] = h < a.heads ? a.t[v * a.heads + h] : 0.f;
        m[h] = -INFINITY;
        den[h] = 0.f;
    }
    // sweep 1: row maximum and soft-max sum per head, 32 entries at a time (lane j scores entry j)
    for (int64_t e0 = 0; e0 < total; e0 += kWarp) {
        const bool valid = e0 + lane < total;
        const int64_t u = !valid ? v : (e0 + lane < deg ? (int64_t)__ldg(a.colidx + beg + e0 + lane) : v);
#pragma unroll
        for (int h = 0; h < kGbMaxHeads; ++h) {
            if (h < a.heads) {
                const float z = a.s[u * a.heads + h] + tv[h];
                const float e = valid ? (z > 0.f ? z : a.slope * z) : -INFINITY;
                const float mn = fmaxf(m[h], warp_max(e));
                den[h] = den[h] * expf(m[h] - mn) + warp_sum(valid ? expf(e - mn) : 0.f);
                m[h] = mn;
            }
        }
    }
    // sweep 2: c_v = sum alpha dalpha, and the two sums that give dt_v = sum alpha (dalpha - c_v) g'
    float csum[kGbMaxHeads], a1[kGbMaxHeads], a2[kGbMaxHeads];
#pragma unroll
    for (int h = 0; h < kGbMaxHeads; ++h) { csum[h] = 0.f; a1[h] = 0.f; a2[h] = 0.f; }
    for (int64_t e = 0; e < total; ++e) {
        const int64_t u = e < deg ? (int64_t)__ldg(a.colidx + beg + e) : v;
        float x[NC], dalpha[kGbMaxHeads];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int col = c * kWarp + lane;
            x[c] = col < a.dim ? __ldg(a.p + u * a.ldp + col) : 0.f;
        }
        head_dots<NC>(g, x, head_of, a.heads, dalpha);
#pragma unroll
        for (int h = 0; h < kGbMaxHeads; ++h) {
            if (h < a.heads) {
                const float z = a.s[u * a.heads + h] + tv[h];
                const float alpha = expf((z > 0.f ? z : a.slope * z) - m[h]) / den[h];
                const float gp = z > 0.f ? 1.f : a.slope;
                csum[h] = fmaf(alpha, dalpha[h], csum[h]);
                a1[h] = fmaf(alpha * gp, dalpha[h], a1[h]);
                a2[h] = fmaf(alpha, gp, a2[h]);
            }
        }
    }
#pragma unroll
    for (int h = 0; h < kGbMaxHeads; ++h)
        if (h < a.heads && lane == h) a.stats[v * a.heads + h] = make_float4(m[h], 1.f / den[h], csum[h], a1[h] - csum[h] * a2[h]);
}

// Pass over sources: one warp per u walks the destinations that attend over u (its own row, and itself).
template <int NC>
__global__ void __launch_bounds__(kGbThreads) gat_bwd_src_kernel(GatBwdArgs a) {
    __shared__ float sm_part[kGbWarps][2][NC * kWarp];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t u = blockIdx.x * (int64_t)kGbWarps + warp;
    int head_of[NC];
    float px[NC], acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int col = c * kWarp + lane;
        head_of[c] = col < a.dim ? col / a.head_dim : -1;
        px[c] = (u < a.n && col < a.dim) ? a.p[u * a.ldp + col] : 0.f;
        acc[c] = 0.f;
    }
    float ds[kGbMaxHeads], dtu[kGbMaxHeads], su[kGbMaxHeads];
#pragma unroll
    for (int h = 0; h < kGbMaxHeads; ++h) { ds[h] = 0.f; dtu[h] = 0.f; su[h] = 0.f; }
    if (u < a.n) {
#pragma unroll
        for (int h = 0; h < kGbMaxHeads; ++h) {
            if (h < a.heads) {
                su[h] = a.s[u * a.heads + h];
                dtu[h] = a.stats[u * a.heads + h].w;
            }
        }
        const int64_t beg = a.rowptr[u];
        const int64_t deg = a.rowptr[u + 1] - beg;
        const int64_t total = deg + (a.self_loop ? 1 : 0);
        for (int64_t e = 0; e < total; ++e) {
            const int64_t v = e < deg ? (int64_t)__ldg(a.colidx + beg + e) : u;
            if (a.stats[v * a.heads].y == 0.f) continue;      // dz_v is zero (the same for every lane)
            float g[NC], dalpha[kGbMaxHeads], alpha[kGbMaxHeads];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int col = c * kWarp + lane;
                g[c] = col < a.dim ? __ldg(a.dz + v * a.lddz + col) : 0.f;
            }
            head_dots<NC>(g, px, head_of, a.heads, dalpha);
#pragma unroll
            for (int h = 0; h < kGbMaxHeads; ++h) {
                alpha[h] = 0.f;
                if (h < a.heads) {
                    const float4 st = a.stats[v * a.heads + h];
                    const float z = su[h] + a.t[v * a.heads + h];
                    alpha[h] = expf((z > 0.f ? z : a.slope * z) - st.x) * st.y;
                    ds[h] = fmaf(alpha[h] * (z > 0.f ? 1.f : a.slope), dalpha[h] - st.z, ds[h]);
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                float al = 0.f;
#pragma unroll
                for (int h = 0; h < kGbMaxHeads; ++h) al = head_of[c] == h ? alpha[h] : al;
                acc[c] = fmaf(al, g[c], acc[c]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int col = c * kWarp + lane;
        float dsc = 0.f, dtc = 0.f;
#pragma unroll
        for (int h = 0; h < kGbMaxHeads; ++h) { dsc = head_of[c] == h ? ds[h] : dsc; dtc = head_of[c] == h ? dtu[h] : dtc; }
        if (u < a.n && col < a.dim) {
            const float val = acc[c] + dsc * a.a_src[col] + dtc * a.a_dst[col];
            if (a.dp) a.dp[u * a.lddp + col] = val;
            if (a.dp16) a.dp16[u * a.lddp16 + col] = f32_to_bf16(val);
        }
        sm_part[warp][0][c * kWarp + lane] = dsc * px[c];       // (zero beyond the last node / column)
        sm_part[warp][1][c * kWarp + lane] = dtc * px[c];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * a.dim; i += kGbThreads) {
        const int which = i / a.dim, col = i % a.dim;
        float sum = 0.f;
        for (int w = 0; w < kGbWarps; ++w) sum += sm_part[w][which][col];
        a.partial[((int64_t)blockIdx.x * 2 + which) * a.dim + col] = sum;
    }
}

// da_src / da_dst: one block per column sums the per-block partials, each thread its share in index order,
// then the 256 shares in thread order.
__global__ void __launch_bounds__(256) gat_bwd_reduce_kernel(const float* partial, int64_t n_blocks, int32_t dim,
                                                             float* da_src, float* da_dst) {
    __shared__ float share[256];
    const int which = blockIdx.x / dim, col = blockIdx.x % dim;
    float sum = 0.f;
    for (int64_t b = threadIdx.x; b < n_blocks; b += 256) sum += partial[(b * 2 + which) * dim + col];
    share[threadIdx.x] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        float total = 0.f;
        for (int t = 0; t < 256; ++t) total += share[t];
        (which ? da_dst : da_src)[col] = total;
    }
}

// ---------------------------------------------------------------- lane layout (gat_lanes.cuh)
// Destinations: for row v, with its own gradient dz_v in registers, the soft-max statistics and the sums
//   c_v = sum alpha dalpha,   dt_v = sum alpha g' dalpha - c_v sum alpha g'      (g' = 1 or the slope)
// in one pass over the entries with a running maximum.  dalpha = <dz_v, p_u> over the head's columns enters linearly, so a lane
// keeps the share of its own columns and the head's lanes are added once per row.  All four sums are compensated: c_v and dt_v are
// what is left of sums that cancel.
template <int LPG, int W>
struct GatDstPass {
    const GatBwdArgs& a;
    const float* p;
    const float* s;
    int head, col;
    bool on;
    float tv, m, den, c, b1, b2, den_lost, c_lost, b1_lost, b2_lost;
    Cols<W> g;
    __device__ __forceinline__ GatDstPass(const GatBwdArgs& a_, const GatLanes<LPG, W>& L)
        : a(a_), p(a_.p + L.col), s(a_.s + L.head), head(L.head), col(L.col), on(L.on) {}
    // Returns whether this lane's part of the gradient has a non-zero entry.
    __device__ __forceinline__ bool begin(int64_t v) {
        tv = __ldg(a.t + v * a.heads + head);
        m = -INFINITY; den = c = b1 = b2 = den_lost = c_lost = b1_lost = b2_lost = 0.f;
        g.load(a.dz + v * a.lddz + col);
        bool any = false;
#pragma unroll
        for (int i = 0; i < W; ++i) any = any || g.v[i] != 0.f;
        return on && any;
    }
    template <int U>
    __device__ __forceinline__ void batch(const int32_t (&u)[U], const bool (&ok)[U]) {
        Cols<W> x[U];
        float z[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
            z[t] = __ldg(s + (int64_t)u[t] * a.heads);
            x[t].load(p + (int64_t)u[t] * a.ldp);
        }
        float big = m, e[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
            z[t] += tv;
            e[t] = ok[t] ? leaky(z[t], a.slope) : -INFINITY;
            big = fmaxf(big, e[t]);
        }
        const float f = exp_rel(m, big), ref = big == -INFINITY ? 0.f : big;
        m = big;
        den *= f; c *= f; b1 *= f; b2 *= f;
        den_lost *= f; c_lost *= f; b1_lost *= f; b2_lost *= f;
        float den_more = -den_lost, c_more = -c_lost, b1_more = -b1_lost, b2_more = -b2_lost;
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const float w = exp_below(e[t], ref), wg = z[t] > 0.f ? w : w * a.slope, d = g.dot(x[t]);
            den_more += w;
            b2_more += wg;
            c_more = fmaf(w, d, c_more);
            b1_more = fmaf(wg, d, b1_more);
        }
        if (!ok[0]) return;      // (beyond the row's end nothing may change, not even what is lost)
        add_compensated(den, den_lost, den_more);
        add_compensated(c, c_lost, c_more);
        add_compensated(b1, b1_lost, b1_more);
        add_compensated(b2, b2_lost, b2_more);
    }
    __device__ __forceinline__ void merge(float m2, float den2, float c2, float b12, float b22) {
        const float big = fmaxf(m, m2), f = exp_rel(m, big), f2 = exp_rel(m2, big);
        den = den * f + den2 * f2; c = c * f + c2 * f2; b1 = b1 * f + b12 * f2; b2 = b2 * f + b22 * f2;
        m = big;
    }
    // Adds the states of the warp's groups (for a row of the whole warp) in a fixed tree.
    __device__ __forceinline__ void merge_groups() {
#pragma unroll
        for (int o = LPG; o < kWarp; o <<= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, m, o), den2 = __shfl_xor_sync(0xffffffffu, den, o);
            const float c2 = __shfl_xor_sync(0xffffffffu, c, o), b12 = __shfl_xor_sync(0xffffffffu, b1, o);
            const float b22 = __shfl_xor_sync(0xffffffffu, b2, o);
            merge(m2, den2, c2, b12, b22);
        }
    }
    // The lanes of a head add their columns' shares and its first lane writes the row's statistics; warp-uniform call.
    __device__ __forceinline__ void finish(int64_t v, bool live, bool write, int hw) {
        for (int o = 1; o < hw; o <<= 1) {
            c += __shfl_xor_sync(0xffffffffu, c, o);
            b1 += __shfl_xor_sync(0xffffffffu, b1, o);
        }
        if (!write || !on || col % a.head_dim != 0) return;
        const float inv = live ? 1.f / den : 0.f, cn = live ? c * inv : 0.f;
        a.stats[v * a.heads + head] = make_float4(live ? m : 0.f, inv, cn, tv);
        a.dt[v * a.heads + head] = live ? b1 * inv - cn * (b2 * inv) : 0.f;
    }
};

// Bound like the forward pass by the gather of p_u (4 dim + 4 heads bytes an entry); rows whose gradient is zero gather nothing.
// Measured, whole backward pass (a lane per entry reading its own row in 16-byte pieces before; heads of other shapes a warp
// per entry): 717 k nodes, 14 M entries, 4 x 16: 5319 -> 1936 us, in order of lengths 1350; 60 k nodes, 12 M entries: 2960 -> 733 us; 100 k nodes, 3 M
// entries, 8 x 32: 26.6 -> 0.92 ms; 200 k nodes, 4 M entries, 1 x 8: 834 -> 160 us.
template <int LPG, int W>
__global__ void __launch_bounds__(kGatThreads, kGatBlocksPerSm) gat_lane_dst_kernel(GatBwdArgs a, GatRowOrder order, GatGrid grid) {
    __shared__ float sm[2][kGatWarps][5][LPG];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const GatLanes<LPG, W> L(lane, a.dim, a.head_dim);
    GatDstPass<LPG, W> pass(a, L);
    const int hw = a.head_dim / W;
    if ((int)blockIdx.x >= grid.hub_blocks) {
        int rows;
        const int64_t i0 = gat_first_row<LPG>(order, grid, (int64_t)((int)blockIdx.x - grid.hub_blocks) * kGatWarps + warp, rows);
        if (rows == 0) return;
        const GatRow row = load_row_entry(order.rows + i0 + min(L.g, rows - 1));
        const int64_t v = row.v, beg = row.beg;
        const int32_t deg = row.deg;
        const int32_t total = L.g < rows ? deg + a.self_loop : INT32_MAX;
        const bool mine = total <= kGatGroupEntries;
        const unsigned lanes = __ballot_sync(0xffffffffu, pass.begin(v));
        const unsigned group = LPG == 32 ? 0xffffffffu : ((1u << (LPG & 31)) - 1u) << (L.g * LPG);
        const bool live = (lanes & group) != 0 && total > 0;      // else nothing flows back through this row
        const int32_t take = mine && live ? total : 0;
        gat_walk_by_group<LPG, W>(pass, L, a.colidx, (int32_t)v, beg, deg, take, __reduce_max_sync(0xffffffffu, take));
        pass.finish(v, live, mine, hw);
        unsigned longer = __ballot_sync(0xffffffffu, L.li == 0 && !mine && L.g < rows);
        while (longer) {
            const int src = __ffs(longer) - 1;
            longer &= longer - 1;
            const int64_t w = __shfl_sync(0xffffffffu, v, src), w_beg = __shfl_sync(0xffffffffu, beg, src);
            const int32_t w_deg = __shfl_sync(0xffffffffu, deg, src);
            const bool w_live = __any_sync(0xffffffffu, pass.begin(w));
            if (w_live) {
                gat_walk_by_warp<LPG, W>(pass, L, a.colidx, (int32_t)w, w_beg, w_deg, w_deg + a.self_loop, 0, kWarp, lane);
                pass.merge_groups();
            }
            pass.finish(w, w_live, L.g == 0, hw);
        }
        return;
    }
    const int n_hubs = *order.counts;
    int turn = 0;      // (of the rows that meet a barrier)
    for (int hub = blockIdx.x; hub < n_hubs; hub += grid.hub_blocks) {
        const GatRow row = order.rows[hub];
        const int64_t v = row.v, beg = row.beg;
        const int32_t deg = row.deg;
        const bool live = __any_sync(0xffffffffu, pass.begin(v));      // (the same in every warp)
        if (live) {
            gat_walk_by_warp<LPG, W>(pass, L, a.colidx, (int32_t)v, beg, deg, deg + a.self_loop, warp * kWarp, kGatWarps * kWarp, lane);
            pass.merge_groups();
            if (L.g == 0) {
                sm[turn][warp][0][L.li] = pass.m; sm[turn][warp][1][L.li] = pass.den; sm[turn][warp][2][L.li] = pass.c;
                sm[turn][warp][3][L.li] = pass.b1; sm[turn][warp][4][L.li] = pass.b2;
            }
            __syncthreads();
        }
        if (warp == 0) {      // the warps' states in warp order
            if (live) {
                for (int w = 1; w < kGatWarps; ++w)
                    pass.merge(sm[turn][w][0][L.li], sm[turn][w][1][L.li], sm[turn][w][2][L.li], sm[turn][w][3][L.li], sm[turn][w][4][L.li]);
            }
            pass.finish(v, live, L.g == 0, hw);
        }
        turn ^= live ? 1 : 0;
    }
}

// Sources: the rows v that attend over u are u's own row (the graph is symmetric) and u itself; with p_u in registers
//   acc_u = sum alpha_uv dz_v,   ds_u = sum alpha g' (<dz_v, p_u> - c_v),   dp_u = acc_u + ds_u a_src + dt_u a_dst.
// A destination whose gradient is zero (1 / den = 0 in its statistics) is not read.
template <int LPG, int W>
struct GatSrcPass {
    const GatBwdArgs& a;
    const float* dz;
    const float4* stats;
    int head, col, hw;
    float su, ds, ds_lost;            // (the same in all lanes of a head)
    Cols<W> px, acc;
    __device__ __forceinline__ GatSrcPass(const GatBwdArgs& a_, const GatLanes<LPG, W>& L)
        : a(a_), dz(a_.dz + L.col), stats(a_.stats + L.head), head(L.head), col(L.col), hw(a_.head_dim / W) {}
    __device__ __forceinline__ void begin(int64_t u) {
        su = __ldg(a.s + u * a.heads + head);
        px.load(a.p + u * a.ldp + col);
        ds = ds_lost = 0.f;
        acc.zero();
    }
    template <int U>
    __device__ __forceinline__ void batch(const int32_t (&v)[U], const bool (&ok)[U]) {
        Cols<W> g[U];
        float4 st[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
            st[t] = __ldg(stats + (int64_t)v[t] * a.heads);
            if (!ok[t]) st[t].y = 0.f;
        }
#pragma unroll
        for (int t = 0; t < U; ++t) {
            g[t].zero();
            if (st[t].y != 0.f) g[t].load(dz + (int64_t)v[t] * a.lddz);
        }
        float more = -ds_lost;
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const float z = su + st[t].w;
            const float alpha = st[t].y != 0.f ? exp_below(leaky(z, a.slope), st[t].x) * st[t].y : 0.f;
            const float ag = z > 0.f ? alpha : alpha * a.slope;
            float d = px.dot(g[t]);           // of the whole head: what d and c_v have in common goes before anything is added up
            for (int o = 1; o < hw; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            more = fmaf(ag, d - st[t].z, more);
            acc.fma(alpha, g[t]);
        }
        if (ok[0]) add_compensated(ds, ds_lost, more);
    }
    __device__ __forceinline__ void merge_groups() {
#pragma unroll
        for (int o = LPG; o < kWarp; o <<= 1) {
            ds += __shfl_xor_sync(0xffffffffu, ds, o);
            acc.add_xor(o);
        }
    }
    // (the attention vectors are read here: held through the walk, their 16 registers a lane were spilled)
    __device__ __forceinline__ void finish(int64_t u, bool write, bool vec, bool vec16) {
        if (!write) return;
        const float dt = __ldg(a.dt + u * a.heads + head);
        Cols<W> att;
        att.load_unaligned(a.a_src + col);
        acc.fma(ds, att);
        att.load_unaligned(a.a_dst + col);
        acc.fma(dt, att);
        if (a.dp) acc.store(a.dp + u * a.lddp + col, vec);
        if (a.dp16) acc.store(a.dp16 + u * a.lddp16 + col, vec16);
        if (col % a.head_dim == 0) a.ds[u * a.heads + head] = ds;
    }
};

// Bound by the gather of dz_v and the statistics (4 dim + 16 heads bytes an entry).
template <int LPG, int W>
__global__ void __launch_bounds__(kGatThreads, kGatBlocksPerSm) gat_lane_src_kernel(GatBwdArgs a, GatRowOrder order, GatGrid grid,
                                                                                    int vec, int vec16) {
    __shared__ Cols<W> sm_acc[2][kGatWarps][LPG];
    __shared__ float sm_ds[2][kGatWarps][LPG];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const GatLanes<LPG, W> L(lane, a.dim, a.head_dim);
    GatSrcPass<LPG, W> pass(a, L);
    if ((int)blockIdx.x >= grid.hub_blocks) {
        int rows;
        const int64_t i0 = gat_first_row<LPG>(order, grid, (int64_t)((int)blockIdx.x - grid.hub_blocks) * kGatWarps + warp, rows);
        if (rows == 0) return;
        const GatRow row = load_row_entry(order.rows + i0 + min(L.g, rows - 1));
        const int64_t u = row.v, beg = row.beg;
        const int32_t deg = row.deg;
        const int32_t total = L.g < rows ? deg + a.self_loop : INT32_MAX;
        const bool mine = total <= kGatGroupEntries;
        pass.begin(u);
        gat_walk_by_group<LPG, W>(pass, L, a.colidx, (int32_t)u, beg, deg, mine ? total : 0, __reduce_max_sync(0xffffffffu, mine ? total : 0));
        pass.finish(u, mine && L.on, vec != 0, vec16 != 0);
        unsigned longer = __ballot_sync(0xffffffffu, L.li == 0 && !mine && L.g < rows);
        while (longer) {
            const int src = __ffs(longer) - 1;
            longer &= longer - 1;
            const int64_t w = __shfl_sync(0xffffffffu, u, src), w_beg = __shfl_sync(0xffffffffu, beg, src);
            const int32_t w_deg = __shfl_sync(0xffffffffu, deg, src);
            pass.begin(w);
            gat_walk_by_warp<LPG, W>(pass, L, a.colidx, (int32_t)w, w_beg, w_deg, w_deg + a.self_loop, 0, kWarp, lane);
            pass.merge_groups();
            pass.finish(w, L.g == 0 && L.on, vec != 0, vec16 != 0);
        }
        return;
    }
    const int n_hubs = *order.counts;
    int turn = 0;
    for (int hub = blockIdx.x; hub < n_hubs; hub += grid.hub_blocks, turn ^= 1) {
        const GatRow row = order.rows[hub];
        const int64_t u = row.v, beg = row.beg;
        const int32_t deg = row.deg;
        pass.begin(u);
        gat_walk_by_warp<LPG, W>(pass, L, a.colidx, (int32_t)u, beg, deg, deg + a.self_loop, warp * kWarp, kGatWarps * kWarp, lane);
        pass.merge_groups();
        if (L.g == 0) {
            sm_acc[turn][warp][L.li] = pass.acc;
            sm_ds[turn][warp][L.li] = pass.ds;
        }
        __syncthreads();
        if (warp == 0) {      // the warps' sums in warp order
            for (int w = 1; w < kGatWarps; ++w) {
                pass.acc.fma(1.f, sm_acc[turn][w][L.li]);
                pass.ds += sm_ds[turn][w][L.li];
            }
            pass.finish(u, L.g == 0 && L.on, vec != 0, vec16 != 0);
        }
    }
}

// da_src = sum_u ds_u p_u, da_dst = sum_u dt_u p_u: one stream over p (the sums of a hub row come from whichever block took it, so
// they are added here, where every node has a fixed place), per block, and by the last block to finish in block order.
// Latency on small graphs: four nodes a group and 24 block sums a thread are asked for before the first is added (two and eight
// before): 22 k nodes, 4 x 16: 15.2 -> 6.2 us (2 nodes 6.8, 8 nodes 5.8); 717 k nodes 41 us = 4.7 TB/s (2 nodes 45).
template <int LPG, int W>
__global__ void __launch_bounds__(256) gat_lane_params_kernel(GatBwdArgs a, float* __restrict__ da_src, float* __restrict__ da_dst) {
    constexpr int G = GatLanes<LPG, W>::G, kParts = 256 / LPG;
    __shared__ Cols<W> sm[2][kParts][LPG];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const GatLanes<LPG, W> L(lane, a.dim, a.head_dim);
    Cols<W> s0, s1;
    s0.zero(); s1.zero();
    constexpr int U = 4;      // nodes a group has in flight
    const int64_t step = (int64_t)gridDim.x * 8 * G;
    for (int64_t u0 = ((int64_t)blockIdx.x * 8 + warp) * G + L.g; u0 < a.n; u0 += U * step) {
        Cols<W> x[U];
        float ds[U], dt[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t u = u0 + k * step;
            x[k].zero();
            ds[k] = dt[k] = 0.f;
            if (u < a.n) {
                x[k].load(a.p + u * a.ldp + L.col);
                ds[k] = __ldg(a.ds + u * a.heads + L.head);
                dt[k] = __ldg(a.dt + u * a.heads + L.head);
            }
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            s0.fma(ds[k], x[k]);
            s1.fma(dt[k], x[k]);
        }
    }
    sm[0][warp * G + L.g][L.li] = s0;
    sm[1][warp * G + L.g][L.li] = s1;
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * a.dim; i += 256) {
        const int which = i / a.dim, col = i % a.dim;
        float sum = 0.f;
        for (int k = 0; k < kParts; ++k) sum += sm[which][k][col / W].v[col % W];
        a.partial[(int64_t)blockIdx.x * 2 * a.dim + i] = sum;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(a.done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    if (threadIdx.x == 0) *a.done = 0;      // for the next pass over this scratch
    __threadfence();
    // every column by 256 / (2 dim) threads (one where the columns are more), each its share of the blocks in order
    const int cols = 2 * a.dim, shares = cols < 256 ? 256 / cols : 1;
    float* share_sum = &sm[0][0][0].v[0];
    for (int i = threadIdx.x; i < shares * cols; i += 256) {
        const int col = i % cols, share = i / cols;
        float sum = 0.f;
        for (int b0 = share; b0 < (int)gridDim.x; b0 += 24 * shares) {
            float x[24];
#pragma unroll
            for (int k = 0; k < 24; ++k) x[k] = b0 + k * shares < (int)gridDim.x ? __ldcg(a.partial + (int64_t)(b0 + k * shares) * cols + col) : 0.f;
#pragma unroll
            for (int k = 0; k < 24; ++k) sum += x[k];
        }
        share_sum[i] = sum;
    }
    __syncthreads();
    for (int col = threadIdx.x; col < cols; col += 256) {
        float sum = 0.f;
        for (int share = 0; share < shares; ++share) sum += share_sum[share * cols + col];
        (col < a.dim ? da_src : da_dst)[col % a.dim] = sum;
    }
}

template <int NC>
static int launch_bwd(const GatBwdArgs& a, unsigned blocks, float* da_src, float* da_dst, cudaStream_t st) {
    gat_bwd_dst_kernel<NC><<<blocks, kGbThreads, 0, st>>>(a);
    gat_bwd_src_kernel<NC><<<blocks, kGbThreads, 0, st>>>(a);
    gat_bwd_reduce_kernel<<<(unsigned)(2 * a.dim), 256, 0, st>>>(a.partial, blocks, a.dim, da_src, da_dst);
    return launch_status();
}

}  // namespace retexo

using namespace retexo;

constexpr int64_t kGatParamBlocks = 296;      // blocks of gat_lane_params_kernel at most (the last one adds their sums)

extern "C" size_t retexo_gat_backward_workspace_size(int64_t n_nodes, int64_t n_edges, int32_t heads, int32_t dim) {
    if (n_nodes < 0 || n_edges < 0 || heads <= 0 || dim <= 0) return 0;
    Sizer s;
    s.take<float>((size_t)n_nodes * heads);
    s.take<float>((size_t)n_nodes * heads);
    s.take<float4>((size_t)n_nodes * heads);
    s.take<float>((size_t)std::max<int64_t>((n_nodes + kGbWarps - 1) / kGbWarps, kGatParamBlocks) * 2 * (size_t)dim);
    s.take<float>((size_t)n_nodes * heads);
    s.take<float>((size_t)n_nodes * heads);
    s.take<int32_t>(kGatOrderInts + 64);
    s.take<GatRow>((size_t)n_nodes);
    return s.off + kAlign;
}

extern "C" int retexo_gat_backward(const retexo_csr* g, const float* p, int64_t ldp, const retexo_gat_params* gat,
                                   const float* dz, int64_t lddz, float* dp, int64_t lddp, void* dp_bf16,
                                   int64_t lddp_bf16, float* da_src, float* da_dst, void* workspace,
                                   size_t workspace_bytes, void* stream) {
    return gat_backward(g, p, ldp, gat, dz, lddz, dp, lddp, dp_bf16, lddp_bf16, da_src, da_dst, workspace, workspace_bytes, nullptr,
                        static_cast<cudaStream_t>(stream));
}

// Scratch, in the order retexo_gat_backward_workspace_size lists it.
struct GatBwdScratch { float *s, *t; float4* stats; float* partial; float *ds, *dt; int32_t* bins; GatRow* rows; };
static GatBwdScratch backward_scratch(int64_t n, int32_t heads, int32_t dim, void* workspace, size_t workspace_bytes) {
    Arena ws(workspace, workspace_bytes);
    GatBwdScratch b;
    b.s = ws.take<float>((size_t)n * heads);
    b.t = ws.take<float>((size_t)n * heads);
    b.stats = ws.take<float4>((size_t)n * heads);
    b.partial = ws.take<float>((size_t)std::max<int64_t>((n + kGbWarps - 1) / kGbWarps, kGatParamBlocks) * 2 * (size_t)dim);
    b.ds = ws.take<float>((size_t)n * heads);
    b.dt = ws.take<float>((size_t)n * heads);
    b.bins = ws.take<int32_t>(kGatOrderInts + 64);
    b.rows = ws.take<GatRow>((size_t)n);
    return b;
}

int retexo::gat_backward_prepare(int64_t n_nodes, int64_t n_edges, int32_t heads, int32_t head_dim, void* workspace, size_t workspace_bytes,
                                 cudaStream_t st) {
    if (workspace_bytes < retexo_gat_backward_workspace_size(n_nodes, n_edges, heads, heads * head_dim)) return RETEXO_ERR_WORKSPACE;
    const GatBwdScratch b = backward_scratch(n_nodes, heads, heads * head_dim, workspace, workspace_bytes);
    RETEXO_CUDA_TRY(cudaMemsetAsync(b.stats, 0, sizeof(float4) * (size_t)n_nodes * heads, st));
    RETEXO_CUDA_TRY(cudaMemsetAsync(b.dt, 0, sizeof(float) * (size_t)n_nodes * heads, st));
    RETEXO_CUDA_TRY(cudaMemsetAsync(b.bins, 0, (kGatOrderInts + 64) * sizeof(int32_t), st));
    return RETEXO_OK;
}

int retexo::gat_backward(const retexo_csr* g, const float* p, int64_t ldp, const retexo_gat_params* gat, const float* dz, int64_t lddz,
                         float* dp, int64_t lddp, void* dp_bf16, int64_t lddp_bf16, float* da_src, float* da_dst, void* workspace,
                         size_t workspace_bytes, const GatBackwardKept* kept, cudaStream_t st) {
    if (!g || g->n_nodes < 0 || g->n_edges < 0 || g->n_nodes > INT32_MAX) return RETEXO_ERR_INVALID_ARG;
    if (!gat || gat->heads <= 0 || gat->head_dim <= 0 || !gat->a_src || !gat->a_dst) return RETEXO_ERR_INVALID_ARG;
    const int32_t dim = gat->heads * gat->head_dim;
    if (gat->heads > kGbMaxHeads || dim > 256) return RETEXO_ERR_UNSUPPORTED;
    if (!da_src || !da_dst || (!dp && !dp_bf16)) return RETEXO_ERR_INVALID_ARG;
    if (ldp < dim || lddz < dim || (dp && lddp < dim) || (dp_bf16 && lddp_bf16 < dim)) return RETEXO_ERR_INVALID_ARG;
    if (g->n_nodes == 0) {
        RETEXO_CUDA_TRY(cudaMemsetAsync(da_src, 0, sizeof(float) * dim, st));
        RETEXO_CUDA_TRY(cudaMemsetAsync(da_dst, 0, sizeof(float) * dim, st));
        return RETEXO_OK;
    }
    if (!g->rowptr || !p || !dz || (g->n_edges > 0 && !g->colidx)) return RETEXO_ERR_INVALID_ARG;
    const size_t need = retexo_gat_backward_workspace_size(g->n_nodes, g->n_edges, gat->heads, dim);
    if (!workspace || !aligned_to(workspace, kAlign) || workspace_bytes < need) return RETEXO_ERR_WORKSPACE;
    const int64_t n = g->n_nodes;
    const GatBwdScratch b = backward_scratch(n, gat->heads, dim, workspace, workspace_bytes);
    GatBwdArgs a;
    a.n = n; a.rowptr = g->rowptr; a.colidx = g->colidx; a.p = p; a.ldp = ldp;
    a.heads = gat->heads; a.head_dim = gat->head_dim; a.dim = dim;
    a.a_src = gat->a_src; a.a_dst = gat->a_dst; a.slope = gat->negative_slope; a.self_loop = gat->add_self_loop ? 1 : 0;
    a.dz = dz; a.lddz = lddz;
    a.s = b.s; a.t = b.t; a.stats = b.stats; a.partial = b.partial; a.ds = b.ds; a.dt = b.dt; a.done = b.bins + kGatOrderInts;
    const unsigned blocks = (unsigned)((n + kGbWarps - 1) / kGbWarps);
    a.dp = dp; a.lddp = lddp; a.dp16 = static_cast<__nv_bfloat16*>(dp_bf16); a.lddp16 = lddp_bf16;
    int lpg, w;
    if (gat_lanes_cover(dim, gat->head_dim, p, ldp, dz, lddz, &lpg, &w)) {
        const int n_sm = sm_count();
        if (n_sm <= 0) return RETEXO_ERR_CUDA;
        const int vec = dp && lddp % 4 == 0 && aligned_to(dp, 16), vec16 = dp_bf16 && lddp_bf16 % 4 == 0 && aligned_to(dp_bf16, 8);
        const int hub_entries = gat_hub_entries(g->n_edges, n_sm);
        if (kept) {
            a.s = const_cast<float*>(kept->s); a.t = const_cast<float*>(kept->t);
        } else {
            RETEXO_CUDA_TRY(cudaMemsetAsync(b.bins, 0, (kGatOrderInts + 1) * sizeof(int32_t), st));
            RETEXO_TRY((gat_lanes_dispatch(lpg, w, [&]<int LPG, int W>() {
                gat_lane_scores_kernel<LPG, W><<<gat_lane_scores_grid<LPG, W>(n, n_sm), 256, 0, st>>>(
                    n, a.rowptr, a.p, a.ldp, a.heads, a.head_dim, a.a_src, a.a_dst, a.self_loop, hub_entries, a.s, a.t, b.bins);
                return launch_status();
            })));
            gat_order_kernel<<<gat_order_blocks(n), 256, 0, st>>>(n, nullptr, a.rowptr, a.self_loop, hub_entries, b.bins, b.rows, nullptr, 0);
        }
        const GatRowOrder all{b.rows, b.bins + kGatOrderCounts, nullptr, n}, dst = kept ? kept->dst : all, src = kept ? kept->src : all;
        RETEXO_TRY((gat_lanes_dispatch(lpg, w, [&]<int LPG, int W>() {
            const GatGrid dst_grid = gat_grid<LPG>(dst.n, g->n_edges + n, n_sm, 6 * n_sm), src_grid = gat_grid<LPG>(src.n, g->n_edges + n, n_sm, 6 * n_sm);
            gat_lane_dst_kernel<LPG, W><<<dst_grid.blocks, kGatThreads, 0, st>>>(a, dst, dst_grid);
            if (kept) a.colidx = kept->src_colidx;
            gat_lane_src_kernel<LPG, W><<<src_grid.blocks, kGatThreads, 0, st>>>(a, src, src_grid, vec, vec16);
            return launch_status();
        })));
        return gat_lanes_dispatch(lpg, w, [&]<int LPG, int W>() {
            const int64_t want = (n + 64 * GatLanes<LPG, W>::G - 1) / (64 * GatLanes<LPG, W>::G);      // 8 nodes per group
            gat_lane_params_kernel<LPG, W><<<(unsigned)std::min(want, kGatParamBlocks), 256, 0, st>>>(a, da_src, da_dst);
            return launch_status();
        });
    }
    gat_bwd_scores_kernel<<<blocks, kGbThreads, 0, st>>>(a);
    const int nc = (dim + kWarp - 1) / kWarp;
    if (nc <= 1) return launch_bwd<1>(a, blocks, da_src, da_dst, st);
    if (nc <= 2) return launch_bwd<2>(a, blocks, da_src, da_dst, st);
    if (nc <= 4) return launch_bwd<4>(a, blocks, da_src, da_dst, st);
    return launch_bwd<8>(a, blocks, da_src, da_dst, st);
}
