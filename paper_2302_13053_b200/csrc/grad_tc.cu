// Weight gradients of one training iteration of the per-node model on sm_100a: [dW1 ; db1] = [X | 1]^T dHd and
// [dW2 ; db2] = [Hd | 1]^T dL in one launch.
//
// Both reductions run over the batch, so the operands are read as they lie in memory (M and N contiguous, boxes of 64 rows x 64
// columns by TMA, tcgen05.mma with both operands MN-major).  A block owns one 128 x BN tile and one range of the rows; the
// two products share the grid, cut so that every block takes about the same number of steps.
// A bias gradient is the product of a vector of ones with the same B operand: one more MMA whose A operand is a constant 2 KB
// of ones, instead of a column of ones behind X and Hd, which cost a pass over a caller's batch that had none and a whole
// further row of tiles wherever the width is a multiple of 128 (257 = 3 tiles for 2).  Of the row's steps each row of tiles
// takes an equal share, so that no block has twice the MMAs of another.
// Bound by HBM on large batches, by its latencies on small ones.  Whole iterations, one product per launch with columns of ones
// before -> this kernel: 60 x 1000 (hidden 128) 43 -> 33 us, 2000 x 300 (150) 58 -> 43, 38439 x 512 (256) 91 -> 71,
// 195922 x 100 (256) 206 -> 187, 153757 x 512 (256) 203 -> 181, 153757 x 1204 (256) 275 -> 262; 20000 x 8192 (512), where one
// range of rows fills the device, 443 -> 452.
// Every wait is bounded: a wait that runs out sets *status and the block tears down in order.
#include <string.h>

#include "gemm_tc.h"
#include "grad_tc.h"
#include "tc_common.cuh"

namespace retexo {

constexpr int kGradEpiWarps = 8, kGradThreads = 64 + 32 * kGradEpiWarps;
constexpr uint32_t kGradBoxBytes = kTcBK * 64 * 2;      // 64 reduction rows of 64 elements
constexpr uint32_t kOnesBytes = 16 * 64 * 2;            // 16 reduction rows of 64 ones

struct GradDims {
    int32_t M, N, bn, n_m, n_n, splits, kb_per_split, tiles, bias_shares;
    float* partial; float* bias_partial;
};
struct GradArgs {
    GradDims p[2];
    int32_t kb_total, n_tiles;
    int32_t* status;
};

struct GradTile { int which, m, n, z; };
__device__ __forceinline__ GradTile grad_tile(const GradArgs& g, int t) {
    GradTile r;
    r.which = t >= g.p[0].tiles ? 1 : 0;
    const GradDims& d = g.p[r.which];
    const int i = t - (r.which ? g.p[0].tiles : 0), per_split = d.n_m * d.n_n;
    r.z = i / per_split;
    r.m = (i % per_split) % d.n_m;
    r.n = (i % per_split) / d.n_m;
    return r;
}

template <int BN, int STAGES>
__global__ void __launch_bounds__(kGradThreads, 1)
grad_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_b0,
            const __grid_constant__ CUtensorMap map_a1, const __grid_constant__ CUtensorMap map_b1, GradArgs g) {
    constexpr uint32_t kABytes = 2 * kGradBoxBytes, kStageBytes = kABytes + (BN / 64) * kGradBoxBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* ones = tiles + STAGES * kStageBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(ones + kOnesBytes);
    uint64_t* empty = full + STAGES;
    uint64_t* acc_full = empty + STAGES;
    uint64_t* acc_empty = acc_full + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, kGradEpiWarps);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x == 32) { prefetch_map(&map_a0); prefetch_map(&map_b0); if (g.p[1].tiles) { prefetch_map(&map_a1); prefetch_map(&map_b1); } }
    if (warp == 1) {      // tensor memory: the tile's accumulator and the bias row's, BN columns each
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(2 * BN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    for (uint32_t i = threadIdx.x; i < kOnesBytes / 4; i += kGradThreads) reinterpret_cast<uint32_t*>(ones)[i] = 0x3f803f80u;
    fence_proxy_async_smem();
    grid_dependency_wait();          // everything from here on may read what the previous kernel wrote
    grid_dependency_release();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        const bool leader = elect_one();
        RingPos r;
        int issued = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < g.n_tiles && ok; t += gridDim.x) {
            const GradTile tile = grad_tile(g, t);
            const GradDims& d = g.p[tile.which];
            const CUtensorMap* ma = tile.which ? &map_a1 : &map_a0;
            const CUtensorMap* mb = tile.which ? &map_b1 : &map_b0;
            const int m0 = tile.m * 128, n0 = tile.n * d.bn;
            const int na = d.M - m0 > 64 ? 2 : 1, nb = min(d.bn / 64, (d.N - n0 + 63) / 64);      // boxes that hold anything
            const int kb0 = tile.z * d.kb_per_split, kb1 = min(g.kb_total, kb0 + d.kb_per_split);
            const uint32_t bytes = (uint32_t)(na + nb) * kGradBoxBytes;
            for (int kb = kb0; kb < kb1; ++kb, ++issued, r.next(STAGES)) {
                uint64_t* bar = full + r.s;
                if (!mbar_wait_warp(empty + r.s, r.ph ^ 1, g.status, abort_flag)) { ok = false; break; }
                uint8_t* dst = tiles + r.s * kStageBytes;
                if (!leader) continue;
                mbar_expect_tx(bar, bytes);
                tma_load_2d(dst, ma, m0, kb * kTcBK, bar);
                if (na > 1) tma_load_2d(dst + kGradBoxBytes, ma, m0 + 64, kb * kTcBK, bar);
#pragma unroll
                for (int i = 0; i < BN / 64; ++i)
                    if (i < nb) tma_load_2d(dst + kABytes + i * kGradBoxBytes, mb, n0 + 64 * i, kb * kTcBK, bar);
            }
        }
        if (*abort_flag) {      // await (bounded) what was issued and not consumed, so that nothing lands after the block has left
            for (int i = issued > STAGES ? issued - STAGES : 0; i < issued; ++i)
                for (uint32_t w = 0; w < (1u << 20); ++w) if (mbar_try_wait(full + i % STAGES, (uint32_t)(i / STAGES) & 1)) break;
        }
    } else if (warp == 1) {
        const bool leader = elect_one();
        const uint64_t ones_desc = make_smem_desc_mn(smem_u32(ones), 0);      // (both halves of M read the same 64 ones)
        const uint32_t tiles_addr = smem_u32(tiles);
        RingPos r;
        int lt = 0;
        bool ok = true, ready = false;      // ready: the stage at r has been seen full
        for (int t = blockIdx.x; t < g.n_tiles && ok; t += gridDim.x, ++lt) {
            const GradTile tile = grad_tile(g, t);
            const GradDims& d = g.p[tile.which];
            const int kb0 = tile.z * d.kb_per_split, kb1 = min(g.kb_total, kb0 + d.kb_per_split);
            const uint32_t idesc = make_idesc(d.bn, true, true);
            ok = mbar_wait_warp(acc_empty, ((uint32_t)lt & 1) ^ 1, g.status, abort_flag);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            bool bias_begun = false;
            const int shares = d.bias_shares;
            int next_share = kb0 + (tile.m - kb0 % shares + shares) % shares;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!ready) ok = mbar_wait_warp(full + r.s, r.ph, g.status, abort_flag);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a_addr = tiles_addr + (uint32_t)r.s * kStageBytes;
                const uint64_t adesc = make_smem_desc_mn(a_addr, kGradBoxBytes), bdesc = make_smem_desc_mn(a_addr + kABytes, kGradBoxBytes);
                uint64_t* const used = empty + r.s;
                r.next(STAGES);
                const bool next_ready = mbar_test(full + r.s, r.ph);
                const bool share = kb == next_share;      // (the first step this block takes clears its row)
                if (leader) {
#pragma unroll
                    for (int k = 0; k < kTcBK / 16; ++k)      // 16 reduction rows = two 1024-byte atoms: +128 in 16-byte units
                        umma_bf16(tmem, adesc + 128 * k, bdesc + 128 * k, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
                    if (share) {
#pragma unroll
                        for (int k = 0; k < kTcBK / 16; ++k)
                            umma_bf16(tmem + BN, ones_desc, bdesc + 128 * k, idesc, (bias_begun || k > 0) ? 1u : 0u);
                    }
                    umma_commit(used);
                }
                ready = __all_sync(0xffffffffu, next_ready);
                if (share) { next_share += shares; bias_begun = true; }
            }
            if (ok && leader) umma_commit(acc_full);
        }
    } else {
        const int q = warp & 3, ew = warp - 2, half = ew >> 2;
        int lt = 0;
        for (int t = blockIdx.x; t < g.n_tiles; t += gridDim.x, ++lt) {
            const GradTile tile = grad_tile(g, t);
            const GradDims& d = g.p[tile.which];
            const int m0 = tile.m * 128, n0 = tile.n * d.bn;
            const int kb0 = tile.z * d.kb_per_split;
            const bool empty_range = kb0 >= g.kb_total;
            const int part = d.bn / 2, c_begin = half * part, c_end = min(c_begin + part, d.N - n0);
            const int row = m0 + q * 32 + lane;
            float* dst_base = d.partial + (int64_t)tile.z * d.M * d.N;
            const int kb1 = min(g.kb_total, kb0 + d.kb_per_split);
            // this block's share of the bias row: empty if none of its steps fell to it
            const int first_share = kb0 + (tile.m - kb0 % d.bias_shares + d.bias_shares) % d.bias_shares;
            const bool no_share = empty_range || first_share >= kb1;
            if (!mbar_wait(acc_full, (uint32_t)lt & 1, g.status, abort_flag)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int c0 = c_begin; c0 < c_end; c0 += 32) {
                uint32_t r[32];
                if (empty_range) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) r[j] = 0u;
                } else {
                    tmem_ld_issue(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, r);
                    tmem_ld_wait(r);
                }
                const int col0 = n0 + c0, n_cols = min(32, d.N - col0);
                if (row < d.M) {
                    float* dst = dst_base + (int64_t)row * d.N + col0;
                    if (n_cols == 32 && (d.N & 3) == 0) {
#pragma unroll
                        for (int j = 0; j < 32; j += 4)
                            *reinterpret_cast<float4*>(dst + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                                              __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j) if (j < n_cols) dst[j] = __uint_as_float(r[j]);
                    }
                }
                if (q == 0) {      // the bias row: row 0 of the second accumulator, in lane 0
                    uint32_t b[32];
                    if (no_share) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) b[j] = 0u;
                    } else {
                        tmem_ld_issue(tmem + BN + (uint32_t)c0, b);
                        tmem_ld_wait(b);
                    }
                    float mine = 0.f;
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float x = __shfl_sync(0xffffffffu, __uint_as_float(b[j]), 0);
                        mine = lane == j ? x : mine;
                    }
                    if (lane < n_cols) d.bias_partial[((int64_t)tile.z * d.bias_shares + tile.m) * d.N + col0 + lane] = mine;
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(acc_empty)) : "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN));
    }
}

// ---------------------------------------------------------------- host side
static int grad_bn(int32_t N) { return N > 128 ? 256 : (N > 64 ? 128 : 64); }

int32_t grad_bias_shares(int32_t M) { return (M + 127) / 128; }      // one share per row of tiles

void grad_splits(int32_t M1, int32_t N1, int32_t M2, int32_t N2, int64_t rows, int64_t* s1, int64_t* s2) {
    const int64_t kb = (rows + 63) / 64;
    *s1 = *s2 = 1;
    const int64_t bn1 = grad_bn(N1), t1 = ((M1 + 127) / 128) * ((N1 + bn1 - 1) / bn1), t2 = N2 > 0 ? (M2 + 127) / 128 : 0;
    const int64_t sms = 148, most = 64;      // (more ranges than 64 cost the update kernel more than they save here)
    // Equal steps per block, as far as one block per SM allows: a step waits for memory about as long whether its stage holds 48 KB or
    // 24, so blocks that shared out the bytes left the ones of the second product behind, with half as many steps again.  (That
    // -> this: 153757 x 1204 (256) 284 -> 262 us an iteration, 153757 x 512 (256) 195 -> 181, 200000 x 512 (512) 541 -> 468,
    // 400000 x 256 (256) 372 -> 338; weights of 0.75 to 1 for the narrow steps are within 2 %.)
    double best = 1e30;
    for (int64_t a = 1; a <= most && a <= kb; ++a) {
        int64_t b = 1;
        if (t2 > 0) {
            b = (sms - t1 * a) / t2;
            b = b < 1 ? 1 : b > most ? most : b > kb ? kb : b;
        }
        const int64_t waves = (t1 * a + t2 * b + sms - 1) / sms;
        const double c1 = (double)((kb + a - 1) / a), c2 = t2 > 0 ? 0.9 * (double)((kb + b - 1) / b) : 0.0;
        const double cost = (double)waves * (c1 > c2 ? c1 : c2);
        if (cost < best * 0.999) { best = cost; *s1 = a; *s2 = b; }
    }
}

template <int BN, int STAGES>
static int launch_grad(const CUtensorMap (&maps)[4], const GradArgs& g, cudaStream_t st) {
    constexpr size_t smem = 1024 + (size_t)STAGES * (2 + BN / 64) * kGradBoxBytes + kOnesBytes + 512;
    static_assert(smem <= 227 * 1024, "shared memory budget");
    auto kernel = grad_kernel<BN, STAGES>;
    const int n_sm = sm_count();
    if (n_sm <= 0 || cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        (void)cudaGetLastError();
        return RETEXO_ERR_CUDA;
    }
    OverlapLaunch ol(dim3((unsigned)(g.n_tiles < n_sm ? g.n_tiles : n_sm)), dim3(kGradThreads), smem, st);
    if (cudaLaunchKernelEx(&ol.cfg, kernel, maps[0], maps[1], maps[2], maps[3], g) != cudaSuccess) {
        (void)cudaGetLastError();
        return RETEXO_ERR_CUDA;
    }
    return launch_status();
}

int grad_launch(const GradProduct* products, int n_products, int64_t rows, int32_t* status, cudaStream_t st) {
    if (n_products < 1 || n_products > 2 || rows < 1 || rows > INT32_MAX - 64) return RETEXO_ERR_INVALID_ARG;
    GradArgs g{};
    CUtensorMap maps[4];
    memset(maps, 0, sizeof(maps));
    g.kb_total = (int32_t)((rows + 63) / 64);
    g.status = status;
    for (int i = 0; i < n_products; ++i) {
        const GradProduct& p = products[i];
        GradDims& d = g.p[i];
        if (i == 1 && p.N > 64) return RETEXO_ERR_UNSUPPORTED;
        d.M = p.M; d.N = p.N; d.bn = i == 0 ? grad_bn(p.N) : 64;
        d.n_m = (p.M + 127) / 128; d.n_n = (p.N + d.bn - 1) / d.bn;
        d.splits = p.splits; d.kb_per_split = (g.kb_total + p.splits - 1) / p.splits;
        d.tiles = d.n_m * d.n_n * p.splits;
        d.partial = p.partial; d.bias_partial = p.bias_partial; d.bias_shares = grad_bias_shares(p.M);
        g.n_tiles += d.tiles;
        if (!tc_make_map_2d(&maps[2 * i], p.A, rows, p.M, p.lda, kTcBK, 64, 128, true)) return RETEXO_ERR_CUDA;
        if (!tc_make_map_2d(&maps[2 * i + 1], p.B, rows, p.N, p.ldb, kTcBK, 64, 128, true)) return RETEXO_ERR_CUDA;
    }
    if (g.p[0].bn == 256) return launch_grad<256, 4>(maps, g, st);
    if (g.p[0].bn == 128) return launch_grad<128, 6>(maps, g, st);
    return launch_grad<64, 8>(maps, g, st);
}

}  // namespace retexo
