// A training iteration of a small batch in two kernels.  The four of a large one (forward product, head_backward_kernel, grad_kernel,
// reduce_update_kernel) are a chain of launches of about 5 us each however little they have to do; here
//   small_forward_kernel   Hd = ReLU(X W1 + b1), logits = Hd W2 + b2, loss, dL, dHd = (dL W2^T) .* [Hd > 0]: a block per 32 rows
//   small_update_kernel    [dW1 ; db1], [dW2 ; db2] over the whole batch, the optimiser on the gradient where it lies, the weights'
//                          bf16 copies: a block per 8 to 32 inputs
// Nothing that is handed on inside a kernel leaves the SM.
// Bound by latencies: the first by its reduction steps one after the other (23 of about 0.2 us at 1433 columns) and a chain of three
// products, the second by one load, one product and the optimiser.  An iteration of 140 + 500 rows in rounds of 1433, 64 and 64
// columns (hidden 64, 7 classes): 22 -> 13 us; of 60 + 500 rows x 1000, 256, 256 (128): 24 -> 15.
// The tensor core always takes 128 rows; those a tile does not have are whatever lies behind it in shared memory, and
// nobody reads their results.
// Every wait is bounded: one that runs out sets *status, and the block goes on to its end (with values nobody will use: the status
// turns the loss into NaN), so that no thread is left at a barrier, and leaves once its copies have landed.
#include <string.h>

#include "class_loss.cuh"
#include "gemm_tc.h"
#include "mlp_kernels.cuh"
#include "mlp_small.h"

namespace retexo {

constexpr int kSmTile = 32;                                   // rows a block of the forward kernel takes
constexpr int kSmMaxHidden = 128, kSmMaxTrain = 512, kSmMaxInputs = 32 * 140;
constexpr uint32_t kSmABytes = kSmTile * 128;                 // [32 rows x 64 columns]
constexpr uint32_t kSmPanelBytes = 64 * 128;                  // [64 rows x 64 columns]
constexpr uint32_t kSmMmaBytes = 128 * 128;                   // what the tensor core reads behind a tile's start
constexpr int kSmMaxStages = 18;
constexpr int kSmThreads = 5 * 32;

struct SmForwardArgs {
    int64_t n_all, n_train;
    int32_t H, O, np, kb_total, stages, x_early;
    const float* b1; const float* b2;
    const int32_t* y; const int32_t* y_eval;
    float inv_rows;
    float* loss_partial;
    unsigned long long* correct;
    int32_t* status;
};

enum SmBarrier { SM_W2_FULL = 0, SM_ACC1 = 1, SM_HD = 2, SM_ACC2 = 3, SM_DL = 4, SM_ACC3 = 5, SM_FULL = 6 };

// Warps: 0 and 4 (lane quarter 0, where the tile's 32 rows are) are the epilogue; 1 issues the MMAs and owns tensor memory; 2 loads W1,
// 3 loads X and W2.
__global__ void __launch_bounds__(kSmThreads, 1)
small_forward_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w1,
                     const __grid_constant__ CUtensorMap map_w2, const __grid_constant__ CUtensorMap map_hd,
                     const __grid_constant__ CUtensorMap map_dl, const __grid_constant__ CUtensorMap map_dhd, SmForwardArgs g) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int np = g.np, stages = g.stages;
    const bool last = g.H == 0;
    const uint32_t stage_bytes = kSmABytes + (uint32_t)np * kSmPanelBytes;
    uint8_t* dl_s = base;                                         // [32 rows x 64 classes]
    uint8_t* hd_s = dl_s + kSmABytes;                             // [np][32 rows x 64 units]
    uint8_t* out_s = hd_s + (uint32_t)np * kSmABytes;             // [np][32 rows x 64 units]: dHd on its way out
    uint8_t* w2_s = out_s + (uint32_t)np * kSmABytes;             // [np][64 classes x 64 units]
    uint8_t* ring = w2_s + (uint32_t)np * kSmPanelBytes;          // [stages][rows of X | rows of W1^T]
    float* bias_s = reinterpret_cast<float*>(ring + (uint32_t)stages * stage_bytes);      // [64]
    float* xch = bias_s + 64;
    uint64_t* bars = reinterpret_cast<uint64_t*>(xch + kClassLossExchange);
    uint64_t* full = bars + SM_FULL;
    uint64_t* empty = full + kSmMaxStages;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(empty + kSmMaxStages);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row0 = (int64_t)blockIdx.x * kSmTile;
    const bool trains = row0 < g.n_train;
    const int ahead = min(stages, g.kb_total);
    if (threadIdx.x == 96) {
        mbar_init(bars + SM_W2_FULL, 1);
        mbar_init(bars + SM_ACC1, 1);
        mbar_init(bars + SM_HD, 2);
        mbar_init(bars + SM_ACC2, 1);
        mbar_init(bars + SM_DL, 1);
        mbar_init(bars + SM_ACC3, 1);
        for (int s = 0; s < stages; ++s) { mbar_init(full + s, 2); mbar_init(empty + s, 1); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x == 64) {
        prefetch_map(&map_w1);
        prefetch_map(&map_dl);
        if (!last) { prefetch_map(&map_w2); prefetch_map(&map_hd); prefetch_map(&map_dhd); }
    }
    if (warp == 1) {      // first product (up to 128 columns), logits (64), dHd (up to 128)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot, acc2 = tmem + (last ? 0u : 128u), acc3 = tmem + 256u;
    auto load_x = [&](int kb, int s) {
        mbar_expect_tx(full + s, kSmABytes);
        tma_load_2d(ring + s * stage_bytes, &map_x, kb * kTcBK, (int32_t)row0, full + s);
    };
    if (warp == 3 && g.x_early && elect_one())
        for (int kb = 0; kb < ahead; ++kb) load_x(kb, kb);
    grid_dependency_wait();          // everything from here on may read what the previous kernel wrote
    grid_dependency_release();

    if (warp == 3) {
        const bool leader = elect_one();
        if (!last && leader) {
            mbar_expect_tx(bars + SM_W2_FULL, (uint32_t)np * kSmPanelBytes);
            for (int p = 0; p < np; ++p) tma_load_2d(w2_s + p * kSmPanelBytes, &map_w2, 64 * p, 0, bars + SM_W2_FULL);
        }
        RingPos r;
        int kb = 0;
        if (g.x_early) {
            kb = ahead;
            if (ahead == stages) r.ph = 1;
            else r.s = ahead;
        }
        for (; kb < g.kb_total; ++kb, r.next(stages)) {
            if (!mbar_wait_warp(empty + r.s, r.ph ^ 1, g.status, abort_flag)) break;
            if (leader) load_x(kb, r.s);
        }
    } else if (warp == 2) {
        const bool leader = elect_one();
        RingPos r;
        int kb = 0;
        for (; kb < g.kb_total; ++kb, r.next(stages)) {
            if (!mbar_wait_warp(empty + r.s, r.ph ^ 1, g.status, abort_flag)) break;
            if (leader) {
                mbar_expect_tx(full + r.s, (uint32_t)np * kSmPanelBytes);
                tma_load_2d(ring + r.s * stage_bytes + kSmABytes, &map_w1, kb * kTcBK, 0, full + r.s);
            }
        }
        if (*abort_flag) {      // await (bounded) what was issued, so that nothing lands after the block has left
            if (!last) for (uint32_t w = 0; w < (1u << 20); ++w) if (mbar_try_wait(bars + SM_W2_FULL, 0)) break;
            for (int i = kb > stages ? kb - stages : 0; i < kb; ++i)
                for (uint32_t w = 0; w < (1u << 20); ++w) if (mbar_try_wait(full + i % stages, (uint32_t)(i / stages) & 1)) break;
        }
    } else if (warp == 1) {
        const bool leader = elect_one();
        const uint32_t idesc1 = make_idesc(64 * np);
        uint64_t adesc = make_smem_desc(smem_u32(ring)), bdesc = make_smem_desc(smem_u32(ring) + kSmABytes);
        const uint64_t desc_step = stage_bytes >> 4, desc_wrap = (uint64_t)(stages - 1) * desc_step;
        RingPos r;
        bool ok = true, ready = false;      // ready: the stage at r has been seen full
        for (int kb = 0; kb < g.kb_total; ++kb) {
            if (!ready) ok = mbar_wait_warp(full + r.s, r.ph, g.status, abort_flag);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint64_t* const used = empty + r.s;
            r.next(stages);
            const bool next_ready = mbar_test(full + r.s, r.ph);
            if (leader) {
#pragma unroll
                for (int k = 0; k < kTcBK / 16; ++k) umma_bf16(tmem, adesc + 2 * k, bdesc + 2 * k, idesc1, (kb > 0 || k > 0) ? 1u : 0u);
                umma_commit(used);
            }
            ready = __all_sync(0xffffffffu, next_ready);
            if (r.s) { adesc += desc_step; bdesc += desc_step; }
            else { adesc -= desc_wrap; bdesc -= desc_wrap; }
        }
        if (ok && leader) umma_commit(bars + SM_ACC1);
        if (ok && !last) {
            const uint32_t w2_addr = smem_u32(w2_s);
            ok = mbar_wait_warp(bars + SM_W2_FULL, 0, g.status, abort_flag) && mbar_wait_warp(bars + SM_HD, 0, g.status, abort_flag);
            if (ok) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t hdesc = make_smem_desc(smem_u32(hd_s)), wdesc = make_smem_desc(w2_addr);
                const uint32_t idesc2 = make_idesc(64);
                if (leader) {
#pragma unroll
                    for (int p = 0; p < 2; ++p)
                        if (p < np) {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                umma_bf16(acc2, hdesc + (uint64_t)(p * (kSmABytes >> 4) + 2 * j), wdesc + (uint64_t)(p * (kSmPanelBytes >> 4) + 2 * j), idesc2, (p | j) ? 1u : 0u);
                        }
                    umma_commit(bars + SM_ACC2);
                }
            }
            if (ok && trains) ok = mbar_wait_warp(bars + SM_DL, 0, g.status, abort_flag);
            if (ok && trains) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t ddesc = make_smem_desc(smem_u32(dl_s)), wdesc = make_smem_desc_mn(w2_addr, kSmPanelBytes);
                const uint32_t idesc3 = make_idesc(64 * np, false, true);
                if (leader) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)      // 16 classes along K: 32 bytes of a dL line, two 1024-byte atoms of W2^T
                        umma_bf16(acc3, ddesc + (uint64_t)(2 * j), wdesc + (uint64_t)(128 * j), idesc3, j ? 1u : 0u);
                    umma_commit(bars + SM_ACC3);
                }
            }
        }
    } else {
        const int part = warp >> 2;                     // which half of every panel of 64 columns, which classes
        const int64_t row = row0 + lane;
        const bool train = row < g.n_train;
        const bool eval = !train && row < g.n_all && g.y_eval != nullptr;
        const int32_t label = train ? g.y[row] : (eval ? g.y_eval[row - g.n_train] : -1);
        const int n1 = last ? g.O : g.H;
        float bias[2] = {0.f, 0.f};                     // of columns 32 part + lane and 64 further on
#pragma unroll
        for (int p = 0; p < 2; ++p)
            if (p < np && 64 * p + 32 * part + lane < n1) bias[p] = __ldg(g.b1 + 64 * p + 32 * part + lane);
        bias_s[32 * part + lane] = last ? bias[0] : (32 * part + lane < g.O ? __ldg(g.b2 + 32 * part + lane) : 0.f);
        ClassLoss cl(g.O, part, 0, lane, xch, 1);
        cl.pair_sync();                                 // both halves of the classes' bias are there
        (void)mbar_wait(bars + SM_ACC1, 0, g.status, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t gate[2] = {0u, 0u};
        if (!last) {
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (p >= np) break;
                uint32_t r[32];
                tmem_ld_issue(tmem + (uint32_t)(64 * p + 32 * part), r);
                tmem_ld_wait(r);
                uint32_t o[16], word = 0u;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float lo = fmaxf(__uint_as_float(r[2 * j]) + __shfl_sync(0xffffffffu, bias[p], 2 * j), 0.f);
                    const float hi = fmaxf(__uint_as_float(r[2 * j + 1]) + __shfl_sync(0xffffffffu, bias[p], 2 * j + 1), 0.f);
                    word |= ((lo > 0.f ? 1u : 0u) << (2 * j)) | ((hi > 0.f ? 1u : 0u) << (2 * j + 1));
                    __nv_bfloat162 b2 = __floats2bfloat162_rn(lo, hi);
                    o[j] = *reinterpret_cast<uint32_t*>(&b2);
                }
                gate[p] = word;
                uint8_t* line = hd_s + (uint32_t)p * kSmABytes + lane * 128;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    *reinterpret_cast<uint4*>(line + (((4 * part + j) ^ (lane & 7)) * 16)) = make_uint4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bars + SM_HD)) : "memory");
            cl.pair_sync();
            if (lane == 0 && part < np && trains) {      // Hd goes out whole panels at a time
                tma_store_2d(&map_hd, hd_s + (uint32_t)part * kSmABytes, 64 * part, (int32_t)row0);
                bulk_commit();
            }
            (void)mbar_wait(bars + SM_ACC2, 0, g.status, abort_flag);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        cl.load(acc2, bias_s);
        cl.reduce(label, eval, g.correct && row0 + 32 > g.n_train, g.correct);
        if (trains) {
            cl.store_dl(label, train, g.inv_rows, dl_s + lane * 128);
            fence_proxy_async_smem();
            cl.pair_sync();
            if (part == 0 && lane == 0) {
                if (!last) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bars + SM_DL)) : "memory");
                tma_store_2d(&map_dl, dl_s, 0, (int32_t)row0);
                bulk_commit();
            }
        }
        if (part == 0) {
            const float loss = warp_sum(cl.loss(train));
            if (lane == 0 && g.loss_partial) g.loss_partial[blockIdx.x] = loss;
        }
        if (!last && trains) {
            (void)mbar_wait(bars + SM_ACC3, 0, g.status, abort_flag);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (p >= np) break;
                uint32_t r[32];
                tmem_ld_issue(acc3 + (uint32_t)(64 * p + 32 * part), r);
                tmem_ld_wait(r);
                uint8_t* line = out_s + (uint32_t)p * kSmABytes + lane * 128;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t o[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int c = 8 * j + 2 * k;
                        __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(r[c] & (0u - ((gate[p] >> c) & 1u))),
                                                                  __uint_as_float(r[c + 1] & (0u - ((gate[p] >> (c + 1)) & 1u))));
                        o[k] = *reinterpret_cast<uint32_t*>(&b2);
                    }
                    *reinterpret_cast<uint4*>(line + (((4 * part + j) ^ (lane & 7)) * 16)) = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
            fence_proxy_async_smem();
            cl.pair_sync();
            if (lane == 0 && part < np) {
                tma_store_2d(&map_dhd, out_s + (uint32_t)part * kSmABytes, 64 * part, (int32_t)row0);
                bulk_commit();
            }
        }
        if (lane == 0) bulk_wait_all();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

// ---------------------------------------------------------------- gradients and update
constexpr int kSmUpdateThreads = 64 + 256;
constexpr uint32_t kSmOnesBytes = 16 * 64 * 2;            // 16 reduction rows of 64 ones

// Shared memory of the operands, or of the gradient that takes their place.
template <int NP>
__host__ __device__ constexpr uint32_t small_update_operands(int kb_total) {
    const uint32_t operands = (uint32_t)kb_total * (1 + NP) * kSmPanelBytes, gradient = (32 * (64 * NP + 1) * 4 + 1023) / 1024 * 1024;
    return operands > gradient ? operands : gradient;
}

// A block owns FR inputs (rows) of one product's result, all of its columns and the whole batch: [FR x N] = A^T B, one accumulator.
// (Of the tensor core's 128 rows the halves read the same 64 inputs, so that lane quarters 0 and 2 hold the same results and share the
// columns; boxes are 64 inputs wide whatever FR.)  The gradient goes through shared memory to threads that lie along theta's rows.  Few
// inputs a block, because what takes the time is the optimiser: more than a hundred instructions an element.
template <int NP, int FR>
__device__ __forceinline__ void small_update_block(const CUtensorMap& map_a, const CUtensorMap& map_b, int which, int m0, int kb_total, bool a_early,
                                                   const UpdateArgs& u) {
    constexpr int kCols = 64 * NP, kPer = FR * kCols / 256, kPitch = kCols + 1;      // kPer: elements a thread updates
    constexpr uint32_t kStage = (1 + NP) * kSmPanelBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float* grad_s = reinterpret_cast<float*>(base);                                  // once the product is done: [FR][kPitch]
    bf16* t16_s = reinterpret_cast<bf16*>(base);                                     // later: [kCols][FR + 2]
    uint8_t* ones = base + small_update_operands<NP>(kb_total);
    float* bias_s = reinterpret_cast<float*>(ones + kSmOnesBytes);                   // [kCols]
    uint64_t* full = reinterpret_cast<uint64_t*>(bias_s + kCols);
    uint64_t* acc_full = full + kSmMaxTrain / 64;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    float* corr_s = reinterpret_cast<float*>(tmem_slot + 2);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t M = which ? u.hidden : u.d_in, N = which ? u.n_classes : u.out1;
    const bool has_bias = m0 == 0;
    const bool adam = u.optimizer != RETEXO_SGD;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kb_total; ++s) mbar_init(full + s, 1);
        mbar_init(acc_full, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int s = 0; s < kb_total; ++s) {
            mbar_expect_tx(full + s, kStage);
            if (a_early) tma_load_2d(base + s * kStage, &map_a, m0, s * kTcBK, full + s);
        }
    }
    if (threadIdx.x == 32) { prefetch_map(&map_a); prefetch_map(&map_b); }
    if (warp == 1) {      // the accumulator and the bias row's
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(256));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    for (uint32_t i = threadIdx.x; i < kSmOnesBytes / 4; i += kSmUpdateThreads) reinterpret_cast<uint32_t*>(ones)[i] = 0x3f803f80u;
    fence_proxy_async_smem();

    // ---- what is older than the kernel before this one: parameters, moments, iteration state (left by the previous update)
    const int t = (int)threadIdx.x - 64;
    const int c = t & (kCols - 1), r_first = t / kCols;
    constexpr int kRowStep = 256 / kCols;
    const int64_t p0 = which ? u.seg[0].size : 0;
    float theta[kPer], m[kPer], v[kPer];
    float b_theta = 0.f, b_m = 0.f, b_v = 0.f;
    unsigned long long step_now = 0, snap_best = 0;
    int32_t snap_have = 1;
    if (u.step_dev) step_now = *u.step_dev;
    if (u.snap_cur) { snap_have = *u.snap_have; snap_best = *u.snap_best; }
    if (t >= 0) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int r = m0 + r_first + kRowStep * i;
            const bool live = r < M && c < N;
            const int64_t p = p0 + (int64_t)r * N + c;
            theta[i] = live ? u.theta[p] : 0.f;
            m[i] = live && adam ? u.m[p] : 0.f;
            v[i] = live && adam ? u.v[p] : 0.f;
        }
        if (has_bias && t < N) {
            const int64_t p = p0 + (int64_t)M * N + t;
            b_theta = u.theta[p];
            if (adam) { b_m = u.m[p]; b_v = u.v[p]; }
        }
        if (u.step_dev) {
            if (t == 0) corr_s[0] = (float)(1.0 - pow_whole((double)u.beta1, step_now + 1));
            if (t == 32) corr_s[1] = (float)(1.0 - pow_whole((double)u.beta2, step_now + 1));
        }
    }
    grid_dependency_wait();
    grid_dependency_release();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kb_total; ++s) {
            if (!a_early) tma_load_2d(base + s * kStage, &map_a, m0, s * kTcBK, full + s);
#pragma unroll
            for (int i = 0; i < NP; ++i)
                tma_load_2d(base + s * kStage + (1 + i) * kSmPanelBytes, &map_b, 64 * i, s * kTcBK, full + s);
        }
    }
    // (the validation count was written by the kernel before this one)
    const unsigned long long snap_cur = u.snap_cur ? *u.snap_cur : 0;
    const bool snapshot = u.theta_best && (!snap_have || snap_cur > snap_best);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    if (u.done && threadIdx.x == 32) update_bookkeeping(u, step_now, snap_cur, snap_best, snap_have, snapshot);

    if (warp == 0) {
        const bool leader = elect_one();
        const uint64_t ones_desc = make_smem_desc_mn(smem_u32(ones), 0);
        const uint32_t idesc = make_idesc(kCols, true, true);
        uint64_t adesc = make_smem_desc_mn(smem_u32(base), 0), bdesc = make_smem_desc_mn(smem_u32(base) + kSmPanelBytes, kSmPanelBytes);
        bool ok = true;
        for (int s = 0; s < kb_total; ++s, adesc += kStage >> 4, bdesc += kStage >> 4) {
            ok = mbar_wait_warp(full + s, 0, u.status_word, abort_flag);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (leader) {
#pragma unroll
                for (int k = 0; k < kTcBK / 16; ++k) umma_bf16(tmem, adesc + 128 * k, bdesc + 128 * k, idesc, (s > 0 || k > 0) ? 1u : 0u);
                if (has_bias) {
#pragma unroll
                    for (int k = 0; k < kTcBK / 16; ++k) umma_bf16(tmem + 128, ones_desc, bdesc + 128 * k, idesc, (s > 0 || k > 0) ? 1u : 0u);
                }
            }
        }
        if (ok) {
            if (leader) umma_commit(acc_full);
        } else {      // await (bounded) what was issued, so that nothing lands after the block has left
            for (int s = 0; s < kb_total; ++s)
                for (uint32_t w = 0; w < (1u << 20); ++w) if (mbar_try_wait(full + s, 0)) break;
        }
    } else if (warp >= 2) {
        if (blockIdx.x == 0 && warp == 9) update_loss(u, step_now, lane);
        (void)mbar_wait(acc_full, 0, u.status_word, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int q = warp & 3, part = (q >> 1) + 2 * ((warp - 2) >> 2);      // quarters 0 and 2 hold the (up to 32) rows
        if ((q & 1) == 0) {
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                uint32_t r[16];
                const int col = 16 * (part * NP + j);
                tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)col, r);
                if (lane < FR) {
#pragma unroll
                    for (int k = 0; k < 16; ++k) grad_s[lane * kPitch + col + k] = __uint_as_float(r[k]);
                }
                if (has_bias) {      // (every row of that accumulator is the bias gradient)
                    tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + 128u + (uint32_t)col, r);
                    if (lane == 0) {
#pragma unroll
                        for (int k = 0; k < 16; ++k) bias_s[col + k] = __uint_as_float(r[k]);
                    }
                }
            }
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const float corr1 = u.step_dev ? corr_s[0] : u.corr1, corr2 = u.step_dev ? corr_s[1] : u.corr2;
        auto update = [&](int64_t p, float g, float theta_p, float m_p, float v_p) -> float {
            if (u.grad_out) u.grad_out[p] = g;
            if (snapshot) u.theta_best[p] = theta_p;
            float now;
            if (adam) {
                m_p = u.beta1 * m_p + (1.f - u.beta1) * g;
                v_p = u.beta2 * v_p + (1.f - u.beta2) * g * g;
                u.m[p] = m_p;
                u.v[p] = v_p;
                now = theta_p - u.lr * (m_p / corr1) / (sqrtf(v_p / corr2) + u.eps);
            } else {
                now = theta_p - u.lr * g;
            }
            u.theta[p] = now;
            return now;
        };
        float g[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) g[i] = grad_s[(r_first + kRowStep * i) * kPitch + c];
        bf16* wr = which ? nullptr : u.w1r16;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int r = m0 + r_first + kRowStep * i;
            if (r < M && c < N) {
                theta[i] = update(p0 + (int64_t)r * N + c, g[i], theta[i], m[i], v[i]);
                if (wr) wr[(int64_t)r * u.ld_o1 + c] = f32_to_bf16(theta[i]);
            }
        }
        if (has_bias && t < N) update(p0 + (int64_t)M * N + t, bias_s[t], b_theta, b_m, b_v);
        bf16* wt = which ? u.w2t16 : u.w1t16;
        const int64_t ld_wt = which ? u.ld_h : u.ld_k;
        if (wt) {      // the transposed copy, runs of FR inputs (its stride covers whole blocks of 64)
            asm volatile("bar.sync 1, 256;" ::: "memory");      // (the gradient has been read)
#pragma unroll
            for (int i = 0; i < kPer; ++i) t16_s[c * (FR + 2) + r_first + kRowStep * i] = f32_to_bf16(theta[i]);
            asm volatile("bar.sync 1, 256;" ::: "memory");
            constexpr int kLanes = FR / 2;
            for (int col = t / kLanes; col < N; col += 256 / kLanes)
                reinterpret_cast<uint32_t*>(wt + col * ld_wt + m0)[t % kLanes] = *reinterpret_cast<const uint32_t*>(t16_s + col * (FR + 2) + 2 * (t % kLanes));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
    }
}

template <int NP, int FR>
__global__ void __launch_bounds__(kSmUpdateThreads, 1)
small_update_kernel(const __grid_constant__ CUtensorMap map_a1, const __grid_constant__ CUtensorMap map_b1,
                    const __grid_constant__ CUtensorMap map_a2, const __grid_constant__ CUtensorMap map_b2, int tiles1, int kb_total, int x_early,
                    UpdateArgs u) {
    if ((int)blockIdx.x < tiles1) small_update_block<NP, FR>(map_a1, map_b1, 0, (int)blockIdx.x * FR, kb_total, x_early != 0, u);
    else small_update_block<1, FR>(map_a2, map_b2, 1, ((int)blockIdx.x - tiles1) * FR, kb_total, false, u);
}

// ---------------------------------------------------------------- host side
// Up to 512 training rows (their operands are all in shared memory at once) and as many rows in all as give every SM one tile.
bool small_step_supported(int32_t d_in, int32_t hidden, int32_t n_classes, int64_t n_train, int64_t n_all) {
    return d_in > 0 && d_in <= kSmMaxInputs && hidden >= 0 && hidden <= kSmMaxHidden && n_classes > 0 && n_classes <= 64 && n_train > 0 &&
           n_train <= kSmMaxTrain && n_all <= 148 * kSmTile;
}

static size_t small_forward_smem(int np, int stages) {
    return 1024 + kSmABytes * (1 + 2 * np) + (size_t)np * kSmPanelBytes + (size_t)stages * (kSmABytes + np * kSmPanelBytes) +
           4 * (64 + kClassLossExchange) + 8 * (SM_FULL + 2 * kSmMaxStages) + 64 + kSmMmaBytes;
}

int small_forward_launch(const SmallForward& f, cudaStream_t st) {
    if (!small_step_supported(f.d_in, f.hidden, f.n_classes, f.n_train, f.n_all)) return RETEXO_ERR_UNSUPPORTED;
    SmForwardArgs g{};
    g.n_all = f.n_all; g.n_train = f.n_train; g.H = f.hidden; g.O = f.n_classes;
    const int32_t out1 = f.hidden > 0 ? f.hidden : f.n_classes;
    g.np = (out1 + 63) / 64;
    g.kb_total = (f.d_in + kTcBK - 1) / kTcBK;
    g.stages = g.kb_total < kSmMaxStages ? g.kb_total : kSmMaxStages;
    while (g.stages > 1 && small_forward_smem(g.np, g.stages) > 227 * 1024) --g.stages;
    g.x_early = f.x_early ? 1 : 0;
    g.b1 = f.b1; g.b2 = f.b2; g.y = f.y; g.y_eval = f.y_eval; g.inv_rows = f.inv_rows;
    g.loss_partial = f.loss_partial; g.correct = f.correct; g.status = f.status;
    CUtensorMap m[6];
    memset(m, 0, sizeof(m));
    if (!tc_make_map_2d(&m[0], f.x, f.n_all, f.d_in, f.ldx, kSmTile, 64, 128, true)) return RETEXO_ERR_CUDA;
    if (!tc_make_map_2d(&m[1], f.w1t, out1, f.d_in, f.ld_w1t, 64 * g.np, 64, 128, true)) return RETEXO_ERR_CUDA;
    if (!tc_make_map_2d(&m[4], f.dl, f.n_train, 64, f.ld_dl, kSmTile, 64, 128, false)) return RETEXO_ERR_CUDA;
    if (f.hidden > 0) {
        if (!tc_make_map_2d(&m[2], f.w2t, f.n_classes, f.hidden, f.ld_w2t, 64, 64, 128, true)) return RETEXO_ERR_CUDA;
        if (!tc_make_map_2d(&m[3], f.hd, f.n_train, f.hidden, f.ld_hd, kSmTile, 64, 128, false)) return RETEXO_ERR_CUDA;
        if (!tc_make_map_2d(&m[5], f.dhd, f.n_train, f.hidden, f.ld_dhd, kSmTile, 64, 128, false)) return RETEXO_ERR_CUDA;
    }
    const size_t smem = small_forward_smem(g.np, g.stages);
    if (smem > 227 * 1024 || cudaFuncSetAttribute(small_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        (void)cudaGetLastError();
        return RETEXO_ERR_CUDA;
    }
    // (before the wait it reads nothing but, where the caller says so, X)
    OverlapLaunch ol(dim3((unsigned)((f.n_all + kSmTile - 1) / kSmTile)), dim3(kSmThreads), smem, st);
    if (cudaLaunchKernelEx(&ol.cfg, small_forward_kernel, m[0], m[1], m[2], m[3], m[4], m[5], g) != cudaSuccess) {
        (void)cudaGetLastError();
        return RETEXO_ERR_CUDA;
    }
    return launch_status();
}

template <int NP, int FR>
static int launch_small_update(const CUtensorMap (&m)[4], int kb_total, bool x_early, const UpdateArgs& u, cudaStream_t st) {
    const int tiles1 = (u.d_in + FR - 1) / FR, tiles2 = u.hidden > 0 ? (u.hidden + FR - 1) / FR : 0;
    const size_t smem = 1024 + small_update_operands<NP>(kb_total) + kSmOnesBytes + 4 * 64 * NP + 256;      // (the second product's blocks need less)
    auto kernel = small_update_kernel<NP, FR>;
    if (smem > 227 * 1024 || cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        (void)cudaGetLastError();
        return RETEXO_ERR_CUDA;
    }
    // (reads parameters, moments and iteration state early: between the update that left them and this lies the forward kernel)
    OverlapLaunch ol(dim3((unsigned)(tiles1 + tiles2)), dim3(kSmUpdateThreads), smem, st);
    if (cudaLaunchKernelEx(&ol.cfg, kernel, m[0], m[1], m[2], m[3], tiles1, kb_total, x_early ? 1 : 0, u) != cudaSuccess) {
        (void)cudaGetLastError();
        return RETEXO_ERR_CUDA;
    }
    return launch_status();
}

int small_update_launch(const SmallGrad& s, const UpdateArgs& u, cudaStream_t st) {
    CUtensorMap m[4];
    memset(m, 0, sizeof(m));
    if (!tc_make_map_2d(&m[0], s.x, s.n_train, u.d_in, s.ldx, kTcBK, 64, 128, true)) return RETEXO_ERR_CUDA;
    if (!tc_make_map_2d(&m[1], s.grad1, s.n_train, u.out1, s.ld_grad1, kTcBK, 64, 128, true)) return RETEXO_ERR_CUDA;
    if (u.hidden > 0) {
        if (!tc_make_map_2d(&m[2], s.hd, s.n_train, u.hidden, s.ld_hd, kTcBK, 64, 128, true)) return RETEXO_ERR_CUDA;
        if (!tc_make_map_2d(&m[3], s.dl, s.n_train, u.n_classes, s.ld_dl, kTcBK, 64, 128, true)) return RETEXO_ERR_CUDA;
    }
    const int kb = (int)((s.n_train + kTcBK - 1) / kTcBK);
    // Blocks as small as lets all of them be resident at once: 8 inputs a block, else 16, else 32.  (A run of 300 iterations of 140 + 500 rows
    // x 1433, 64: 4.26 ms with 16, 3.95 with 8; 512 rows x 1433, 128, whose operands leave room for one block an SM: 12.7 us with 16, 18.9.)
    auto go = [&]<int FR>() { return u.out1 <= 64 ? launch_small_update<1, FR>(m, kb, s.x_early, u, st) : launch_small_update<2, FR>(m, kb, s.x_early, u, st); };
    const int inputs = u.d_in + u.hidden;
    const int per_sm = kb * (u.out1 <= 64 ? 2 : 3) <= 12 ? 2 : 1;      // (8 KB each)
    return inputs <= 8 * 140 * per_sm ? go.template operator()<8>() : inputs <= 16 * 140 * per_sm ? go.template operator()<16>() : go.template operator()<32>();
}

}  // namespace retexo
