// Soft-max cross-entropy over a row of logits in tensor memory, two threads a row: shared by the kernels that turn a class product into
// loss and dL.  The classes are cut into groups of eight, the first half of the groups goes to the one thread, the rest to the other;
// the two sit in two warps of the same tensor-memory lane quarter and exchange row maximum, sum and the label's logit through shared
// memory.  Every reduction is a tree, so that a warp finds independent instructions to issue.
#pragma once
#include "tc_common.cuh"

namespace retexo {

constexpr int kClassLossExchange = 4 * 4 * 2 * 32;      // floats of shared memory: 4 values x 4 lane quarters x 2 threads x 32 rows

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct ClassLoss {
    int O, part, lane, pair_bar;
    int g_first, g_count, g_split;      // this thread's groups (<= 4)
    float* x;                           // the exchange values of this lane quarter's rows
    float v[32], mx, den, ly;

    // q: the warps' lane quarter; pair_bar: a named barrier of the two warps
    __device__ __forceinline__ ClassLoss(int O_, int part_, int q, int lane_, float* xch, int pair_bar_)
        : O(O_), part(part_), lane(lane_), pair_bar(pair_bar_) {
        const int ng = (O + 7) >> 3;
        g_split = (ng + 1) >> 1;
        g_first = part ? g_split : 0;
        g_count = part ? ng - g_split : g_split;
        x = xch + q * 64 + lane;
    }
    __device__ __forceinline__ void pair_sync() { asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory"); }

    // The thread's logits: accumulator columns plus bias (64 floats in shared memory); columns beyond the last class hold -inf.
    __device__ __forceinline__ void load(uint32_t taddr, const float* bias_s) {
        uint32_t r[32];
        tmem_ld_issue(taddr + (uint32_t)(8 * g_first), r);
        tmem_ld_wait(r);
#pragma unroll
        for (int gi = 0; gi < 4; ++gi) {
            if (gi < g_count) {
                const int c0 = 8 * (g_first + gi);
                const float4 b0 = *reinterpret_cast<const float4*>(bias_s + c0);
                const float4 b1 = *reinterpret_cast<const float4*>(bias_s + c0 + 4);
                const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int k = 0; k < 8; ++k) v[8 * gi + k] = c0 + k < O ? __uint_as_float(r[8 * gi + k]) + bb[k] : -INFINITY;
            }
        }
    }
    // Loss terms of the row; has_eval: rows of this warp are evaluated, their hits (arg-max = label) go to *correct.
    __device__ __forceinline__ void reduce(int32_t label, bool eval, bool has_eval, unsigned long long* correct) {
        mx = -INFINITY;
#pragma unroll
        for (int gi = 0; gi < 4; ++gi) {
            if (gi < g_count) {
                const float m01 = fmaxf(v[8 * gi], v[8 * gi + 1]), m23 = fmaxf(v[8 * gi + 2], v[8 * gi + 3]);
                const float m45 = fmaxf(v[8 * gi + 4], v[8 * gi + 5]), m67 = fmaxf(v[8 * gi + 6], v[8 * gi + 7]);
                mx = fmaxf(mx, fmaxf(fmaxf(m01, m23), fmaxf(m45, m67)));
            }
        }
        if (has_eval) {      // arg-max: the lowest index that reaches this thread's maximum
            int best = 0;
#pragma unroll
            for (int gi = 3; gi >= 0; --gi) {
                if (gi < g_count) {
#pragma unroll
                    for (int k = 7; k >= 0; --k) best = v[8 * gi + k] == mx ? 8 * (g_first + gi) + k : best;
                }
            }
            x[768 + part * 32] = __int_as_float(best);
        }
        x[part * 32] = mx;
        pair_sync();
        const float m0 = x[0], m1 = x[32];
        mx = fmaxf(m0, m1);
        if (has_eval && part == 0) {      // the lower classes win ties
            const int arg = __float_as_int(m1 > m0 ? x[768 + 32] : x[768]);
            const unsigned hits = __ballot_sync(0xffffffffu, eval && arg == label);
            if (lane == 0 && hits) atomicAdd(correct, (unsigned long long)__popc(hits));
        }
        // exp(v - mx) as one multiply-add and one exponential per column; the label's logit is picked up on the way
        const float kLog2e = 1.4426950408889634f;
        const float shift = -mx * kLog2e;
        den = 0.f;
        ly = 0.f;
#pragma unroll
        for (int gi = 0; gi < 4; ++gi) {
            if (gi < g_count) {
                float e[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    ly = 8 * (g_first + gi) + k == label ? v[8 * gi + k] : ly;
                    e[k] = fast_exp2(fmaf(v[8 * gi + k], kLog2e, shift));
                    v[8 * gi + k] = e[k];
                }
                den += ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7]));
            }
        }
        x[256 + part * 32] = den;
        x[512 + part * 32] = ly;
        pair_sync();
        den = x[256] + x[256 + 32];
        ly = x[512] + x[512 + 32];
    }
    // The thread's columns of dL as bf16 into the row's 128-byte line (128-byte swizzle); padding columns are zero.
    __device__ __forceinline__ void store_dl(int32_t label, bool train, float inv_rows, uint8_t* line) const {
        const float scale = train ? inv_rows / den : 0.f;
        const float hot = train ? inv_rows : 0.f;
#pragma unroll
        for (int gi = 0; gi < 4; ++gi) {      // one 16-byte piece of the row's line per group of eight classes
            const int piece = part ? g_split + gi : gi;      // part 1 also clears the pieces beyond the last class
            if (piece < 8 && (part || gi < g_split)) {
                uint32_t pk[4] = {0u, 0u, 0u, 0u};
                if (gi < g_count) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int c = 8 * piece + 2 * k;
                        const float lo = fmaf(v[8 * gi + 2 * k], scale, c == label ? -hot : 0.f);
                        const float hi = fmaf(v[8 * gi + 2 * k + 1], scale, c + 1 == label ? -hot : 0.f);
                        __nv_bfloat162 b2 = __floats2bfloat162_rn(lo, hi);
                        pk[k] = *reinterpret_cast<uint32_t*>(&b2);
                    }
                }
                *reinterpret_cast<uint4*>(line + ((piece ^ (lane & 7)) * 16)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
        }
        if (part == 1) {      // pieces that neither thread's four groups reach (few classes): zeros
            for (int piece = g_split + 4; piece < 8; ++piece)
                *reinterpret_cast<uint4*>(line + ((piece ^ (lane & 7)) * 16)) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    __device__ __forceinline__ float loss(bool train) const { return train ? (mx + __logf(den)) - ly : 0.f; }
};

}  // namespace retexo
