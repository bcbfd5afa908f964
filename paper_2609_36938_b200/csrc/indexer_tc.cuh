// Parts shared by the tensor-core indexer kernels (indexer_tc.cu, indexer_tc_batch.cu).
#pragma once

#include "janus_common.cuh"
#include "sm100_ptx.cuh"

namespace janus {

using namespace ptx;

constexpr int TC_KEYS = 128;        // keys per tile = MMA M
constexpr int TC_SMEM_BUDGET = 227 * 1024;
constexpr int TC_MAX_CTAS = 148;      // SMs: CTAs of a persistent launch that are resident at once

// Barrier of the epilogue warps alone.
template <int THREADS>
__device__ __forceinline__ void epilogue_barrier() {
    asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// One 32-column chunk of accumulators: 2 * ReLU, half weight, reduce over heads; a token's sum is complete every H columns.
// Pairs of columns go through packed fp32 FMAs into up to four independent accumulator pairs, so the reduction is
// neither one long dependent chain nor one instruction per element.
template <int H, class Store>
__device__ __forceinline__ void reduce_chunk(const uint32_t (&r)[32], const float* __restrict__ wchunk, int col0, float2 (&acc)[4], Store&& store) {
    constexpr int NACC = (H / 2 < 4) ? H / 2 : 4;
#pragma unroll
    for (int i4 = 0; i4 < 8; ++i4) {
        const float4 wv = *reinterpret_cast<const float4*>(wchunk + 4 * i4);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int i = 4 * i4 + 2 * j;                      // first column of the pair inside the chunk
            const int col = col0 + i;
            const float2 w2 = j == 0 ? make_float2(wv.x, wv.y) : make_float2(wv.z, wv.w);
            // 2 * max(x, 0) = x + |x|, exactly: an add (full-rate FMA pipe, |x| is an operand modifier) instead of a max (the
            // half-rate pipe, which 256 of them per thread and tile would saturate before the tensor pipe); the weights
            // carry the factor 1/2
            const float xa = __uint_as_float(r[i]), xb = __uint_as_float(r[i + 1]);
            const float2 x2 = make_float2(xa + fabsf(xa), xb + fabsf(xb));
            float2& a = acc[(col / 2) % NACC];
            a = ffma2(w2, x2, a);
            if (((col + 2) % H) == 0) {
                float v = 0.f;
#pragma unroll
                for (int q = 0; q < NACC; ++q) {
                    v += acc[q].x + acc[q].y;
                    acc[q] = make_float2(0.f, 0.f);
                }
                store(col / H, v);
            }
        }
    }
}

}  // namespace janus
