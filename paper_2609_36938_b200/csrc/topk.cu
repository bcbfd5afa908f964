// janus_topk: per-row selection of the k largest scores over the causal prefix (Eq. 1, Sec. 2.2).
//
// A CTA works on one query row at a time; the CTAs resident on the device walk the rows with stride gridDim.x, or, while rows
// are few, a cluster of CTAs shares a row.  The row (0.5-1 MB of fp32 at 128K-256K keys) is read from HBM once:
//   1. a strided sample of the row (512 x 32-byte sectors) gives a conservative threshold whose
//      expected rank is a little above k;
//   2. one streaming pass with 16-byte loads keeps only the elements at or above that threshold
//      in a shared-memory candidate buffer (~1.5-3 % of the row pass the one-compare filter);
//   3. a 2048-bucket histogram of the candidates (linear in the order-preserving integer key) gives the bucket of the k-th
//      key; one pass emits everything above it and the keys inside are ranked directly.
// If the sample misjudges the row (fewer than k candidates, or more than the buffer holds) an exact selection over repeated
// histograms runs over the row in global memory instead; that path is slower, never wrong.  A threshold with thousands of copies has a
// way of its own (topk_row).  Rows that fit the buffer may skip the sampling step (janus_topk).
#include <algorithm>

#include "topk_plan.h"
#include "topk_select.cuh"

namespace janus {

// Three CTAs share an SM (registers).  With 73 KB of shared memory each they leave next to nothing of it to L1, through which the
// streaming loads pass, with 54 KB a third: 4096 rows of 135168 390 us against 498, 1024 of 16384 28 against 35.  (Four CTAs of 54 KB and
// 32 registers: 497.)
constexpr int TK_CAP = 8192;
constexpr int TK_CAP_SMALLEST = 3840;

template <int CAP>
__global__ void __launch_bounds__(TK_THREADS)
topk_rows_kernel(const float* scores, int64_t ld, int M, int64_t n_keys, int64_t q_pos0, int causal, int k,
                 int32_t* __restrict__ idx, int32_t* __restrict__ count, float* __restrict__ kth) {
    grid_launch_next();
    grid_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using TopkShared = TopkSharedT<CAP>;
    TopkShared& sh = *reinterpret_cast<TopkShared*>(smem_raw);
    // resident CTAs walk the rows with stride gridDim.x, each asking for the head of its next row ahead of time
    for (int t = blockIdx.x; t < M; t += gridDim.x) {
        const int64_t prefix64 = causal ? min(n_keys, q_pos0 + t + 1) : n_keys;
        const int t_next = t + gridDim.x;
        const int64_t prefix_next = t_next < M ? (causal ? min(n_keys, q_pos0 + t_next + 1) : n_keys) : 0;
        topk_row<CAP == TK_CAP_SMALLEST>(scores + static_cast<int64_t>(t) * ld, static_cast<int>(prefix64), k, idx + static_cast<int64_t>(t) * k,
                 count != nullptr ? count + t : nullptr, kth != nullptr ? kth + t : nullptr, sh, t_next < M ? scores + static_cast<int64_t>(t_next) * ld : nullptr, static_cast<int>(prefix_next));
        __syncthreads();   // the selection state in shared memory is reused by the next row
    }
}

// Few rows: one cluster of CTAs per row.
__global__ void __launch_bounds__(TK_THREADS)
topk_rows_cluster_kernel(const float* scores, int64_t ld, int64_t n_keys, int64_t q_pos0, int causal, int k,
                         int32_t* __restrict__ idx, int32_t* __restrict__ count, float* __restrict__ kth) {
    grid_launch_next();
    grid_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TopkSharedT<TK_CAP>& sh = *reinterpret_cast<TopkSharedT<TK_CAP>*>(smem_raw);
    const int t = blockIdx.x / ptx::cluster_nctarank();
    const int64_t prefix = causal ? min(n_keys, q_pos0 + t + 1) : n_keys;
    topk_row_cluster(scores + static_cast<int64_t>(t) * ld, static_cast<int>(prefix), k, idx + static_cast<int64_t>(t) * k,
                     count != nullptr ? count + t : nullptr, kth != nullptr ? kth + t : nullptr, sh);
}

// Entry granularity (footnote of Sec. 2.2): columns are entries of `entry_size` consecutive tokens; row t (position
// q_pos0 + t) may select the entries that hold a token at or before its position: entries 0 .. (q_pos0 + t) / entry_size.
template <int CAP>
__global__ void __launch_bounds__(TK_THREADS)
topk_entries_kernel(const float* scores, int64_t ld, int M, int64_t n_entries, int64_t q_pos0, int entry_size, int k,
                    int32_t* __restrict__ idx, int32_t* __restrict__ count, float* __restrict__ kth) {
    grid_launch_next();
    grid_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using TopkShared = TopkSharedT<CAP>;
    TopkShared& sh = *reinterpret_cast<TopkShared*>(smem_raw);
    const int t = blockIdx.x;
    int64_t prefix = (q_pos0 + t) / entry_size + 1;
    if (prefix > n_entries) prefix = n_entries;
    topk_row(scores + static_cast<int64_t>(t) * ld, static_cast<int>(prefix), k, idx + static_cast<int64_t>(t) * k,
             count != nullptr ? count + t : nullptr, kth != nullptr ? kth + t : nullptr, sh);
}

// Token selection of an entry selection: slot e * E + j of row t = entry * E + j if that token is at or before q_pos0 + t.
__global__ void entry_expand_kernel(const int32_t* idx_e, int M, int k_e, int entry_size, int64_t q_pos0,
                                    int32_t* __restrict__ idx_tok) {
    grid_launch_next();
    grid_wait();
    const int64_t n = static_cast<int64_t>(M) * k_e * entry_size;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t slot = i / entry_size;            // (t, e)
        const int j = static_cast<int>(i - slot * entry_size);
        const int64_t t = slot / k_e;
        const int32_t ent = ld_input(idx_e + slot);
        const int64_t tok = static_cast<int64_t>(ent) * entry_size + j;
        idx_tok[i] = (ent >= 0 && tok <= q_pos0 + t) ? static_cast<int32_t>(tok) : -1;
    }
}

// Pooled entry scores (the second reading of the entry footnote of Sec. 2.2): an entry scores as the best of its tokens the
// row may see.  Bound by the bytes of the score matrix.
//
// Entries of 4, 8, .. 128 tokens in 16-byte aligned rows: a warp takes 128 U consecutive scores with U 16-byte loads per lane,
// all in flight together; ENTRY / 4 neighbouring lanes hold an entry of each load.  512 rows x 40512 in entries of 128: 32.8 us with
// a warp per entry (four 4-byte loads and a 64-bit division each), 19 us so; entries of 16 tokens 200 and 18.
template <int ENTRY, int U>
__global__ void __launch_bounds__(256)
entry_pool_vec_kernel(const float* scores, int64_t ld, int M, int64_t n_keys, int64_t q_pos0, int causal, int n_entries,
                      float* __restrict__ out, int64_t out_ld) {
    grid_launch_next();
    grid_wait();
    constexpr int LANES = ENTRY / 4, STRIP = 128 * U;
    const int lane = threadIdx.x & 31;
    const int strip = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int64_t s0 = static_cast<int64_t>(strip) * STRIP + 4 * lane;
    const float neg_inf = __int_as_float(0xff800000);
    for (int t = blockIdx.y; t < M; t += gridDim.y) {
        const int64_t prefix = causal ? (n_keys < q_pos0 + t + 1 ? n_keys : q_pos0 + t + 1) : n_keys;
        const float* row = scores + static_cast<int64_t>(t) * ld;
        float4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t s = s0 + 128 * u;
            x[u] = make_float4(neg_inf, neg_inf, neg_inf, neg_inf);
            if (s + 3 < prefix) {
                x[u] = __ldcs(reinterpret_cast<const float4*>(row + s));
            } else {
                if (s < prefix) x[u].x = row[s];
                if (s + 1 < prefix) x[u].y = row[s + 1];
                if (s + 2 < prefix) x[u].z = row[s + 2];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float m = fmaxf(fmaxf(x[u].x, x[u].y), fmaxf(x[u].z, x[u].w));
            if constexpr (LANES == 32) {
                asm volatile("redux.sync.max.f32 %0, %0, 0xffffffff;" : "+f"(m));
            } else {
#pragma unroll
                for (int d = LANES / 2; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
            }
            const int e = static_cast<int>((s0 + 128 * u) / ENTRY);
            if ((lane & (LANES - 1)) == 0 && e < n_entries) out[static_cast<int64_t>(t) * out_ld + e] = m;
        }
    }
}

// Any entry size: one warp per (row, entry) strip, lanes read consecutive floats, a warp shuffle takes the maximum.
__global__ void __launch_bounds__(256)
entry_pool_kernel(const float* scores, int64_t ld, int M, int64_t n_keys, int64_t q_pos0, int causal, int entry_size,
                  int64_t n_entries, float* __restrict__ out, int64_t out_ld) {
    grid_launch_next();
    grid_wait();
    const int lane = threadIdx.x & 31;
    const int64_t warp_id = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t n_warps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const float neg_inf = __int_as_float(0xff800000);
    for (int64_t item = warp_id; item < static_cast<int64_t>(M) * n_entries; item += n_warps) {
        const int64_t t = item / n_entries, e = item - t * n_entries;
        const int64_t prefix = causal ? (n_keys < q_pos0 + t + 1 ? n_keys : q_pos0 + t + 1) : n_keys;
        const int64_t a = e * entry_size;
        const int64_t b = a + entry_size < prefix ? a + entry_size : prefix;
        const float* row = scores + t * ld;
        float m = neg_inf;
        for (int64_t s = a + lane; s < b; s += 32) m = fmaxf(m, ld_input(row + s));
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
        if (lane == 0) out[t * out_ld + e] = m;
    }
}

// Batch form (decode over many sessions): row b starts at scores[row_offsets[b]] and has row_lengths[b] elements (or runs
// up to the next row's start when row_lengths is NULL), every element visible.
template <bool CLUSTER>
__global__ void __launch_bounds__(TK_THREADS)
topk_ragged_kernel(const float* scores, const int64_t* row_offsets, const int64_t* row_lengths, int k,
                   int32_t* __restrict__ idx, int32_t* __restrict__ count, float* __restrict__ kth, int32_t* dev_status) {
    grid_launch_next();
    grid_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TopkSharedT<TK_CAP>& sh = *reinterpret_cast<TopkSharedT<TK_CAP>*>(smem_raw);
    const int b = CLUSTER ? blockIdx.x / ptx::cluster_nctarank() : blockIdx.x;
    const int64_t off = row_offsets[b];
    const int64_t n = row_lengths != nullptr ? row_lengths[b] : row_offsets[b + 1] - off;
    // the offsets come from device memory: a row that starts before the array, off a 16-byte boundary (the row is read with
    // 16-byte loads) or has a negative or unrepresentable length is reported and left empty, never read
    if (off < 0 || (off & 3) != 0 || n < 0 || n > 2147483639) {
        for (int i = threadIdx.x; i < k; i += blockDim.x) idx[static_cast<int64_t>(b) * k + i] = -1;      // (every CTA of a cluster: the same values)
        if (threadIdx.x == 0) {
            if (count != nullptr) count[b] = 0;
            if (kth != nullptr) kth[b] = __int_as_float(0xff800000);
            report(dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);
        }
        return;
    }
    int32_t* out = idx + static_cast<int64_t>(b) * k;
    if constexpr (CLUSTER)
        topk_row_cluster(scores + off, static_cast<int>(n), k, out, count != nullptr ? count + b : nullptr, kth != nullptr ? kth + b : nullptr, sh);
    else
        topk_row(scores + off, static_cast<int>(n), k, out, count != nullptr ? count + b : nullptr, kth != nullptr ? kth + b : nullptr, sh);
}

// The forms of topk_rows_kernel, by candidate slots.
struct TopkForm {
    void (*kernel)(const float*, int64_t, int, int64_t, int64_t, int, int, int32_t*, int32_t*, float*);
    int cap, smem;
};
template <int CAP>
constexpr TopkForm topk_form() { return {topk_rows_kernel<CAP>, CAP, static_cast<int>(sizeof(TopkSharedT<CAP>))}; }
constexpr int TK_FORMS = 3;
static const TopkForm topk_forms[TK_FORMS] = {topk_form<TK_CAP_SMALLEST>(), topk_form<5632>(), topk_form<TK_CAP>()};

// Kernel attributes, set once in every context, and the number of resident CTAs, a property of the device.
struct TopkDevice {
    int n_sm, resident[TK_FORMS];
};
static cudaError_t topk_device(TopkDevice& d) {
    static once_per_context once;
    static std::atomic<int> sms[64], resident[64][TK_FORMS];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    e = once.run([&] {
        const int smem = static_cast<int>(sizeof(TopkSharedT<TK_CAP>));
        int n_sm = 0;
        cudaError_t r = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        auto limit = [&](const void* f, int bytes) { if (r == cudaSuccess) r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); };
        limit(reinterpret_cast<const void*>(topk_rows_cluster_kernel), smem);
        limit(reinterpret_cast<const void*>(topk_entries_kernel<TK_CAP>), smem);
        limit(reinterpret_cast<const void*>(topk_ragged_kernel<true>), smem);
        limit(reinterpret_cast<const void*>(topk_ragged_kernel<false>), smem);
        sms[dev] = n_sm;
        for (int f = 0; f < TK_FORMS; ++f) {
            int per = 0;
            limit(reinterpret_cast<const void*>(topk_forms[f].kernel), topk_forms[f].smem);
            if (r == cudaSuccess) r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, topk_forms[f].kernel, TK_THREADS, topk_forms[f].smem);
            resident[dev][f] = std::max(1, per) * n_sm;
        }
        return r;
    });
    d.n_sm = sms[dev];
    for (int f = 0; f < TK_FORMS; ++f) d.resident[f] = resident[dev][f];
    return e;
}

}  // namespace janus

extern "C" int janus_topk_entries(const float* scores, int64_t scores_ld, int M, int64_t n_entries, int64_t q_pos0, int entry_size, int k,
                                  int32_t* idx, int32_t* count, float* kth, int32_t* /*dev_status*/, void* stream_) {
    using namespace janus;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (M < 0 || n_entries < 0 || k <= 0 || q_pos0 < 0 || entry_size <= 0 || scores_ld < n_entries) return JANUS_ERR_INVALID_ARG;
    if (n_entries >= (int64_t(1) << 31) - 8) return JANUS_ERR_UNSUPPORTED;
    if (M == 0) return JANUS_OK;
    if (!idx) return JANUS_ERR_INVALID_ARG;
    if (n_entries > 0 && (!scores || !aligned16(scores) || (scores_ld & 3) != 0)) return JANUS_ERR_INVALID_ARG;
    const size_t smem = sizeof(TopkSharedT<TK_CAP>);
    TopkDevice d;
    JANUS_CUDA_CHECK(topk_device(d));
    JANUS_CUDA_CHECK(launch_kernel(topk_entries_kernel<TK_CAP>, dim3(M), TK_THREADS, smem, stream, 1, scores, scores_ld, M, n_entries, q_pos0,
                                   entry_size, k, idx, count, kth));
    return JANUS_OK;
}

extern "C" int janus_entry_pool_scores(const float* scores, int64_t scores_ld, int M, int64_t n_keys, int64_t q_pos0, int causal, int entry_size,
                                       float* entry_scores, int64_t entry_ld, void* stream_) {
    using namespace janus;
    if (M < 0 || n_keys < 0 || q_pos0 < 0 || entry_size <= 0 || scores_ld < n_keys) return JANUS_ERR_INVALID_ARG;
    const int64_t n_entries = (n_keys + entry_size - 1) / entry_size;
    if (entry_ld < n_entries) return JANUS_ERR_INVALID_ARG;
    if (M == 0 || n_entries == 0) return JANUS_OK;
    if (!scores || !entry_scores) return JANUS_ERR_INVALID_ARG;
    const cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (aligned16(scores) && (scores_ld & 3) == 0 && n_keys < (int64_t(1) << 31) - 8192) {
        // Eight loads per lane keep the most bytes in flight; two while eight would leave the chip short of warps (512 rows of 1000 in
        // entries of 64 2.3 us against 4.6, 2000 rows of 200 3.8 against 12.9).
        const bool few = M * ((n_keys + 1023) / 1024) < 148 * 16;
        const int per_block = 8 * 128 * (few ? 2 : 8);
        const dim3 grid(static_cast<unsigned>((n_keys + per_block - 1) / per_block), static_cast<unsigned>(M < 65535 ? M : 65535));
        const int n = static_cast<int>(n_entries);
        switch (entry_size) {
#define JANUS_POOL_CASE(E)                                                                                                                    \
    case E:                                                                                                                                   \
        if (few) JANUS_CUDA_CHECK(launch_kernel(entry_pool_vec_kernel<E, 2>, grid, 256, 0, stream, 1, scores, scores_ld, M, n_keys, q_pos0,   \
                                                causal, n, entry_scores, entry_ld));                                                          \
        else JANUS_CUDA_CHECK(launch_kernel(entry_pool_vec_kernel<E, 8>, grid, 256, 0, stream, 1, scores, scores_ld, M, n_keys, q_pos0,       \
                                            causal, n, entry_scores, entry_ld));                                                              \
        return JANUS_OK;
            JANUS_POOL_CASE(4)
            JANUS_POOL_CASE(8)
            JANUS_POOL_CASE(16)
            JANUS_POOL_CASE(32)
            JANUS_POOL_CASE(64)
            JANUS_POOL_CASE(128)
#undef JANUS_POOL_CASE
        }
    }
    const int64_t items = static_cast<int64_t>(M) * n_entries;
    int64_t blocks = (items + 7) / 8;                        // eight warps per block, one strip each
    if (blocks > 148 * 16) blocks = 148 * 16;
    JANUS_CUDA_CHECK(launch_kernel(entry_pool_kernel, dim3(static_cast<unsigned>(blocks)), 256, 0, stream, 1, scores,
                                   scores_ld, M, n_keys, q_pos0, causal, entry_size, n_entries, entry_scores, entry_ld));
    return JANUS_OK;
}

extern "C" int janus_entry_expand(const int32_t* idx_entries, int M, int k_e, int entry_size, int64_t q_pos0, int32_t* idx_tokens,
                                  void* stream_) {
    using namespace janus;
    if (M < 0 || k_e < 0 || entry_size <= 0 || q_pos0 < 0) return JANUS_ERR_INVALID_ARG;
    const int64_t n = static_cast<int64_t>(M) * k_e * entry_size;
    if (n == 0) return JANUS_OK;
    if (!idx_entries || !idx_tokens) return JANUS_ERR_INVALID_ARG;
    if (static_cast<int64_t>(k_e) * entry_size > 2147483647) return JANUS_ERR_UNSUPPORTED;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 148 * 16) blocks = 148 * 16;
    JANUS_CUDA_CHECK(launch_kernel(entry_expand_kernel, dim3(static_cast<unsigned>(blocks)), 256, 0, static_cast<cudaStream_t>(stream_), 1,
                                   idx_entries, M, k_e, entry_size, q_pos0, idx_tokens));
    return JANUS_OK;
}

extern "C" int janus_topk_batch(const float* scores, const int64_t* row_offsets, const int64_t* row_lengths, int B, int k, int32_t* idx,
                                int32_t* count, float* kth, int32_t* dev_status, void* stream_) {
    using namespace janus;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (B < 0 || k <= 0) return JANUS_ERR_INVALID_ARG;
    if (B == 0) return JANUS_OK;
    if (!idx || !row_offsets || !scores || !aligned16(scores)) return JANUS_ERR_INVALID_ARG;
    // row lengths live on the device: the large candidate buffer serves any length
    TopkDevice d;
    JANUS_CUDA_CHECK(topk_device(d));
    const int cluster = topk_cluster_size(B, -1.);
    if (cluster > 1) {
        JANUS_CUDA_CHECK(launch_kernel(topk_ragged_kernel<true>, dim3(B * cluster), TK_THREADS, sizeof(TopkSharedT<TK_CAP>), stream, cluster, scores,
                                       row_offsets, row_lengths, k, idx, count, kth, dev_status));
    } else {
        JANUS_CUDA_CHECK(launch_kernel(topk_ragged_kernel<false>, dim3(B), TK_THREADS, sizeof(TopkSharedT<TK_CAP>), stream, 1, scores, row_offsets,
                                       row_lengths, k, idx, count, kth, dev_status));
    }
    return JANUS_OK;
}

extern "C" size_t janus_topk_workspace_size(int, int64_t, int) { return 0; }

extern "C" int janus_topk(const float* scores, int64_t scores_ld, int M, int64_t n_keys, int64_t q_pos0, int causal, int k,
                          int32_t* idx, int32_t* count, float* kth, void* /*ws*/, size_t /*ws_bytes*/,
                          int32_t* /*dev_status*/, void* stream_) {
    using namespace janus;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (M < 0 || n_keys < 0 || k <= 0 || q_pos0 < 0 || scores_ld < n_keys) return JANUS_ERR_INVALID_ARG;
    if (n_keys >= (int64_t(1) << 31) - 8) return JANUS_ERR_UNSUPPORTED;
    if (M == 0) return JANUS_OK;
    if (!idx) return JANUS_ERR_INVALID_ARG;
    if (n_keys > 0 && (!scores || !aligned16(scores) || (scores_ld & 3) != 0)) return JANUS_ERR_INVALID_ARG;
    // The candidate list of a row holds what passes the sampled threshold: about n * r / 4096 elements for the sample rank
    // r = e + 4 sqrt(e) + 8, e = 4096 k / n, give or take n sqrt(r) / 4096 and what the lower edge of the threshold's bucket lets in
    // besides (3 + r / 16 sample keys at most; drawn normal, gamma and narrow rows had lists under 2 % longer than expected).  The smallest
    // form is taken into which the list plus five deviations fits for the longest row, since less shared memory leaves more of it to L1
    // (2048 rows of 34816 102.7 us with 5632 slots, 96.7 with 3840; 777 of 20788 34.7 and 32.3; 4096 of 135168 498 with 8192 and 396 with
    // 5632); a row that overflows all the same is selected from global memory.  Rows that fit a form whole are taken whole where CTAs have
    // an SM each, half of the row is on the list anyway or the list needs more than the smallest form, which alone is safe against a crowd at
    // the threshold (256 of 4000, k = 2048, 8.9 us, 11.3 through the sample; 256 of 8000 17.8 and 12.5; 4000 of 6000, k = 512, 216 and 85;
    // of values in steps of one half 169 and 156, but with few to select the sample's further passes show: 4000 of 3900, k = 64, 100 and 128).
    const double n_max = static_cast<double>(causal ? (n_keys < q_pos0 + M ? n_keys : q_pos0 + M) : n_keys);
    const double e = n_max > 0. ? 4096.0 * k / n_max : 0., r = e + 4.0 * sqrt(e) + 8.0, list = n_max * (r + 5.0 * sqrt(r)) / 4096.0;
    TopkDevice d;
    JANUS_CUDA_CHECK(topk_device(d));
    const bool share = M > d.n_sm;
    auto fits = [&](int f) { return list <= topk_forms[f].cap && k <= topk_forms[f].cap / 2 + 256; };
    const bool whole = n_max <= TK_CAP && (!share || list > n_max / 2 || !fits(0));
    int form = share ? 0 : 1;
    while (form < TK_FORMS - 1 && !(whole ? n_max <= topk_forms[form].cap : fits(form))) ++form;
    const int cluster = topk_cluster_size(M, n_max);
    if (cluster > 1) {
        JANUS_CUDA_CHECK(launch_kernel(topk_rows_cluster_kernel, dim3(M * cluster), TK_THREADS, sizeof(TopkSharedT<TK_CAP>), stream, cluster, scores,
                                       scores_ld, n_keys, q_pos0, causal, k, idx, count, kth));
        return JANUS_OK;
    }
    const TopkForm& f = topk_forms[form];
    JANUS_CUDA_CHECK(launch_kernel(f.kernel, dim3(std::min(M, d.resident[form])), TK_THREADS, f.smem, stream, 1, scores, scores_ld, M, n_keys, q_pos0, causal, k,
                                   idx, count, kth));
    return JANUS_OK;
}
