// Shared device code of the top-k selection (Eq. 1, Sec. 2.2, selection part): the sampled single-pass top-k of one fp32 row,
// by one CTA or by a cluster, and exact k-th selection over a candidate set.
// Used by janus_topk (materialised scores) and by janus_indexer_topk (candidates appended by the indexer epilogue).
//
// A row's time beyond its bytes is the chain of block-wide steps of its two selections, so both are kept short: the threshold is
// the lower edge of a bucket of one histogram over the sample (held in registers; a conservative threshold need not be a
// sample value), candidates are counted into the buckets of a second histogram as they are found, and one pass over them then
// emits what lies above the k-th key's bucket while the few keys inside it are ranked directly.  Against two selections of repeated
// histogram passes (B200, k = 2048, the kernel alone in a loop): 4096 rows of 135168 0.442 -> 0.385 ms (5.7 TB/s, 0.86 of the copy bandwidth; what is left
// is that a CTA between two streaming passes reads nothing; inside a step, after the indexer, 0.483 -> 0.42 = 0.81), 2048 rows of 34816 122 -> 100 us, one row of 32768 (a cluster) 15.4 -> 9.6, and 8.2 us
// with its first loads issued before the sample and counts of 16 bits exchanged.  The exact selection over
// repeated histogram passes (select_kth) remains for what this cannot settle: a misjudged sample, or hundreds of keys in one bucket.
#pragma once

#include "janus_common.cuh"
#include "sm100_ptx.cuh"
#include "topk_plan.h"

namespace janus {

constexpr int TK_THREADS = 512;
constexpr int TK_WARPS = TK_THREADS / 32;
constexpr int TK_MAX_CLUSTER = 8;   // CTAs that share a row
constexpr int TK_BUCKETS = 2048;
constexpr int TK_SAMPLE = 4096;     // 512 threads x 8 floats (one 32-byte sector each)
constexpr int TK_FULL = 1 << 26;    // more than the counts of all buckets of a cluster
constexpr int TK_DIRECT = 256;      // a bucket of at most this many keys is ranked directly instead of split further

template <int CAP>
struct TopkSharedT {
    static constexpr int kCap = CAP;      // candidate slots (key + index = 8 bytes each)
    uint32_t cand_key[CAP];
    int32_t cand_idx[CAP];
    alignas(16) int hist[TK_BUCKETS];
    uint32_t small_key[TK_DIRECT];        // the keys of the k-th key's bucket
    int32_t small_idx[TK_DIRECT];
    int scan[40];
    uint32_t warp_lo[TK_WARPS], warp_hi[TK_WARPS];
    int n_cand;
    int out_pos;
    int eq_taken;
    uint32_t red_lo, red_hi;
    int sel_bucket, sel_above, sel_count;
    int n_small;
    int crowd;                            // see sample_threshold
    int sel_out;                          // cluster form: next free slot of the row's output
};

struct SmemSource {
    const uint32_t* key;
    const int32_t* idx;
    int n;
    __device__ __forceinline__ int size() const { return n; }
    __device__ __forceinline__ uint32_t key_at(int i) const { return key[i]; }
    __device__ __forceinline__ int32_t idx_at(int i) const { return idx ? idx[i] : i; }
};
struct GlobalSource {
    const float* row;
    int n;
    __device__ __forceinline__ int size() const { return n; }
    __device__ __forceinline__ uint32_t key_at(int i) const { return float_to_key(__ldcg(row + i)); }
    __device__ __forceinline__ int32_t idx_at(int i) const { return i; }
};

// Exact `need`-th largest key of a source (1 <= need <= number of elements).
// Returns the threshold key T and, in *n_eq_take, how many elements equal to T belong to the selection.
// Every thread of the CTA must call it; results are uniform.
template <class Src, class Sh>
__device__ __noinline__ uint32_t select_kth(const Src& src, int need, Sh& sh, int* n_eq_take) {
    const int tid = threadIdx.x;
    const int n = src.size();
    // range of the active keys
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int i = tid; i < n; i += TK_THREADS) {
        const uint32_t key = src.key_at(i);
        lo = min(lo, key);
        hi = max(hi, key);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, d));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, d));
    }
    if (tid == 0) { sh.red_lo = 0xffffffffu; sh.red_hi = 0u; }
    __syncthreads();
    if ((tid & 31) == 0) { atomicMin(&sh.red_lo, lo); atomicMax(&sh.red_hi, hi); }
    __syncthreads();
    lo = sh.red_lo;
    hi = sh.red_hi;
    __syncthreads();

    for (int iter = 0; iter < 8 && lo < hi; ++iter) {
        const uint32_t range = hi - lo;
        const int bits = 32 - __clz(range);                   // range < 2^bits
        const int shift = bits > 11 ? bits - 11 : 0;          // (range >> shift) < 2048
        for (int i = tid; i < TK_BUCKETS; i += TK_THREADS) sh.hist[i] = 0;
        __syncthreads();
        for (int i = tid; i < n; i += TK_THREADS) {
            const uint32_t key = src.key_at(i);
            if (key >= lo && key <= hi) atomicAdd(&sh.hist[(key - lo) >> shift], 1);
        }
        __syncthreads();
        // walk the buckets from the top: thread t owns the 4 buckets 2047-4t .. 2044-4t
        int c[4];
        int mine = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) { c[j] = sh.hist[TK_BUCKETS - 1 - (4 * tid + j)]; mine += c[j]; }
        int total;
        int above = block_exclusive_scan<TK_THREADS>(mine, sh.scan, &total);
        if (above < need && need <= above + mine) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (above < need && need <= above + c[j]) { sh.sel_bucket = TK_BUCKETS - 1 - (4 * tid + j); sh.sel_above = above; sh.sel_count = c[j]; }
                above += c[j];
            }
        }
        __syncthreads();
        const uint32_t b = static_cast<uint32_t>(sh.sel_bucket);
        need -= sh.sel_above;
        const uint32_t new_lo = lo + (b << shift);
        if (b < (range >> shift)) hi = new_lo + ((1u << shift) - 1u);   // the top bucket keeps hi (and cannot overflow)
        lo = new_lo;
        const int m = sh.sel_count;                                    // keys inside [lo, hi]
        __syncthreads();
        if (lo < hi && m <= TK_DIRECT) {
            // Few keys are left: instead of two more histogram passes (each a sweep over the source plus a block scan), copy
            // them out (the histogram array is free) and count, for every key, the keys above and equal to it.
            uint32_t* small = reinterpret_cast<uint32_t*>(sh.hist);
            if (tid == 0) sh.n_small = 0;
            __syncthreads();
            for (int i = tid; i < n; i += TK_THREADS) {
                const uint32_t key = src.key_at(i);
                if (key >= lo && key <= hi) small[atomicAdd(&sh.n_small, 1)] = key;
            }
            __syncthreads();
            for (int i = tid >> 5; i < m; i += TK_THREADS / 32) {      // a warp per key, its lanes striding over the others
                const uint32_t mine = small[i];
                int g = 0, e = 0;
                for (int j = tid & 31; j < m; j += 32) {
                    const uint32_t other = small[j];
                    g += other > mine ? 1 : 0;
                    e += other == mine ? 1 : 0;
                }
                g = __reduce_add_sync(0xffffffffu, g);
                e = __reduce_add_sync(0xffffffffu, e);
                if ((tid & 31) == 0 && g < need && need <= g + e) { sh.red_lo = mine; sh.sel_above = need - g; }   // equal keys write equal values
            }
            __syncthreads();
            const uint32_t T = sh.red_lo;
            *n_eq_take = sh.sel_above;
            __syncthreads();
            return T;
        }
    }
    *n_eq_take = need;   // lo == hi: `need` of the elements equal to lo complete the selection
    return lo;
}

// Writes the selection (all keys > T, plus n_eq of the keys == T) to out[0..k).
template <class Src, class Sh>
__device__ __noinline__ void emit_selection(const Src& src, uint32_t T, int n_eq, int32_t* out, Sh& sh) {
    const int n = src.size();
    for (int i = threadIdx.x; i < n; i += TK_THREADS) {
        const uint32_t key = src.key_at(i);
        if (key > T) {
            out[atomicAdd(&sh.out_pos, 1)] = src.idx_at(i);
        } else if (key == T) {
            if (atomicAdd(&sh.eq_taken, 1) < n_eq) out[atomicAdd(&sh.out_pos, 1)] = src.idx_at(i);
        }
    }
}

// ---- short selections ---------------------------------------------------------------------------------------------------------
// Smallest and largest key of the block (every thread gets them; one barrier).
template <class Sh>
__device__ __forceinline__ void block_key_range(uint32_t& lo, uint32_t& hi, Sh& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { sh.warp_lo[warp] = lo; sh.warp_hi[warp] = hi; }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, sh.warp_lo[lane & (TK_WARPS - 1)]);
    hi = __reduce_max_sync(0xffffffffu, sh.warp_hi[lane & (TK_WARPS - 1)]);
}

// Buckets linear in the key over [lo, hi], at most TK_BUCKETS of them; keys above hi count into the last.
struct BucketMap {
    uint32_t lo;
    int shift;
    __device__ __forceinline__ BucketMap(uint32_t lo_, uint32_t hi) : lo(lo_) {
        const int bits = 32 - __clz(hi - lo_);
        shift = bits > 11 ? bits - 11 : 0;
    }
    __device__ __forceinline__ int operator()(uint32_t key) const { return static_cast<int>(min((key - lo) >> shift, static_cast<uint32_t>(TK_BUCKETS - 1))); }
    __device__ __forceinline__ uint32_t first(int b) const { return lo + (static_cast<uint32_t>(b) << shift); }
    __device__ __forceinline__ uint32_t last(int b) const { return b == TK_BUCKETS - 1 ? 0xffffffffu : first(b) + ((1u << shift) - 1u); }
};

template <class Sh>
__device__ __forceinline__ void clear_hist(Sh& sh) {
    reinterpret_cast<int4*>(sh.hist)[threadIdx.x] = make_int4(0, 0, 0, 0);
}

// The bucket that holds the `need`-th key from the top: sh.sel_bucket, the keys above it (sel_above) and in it (sel_count).
// c: this thread's four buckets, 4 * (511 - tid) .. + 3.  Returns the number of keys in all buckets.  Two barriers.
template <class Sh>
__device__ __forceinline__ int find_bucket(const int4& c, int need, Sh& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int mine = c.x + c.y + c.z + c.w;
    int incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) sh.scan[warp] = incl;
    __syncthreads();
    const int w = lane < TK_WARPS ? sh.scan[lane] : 0;
    int above = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0) + incl - mine;
    const int total = __reduce_add_sync(0xffffffffu, w);
    if (above < need && need <= above + mine) {
        const int b[4] = {c.w, c.z, c.y, c.x};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (above < need && need <= above + b[j]) { sh.sel_bucket = TK_BUCKETS - 1 - (4 * tid + j); sh.sel_above = above; sh.sel_count = b[j]; }
            above += b[j];
        }
    }
    __syncthreads();
    return total;
}
template <class Sh>
__device__ __forceinline__ int4 own_buckets(const Sh& sh) { return reinterpret_cast<const int4*>(sh.hist)[TK_THREADS - 1 - threadIdx.x]; }

// Streaming threshold out of a sample of which every thread holds N keys: the lower edge of the bucket that holds the sample's
// r-th key, once that bucket holds no more than `slack` keys; a fuller one is split further, up to a width of one key.  `hi` receives
// the largest sample key, sh.crowd (after a barrier) zero or, where the threshold is one value of which there are more than `slack`, the
// number of sample keys from it on.
template <int N, class Sh>
__device__ __forceinline__ uint32_t sample_threshold(const uint32_t (&key)[N], int r, int slack, uint32_t& hi, Sh& sh) {
    uint32_t lo = key[0];
    hi = key[0];
#pragma unroll
    for (int j = 1; j < N; ++j) { lo = min(lo, key[j]); hi = max(hi, key[j]); }
    clear_hist(sh);
    block_key_range(lo, hi, sh);
    uint32_t top = hi;
    int above = 0;
    for (;;) {
        const BucketMap map(lo, top);
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (key[j] >= lo && key[j] <= top) atomicAdd(&sh.hist[map(key[j])], 1);
        __syncthreads();
        find_bucket(own_buckets(sh), r - above, sh);
        const int b = sh.sel_bucket, count = sh.sel_count;
        above += sh.sel_above;
        if (count <= slack || map.shift == 0) {
            if (threadIdx.x == 0) sh.crowd = count <= slack ? 0 : above + count;
            return map.first(b);
        }
        if (b < TK_BUCKETS - 1) top = min(top, map.last(b));
        lo = map.first(b);
        clear_hist(sh);
        __syncthreads();
    }
}

// One pass over n candidates once the k-th key's bucket [b_lo, b_hi] is known: keys above it leave for out[at .. ), the keys in
// it to small(key, index).  sh.out_pos is zero on entry.
template <class Src, class Sh, class Small>
__device__ __forceinline__ void emit_above(const Src& src, uint32_t b_lo, uint32_t b_hi, int32_t* __restrict__ out, int at, Sh& sh, Small&& small) {
    const int n = src.size(), lane = threadIdx.x & 31;
    for (int i0 = threadIdx.x - lane; i0 < n; i0 += TK_THREADS) {
        const int i = i0 + lane;
        const uint32_t key = i < n ? src.key_at(i) : 0u;
        const bool above = i < n && key > b_hi, in = i < n && key >= b_lo && key <= b_hi;
        const uint32_t m = __ballot_sync(0xffffffffu, above);
        if (m != 0u) {
            int base = 0;
            if (lane == 0) base = atomicAdd(&sh.out_pos, __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (above) out[at + base + __popc(m & ((1u << lane) - 1u))] = src.idx_at(i);
        }
        if (in) small(key, src.idx_at(i));
    }
}

// The `need` largest of the m keys in the small list go to out[0 .. need); the last of them is the row's k-th value.
template <class Sh>
__device__ __forceinline__ void emit_small(int m, int need, int32_t* __restrict__ out, float* __restrict__ kth, Sh& sh) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < m; i += TK_WARPS) {        // a warp per key, its lanes striding over the others
        const uint32_t mine = sh.small_key[i];
        int rank = 0;
        for (int j = lane; j < m; j += 32) {
            const uint32_t other = sh.small_key[j];
            rank += (other > mine || (other == mine && j < i)) ? 1 : 0;
        }
        rank = __reduce_add_sync(0xffffffffu, rank);
        if (lane == 0 && rank < need) {
            out[rank] = sh.small_idx[i];
            if (rank == need - 1 && kth != nullptr) *kth = key_to_float(mine);
        }
    }
}

// Top k of the n >= k candidates of `src`, counted into sh.hist with `map` (complete, barrier passed).
template <class Src, class Sh>
__device__ __forceinline__ void select_and_emit(const Src& src, const BucketMap& map, int k, int32_t* __restrict__ out, float* __restrict__ kth, Sh& sh) {
    if (threadIdx.x == 0) { sh.out_pos = 0; sh.n_small = 0; sh.eq_taken = 0; }
    find_bucket(own_buckets(sh), k, sh);
    const int b = sh.sel_bucket, above = sh.sel_above, count = sh.sel_count;
    if (count <= TK_DIRECT) {
        emit_above(src, map.first(b), map.last(b), out, 0, sh, [&](uint32_t key, int32_t i) {
            const int s = atomicAdd(&sh.n_small, 1);
            if (s < TK_DIRECT) { sh.small_key[s] = key; sh.small_idx[s] = i; }
        });
        __syncthreads();
        emit_small(count, k - above, out + above, kth, sh);
    } else {
        int n_eq;
        const uint32_t T = select_kth(src, k, sh, &n_eq);
        emit_selection(src, T, n_eq, out, sh);
        if (threadIdx.x == 0 && kth != nullptr) *kth = key_to_float(T);
    }
}

// The sixteen elements a thread holds after four 16-byte loads (x[u] = elements e0 + u * e_step .. + 3): those at or above the
// streaming threshold become candidates (value bits and position).  The thread counts them, reserves that many slots with one
// atomic and writes them: one element in thirty passes, so an atomic per element (even aggregated over the warp) costs several
// times the instructions of the comparison itself and made the streaming pass issue-bound rather than memory-bound; for the
// same reason keys and buckets are made of the candidates afterwards.  A list that is full stays incomplete (n_cand tells).
// The float comparison admits a superset of the exact key comparison (it treats -0 and +0 alike).
template <class Sh>
__device__ __forceinline__ void keep_candidates16(const float4 (&x)[4], int e0, int e_step, float thr_f, Sh& sh) {
    int c = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
        c += (x[u].x >= thr_f ? 1 : 0) + (x[u].y >= thr_f ? 1 : 0) + (x[u].z >= thr_f ? 1 : 0) + (x[u].w >= thr_f ? 1 : 0);
    if (c == 0) return;
    const int o = atomicAdd(&sh.n_cand, c);
    if (o + c > Sh::kCap) return;
    uint32_t* slot = sh.cand_key + o;
    auto put = [&](float v, int e) {
        if (v >= thr_f) {
            slot[0] = __float_as_uint(v);
            slot[Sh::kCap] = static_cast<uint32_t>(e);      // cand_idx
            ++slot;
        }
    };
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * e_step;
        put(x[u].x, e); put(x[u].y, e + 1); put(x[u].z, e + 2); put(x[u].w, e + 3);
    }
}

// After the streaming pass (barrier passed): candidates become keys and are counted into their buckets (sh.hist is zero).
template <class Sh>
__device__ __forceinline__ void count_candidates(int n, const BucketMap& map, Sh& sh) {
    for (int i = threadIdx.x; i < n; i += TK_THREADS) {
        const uint32_t key = max(float_to_key(__uint_as_float(sh.cand_key[i])), map.lo);      // -0 at a threshold of +0: the same value
        sh.cand_key[i] = key;
        atomicAdd(&sh.hist[map(key)], 1);
    }
}

__device__ __forceinline__ void topk_prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// First float of the 8-float group that thread i samples of a row of n elements.
__device__ __forceinline__ int64_t sample_offset(int n) {
    return 8 * ((static_cast<int64_t>(threadIdx.x) * ((n >> 3) - 1)) / (TK_THREADS - 1));
}

// Streaming threshold of a row as an order-preserving key: the sample value of a rank a few standard deviations below where the
// row's k-th value is expected.  Thread i reads 8 consecutive floats at an evenly spread, 32-byte aligned offset.  Every
// thread of the CTA calls it; the result is uniform and depends on the row only.  False: no threshold is low enough.
template <class Sh>
__device__ __forceinline__ bool topk_sample(const float* row, int n, int k, uint32_t& thr, uint32_t& hi, Sh& sh) {
    const float expect = static_cast<float>(TK_SAMPLE) * static_cast<float>(k) / static_cast<float>(n);
    const int r = static_cast<int>(expect + 4.0f * sqrtf(expect) + 8.0f);
    if (r >= TK_SAMPLE) return false;
    const float4* src = reinterpret_cast<const float4*>(row + sample_offset(n));
    const float4 a = __ldcg(src), b = __ldcg(src + 1);
    const uint32_t key[8] = {float_to_key(a.x), float_to_key(a.y), float_to_key(a.z), float_to_key(a.w),
                             float_to_key(b.x), float_to_key(b.y), float_to_key(b.z), float_to_key(b.w)};
    thr = sample_threshold(key, r, 4 + r / 16, hi, sh);
    return true;
}

// Four 16-byte groups of a thread: i, i + TK_THREADS, ..; past the end NaN, which no threshold lets in.
__device__ __forceinline__ void load_groups(const float4* row4, int i, int f4_end, float4 (&x)[4]) {
    if (i + 3 * TK_THREADS < f4_end) {
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = __ldcs(row4 + i + u * TK_THREADS);
    } else {
        const float nan = __int_as_float(0x7fffffff);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            x[u] = make_float4(nan, nan, nan, nan);
            if (i + u * TK_THREADS < f4_end) x[u] = __ldcs(row4 + i + u * TK_THREADS);
        }
    }
}

// One streaming pass over the 16-byte groups [f4_begin, f4_end) of the row (and, with `tail`, the n % 4 elements after the
// last whole group).
template <class Sh>
__device__ __forceinline__ void topk_stream(const float* row, int n, int f4_begin, int f4_end, bool tail, float thr_f, Sh& sh) {
    const int tid = threadIdx.x;
    const float4* row4 = reinterpret_cast<const float4*>(row);
    int i = f4_begin + tid;
    for (; i + 3 * TK_THREADS < f4_end; i += 4 * TK_THREADS) {
        float4 x[4];                              // 16-byte loads in flight per thread
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = __ldcs(row4 + i + u * TK_THREADS);
        keep_candidates16(x, 4 * i, 4 * TK_THREADS, thr_f, sh);
    }
    if (i < f4_end) {
        float4 x[4];
        load_groups(row4, i, f4_end, x);
        keep_candidates16(x, 4 * i, 4 * TK_THREADS, thr_f, sh);
    }
    const int n4 = n >> 2;
    if (tail && tid < n - 4 * n4) {
        const float v = __ldcg(row + 4 * n4 + tid);
        if (v >= thr_f) {
            const int o = atomicAdd(&sh.n_cand, 1);
            if (o < Sh::kCap) { sh.cand_key[o] = __float_as_uint(v); sh.cand_idx[o] = 4 * n4 + tid; }
        }
    }
}

// A row of at most k elements: all of them, and the smallest value.
template <class Sh>
__device__ __noinline__ void topk_whole_row(const float* row, int n, int k, int32_t* __restrict__ out, int32_t* __restrict__ count,
                               float* __restrict__ kth, Sh& sh) {
    const int tid = threadIdx.x;
    for (int i = tid; i < k; i += TK_THREADS) out[i] = i < n ? i : -1;
    if (count != nullptr && tid == 0) *count = n;
    if (kth != nullptr) {
        uint32_t lo = 0xffffffffu, hi = 0u;
        for (int i = tid; i < n; i += TK_THREADS) lo = min(lo, float_to_key(__ldcg(row + i)));
        block_key_range(lo, hi, sh);
        if (tid == 0) *kth = n > 0 ? key_to_float(lo) : __int_as_float(0xff800000);
        __syncthreads();
    }
}

// The exact selection over the row in global memory.
template <class Sh>
__device__ __noinline__ void topk_exact_row(const float* row, int n, int k, int32_t* __restrict__ out, float* __restrict__ kth, Sh& sh) {
    if (threadIdx.x == 0) { sh.out_pos = 0; sh.eq_taken = 0; }
    int n_eq;
    GlobalSource s{row, n};
    const uint32_t T = select_kth(s, k, sh, &n_eq);
    emit_selection(s, T, n_eq, out, sh);
    if (threadIdx.x == 0 && kth != nullptr) *kth = key_to_float(T);
}

// Positions of `need` elements of the row that equal t to out[0 .. need), whichever come first.  sh.n_small, zero on entry, counts those
// found; at the end it is below `need` if the row has no more.
template <class Sh>
__device__ __noinline__ void topk_copies(const float* row, int n, float t, int need, int32_t* __restrict__ out, Sh& sh) {
    const float nan = __int_as_float(0x7fffffff);
    const int n4 = n >> 2;
    for (int i = threadIdx.x; i <= n4 && *reinterpret_cast<volatile int*>(&sh.n_small) < need; i += TK_THREADS) {
        float4 x = make_float4(nan, nan, nan, nan);
        if (i < n4) {
            x = __ldcg(reinterpret_cast<const float4*>(row) + i);
        } else {                                   // the n % 4 elements after the last whole group
            if (4 * n4 < n) x.x = __ldcg(row + 4 * n4);
            if (4 * n4 + 1 < n) x.y = __ldcg(row + 4 * n4 + 1);
            if (4 * n4 + 2 < n) x.z = __ldcg(row + 4 * n4 + 2);
        }
        const int c = (x.x == t ? 1 : 0) + (x.y == t ? 1 : 0) + (x.z == t ? 1 : 0) + (x.w == t ? 1 : 0);
        if (c == 0) continue;
        int o = atomicAdd(&sh.n_small, c);
        auto put = [&](float v, int e) {
            if (v == t && o < need) out[o++] = e;
        };
        put(x.x, 4 * i); put(x.y, 4 * i + 1); put(x.z, 4 * i + 2); put(x.w, 4 * i + 3);
    }
}

// Top-k of one fp32 row of n elements (16-byte aligned) by the whole CTA (TK_THREADS threads): out[0..k) receives the
// indices (-1 padded), *count / *kth the number selected and the smallest selected value (either may be NULL).
// `next_row` (may be NULL): the row this CTA takes next.  The sample sectors of that row are requested into L2 once this
// row's streaming pass is over, so the next sample does not start with a DRAM round trip.  (Requesting the head of the next
// row as well, 96 to 512 KB, made the kernel slower: 0.49 -> 0.50 .. 0.58 ms at 4096 rows of 135168.)
// COPIES: a threshold that is one value with more copies than the list holds (scores cut off at zero, coarse ones) is met by a list of what
// lies above it; if that is less than k, copies are looked for afterwards, as many as are missing.  For the small lists: 4000 rows of 8000,
// k = 512, of which 7 % above zero 105 us, 270 when the list overflows and the row is selected from global memory, 148 with the row in
// shared memory.  The larger ones seldom overflow, and the few instructions cost them 1 to 3 %.
template <bool COPIES = false, class Sh>
__device__ __forceinline__ void topk_row(const float* row, int n, int k, int32_t* __restrict__ out, int32_t* __restrict__ count,
                         float* __restrict__ kth, Sh& sh, const float* next_row = nullptr, int next_n = 0) {
    const int tid = threadIdx.x;
    if (n <= k) {
        topk_whole_row(row, n, k, out, count, kth, sh);
        return;
    }
    if (count != nullptr && tid == 0) *count = k;
    if (n <= Sh::kCap) {                           // the whole row is the candidate list
        uint32_t lo = 0xffffffffu, hi = 0u;
        auto take = [&](float v, int i) {
            const uint32_t key = float_to_key(v);
            sh.cand_key[i] = key;
            lo = min(lo, key);
            hi = max(hi, key);
        };
        const float4* row4 = reinterpret_cast<const float4*>(row);
        for (int i = tid; i < (n >> 2); i += TK_THREADS) {
            const float4 x = __ldcs(row4 + i);
            take(x.x, 4 * i); take(x.y, 4 * i + 1); take(x.z, 4 * i + 2); take(x.w, 4 * i + 3);
        }
        if (tid < (n & 3)) take(__ldcg(row + (n & ~3) + tid), (n & ~3) + tid);
        clear_hist(sh);
        block_key_range(lo, hi, sh);
        const BucketMap map(lo, hi);
        for (int i = tid; i < n; i += TK_THREADS) atomicAdd(&sh.hist[map(sh.cand_key[i])], 1);
        __syncthreads();
        select_and_emit(SmemSource{sh.cand_key, nullptr, n}, map, k, out, kth, sh);
        return;
    }
    uint32_t thr, hi;
    if (tid == 0) { sh.n_cand = 0; sh.n_small = 0; }
    const bool sampled = topk_sample(row, n, k, thr, hi, sh);
    if (sampled) {
        clear_hist(sh);
        __syncthreads();
        auto tied = [&]() { return COPIES && static_cast<int64_t>(sh.crowd) * n > static_cast<int64_t>(Sh::kCap) * (TK_SAMPLE - TK_SAMPLE / 8); };
        if (tied()) thr += thr == float_to_key(-0.f) ? 2u : 1u;      // (-0 and +0 are the same value)
        const BucketMap map(thr, max(thr, hi));
        topk_stream(row, n, 0, n >> 2, true, key_to_float(thr), sh);
        if (next_row != nullptr && next_n > Sh::kCap) topk_prefetch_l2(next_row + sample_offset(next_n));
        __syncthreads();
        const int n_cand = sh.n_cand;
        if (n_cand >= k && n_cand <= Sh::kCap) {
            count_candidates(n_cand, map, sh);
            __syncthreads();
            select_and_emit(SmemSource{sh.cand_key, sh.cand_idx, n_cand}, map, k, out, kth, sh);
            return;
        }
        if (n_cand < k && n_cand <= Sh::kCap && tied()) {
            const float t = key_to_float(thr - 1u);
            topk_copies(row, n, t, k - n_cand, out + n_cand, sh);
            __syncthreads();
            if (sh.n_small >= k - n_cand) {
                for (int i = tid; i < n_cand; i += TK_THREADS) out[i] = sh.cand_idx[i];
                if (tid == 0 && kth != nullptr) *kth = t;
                return;
            }
        }
    }
    __syncthreads();
    topk_exact_row(row, n, k, out, kth, sh);       // the sample misjudged the row
}

// The same by a cluster of CTAs (few rows): each CTA samples alike, streams its share of the row into its own candidates and
// histogram, the histograms are added through distributed shared memory, every CTA emits its own keys above the k-th key's
// bucket, and CTA 0 ranks the bucket's keys of all of them.  CTA 0 takes a short row alone.
template <class Sh>
__device__ __forceinline__ void topk_row_cluster(const float* row, int n, int k, int32_t* __restrict__ out, int32_t* __restrict__ count,
                                 float* __restrict__ kth, Sh& sh) {
    using namespace ptx;
    const int tid = threadIdx.x, lane = tid & 31;
    const int rank = static_cast<int>(cluster_ctarank()), n_cta = static_cast<int>(cluster_nctarank());
    uint32_t thr = 0u, hi = 0u;
    if (tid == 0) { sh.n_cand = 0; sh.out_pos = 0; sh.n_small = 0; sh.sel_out = 0; }
    // the first of this CTA's share is on its way while the sample is worked on
    const int64_t n4 = n >> 2;
    const int f4_begin = static_cast<int>(n4 * rank / n_cta), f4_end = static_cast<int>(n4 * (rank + 1) / n_cta);
    float4 x[4];
    bool split = n >= topk_split_from(n_cta) && n > k;      // the same answer in every CTA
    if (split) {
        load_groups(reinterpret_cast<const float4*>(row), f4_begin + tid, f4_end, x);
        split = topk_sample(row, n, k, thr, hi, sh);
    }
    if (!split) {
        if (rank == 0) topk_row(row, n, k, out, count, kth, sh);
        return;
    }
    const BucketMap map(thr, max(thr, hi));
    clear_hist(sh);
    __syncthreads();
    keep_candidates16(x, 4 * (f4_begin + tid), 4 * TK_THREADS, key_to_float(thr), sh);
    topk_stream(row, n, f4_begin + 4 * TK_THREADS, f4_end, rank == n_cta - 1, key_to_float(thr), sh);
    __syncthreads();
    count_candidates(min(sh.n_cand, Sh::kCap), map, sh);
    __syncthreads();
    static_assert(Sh::kCap < 0x8000, "a bucket's count and the flag share 16 bits");
    // The counts travel as 16 bits each, four buckets in 8 bytes where the histogram was (its bytes are what the exchange takes); bit 15 of
    // the lowest bucket says that the list was full.
    const int4 own = own_buckets(sh);
    __syncthreads();
    const uint32_t full = tid == TK_THREADS - 1 && sh.n_cand > Sh::kCap ? 0x8000u : 0u;
    reinterpret_cast<uint2*>(sh.hist)[TK_THREADS - 1 - tid] = make_uint2(static_cast<uint32_t>(own.x) | full | static_cast<uint32_t>(own.y) << 16,
                                                                         static_cast<uint32_t>(own.z) | static_cast<uint32_t>(own.w) << 16);
    cluster_sync_all();                            // every CTA's candidates and counts
    // remote loads of all CTAs are issued together: one after the other each would cost the round trip
    int4 c = make_int4(0, 0, 0, 0);
    {
        const uint32_t my_buckets = smem_u32(sh.hist) + 8u * (TK_THREADS - 1 - tid);
        uint64_t v[TK_MAX_CLUSTER];
#pragma unroll
        for (int r = 0; r < TK_MAX_CLUSTER; ++r) v[r] = ld_cluster_u64(mapa_shared(my_buckets, min(r, n_cta - 1)));
#pragma unroll
        for (int r = 0; r < TK_MAX_CLUSTER; ++r) {
            if (r >= n_cta) continue;
            const uint32_t lo = static_cast<uint32_t>(v[r]), up = static_cast<uint32_t>(v[r] >> 32);
            c.x += static_cast<int>(lo & 0x7fffu) + ((lo & 0x8000u) != 0u ? TK_FULL : 0);
            c.y += static_cast<int>(lo >> 16);
            c.z += static_cast<int>(up & 0xffffu);
            c.w += static_cast<int>(up >> 16);
        }
    }
    const int total = find_bucket(c, k, sh);
    const int b = sh.sel_bucket, above = sh.sel_above, in = sh.sel_count;
    if (total >= TK_FULL || total < k || in > TK_DIRECT) {    // uniform over the cluster: everybody read the same counts
        cluster_sync_all();                        // which may change only now
        if (rank == 0) {
            if (count != nullptr && tid == 0) *count = k;
            topk_exact_row(row, n, k, out, kth, sh);
        }
        return;
    }
    // this CTA's keys above the bucket, and where they go: one reservation in CTA 0
    const int first = TK_BUCKETS - 4 - 4 * tid;
    int mine = (first > b ? own.x : 0) + (first + 1 > b ? own.y : 0) + (first + 2 > b ? own.z : 0) + (first + 3 > b ? own.w : 0);
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) sh.warp_lo[tid >> 5] = static_cast<uint32_t>(mine);
    __syncthreads();
    if (tid < 32) {
        const int n_above = __reduce_add_sync(0xffffffffu, lane < TK_WARPS ? static_cast<int>(sh.warp_lo[lane]) : 0);
        if (lane == 0) sh.eq_taken = atomic_add_cluster_s32(mapa_shared(smem_u32(&sh.sel_out), 0), n_above);
    }
    __syncthreads();
    // the keys inside the bucket (a handful) go straight to CTA 0's small list
    const uint32_t n_small0 = mapa_shared(smem_u32(&sh.n_small), 0), key0 = mapa_shared(smem_u32(sh.small_key), 0), idx0 = mapa_shared(smem_u32(sh.small_idx), 0);
    emit_above(SmemSource{sh.cand_key, sh.cand_idx, sh.n_cand}, map.first(b), map.last(b), out, sh.eq_taken, sh, [&](uint32_t key, int32_t i) {
        const int s = atomic_add_cluster_s32(n_small0, 1);
        if (s < TK_DIRECT) { st_cluster_u32(key0 + 4 * s, key); st_cluster_u32(idx0 + 4 * s, static_cast<uint32_t>(i)); }
    });
    cluster_sync_all();                            // CTA 0 has the list; nobody is read any more
    if (rank == 0) {
        emit_small(in, k - above, out + above, kth, sh);
        if (count != nullptr && tid == 0) *count = k;
    }
}

}  // namespace janus
