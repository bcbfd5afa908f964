// janus_page_demand: union of selected tokens -> physical page bitmap, ascending page list,
// maximal runs of adjacent physical pages, and the miss set "exact minus predicted"
// (union of selections: Sec. 2.2; corrective reads: Sec. 4.2; read packing: Sec. 4.3).
//
// Latency bounds all of it: a few hundred kilobytes in, a few kilobytes out, but several dependent steps.  Up to 128 K
// indices one launch of one cluster does everything (page_demand_kernel): every CTA marks its share of the indices in a private
// bitmap in shared memory, the cluster ORs the bitmaps slice by slice through distributed shared memory, and each CTA
// turns its slice of the set into its part of the lists, offsets coming from one exchange of the CTAs' counts (page_demand_few_kernel: a
// small pool's lists come from one CTA, without the exchange).  Larger blocks of
// indices are marked by the whole chip first (page_mark_kernel, one bitmap of *logical* pages per CTA, so that an index costs
// one shared-memory test and the page table is read once per page and CTA), and the same kernel then only makes the lists, for large pools
// in several clusters.  Which of them, and how many CTAs: page_demand_plan.h.
#include <algorithm>

#include "janus_common.cuh"
#include "page_demand_plan.h"
#include "sm100_ptx.cuh"

namespace janus {

using namespace ptx;

constexpr int MARK_THREADS = 1024;
constexpr int MARK_SMEM_WORDS = 24576;             // bitmaps of logical and physical pages of a marking CTA together: 96 KB, two CTAs per SM

enum { PD_LISTS = 0, PD_MARK = 1, PD_MARK_ROWS = 2 };      // what page_demand_kernel does before the lists

struct PdParams {
    const int32_t* idx;
    int64_t n_idx;
    int k;
    int64_t demand_limit;                 // PD_MARK
    const int64_t* demand_limits;         // PD_MARK_ROWS: per row
    int page_size, page_shift;
    const int32_t* page_table;
    int64_t n_logical_pages;              // PD_MARK
    const int64_t* table_offsets;         // PD_MARK_ROWS: row r uses page_table[table_offsets[r] .. table_offsets[r + 1])
    int64_t n_phys_pages;
    int n_words;
    const uint32_t* predicted;            // may be NULL
    uint32_t* bitmap;
    int32_t *pages, *n_pages, *runs, *n_runs, *miss_pages, *n_miss, *miss_runs, *n_miss_runs;
    int64_t capacity;
    int32_t* dev_status;
};

struct PageDiv {      // token -> logical page
    int size, shift;
    __device__ __forceinline__ int64_t operator()(int s) const { return shift >= 0 ? (s >> shift) : (s / size); }
};

// Sets bit p of a bitmap in shared memory; tested first, because most pages are already there.
__device__ __forceinline__ void set_bit_shared(uint32_t* bm, int p) {
    const uint32_t bit = 1u << (p & 31);
    uint32_t* w = bm + (p >> 5);
    if ((*reinterpret_cast<volatile uint32_t*>(w) & bit) == 0u) atomicOr(w, bit);
}

// Empties the global bitmap before it is marked.  A kernel and not a memset: it and the marking start while their predecessors run
// (777 x 2048 indices of 658 pages, whole call: 12.4 us with a memset, 8.9 with this; 4096 x 2048 of 2112 pages 22.7 and 20.3).
__global__ void __launch_bounds__(256)
page_clear_kernel(uint32_t* bitmap, int n_words) {
    grid_launch_next();
    grid_wait();
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n_words; i += gridDim.x * 256) bitmap[i] = 0u;
}

// ---- marking by the whole chip ----------------------------------------------------------------------------------------------
// A CTA's tokens become bits of its own bitmap of logical pages; at the end its set pages go through the page table into a
// bitmap of physical pages, whose words are ORed into the global one (page by page they would be a contended atomic each:
// 109 us).
// Whole call at 4096 x 2048 indices, in a loop: 35 us when every index went through the page table, 24.7 now (32 inside a step, whose
// other calls leave nothing of the indices in L2); 8192 x 2048: 65.8 and 35.7.
__global__ void __launch_bounds__(MARK_THREADS)
page_mark_kernel(const PdParams p, int n_log_words) {
    extern __shared__ uint32_t lbm[];
    uint32_t* pbm = lbm + n_log_words;
    grid_launch_next();
    for (int i = threadIdx.x; i < n_log_words + p.n_words; i += MARK_THREADS) lbm[i] = 0u;
    grid_wait();
    __syncthreads();
    const PageDiv page{p.page_size, p.page_shift};
    bool bad = false;
    // four tokens at a time: their words are read together, and a bit is set only where it is not there yet
    auto mark4 = [&](const int4& v) {
        const int s[4] = {v.x, v.y, v.z, v.w};
        int lp[4];
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            lp[e] = -1;
            if (s[e] >= 0 && s[e] < p.demand_limit) {
                const int64_t l = page(s[e]);
                if (l >= p.n_logical_pages) bad = true;
                else lp[e] = static_cast<int>(l);
            }
            w[e] = lp[e] >= 0 ? lbm[lp[e] >> 5] : 0xffffffffu;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (((w[e] >> (lp[e] & 31)) & 1u) == 0u) atomicOr(lbm + (lp[e] >> 5), 1u << (lp[e] & 31));
    };
    const int4* idx4 = reinterpret_cast<const int4*>(p.idx);      // 16-byte aligned
    const int64_t n_vec = p.n_idx >> 2, stride = static_cast<int64_t>(gridDim.x) * MARK_THREADS;
    int64_t i = static_cast<int64_t>(blockIdx.x) * MARK_THREADS + threadIdx.x;
    for (; i + 3 * stride < n_vec; i += 4 * stride) {
        int4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = ld_input(idx4 + i + u * stride);
#pragma unroll
        for (int u = 0; u < 4; ++u) mark4(v[u]);
    }
    for (; i < n_vec; i += stride) mark4(ld_input(idx4 + i));
    if (blockIdx.x == 0 && threadIdx.x < (p.n_idx & 3)) mark4(make_int4(p.idx[(n_vec << 2) + threadIdx.x], -1, -1, -1));
    __syncthreads();
    for (int lp = threadIdx.x; lp < n_log_words * 32; lp += MARK_THREADS) {
        if (((lbm[lp >> 5] >> (lp & 31)) & 1u) == 0u) continue;
        const int32_t q = ld_input(p.page_table + lp);
        if (q < 0 || q >= p.n_phys_pages) bad = true;
        else atomicOr(pbm + (q >> 5), 1u << (q & 31));
    }
    __syncthreads();
    for (int w = threadIdx.x; w < p.n_words; w += MARK_THREADS) {
        const uint32_t v = pbm[w];
        if (v != 0u && (__ldcg(p.bitmap + w) & v) != v) atomicOr(p.bitmap + w, v);
    }
    if (bad) report(p.dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);
}

// Physical page of a token, -1 for none (padding, past the limit) and after reporting what is out of range.
__device__ __forceinline__ int32_t page_of_token(int s, int64_t limit, const PageDiv& page, const int32_t* table, int64_t n_logical,
                                                 int64_t n_phys, bool& bad) {
    if (s < 0 || s >= limit) return -1;
    const int64_t lp = page(s);
    const int32_t q = lp < n_logical ? ld_input(table + lp) : -1;
    if (q < 0 || q >= n_phys) { bad = true; return -1; }
    return q;
}

// Tables or pools whose bitmaps do not fit shared memory: straight into the global bitmap.
template <int MODE>
__global__ void __launch_bounds__(256)
page_mark_global_kernel(const PdParams p) {
    grid_launch_next();
    grid_wait();
    const PageDiv page{p.page_size, p.page_shift};
    bool bad = false;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; e < p.n_idx; e += static_cast<int64_t>(gridDim.x) * 256) {
        const int32_t* table = p.page_table;
        int64_t n_log = p.n_logical_pages, limit = p.demand_limit;
        if (MODE == PD_MARK_ROWS) {
            const int64_t r = e / p.k, off = ld_input(p.table_offsets + r);
            n_log = off < 0 ? 0 : ld_input(p.table_offsets + r + 1) - off;       // a table that starts before the array has no pages
            table += off < 0 ? 0 : off;
            limit = ld_input(p.demand_limits + r);
        }
        const int32_t q = page_of_token(ld_input(p.idx + e), limit, page, table, n_log, p.n_phys_pages, bad);
        if (q < 0) continue;
        const uint32_t bit = 1u << (q & 31);
        if ((__ldcg(p.bitmap + (q >> 5)) & bit) == 0u) atomicOr(p.bitmap + (q >> 5), bit);
    }
    if (bad) report(p.dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);
}

// ---- one cluster: marking (optional) and the lists -----------------------------------------------------------------------------
// Counts of a set up to some place, both in one 64-bit word so that they are scanned together: ids in the high half, run
// starts in the low half.  The run ends before a word are the starts before it less the run that reaches into it.
struct PdShared {
    uint64_t warp_sums[2][33];
    uint64_t totals[2];                       // this CTA's slice: the set, the miss set
    uint64_t before[2], all[2];               // the slices before it, all slices up to the cluster's end
    // with several clusters: this CTA's share of the counts before the cluster and of the last run start there, and those of all CTAs
    uint64_t earlier[2], upto[2];
    int last_start[2], open_start[2], last_of_warp[2][32];
    uint64_t at[2][PD_THREADS];               // counts before each word of a chunk
    uint32_t word[2][PD_THREADS + 2];         // the words of a chunk and one neighbour on either side
};

__device__ __forceinline__ void block_scan2_u64(uint64_t (&v)[2], uint64_t (*warp_sums)[33], uint64_t (&excl)[2], uint64_t (&total)[2]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t incl[2] = {v[0], v[1]};
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, incl[q], d);
            if (lane >= d) incl[q] += y;
        }
    }
    __syncthreads();                  // warp_sums is free again
    if (lane == 31) { warp_sums[0][warp] = incl[0]; warp_sums[1][warp] = incl[1]; }
    __syncthreads();
    if (warp < 2) {                   // warp q scans the 32 warp totals of value q
        const uint64_t sv = warp_sums[warp][lane];
        uint64_t si = sv;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, si, d);
            if (lane >= d) si += y;
        }
        warp_sums[warp][lane] = si - sv;
        if (lane == 31) warp_sums[warp][32] = si;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        total[q] = warp_sums[q][32];
        excl[q] = warp_sums[q][warp] + incl[q] - v[q];
    }
}

// Marks the pages of CTA `rank`'s share of the indices in its bitmap in shared memory.  False: something was out of range.
template <int MODE>
__device__ __forceinline__ bool mark_share(const PdParams& p, uint32_t* bm, int rank, int n_cta) {
    const int tid = threadIdx.x;
    const PageDiv page{p.page_size, p.page_shift};
    bool bad = false;
    // Eight indices per thread at a time, in rounds of loads that are all in flight together: indices and their rows' table and
    // limit, then page table entries (one index after the other: 24.2 us instead of 21.9 for 64 decode rows of 2048, when the rest took 5 us longer)
    constexpr int U = 8;
    const int stride = n_cta * PD_THREADS, n_idx = static_cast<int>(p.n_idx);
    for (int base = rank * PD_THREADS + tid; base < n_idx; base += U * stride) {
        int s[U];
        int32_t q[U];
        const int32_t* entry[U];
#pragma unroll
        for (int u = 0; u < U; ++u) s[u] = base + u * stride < n_idx ? ld_input(p.idx + base + u * stride) : -1;
        if constexpr (MODE == PD_MARK_ROWS) {
            int64_t off[U], end[U], limit[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                off[u] = end[u] = limit[u] = 0;
                if (base + u * stride >= n_idx) continue;
                const int r = (base + u * stride) / p.k;
                off[u] = ld_input(p.table_offsets + r);
                end[u] = ld_input(p.table_offsets + r + 1);
                limit[u] = ld_input(p.demand_limits + r);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                entry[u] = nullptr;
                if (s[u] >= 0 && s[u] < limit[u]) {       // a table that starts before the array has no pages
                    const int64_t lp = page(s[u]);
                    if (off[u] >= 0 && lp < end[u] - off[u]) entry[u] = p.page_table + off[u] + lp;
                    else bad = true;
                }
            }
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                entry[u] = nullptr;
                if (s[u] >= 0 && s[u] < p.demand_limit) {
                    const int64_t lp = page(s[u]);
                    if (lp < p.n_logical_pages) entry[u] = p.page_table + lp;
                    else bad = true;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = entry[u] != nullptr ? ld_input(entry[u]) : -1;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (entry[u] == nullptr) continue;
            if (q[u] < 0 || q[u] >= p.n_phys_pages) bad = true;
            else set_bit_shared(bm, q[u]);
        }
    }
    return !bad;
}

// ---- one cluster, a pool of few words --------------------------------------------------------------------------------------------
// The sets of all CTAs are ORed into CTA 0's shared memory, which then makes the lists alone (PD_LISTS: there is one CTA, and the set is
// in global memory): a thread has a word, counts are 16 bits each, runs are put together in shared memory.  One cluster-wide barrier on the
// way instead of four, and no exchange of counts: 7-8 -> 5 us.
constexpr int PD_FEW_RUNS = PD_FEW_WORDS * 16;
struct PdFewShared {
    uint32_t own[PD_FEW_WORDS];
    uint32_t word[2][PD_FEW_WORDS + 2];       // CTA 0: the set, the miss set, with an empty word on either side
    uint32_t at[2][PD_FEW_WORDS];             // ids before a word << 16 | run starts before it
    uint32_t warp_sum[2][PD_FEW_WORDS / 32];
    uint16_t start[2][PD_FEW_RUNS], end[2][PD_FEW_RUNS];
};
static_assert(PD_FEW_WORDS * 32 <= 0xffff && PD_FEW_WORDS <= PD_THREADS, "counts and pages of 16 bits");

template <int MODE>
__global__ void __launch_bounds__(PD_THREADS)
page_demand_few_kernel(const PdParams p) {
    __shared__ PdFewShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = MODE == PD_LISTS ? 0 : static_cast<int>(cluster_ctarank());
    const bool want_miss = p.miss_pages != nullptr;
    grid_launch_next();
    if (tid < PD_FEW_WORDS) sh.own[tid] = 0u;
    if (tid < PD_FEW_WORDS + 2) sh.word[0][tid] = sh.word[1][tid] = 0u;
    if constexpr (MODE != PD_LISTS) cluster_arrive_release();             // (CTA 0's set is empty; waited for before it is written to)
    grid_wait();
    uint32_t predicted = 0u;              // on its way while the indices are marked
    if (rank == 0 && tid < p.n_words && p.predicted != nullptr) predicted = __ldcg(p.predicted + tid);
    __syncthreads();
    if constexpr (MODE == PD_LISTS) {
        if (tid < p.n_words) sh.word[0][tid + 1] = __ldcg(p.bitmap + tid);       // (read back by the same thread)
    } else {
        if (!mark_share<MODE>(p, sh.own, rank, static_cast<int>(cluster_nctarank()))) report(p.dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);
        __syncthreads();
        cluster_wait();
        if (tid < p.n_words && sh.own[tid] != 0u) red_or_cluster_u32(mapa_shared(smem_u32(&sh.word[0][tid + 1]), 0), sh.own[tid]);
        cluster_sync_all();
        if (rank != 0) return;
    }
    if (tid < PD_FEW_WORDS) {
        const uint32_t v = sh.word[0][tid + 1];
        if (MODE != PD_LISTS && tid < p.n_words) p.bitmap[tid] = v;
        if (want_miss) sh.word[1][tid + 1] = v & ~predicted;
    }
    __syncthreads();
    uint32_t incl[2] = {0u, 0u}, mine[2] = {0u, 0u};
    if (tid < PD_FEW_WORDS) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint32_t v = sh.word[q][tid + 1], starts = v & ~((v << 1) | (sh.word[q][tid] >> 31));
            mine[q] = incl[q] = static_cast<uint32_t>(__popc(v)) << 16 | static_cast<uint32_t>(__popc(starts));
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl[q], d);
                if (lane >= d) incl[q] += y;
            }
            if (lane == 31) sh.warp_sum[q][warp] = incl[q];
        }
    }
    __syncthreads();
    uint32_t total[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const uint32_t x = lane < PD_FEW_WORDS / 32 ? sh.warp_sum[q][lane] : 0u;
        total[q] = __reduce_add_sync(0xffffffffu, x);
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? x : 0u);
        if (tid < PD_FEW_WORDS) sh.at[q][tid] = before + incl[q] - mine[q];
    }
    __syncthreads();
    const int cap = static_cast<int>(min(p.capacity, static_cast<int64_t>(0x7fffffff)));
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll
    for (int q = 0; q < 2; ++q) {         // a warp per word, a lane per page
        if (q == 1 && !want_miss) break;
        int32_t* ids = q ? p.miss_pages : p.pages;
        for (int j = warp; j < p.n_words; j += PD_THREADS / 32) {
            const uint32_t w = sh.word[q][j + 1];
            if (((w >> lane) & 1u) == 0u) continue;
            const uint32_t starts = w & ~((w << 1) | (sh.word[q][j] >> 31)), ends = w & ~((w >> 1) | (sh.word[q][j + 2] << 31));
            const uint32_t o = sh.at[q][j];
            const int o_id = static_cast<int>(o >> 16) + __popc(w & below);
            const int run = static_cast<int>(o & 0xffffu) + __popc(starts & (below | (1u << lane))) - 1;      // the page's run
            const int page = j * 32 + lane;
            if (o_id < cap) ids[o_id] = page;
            if ((starts >> lane) & 1u) sh.start[q][run] = static_cast<uint16_t>(page);
            if ((ends >> lane) & 1u) sh.end[q][run] = static_cast<uint16_t>(page);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (q == 1 && !want_miss) break;
        int32_t* runs = q ? p.miss_runs : p.runs;
        const int n_runs = static_cast<int>(total[q] & 0xffffu), n_ids = static_cast<int>(total[q] >> 16);
        for (int j = tid; j < min(n_runs, cap); j += PD_THREADS) {
            runs[2 * j] = sh.start[q][j];
            runs[2 * j + 1] = sh.end[q][j] - sh.start[q][j] + 1;
        }
        if (tid == 0) {
            *(q ? p.n_miss : p.n_pages) = n_ids;
            *(q ? p.n_miss_runs : p.n_runs) = n_runs;
            if (n_ids > p.capacity || n_runs > p.capacity) report(p.dev_status, JANUS_DEV_CAPACITY_EXCEEDED);
        }
    }
}

template <int MODE>
__global__ void __launch_bounds__(PD_THREADS)
page_demand_kernel(const PdParams p) {
    extern __shared__ uint32_t bm[];      // private bitmap (marking modes)
    __shared__ PdShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = static_cast<int>(cluster_ctarank()), n_cta = static_cast<int>(cluster_nctarank());
    // words of a CTA's slice; at most one chunk of PD_THREADS in the marking modes, which are one cluster
    const int wps = (p.n_words + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
    const int w0 = static_cast<int>(min(static_cast<int64_t>(p.n_words), static_cast<int64_t>(blockIdx.x) * wps)), w1 = min(p.n_words, w0 + wps);
    // the cluster's words [c_begin, c_end)
    const int64_t first_cta = static_cast<int64_t>(blockIdx.x) - rank;
    const int c_begin = MODE == PD_LISTS ? static_cast<int>(min(static_cast<int64_t>(p.n_words), first_cta * wps)) : 0;
    const int c_end = MODE == PD_LISTS ? static_cast<int>(min(static_cast<int64_t>(p.n_words), (first_cta + n_cta) * wps)) : p.n_words;

    grid_launch_next();
    if constexpr (MODE != PD_LISTS) {
        for (int i = tid; i < p.n_words; i += PD_THREADS) bm[i] = 0u;
        grid_wait();
        __syncthreads();
        if (!mark_share<MODE>(p, bm, rank, n_cta)) report(p.dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);
        cluster_sync_all();               // every private bitmap is complete
    }

    if constexpr (MODE == PD_LISTS) grid_wait();
    // ---- lists of this CTA's slice, a chunk of words at a time
    const bool want_miss = p.miss_pages != nullptr;
    // word i of the set: ORed over the CTAs' bitmaps, or as page_mark_kernel left it
    auto union_word = [&](int i) -> uint32_t {
        if (i < 0 || i >= p.n_words) return 0u;
        if constexpr (MODE == PD_LISTS) {
            return __ldcg(p.bitmap + i);
        } else {
            const uint32_t addr = smem_u32(bm + i);
            uint32_t v = 0u;
            for (int r0 = 0; r0 < n_cta; r0 += 4) {      // clusters of 4, 8 or 16; four round trips overlap
                uint32_t x[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) x[r] = ld_cluster_u32(mapa_shared(addr, r0 + r));
                v |= (x[0] | x[1]) | (x[2] | x[3]);
            }
            return v;
        }
    };
    auto load_chunk = [&](int c0) {       // words c0 - 1 .. c0 + PD_THREADS, cut off at the slice's end + 1
        __syncthreads();
        for (int j = tid; j < PD_THREADS + 2; j += PD_THREADS) {
            const int i = c0 - 1 + j;
            const uint32_t v = i <= w1 ? union_word(i) : 0u;
            sh.word[0][j] = v;
            if (want_miss) sh.word[1][j] = v == 0u || p.predicted == nullptr ? v : v & ~__ldcg(p.predicted + i);
            if (MODE != PD_LISTS && i >= w0 && i < w1) p.bitmap[i] = v;
        }
        __syncthreads();
    };
    auto count_chunk = [&](int c0, uint64_t (&mine)[2]) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            mine[q] = 0;
            if (c0 + tid < w1 && (q == 0 || want_miss)) {
                const uint32_t v = sh.word[q][tid + 1];
                mine[q] = static_cast<uint64_t>(__popc(v)) << 32 | static_cast<uint64_t>(__popc(v & ~((v << 1) | (sh.word[q][tid] >> 31))));
            }
        }
    };
    const bool one_chunk = wps <= PD_THREADS;
    uint64_t excl[2] = {0, 0}, sum[2] = {0, 0};
    if (one_chunk) {                      // the scan of the only chunk gives the slice's counts as well
        uint64_t mine[2];
        load_chunk(w0);
        count_chunk(w0, mine);
        block_scan2_u64(mine, sh.warp_sums, excl, sum);
    } else {
        uint64_t mine[2] = {0, 0};
        for (int c0 = w0; c0 < w1; c0 += PD_THREADS) {
            uint64_t part[2];
            load_chunk(c0);
            count_chunk(c0, part);
            mine[0] += part[0];
            mine[1] += part[1];
        }
        block_scan2_u64(mine, sh.warp_sums, excl, sum);
    }
    if (tid == 0) { sh.totals[0] = sum[0]; sh.totals[1] = sum[1]; }
    // Later clusters count what lies before them by themselves, a share of the words per CTA (clusters do not wait for one another), and
    // note the last run start, of which a run that reaches into the cluster's words needs its length.
    const bool later = MODE == PD_LISTS && c_begin > 0;
    auto miss_word = [&](int i, uint32_t v) -> uint32_t { return v == 0u || p.predicted == nullptr ? v : v & ~__ldcg(p.predicted + i); };
    if (later) {
        uint64_t part[2] = {0, 0}, dummy[2], before[2];
        int last[2] = {-1, -1};
        for (int i = rank * PD_THREADS + tid; i < c_begin; i += n_cta * PD_THREADS) {
            const uint32_t v0 = union_word(i), u0 = union_word(i - 1);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (q == 1 && !want_miss) break;
                const uint32_t v = q ? miss_word(i, v0) : v0, u = q ? miss_word(i - 1, u0) : u0;
                const uint32_t starts = v & ~((v << 1) | (u >> 31));
                part[q] += static_cast<uint64_t>(__popc(v)) << 32 | static_cast<uint64_t>(__popc(starts));
                if (starts != 0u) last[q] = i * 32 + 31 - __clz(starts);
            }
        }
        block_scan2_u64(part, sh.warp_sums, dummy, before);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            last[q] = __reduce_max_sync(0xffffffffu, last[q]);
            if (lane == 0) sh.last_of_warp[q][warp] = last[q];
        }
        __syncthreads();
        if (warp < 2) {
            const int m = __reduce_max_sync(0xffffffffu, sh.last_of_warp[warp][lane]);
            if (lane == 0) { sh.earlier[warp] = before[warp]; sh.last_start[warp] = m; }
        }
    }
    cluster_sync_all();                   // counts are there; nobody reads the private bitmaps any more
    // Warp 0 fetches everybody's counts, lane r those of CTA r: from all 32 warps they were a thousand small remote loads per CTA, which
    // took 4 us with sixteen CTAs.
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint64_t x = lane < n_cta ? ld_cluster_u64(mapa_shared(smem_u32(&sh.totals[q]), lane)) : 0;
            uint64_t y = lane < rank ? x : 0, z = 0;
            int last = -1;
            if (later && lane < n_cta) {
                z = ld_cluster_u64(mapa_shared(smem_u32(&sh.earlier[q]), lane));
                last = static_cast<int>(ld_cluster_u32(mapa_shared(smem_u32(&sh.last_start[q]), lane)));
            }
#pragma unroll
            for (int d = PD_MAX_CLUSTER / 2; d > 0; d >>= 1) {
                x += __shfl_xor_sync(0xffffffffu, x, d);
                y += __shfl_xor_sync(0xffffffffu, y, d);
                if (later) z += __shfl_xor_sync(0xffffffffu, z, d);
            }
            if (later) last = __reduce_max_sync(0xffffffffu, last);
            if (lane == 0) { sh.upto[q] = z; sh.all[q] = x + z; sh.before[q] = y + z; sh.open_start[q] = last; }
        }
    }
    __syncthreads();
    uint64_t base[2] = {sh.before[0], sh.before[1]};
    const int cap = static_cast<int>(min(p.capacity, static_cast<int64_t>(0x7fffffff)));
    for (int c0 = w0; c0 < w1; c0 += PD_THREADS) {
        if (!one_chunk) {
            uint64_t mine[2];
            load_chunk(c0);
            count_chunk(c0, mine);
            block_scan2_u64(mine, sh.warp_sums, excl, sum);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) sh.at[q][tid] = base[q] + excl[q];
        __syncthreads();
        // A warp writes one word's entries at a time, a lane per page: neighbouring entries leave in one store.  Bound by its instructions.
        const int n_in = min(PD_THREADS, w1 - c0);
        const uint32_t below = (1u << lane) - 1u;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (q == 1 && !want_miss) break;
            int32_t* ids = q ? p.miss_pages : p.pages;
            int32_t* runs = q ? p.miss_runs : p.runs;
            for (int j = warp; j < n_in; j += PD_THREADS / 32) {
                const uint32_t w = sh.word[q][j + 1];
                if (((w >> lane) & 1u) == 0u) continue;
                const uint32_t starts = w & ~((w << 1) | (sh.word[q][j] >> 31)), ends = w & ~((w >> 1) | (sh.word[q][j + 2] << 31));
                const uint64_t o = sh.at[q][j];
                const int o_id = static_cast<int>(o >> 32) + __popc(w & below);
                const int run = static_cast<int>(o & 0xffffffffu) + __popc(starts & (below | (1u << lane))) - 1;      // the page's run
                const int32_t page = (c0 + j) * 32 + lane;
                if (o_id < cap) ids[o_id] = page;
                if (run < cap) {
                    if ((starts >> lane) & 1u) runs[2 * static_cast<int64_t>(run)] = page;
                    if ((ends >> lane) & 1u) runs[2 * static_cast<int64_t>(run) + 1] = page + 1;        // becomes a length below
                }
            }
        }
        base[0] += sum[0];
        base[1] += sum[1];
    }
    cluster_sync_all();                   // every start and end is written (and every CTA has read the counts)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (q == 1 && !want_miss) break;
        int32_t* runs = q ? p.miss_runs : p.runs;
        // The runs that end in the cluster's words: one may have begun before them, and one may go on after them.
        auto open_at = [&](int i) {       // page 32 i belongs to the run of the page before it
            if (MODE != PD_LISTS || i <= 0 || i >= p.n_words) return false;
            const uint32_t u = union_word(i - 1), v = union_word(i);
            return ((q ? miss_word(i - 1, u) : u) >> 31) != 0u && ((q ? miss_word(i, v) : v) & 1u) != 0u;
        };
        const bool begun = later && open_at(c_begin);
        const int64_t n_runs = static_cast<int64_t>(sh.all[q] & 0xffffffffu), n_ids = static_cast<int64_t>(sh.all[q] >> 32);
        const int64_t j_begin = later ? static_cast<int64_t>(sh.upto[q] & 0xffffffffu) - (begun ? 1 : 0) : 0;
        const int64_t j_end = min(n_runs - (open_at(c_end) ? 1 : 0), p.capacity);
        for (int64_t j = j_begin + static_cast<int64_t>(rank) * PD_THREADS + tid; j < j_end; j += static_cast<int64_t>(n_cta) * PD_THREADS)
            runs[2 * j + 1] = __ldcg(runs + 2 * j + 1) - (begun && j == j_begin ? sh.open_start[q] : __ldcg(runs + 2 * j));
        if (c_end == p.n_words && c_begin < c_end && rank == 0 && tid == 0) {
            *(q ? p.n_miss : p.n_pages) = static_cast<int32_t>(n_ids);
            *(q ? p.n_miss_runs : p.n_runs) = static_cast<int32_t>(n_runs);
            if (n_ids > p.capacity || n_runs > p.capacity) report(p.dev_status, JANUS_DEV_CAPACITY_EXCEEDED);
        }
    }
}

__global__ void page_union_kernel(uint32_t* __restrict__ dst, const uint32_t* src, int n_words) {
    grid_launch_next();
    grid_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_words; i += gridDim.x * blockDim.x) dst[i] |= src[i];
}

template <int MODE>
static int launch_page_demand(const PdParams& p, const PdPlan& plan, cudaStream_t stream) {
    if (plan.few) {
        static once_per_context few_attributes;
        JANUS_CUDA_CHECK(few_attributes.run([] { return cudaFuncSetAttribute(page_demand_few_kernel<MODE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1); }));
        const int n_cta = MODE == PD_LISTS ? 1 : plan.cluster;
        JANUS_CUDA_CHECK(launch_kernel(page_demand_few_kernel<MODE>, dim3(n_cta), PD_THREADS, 0, stream, n_cta, p));
        return JANUS_OK;
    }
    const size_t smem = MODE == PD_LISTS ? 0 : sizeof(uint32_t) * static_cast<size_t>(p.n_words);
    static once_per_context attributes;
    JANUS_CUDA_CHECK(attributes.run([] {
        cudaError_t e = cudaFuncSetAttribute(page_demand_kernel<MODE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess && MODE != PD_LISTS)
            e = cudaFuncSetAttribute(page_demand_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, PD_SMEM_WORDS * static_cast<int>(sizeof(uint32_t)));
        return e;
    }));
    JANUS_CUDA_CHECK(launch_kernel(page_demand_kernel<MODE>, dim3(plan.cluster * plan.clusters), PD_THREADS, smem, stream, plan.cluster, p));
    return JANUS_OK;
}

// CTAs of the largest cluster that the device takes: clusters above eight are not granted everywhere (a part of a GPU may have fewer
// SMs side by side).  A property of the device, asked for on its first call.
static cudaError_t largest_cluster(int& largest) {
    static once_per_context once;
    static std::atomic<int> known[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) {
        largest = PD_PORTABLE_CLUSTER;
        return cudaSuccess;
    }
    e = once.run([&] {
        cudaError_t r = cudaFuncSetAttribute(page_demand_kernel<PD_MARK>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(page_demand_kernel<PD_MARK>, cudaFuncAttributeMaxDynamicSharedMemorySize, PD_SMEM_WORDS * static_cast<int>(sizeof(uint32_t)));
        if (r != cudaSuccess) return r;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = PD_MAX_CLUSTER;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(PD_MAX_CLUSTER);
        cfg.blockDim = dim3(PD_THREADS);
        cfg.dynamicSmemBytes = sizeof(uint32_t) * PD_SMEM_WORDS;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, page_demand_kernel<PD_MARK>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        known[dev] = n > 0 ? PD_MAX_CLUSTER : PD_PORTABLE_CLUSTER;
        return cudaSuccess;
    });
    largest = known[dev];
    return e;
}

template <int MODE>
static int run_page_demand(const PdParams& p, cudaStream_t stream) {
    int largest = 0;
    JANUS_CUDA_CHECK(largest_cluster(largest));
    const PdPlan plan = page_demand_plan(p.n_idx, p.n_words, largest);
    if (plan.one_launch) return launch_page_demand<MODE>(p, plan, stream);
    JANUS_CUDA_CHECK(launch_kernel(page_clear_kernel, dim3(std::min((p.n_words + 255) / 256, 148)), 256, 0, stream, 1, p.bitmap, p.n_words));
    const int64_t n_log_words = (p.n_logical_pages + 31) / 32;
    if (MODE == PD_MARK && n_log_words + p.n_words <= MARK_SMEM_WORDS) {
        static once_per_context attributes;
        JANUS_CUDA_CHECK(attributes.run([] {
            return cudaFuncSetAttribute(page_mark_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MARK_SMEM_WORDS * static_cast<int>(sizeof(uint32_t)));
        }));
        const int64_t want = ((p.n_idx >> 2) + MARK_THREADS - 1) / MARK_THREADS;
        const unsigned grid = static_cast<unsigned>(want < 1 ? 1 : want < 148 * 2 ? want : 148 * 2);
        JANUS_CUDA_CHECK(launch_kernel(page_mark_kernel, dim3(grid), MARK_THREADS, sizeof(uint32_t) * (n_log_words + p.n_words), stream, 1, p,
                                       static_cast<int>(n_log_words)));
    } else if (p.n_idx > 0) {
        const int64_t want = (p.n_idx + 1023) / 1024;
        JANUS_CUDA_CHECK(launch_kernel(page_mark_global_kernel<MODE>, dim3(static_cast<unsigned>(want < 148 * 8 ? want : 148 * 8)), 256, 0, stream, 1,
                                       p));
    }
    return launch_page_demand<PD_LISTS>(p, plan, stream);
}

static int page_shift_of(int page_size) {
    if ((page_size & (page_size - 1)) != 0) return -1;
    int shift = 0;
    while ((1 << shift) < page_size) ++shift;
    return shift;
}

}  // namespace janus

extern "C" int janus_page_union(uint32_t* dst, const uint32_t* src, int64_t n_phys_pages, void* stream_) {
    using namespace janus;
    if (!dst || !src || n_phys_pages <= 0) return JANUS_ERR_INVALID_ARG;
    if (n_phys_pages > (int64_t(1) << 31) - 64) return JANUS_ERR_UNSUPPORTED;
    const int n_words = static_cast<int>((n_phys_pages + 31) / 32);
    const int blocks = n_words < 256 * 148 ? (n_words + 255) / 256 : 148;
    JANUS_CUDA_CHECK(launch_kernel(page_union_kernel, dim3(blocks), 256, 0, static_cast<cudaStream_t>(stream_), 1, dst, src, n_words));
    return JANUS_OK;
}

extern "C" size_t janus_page_demand_workspace_size(int64_t, int, int64_t) { return 0; }

extern "C" int janus_page_demand(const int32_t* idx, int64_t n_rows, int k, int64_t demand_limit, int page_size,
                                 const int32_t* page_table, int64_t n_logical_pages, int64_t n_phys_pages,
                                 const uint32_t* predicted_bitmap, uint32_t* bitmap, int32_t* pages, int32_t* n_pages,
                                 int32_t* runs, int32_t* n_runs, int32_t* miss_pages, int32_t* n_miss, int32_t* miss_runs,
                                 int32_t* n_miss_runs, int64_t capacity, void* /*ws*/, size_t /*ws_bytes*/,
                                 int32_t* dev_status, void* stream_) {
    using namespace janus;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (n_rows < 0 || k < 0 || page_size <= 0 || n_logical_pages < 0 || n_phys_pages <= 0 || capacity < 0 || demand_limit < 0)
        return JANUS_ERR_INVALID_ARG;
    if (n_phys_pages > (int64_t(1) << 31) - 64) return JANUS_ERR_UNSUPPORTED;
    if (!bitmap || !pages || !n_pages || !runs || !n_runs || !page_table) return JANUS_ERR_INVALID_ARG;
    const int n_miss_ptrs = (miss_pages != nullptr) + (n_miss != nullptr) + (miss_runs != nullptr) + (n_miss_runs != nullptr);
    if (n_miss_ptrs != 0 && n_miss_ptrs != 4) return JANUS_ERR_INVALID_ARG;
    const int64_t n_idx = n_rows * static_cast<int64_t>(k);
    if (n_idx > 0 && (!idx || !aligned16(idx))) return JANUS_ERR_INVALID_ARG;

    PdParams p = {};
    p.idx = idx; p.n_idx = n_idx; p.k = k;
    p.demand_limit = demand_limit;
    p.page_size = page_size; p.page_shift = page_shift_of(page_size);
    p.page_table = page_table; p.n_logical_pages = n_logical_pages;
    p.n_phys_pages = n_phys_pages; p.n_words = static_cast<int>((n_phys_pages + 31) / 32);
    p.predicted = predicted_bitmap; p.bitmap = bitmap;
    p.pages = pages; p.n_pages = n_pages; p.runs = runs; p.n_runs = n_runs;
    p.miss_pages = miss_pages; p.n_miss = n_miss; p.miss_runs = miss_runs; p.n_miss_runs = n_miss_runs;
    p.capacity = capacity; p.dev_status = dev_status;
    return run_page_demand<PD_MARK>(p, stream);
}

extern "C" int janus_page_demand_batch(const int32_t* idx, int64_t n_rows, int k, const int64_t* demand_limits, int page_size,
                                       const int32_t* page_tables, const int64_t* table_offsets, int64_t n_phys_pages,
                                       const uint32_t* predicted_bitmap, uint32_t* bitmap, int32_t* pages, int32_t* n_pages,
                                       int32_t* runs, int32_t* n_runs, int32_t* miss_pages, int32_t* n_miss, int32_t* miss_runs,
                                       int32_t* n_miss_runs, int64_t capacity, int32_t* dev_status, void* stream_) {
    using namespace janus;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (n_rows < 0 || k < 0 || page_size <= 0 || n_phys_pages <= 0 || capacity < 0) return JANUS_ERR_INVALID_ARG;
    if (n_phys_pages > (int64_t(1) << 31) - 64) return JANUS_ERR_UNSUPPORTED;
    if (!bitmap || !pages || !n_pages || !runs || !n_runs) return JANUS_ERR_INVALID_ARG;
    const int n_miss_ptrs = (miss_pages != nullptr) + (n_miss != nullptr) + (miss_runs != nullptr) + (n_miss_runs != nullptr);
    if (n_miss_ptrs != 0 && n_miss_ptrs != 4) return JANUS_ERR_INVALID_ARG;
    const int64_t n_idx = n_rows * static_cast<int64_t>(k);
    if (n_idx > 0 && (!idx || !demand_limits || !page_tables || !table_offsets)) return JANUS_ERR_INVALID_ARG;

    PdParams p = {};
    p.idx = idx; p.n_idx = n_idx; p.k = k;
    p.demand_limits = demand_limits; p.table_offsets = table_offsets;
    p.page_size = page_size; p.page_shift = page_shift_of(page_size);
    p.page_table = page_tables;
    p.n_phys_pages = n_phys_pages; p.n_words = static_cast<int>((n_phys_pages + 31) / 32);
    p.predicted = predicted_bitmap; p.bitmap = bitmap;
    p.pages = pages; p.n_pages = n_pages; p.runs = runs; p.n_runs = n_runs;
    p.miss_pages = miss_pages; p.n_miss = n_miss; p.miss_runs = miss_runs; p.n_miss_runs = n_miss_runs;
    p.capacity = capacity; p.dev_status = dev_status;
    return run_page_demand<PD_MARK_ROWS>(p, stream);
}
