// Tensor-core sparse attention for the latent layout (Sec. 2.2, "core attention"): one shared KV row of 576 bf16
// per token (keys = all 576 dims, values = the first 512), 128 query heads, selection idx[t, 0:k).
//
//     out[t,h,:] = sum_{s in idx[t]} softmax_s(scale * <q[t,h,:576], row_s[:576]>) * row_s[:512]
//
// Shape of the problem.  The fp32 output of one token, 128 heads x 512 columns, is all of one SM's tensor memory, so a token is handled
// by a pair of CTAs.  They split the *heads*: CTA c owns heads [64 c, 64 c + 64) with their logits, softmax and output, and the MMAs
// are those of a CTA pair (M = 128, 64 rows in each SM, at the full rate of both), whose B operand is read half from each SM:
//
//   logits  S = Q . K^T, 128 keys at a time, N = 128: CTA c holds all 576 dims of keys [64 c, 64 c + 64) of the tile;
//   output  O += P . V, N = 256 twice: CTA c holds value dims [256 c, 256 c + 256) of all 128 keys.
//
// Nothing but barrier arrivals crosses between the SMs.  The price is that a CTA's own keys are gathered twice, once as rows of K and
// once (their owned half of the values) as rows of V, which the MMA cannot read from one place: for the logits the same address holds
// different keys in the two CTAs, for the output the same keys.  139 KB come in per 128 keys and CTA, beside 2185 cycles of MMAs.
// Splitting the feature axis instead (each byte gathered once, partial logits exchanged through distributed shared memory as fp16, the
// softmax of every head computed in both CTAs) took 4500-5200 cycles for the same keys, the softmax being the period; this takes 2700.
// 4096 tokens x 2048 keys 2.83 -> 2.04 ms (1150 TFLOP/s at the 1.37 GHz that the power limit leaves), 512 x 2048 332 -> 266 us,
// 64 x 2048 57 -> 35, 700 x 256 96 -> 79.
//
// What the 2700 cycles hang on: the turn of a K unit (its MMAs, 200 to the copy warps, 500 of issue, 1400 of L2 latency, 300 back to
// the MMA warp) over a ring of four thirds of a tile, that of a V unit over a tile, and S, of which there is one.
//
// Per CTA: tensor memory = O 256 | S 64 | Q 192 columns (query atoms of 64 dims 0-5 as the A operand; both lane halves hold them).  A lane
// is (head = lane % 64, half = lane / 64): S holds the keys, O the value dims of that half.  Shared memory: query atoms 6-8, two buffers
// of P, a ring of K units (64 rows x 3 atoms) and one of V units (32 rows x 4 atoms).  Warp roles (19 warps, 96 registers per thread):
//   warps 0-7    softmax and output (thread = head and a quarter of the tile's keys; the four warps of 32 heads exchange their maxima):
//                fp32 online softmax, P rounded to bf16 into shared memory;
//   warp 8       resolves the rows of the tiles through the page table, two tiles ahead;
//   warps 9-12   copies of K: the TMA unit gathers 4 rows x 128 bytes per instruction, counted on the even CTA's barriers; the queries
//                of a token come through the same ring;
//   warps 13-16  copies of V with 16-byte cp.async.  Either unit alone for both is slower: 272 gathers a tile keep their warps busy for
//                3100 cycles, and 272 cp.async of 512 bytes keep the load/store unit busy for 2000, behind which every barrier and
//                shared-memory access of the other warps queues (740 x 2048: 330, 333 and 322 us);
//   warps 17-18  in the even CTA issue the MMAs, one Q . K and one P . V; in the odd one pass on the news that a unit has landed.
// The kernel is persistent: one pair loops over tokens, and the rings and all barrier phases run on across tokens (1100 cycles a token
// beside its tiles; queries brought in by the head warps, lane by lane, cost 9000).
// The running max only moves when a tile exceeds it by more than 2^8, so O is rescaled (in tensor memory) a handful of
// times per row.  Every wait is bounded; on a timeout the CTA reports JANUS_DEV_WAIT_TIMEOUT, and all CTAs of the
// cluster still meet at the final cluster barrier.
#include <mutex>
#include <type_traits>

#include "janus_common.cuh"
#include "sm100_ptx.cuh"

namespace janus {

using namespace ptx;

constexpr int LP_HEADS = 128;
constexpr int LP_OWN = 64;                  // heads of a CTA; keys of a tile whose K rows it holds
constexpr int LP_DQK = 576;
constexpr int LP_DV = 512;
constexpr int LP_DVH = 256;
constexpr int LP_TILE = 128;                // keys per tile
constexpr int LP_ATOM_BYTES = LP_OWN * 128;                      // 8 KB: 64 rows x 64 dims
constexpr int LP_KPARTS = 3;                // K units of a tile: atoms 6-8 (their queries lie in shared memory), 0-2, 3-5
constexpr int LP_QPARTS = 2;                // units of a token that bring query atoms 0-2, 3-5 through the ring of K units
constexpr int LP_KU = 4;                    // K units in the ring
static_assert(LP_KU - LP_QPARTS >= 1 && LP_KU - LP_QPARTS <= LP_KPARTS, "a copy warp passes over the query units' places without a wait");
constexpr int LP_K_BYTES = 3 * LP_ATOM_BYTES;
constexpr int LP_VROWS = 32;                // keys of a V unit
constexpr int LP_VPARTS = LP_TILE / LP_VROWS;
constexpr int LP_VU = 4;                    // V units in the ring
constexpr int LP_V_ATOM_BYTES = LP_VROWS * 128;
constexpr int LP_V_BYTES = 4 * LP_V_ATOM_BYTES;
constexpr int LP_P_BYTES = 2 * LP_ATOM_BYTES;                    // 16 KB: 64 heads x 128 keys; two of them, by parity of the tile
constexpr int LP_Q_BYTES = 3 * LP_ATOM_BYTES;                    // 24 KB: query atoms 6-8
constexpr int LP_SMEM_TILES = LP_KU * LP_K_BYTES + LP_VU * LP_V_BYTES;
constexpr int LP_HEAD_WARPS = 8, LP_ROWS_WARP = LP_HEAD_WARPS, LP_COPY_WARPS = 4;    // copy warps for K, and as many for V
constexpr int LP_K_WARP0 = LP_ROWS_WARP + 1, LP_V_WARP0 = LP_K_WARP0 + LP_COPY_WARPS, LP_QK_WARP = LP_V_WARP0 + LP_COPY_WARPS, LP_PV_WARP = LP_QK_WARP + 1;
constexpr int LP_THREADS = 32 * (LP_PV_WARP + 1);
constexpr int LP_RROWS = 4;                 // tiles whose row numbers and validity masks are kept
constexpr int LP_MAX_SPLIT = 8;             // pairs of a cluster that share the keys of one token
constexpr uint32_t LP_COL_O = 0, LP_COL_S = 256, LP_COL_Q = 320;

struct LpShared {
    uint64_t k_full[LP_KU], k_empty[LP_KU];       // rows landed (the odd CTA's are passed on to the even one's) / read by the MMAs of both
    uint64_t v_full[LP_VU], v_empty[LP_VU];
    uint64_t r_full[LP_RROWS], r_empty[LP_RROWS]; // rows and masks of a tile are written / no longer needed
    uint64_t s_full, s_free;                      // logits complete / in the registers of all head warps of both CTAs
    uint64_t p_full[2], pv_done[2];               // by parity of the tile: P of both CTAs is written / P.V is done
    uint64_t q_full, q_free;                      // query atoms 6-8: in shared memory of both CTAs / read by the token's last logits
    uint64_t q_idle;                              // the token's last logits are complete: nothing reads its queries in tensor memory
    uint64_t o_free;                              // O of the token before has been read in both CTAs
    uint64_t x_full[2];                           // the four head warps of 32 heads exchange their maxima (and, before that, left their sums)
    uint64_t drain[2];
    uint32_t vmask[LP_RROWS][LP_TILE / 32];       // bit = key of the tile
    alignas(16) int32_t row[LP_RROWS][LP_TILE];   // number of the row in the pool; -1 = none
    int64_t offset[LP_RROWS][LP_TILE];            // its byte offset; INT64_MIN = none
    float mx[2][4][LP_OWN];                       // by parity of the exchange, quarter of the tile's keys
    float l[2][4][LP_OWN];                        // by parity of the token: sum over a quarter of the keys of each tile
    uint32_t tmem_base;
    uint32_t start_abort[2 * LP_MAX_SPLIT];       // by CTA of the cluster
    // reference maximum and row sum of every head, for the merge; the sum is negative until the pair has left its output
    float split_m[LP_OWN], split_l[LP_OWN];
};

// Keys of one token split over several pairs of a cluster (few query rows): a CTA leaves its fp32 output for the merge where its
// rings were, [column / 4][lane][4], and LpShared::split_m / split_l.
static_assert(LP_DVH * LP_TILE * 4 <= LP_SMEM_TILES, "the merge buffer reuses the rings");

struct LpParams {
    const uint16_t* q;
    const uint16_t* pool;
    int64_t page_stride, tok_stride;
    const int32_t* idx;
    int k;
    int page_size, page_shift;
    const int32_t* page_table;
    int64_t n_logical_pages;
    const int64_t* table_offsets;   // NULL, or [M + 1]: row t uses page_table[table_offsets[t] .. table_offsets[t + 1])
    float scale_log2e;        // softmax_scale * log2(e)
    uint16_t* out;
    float* lse;
    int M;
    int32_t* dev_status;
};

__device__ __forceinline__ float lp_exp2(float x) {   // ex2.approx: 2 ulp, exp2(-inf) = 0
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t lp_pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ float lp_ld_cluster(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ float4 lp_ld_cluster4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}

// Element of `out` that lane (head, half) of CTA c starts its 256 columns at, for token t.
__device__ __forceinline__ int64_t lp_out_offset(int t, uint32_t c, int lane128) {
    return (static_cast<int64_t>(t) * LP_HEADS + LP_OWN * static_cast<int>(c) + (lane128 & (LP_OWN - 1))) * LP_DV + (lane128 / LP_OWN) * LP_DVH;
}

// Output of token t from the N pairs' unnormalised outputs: CTA (s, c) takes every N-th block of 16 columns of its 128 lanes, a
// thread one block of one lane at a time.  N is a compile-time number so that all remote loads are issued together.
template <int N>
__device__ __forceinline__ void lp_merge_splits(const LpParams& p, int t, int s, uint32_t c, uint32_t o_addr, uint32_t m_addr, uint32_t l_addr) {
    const int ln = threadIdx.x & (LP_TILE - 1), h = ln & (LP_OWN - 1);
    const float neg_inf = __int_as_float(0xff800000);
    float f[N], l[N];
    float m_all = neg_inf, l_all = 0.f;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        f[r] = lp_ld_cluster(mapa_shared(m_addr + 4 * h, 2 * r + c));
        l[r] = lp_ld_cluster(mapa_shared(l_addr + 4 * h, 2 * r + c));
    }
#pragma unroll
    for (int r = 0; r < N; ++r)
        if (l[r] < 0.f) return;      // a pair gave up (reported): what lies in its buffer may be anything, and the row stays unwritten
#pragma unroll
    for (int r = 0; r < N; ++r) m_all = fmaxf(m_all, f[r]);
#pragma unroll
    for (int r = 0; r < N; ++r) {
        f[r] = m_all == neg_inf ? 0.f : lp_exp2(f[r] - m_all);
        l_all = fmaf(f[r], l[r], l_all);
    }
    const float inv = l_all != 0.f ? 1.f / l_all : 0.f;        // (a NaN is a sum)
    constexpr int GROUPS = LP_THREADS / LP_TILE;
    if (threadIdx.x < GROUPS * LP_TILE) {
        for (int blk = s + N * (threadIdx.x / LP_TILE); blk < LP_DVH / 16; blk += N * GROUPS) {
            float4 acc[4] = {};
#pragma unroll
            for (int v2 = 0; v2 < 4; v2 += 2) {
                float4 x[N][2];
#pragma unroll
                for (int r = 0; r < N; ++r) {
                    const uint32_t src = mapa_shared(o_addr + static_cast<uint32_t>(((blk * 4 + v2) * LP_TILE + ln) * 16), 2 * r + c);
#pragma unroll
                    for (int v = 0; v < 2; ++v) x[r][v] = lp_ld_cluster4(src + v * LP_TILE * 16);
                }
#pragma unroll
                for (int r = 0; r < N; ++r)
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        float4& o = acc[v2 + v];
                        o.x = fmaf(f[r], x[r][v].x, o.x); o.y = fmaf(f[r], x[r][v].y, o.y);
                        o.z = fmaf(f[r], x[r][v].z, o.z); o.w = fmaf(f[r], x[r][v].w, o.w);
                    }
            }
            uint4* dst = reinterpret_cast<uint4*>(p.out + lp_out_offset(t, c, ln) + blk * 16);
            uint32_t w[8];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                w[2 * v] = lp_pack_bf16x2(acc[v].x * inv, acc[v].y * inv);
                w[2 * v + 1] = lp_pack_bf16x2(acc[v].z * inv, acc[v].w * inv);
            }
            dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
            dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
    }
    if (p.lse != nullptr && s == 0 && threadIdx.x < LP_OWN)
        p.lse[static_cast<int64_t>(t) * LP_HEADS + LP_OWN * c + h] = l_all != 0.f ? (m_all + log2f(l_all)) * 0.6931471805599453f : neg_inf;
}

// SPLIT = false: clusters of two CTAs, persistent over tokens.  SPLIT = true: a cluster of 2 n CTAs takes one token, pair s of it
// the tiles [s, s + 1) * n_tiles / n, and the pairs' outputs are merged through distributed shared memory at the end.
// ROWS = true: the pool's rows lie at whole multiples of one stride and those of K are gathered by number; false: by address.
template <bool SPLIT, bool ROWS>
__global__ void __launch_bounds__(LP_THREADS, 1) sparse_attn_latent_pair_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_pool,
                                                                              const LpParams p) {
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* k_smem = smem;                                              // units of 3 atoms x [64 keys x 128 B]
    unsigned char* v_smem = smem + LP_KU * LP_K_BYTES;                         // units of 4 atoms x [32 keys x 128 B]
    unsigned char* p_smem = smem + LP_SMEM_TILES;                              // 2 x 2 x [64 heads x 64 keys]
    unsigned char* q_smem = p_smem + 2 * LP_P_BYTES;                               // query atoms 6-8, each [64 heads x 128 B]
    LpShared* sh = reinterpret_cast<LpShared*>(q_smem + LP_Q_BYTES);

    cluster_arrive();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const uint32_t c = rank & 1u;                  // 0 or 1: which heads, keys and value dims this CTA owns
    // persistent: cluster `cid` handles tokens cid, cid + n_clusters, ...; tiles are counted over all of them
    const int n_split = SPLIT ? static_cast<int>(cluster_nctarank() >> 1) : 1;
    const int cid = blockIdx.x / (2 * n_split), n_clusters = gridDim.x / (2 * n_split);
    const int n_my = cid < p.M ? (p.M - cid + n_clusters - 1) / n_clusters : 0;     // SPLIT: one cluster per token, so 1
    const int all_tiles = (p.k + LP_TILE - 1) / LP_TILE;
    const int tile0 = SPLIT ? static_cast<int>(rank >> 1) * all_tiles / n_split : 0;
    const int n_tiles = SPLIT ? (static_cast<int>(rank >> 1) + 1) * all_tiles / n_split - tile0 : all_tiles;
    const int total = n_my * n_tiles;

    if (SPLIT && threadIdx.x < LP_OWN) sh->split_l[threadIdx.x] = -1.f;
    if (threadIdx.x == 0) {
        // copies by cp.async: a "full" barrier counts every copying thread of the CTA, and in the even CTA the odd one's unit as one arrival
        // more; by the TMA unit: the even CTA's barriers count the bytes of both
        const uint32_t by_threads = 32 * LP_COPY_WARPS + (c == 0u ? 1u : 0u), arrivals = ROWS ? 1u : by_threads;
        for (int u = 0; u < LP_KU; ++u) { mbar_init(smem_u32(&sh->k_full[u]), arrivals); mbar_init(smem_u32(&sh->k_empty[u]), 1); }
        for (int u = 0; u < LP_VU; ++u) { mbar_init(smem_u32(&sh->v_full[u]), by_threads); mbar_init(smem_u32(&sh->v_empty[u]), 1); }
        for (int r = 0; r < LP_RROWS; ++r) { mbar_init(smem_u32(&sh->r_full[r]), 1); mbar_init(smem_u32(&sh->r_empty[r]), 2 * LP_COPY_WARPS + LP_HEAD_WARPS); }
        mbar_init(smem_u32(&sh->s_full), 1);
        mbar_init(smem_u32(&sh->s_free), 2 * LP_HEAD_WARPS);
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&sh->p_full[i]), 2 * LP_HEAD_WARPS); mbar_init(smem_u32(&sh->pv_done[i]), 1); }
        mbar_init(smem_u32(&sh->q_full), 1);
        mbar_init(smem_u32(&sh->q_free), 1);
        mbar_init(smem_u32(&sh->q_idle), 1);
        mbar_init(smem_u32(&sh->o_free), 2 * LP_HEAD_WARPS);
        for (int i = 0; i < 2; ++i) mbar_init(smem_u32(&sh->x_full[i]), 4);
        for (int i = 0; i < 2; ++i) mbar_init(smem_u32(&sh->drain[i]), 1);
        fence_mbar_init();
    }
    grid_wait();
    cluster_wait();                                // every CTA of the cluster runs: its shared memory may be written
    if (threadIdx.x == 0) {
        // start-up agreement: if this CTA should not start (misaligned shared memory, or an earlier CTA of the launch gave
        // up on a wait), every CTA of the cluster must skip the work, so the flag is written to all of them
        uint32_t flag = ((smem_u32(smem) & 1023u) != 0u) ? 1u : 0u;
        if (p.dev_status != nullptr && *reinterpret_cast<volatile int32_t*>(p.dev_status) == JANUS_DEV_WAIT_TIMEOUT) flag = 1u;
        for (uint32_t r = 0; r < cluster_nctarank(); ++r) st_cluster_u32(mapa_shared(smem_u32(&sh->start_abort[rank]), r), flag);
    }
    __syncwarp();
    if (warp == LP_QK_WARP) tmem_alloc_pair(smem_u32(&sh->tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                            // barriers of both CTAs are initialised, start flags exchanged
    if constexpr (SPLIT) grid_launch_next();       // (tensor memory is allocated)
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;
    uint32_t abort_flags = 0u;
    for (int r = 0; r < 2 * n_split; ++r) abort_flags |= sh->start_abort[r];
    const bool start_abort = abort_flags != 0u;
    if (start_abort && threadIdx.x == 0 && (smem_u32(smem) & 1023u) != 0u) report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT);

    // bounded wait of a whole warp, which stays together whatever the lanes saw
    auto wait_warp = [](uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(smem_u32(bar), parity)) != 0; };
    // one arrival (by the calling lane) on a barrier of the pair's even CTA
    auto arrive_even = [&](uint64_t* bar) {
        if (c == 0u) mbar_arrive(smem_u32(bar));
        else mbar_arrive_remote(mapa_shared(smem_u32(bar), rank & ~1u));
    };
    bool ok = true;

    if (start_abort) {
        // nothing to do
    } else if (warp >= LP_QK_WARP && c == 0u) {
        // ================================================================== MMA issue (even CTA): one warp for Q . K, one for P . V
        // A warp runs its loop together and one elected lane issues.  Every counter of the loops is known without looking at a barrier:
        // where it is not (one warp that issues what a probe of all barriers finds ready), the operands of an MMA count as different
        // from lane to lane and each takes 60 cycles to issue instead of 20, twice the time it takes to execute.  Two warps, because a
        // wait between MMAs costs some 270 cycles here, ready or not, and seven of them with 52 MMAs were 3200 cycles a tile for one
        // warp.  S of tile j is in the softmax's registers soon after it is complete, so the next logits are computed while that softmax
        // runs.  Rows written by cp.async are published to the MMAs by the fence that follows the wait for them; those of the odd CTA
        // by its own.
        constexpr uint32_t idesc_qk = umma_idesc_major(1u, LP_HEADS, LP_TILE, 0u, 0u);
        constexpr uint32_t idesc_pv = umma_idesc_major(1u, LP_HEADS, LP_DVH, 0u, 1u);
        const uint16_t pair = static_cast<uint16_t>(3u << rank);
        auto commit = [&](uint64_t* bar) { umma_commit_pair(smem_u32(bar), pair); };
        if (warp == LP_QK_WARP) {
            const uint32_t q_lo = umma_desc_lo(smem_u32(q_smem), 16), k_lo = umma_desc_lo(smem_u32(k_smem), 16);
            int n = 0;                                   // units so far, queries among them
            int j = 0;                                   // tiles so far
            auto next_unit = [&]() {
                ok = wait_warp(&sh->k_full[n & (LP_KU - 1)], static_cast<uint32_t>(n / LP_KU) & 1u);
                if constexpr (!ROWS) fence_proxy_async();
                tc_fence_after();
            };
            static_assert((LP_KU & (LP_KU - 1)) == 0, "place of a unit");
            for (int tok = 0; tok < n_my && ok; ++tok) {
                // query atoms 0-5 from the ring to tensor memory, once the last logits of the token before no longer need the old ones
                ok = tok == 0 || wait_warp(&sh->q_idle, static_cast<uint32_t>(tok - 1) & 1u);
                for (int a = 0; a < LP_QPARTS && ok; ++a, ++n) {
                    next_unit();
                    if (!ok) break;
                    const uint32_t qb = k_lo + static_cast<uint32_t>((n & (LP_KU - 1)) * (LP_K_BYTES >> 4));
                    if (elect_one()) {
#pragma unroll
                        for (int i = 0; i < 24; ++i) tmem_copy_rows64_pair(tmem_base + LP_COL_Q + 96 * a + 4 * i, qb + (i >> 3) * (LP_ATOM_BYTES >> 4) + (i & 7));
                        commit(&sh->k_empty[n & (LP_KU - 1)]);
                    }
                    __syncwarp();
                }
                ok = ok && wait_warp(&sh->q_full, static_cast<uint32_t>(tok) & 1u);
                for (int tile = 0; tile < n_tiles && ok; ++tile, ++j) {
                    const bool last = tile + 1 == n_tiles;
                    ok = j == 0 || wait_warp(&sh->s_free, static_cast<uint32_t>(j - 1) & 1u);
#pragma unroll
                    for (int u = 0; u < LP_KPARTS; ++u) {
                        if (ok) next_unit();
                        if (!ok) break;
                        const uint32_t kb = k_lo + static_cast<uint32_t>((n & (LP_KU - 1)) * (LP_K_BYTES >> 4));
                        if (elect_one()) {
#pragma unroll
                            for (int i = 0; i < 12; ++i) {
                                const uint32_t b = kb + (i >> 2) * (LP_ATOM_BYTES >> 4) + (i & 3) * 2;
                                if (u == 0) umma_pair_bf16_ss(tmem_base + LP_COL_S, q_lo + (i >> 2) * (LP_ATOM_BYTES >> 4) + (i & 3) * 2, b, idesc_qk, i > 0 ? 1u : 0u);
                                else umma_pair_bf16_ts(tmem_base + LP_COL_S, tmem_base + LP_COL_Q + 96 * (u - 1) + 8 * i, b, idesc_qk, 1u);
                            }
                            commit(&sh->k_empty[n & (LP_KU - 1)]);
                            if (last && u == 0) commit(&sh->q_free);
                            if (u == LP_KPARTS - 1) commit(&sh->s_full);
                            if (last && u == LP_KPARTS - 1) commit(&sh->q_idle);
                        }
                        __syncwarp();
                        ++n;
                    }
                }
            }
        } else {
            const uint32_t p_lo = umma_desc_lo(smem_u32(p_smem), 16), v_lo = umma_desc_lo(smem_u32(v_smem), LP_V_ATOM_BYTES);
            int vu = 0, tile = 0, tok = 0;
            uint32_t v_ph = 0u;
            for (int j = 0; j < total; ++j) {
                // the token's first waits until the output of the one before has been read out of O
                ok = tile > 0 || tok == 0 || wait_warp(&sh->o_free, static_cast<uint32_t>(tok - 1) & 1u);
#pragma unroll
                for (int v = 0; v < LP_VPARTS; ++v) {
                    if (v == 0) ok = ok && wait_warp(&sh->p_full[j & 1], static_cast<uint32_t>(j >> 1) & 1u);
                    ok = ok && wait_warp(&sh->v_full[vu], v_ph);
                    if (!ok) break;
                    fence_proxy_async();
                    tc_fence_after();
                    const uint32_t vb = v_lo + static_cast<uint32_t>(vu * (LP_V_BYTES >> 4));
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < LP_VROWS / 16; ++ks)
#pragma unroll
                            for (int n = 0; n < 2; ++n)
                                umma_pair_bf16_ss(tmem_base + LP_COL_O + n * 128,
                                                  p_lo + (j & 1) * (LP_P_BYTES >> 4) + (v * LP_VROWS / LP_OWN) * (LP_ATOM_BYTES >> 4) + (v * LP_VROWS % LP_OWN) / 8 + ks * 2,
                                                  vb + n * (2 * LP_V_ATOM_BYTES >> 4) + ks * (2048 >> 4), idesc_pv, (tile > 0 || v > 0 || ks > 0) ? 1u : 0u);
                        commit(&sh->v_empty[vu]);
                        if (v == LP_VPARTS - 1) commit(&sh->pv_done[j & 1]);
                    }
                    __syncwarp();
                    if (++vu == LP_VU) { vu = 0; v_ph ^= 1u; }
                }
                if (!ok) break;
                if (++tile == n_tiles) { tile = 0; ++tok; }
            }
        }
        if (!ok) {                                // what was issued must be through before tensor memory is given back
            uint64_t* bar = &sh->drain[warp == LP_QK_WARP ? 0 : 1];
            if (elect_one()) commit(bar);
            __syncwarp();
            (void)wait_warp(bar, 0u);
        }
    } else if (warp >= LP_QK_WARP) {
        if (!ROWS || warp == LP_PV_WARP) {
            // ============================================================== odd CTA: units landed here -> the even CTA's barriers
            const bool is_v = warp == LP_PV_WARP;
            int unit = 0;
            uint32_t ph = 0u;
            for (int n = 0; n < (is_v ? total * LP_VPARTS : total * LP_KPARTS + n_my * LP_QPARTS); ++n) {
                uint64_t* bar = is_v ? &sh->v_full[unit] : &sh->k_full[unit];
                ok = wait_warp(bar, ph);
                if (!ok) break;
                fence_proxy_async();
                if (lane == 0) mbar_arrive_remote(mapa_shared(smem_u32(bar), rank & ~1u));
                __syncwarp();
                if (++unit == (is_v ? LP_VU : LP_KU)) { unit = 0; ph ^= 1u; }
            }
        }
    } else if (warp == LP_ROWS_WARP) {
        // ================================================================== rows of the tiles, for the copy warps; masks for the softmax
        // Lane l resolves rows l, l + 32, ... of a tile.  Indices are loaded two tiles ahead, page-table entries one, and nothing is looked
        // at before its tile comes up, so that no load is waited for.
        int64_t tbl_nxt = 0, tbl_n_nxt = p.n_logical_pages;     // page table (start, length) of the query row the last load_raw was for
        int raw_tile = 0, raw_tok = 0, raw[4];                  // tile and token of the next load_raw
        auto load_raw = [&]() {
            const bool any = raw_tok < n_my;
            const int64_t t_row = cid + static_cast<int64_t>(raw_tok) * n_clusters;
            if (any && p.table_offsets != nullptr) {           // every query row has a page table of its own (a batch of sessions)
                tbl_nxt = ld_input(p.table_offsets + t_row);
                tbl_n_nxt = ld_input(p.table_offsets + t_row + 1) - tbl_nxt;
                if (tbl_nxt < 0) tbl_n_nxt = 0;                // a table that starts before the array: its tokens are reported and skipped
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int slot = (tile0 + raw_tile) * LP_TILE + 32 * i + lane;
                raw[i] = any && slot < p.k ? ld_input(p.idx + t_row * p.k + slot) : -1;
            }
            if (++raw_tile == n_tiles) { raw_tile = 0; ++raw_tok; }
        };
        int phys[4], within[4];                                 // within: -1 = no row selected; phys < 0 = no such page
        auto look_up = [&]() {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                phys[i] = within[i] = -1;
                if (raw[i] >= 0) {
                    const int64_t lp = p.page_shift >= 0 ? (raw[i] >> p.page_shift) : (raw[i] / p.page_size);
                    within[i] = p.page_shift >= 0 ? (raw[i] & (p.page_size - 1)) : (raw[i] % p.page_size);
                    if (lp < tbl_n_nxt) phys[i] = ld_input(p.page_table + tbl_nxt + lp);
                }
            }
        };
        const int rows_per_page = ROWS ? static_cast<int>(p.page_stride / p.tok_stride) : 0;
        load_raw();
        look_up();
        load_raw();
        for (int s = 0; s < total; ++s) {
            const int slot = s % LP_RROWS;
            ok = wait_warp(&sh->r_empty[slot], static_cast<uint32_t>(s / LP_RROWS) & 1u ^ 1u);
            if (!ok) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool here = phys[i] >= 0;
                if (within[i] >= 0 && !here) report(p.dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);     // beyond the page table, or a negative page id in it
                if constexpr (ROWS) sh->row[slot][32 * i + lane] = here ? phys[i] * rows_per_page + within[i] : -1;
                sh->offset[slot][32 * i + lane] = here ? 2 * (static_cast<int64_t>(phys[i]) * p.page_stride + static_cast<int64_t>(within[i]) * p.tok_stride) : INT64_MIN;
                const uint32_t mask = __ballot_sync(0xffffffffu, here);
                if (lane == 0) sh->vmask[slot][i] = mask;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh->r_full[slot]));
            look_up();
            load_raw();
        }
    } else if (warp >= LP_K_WARP0) {
        // ================================================================== copies: four warps for K, four for V
        // A unit's rows go round the four warps in fours, so that its copies are under way soon after its place is free.  Warps of their
        // own for K and for V, because each waits for places that the other's MMAs free.
        // K with ROWS: an elected lane has the TMA unit gather 4 rows x 128 bytes at a time; otherwise eight lanes copy 128 bytes of a row.
        const bool is_v = warp >= LP_V_WARP0;
        const int w = warp - (is_v ? LP_V_WARP0 : LP_K_WARP0);
        int unit_slot = 0;
        uint32_t unit_ph = 1u;
        const uint32_t even = rank & ~1u;
        auto next_place = [&]() {
            if (++unit_slot == (is_v ? LP_VU : LP_KU)) { unit_slot = 0; unit_ph ^= 1u; }
        };
        // n_rows rows of a tile from row0 on, n_atoms atoms from atom0 on, each of n_rows x 128 bytes
        auto fill = [&](int slot, uint64_t* full, uint64_t* empty, uint32_t dst, int row0, int atom0, auto n_rows, auto n_atoms) {
            ok = wait_warp(empty, unit_ph);
            if (!ok) return;
            if (ROWS && !is_v) {
                const uint32_t bar = mapa_shared(smem_u32(full), even);
                if (elect_one()) {
                    if (c == 0u && w == 0) mbar_expect_tx(smem_u32(full), 2 * n_atoms * n_rows * 128);
#pragma unroll
                    for (int i = 0; i < n_rows / 4 / LP_COPY_WARPS; ++i) {
                        const int q = w + LP_COPY_WARPS * i;
                        const int4 r = *reinterpret_cast<const int4*>(&sh->row[slot][row0 + 4 * q]);
#pragma unroll
                        for (int a = 0; a < n_atoms; ++a)
                            tma_gather4_pair(dst + q * 512 + a * n_rows * 128, &tmap_pool, (atom0 + a) * 64, r.x, r.y, r.z, r.w, bar);
                    }
                }
                __syncwarp();
            } else {
#pragma unroll
                for (int i = 0; i < n_rows / 4 / LP_COPY_WARPS; ++i) {
                    const int r = 4 * (w + LP_COPY_WARPS * i) + (lane >> 3);
                    const int64_t off = sh->offset[slot][row0 + r];
                    const uint32_t bytes = off != INT64_MIN ? 16u : 0u;            // rows that are not there read as zeros
                    const unsigned char* src = reinterpret_cast<const unsigned char*>(p.pool) + (bytes != 0u ? off : 0) + atom0 * 128 + (lane & 7) * 16;
                    const uint32_t d = dst + static_cast<uint32_t>(r * 128 + (((lane & 7) ^ (r & 7)) << 4));
#pragma unroll
                    for (int a = 0; a < n_atoms; ++a) cp_async16(d + a * n_rows * 128, src + a * 128, bytes);
                }
                cp_async_arrive(smem_u32(full));
            }
            next_place();
        };
        // queries of this CTA's heads, token `it`: atoms 0-5 through the ring, atoms 6-8 to their place (warp 0; plain copies of boxes)
        auto fill_q = [&](int it) {
            const int y = (cid + it * n_clusters) * LP_HEADS + LP_OWN * static_cast<int>(c);
            for (int a = 0; a < LP_QPARTS; ++a) {
                uint64_t *const full = &sh->k_full[unit_slot], *const empty = &sh->k_empty[unit_slot];
                // ROWS: only the warp that fills the unit waits for its place.  The unit lands and its place is freed again without the others, so that
                // one of them that looked late would meet the parity of the phase before and wait for good.  They need no wait: the places of the
                // next two units were freed after this one, and they wait for those.
                if (!ROWS || w == 0) ok = wait_warp(empty, unit_ph);
                if (!ok) return;
                if (w == 0 && elect_one()) {
                    if constexpr (!ROWS) mbar_expect_only(smem_u32(full), LP_K_BYTES);
                    else if (c == 0u) mbar_expect_tx(smem_u32(full), 2 * LP_K_BYTES);
                    const uint32_t dst = smem_u32(k_smem) + static_cast<uint32_t>(unit_slot * LP_K_BYTES), bar = ROWS ? mapa_shared(smem_u32(full), even) : mapa_shared(smem_u32(full), rank);
                    for (int i = 0; i < 3; ++i) tma_load_2d_pair(dst + i * LP_ATOM_BYTES, &tmap_q, (3 * a + i) * 64, y, bar);
                }
                __syncwarp();
                if constexpr (!ROWS) cp_async_arrive(smem_u32(full));
                next_place();
            }
            if (w != 0) return;
            ok = it == 0 || wait_warp(&sh->q_free, static_cast<uint32_t>(it - 1) & 1u);
            if (ok && elect_one()) {
                if (c == 0u) mbar_expect_tx(smem_u32(&sh->q_full), 2 * LP_Q_BYTES);
                for (int i = 0; i < 3; ++i) tma_load_2d_pair(smem_u32(q_smem) + i * LP_ATOM_BYTES, &tmap_q, (6 + i) * 64, y, mapa_shared(smem_u32(&sh->q_full), even));
            }
            __syncwarp();
        };
        int tile = 0, tok = 0;
        for (int s = 0; s < total && ok; ++s) {
            const int slot = s % LP_RROWS;
            if (!is_v && tile == 0) fill_q(tok);
            ok = ok && wait_warp(&sh->r_full[slot], static_cast<uint32_t>(s / LP_RROWS) & 1u);
            if (!is_v) {
                for (int u = 0; u < LP_KPARTS && ok; ++u)
                    fill(slot, &sh->k_full[unit_slot], &sh->k_empty[unit_slot], smem_u32(k_smem) + static_cast<uint32_t>(unit_slot * LP_K_BYTES), LP_OWN * static_cast<int>(c),
                         u == 0 ? 6 : 3 * (u - 1), std::integral_constant<int, LP_OWN>(), std::integral_constant<int, 3>());
            } else {
                for (int v = 0; v < LP_VPARTS && ok; ++v)
                    fill(slot, &sh->v_full[unit_slot], &sh->v_empty[unit_slot], smem_u32(v_smem) + static_cast<uint32_t>(unit_slot * LP_V_BYTES), LP_VROWS * v,
                         4 * static_cast<int>(c), std::integral_constant<int, LP_VROWS>(), std::integral_constant<int, 4>());
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh->r_empty[slot]));
            if (++tile == n_tiles) { tile = 0; ++tok; }
        }
        // Nothing may be on its way into shared memory when the CTA leaves, also after a wait somewhere gave up.  Copies of this thread by
        // cp.async are waited for as such.  Rows and queries by the TMA unit have landed once the MMAs have freed every place that was filled;
        // where those no longer come, the limit of one such wait, a quarter of a second, has passed since the last was asked for.
        cp_async_wait_all();
        for (int u = 0; !is_v && u < LP_KU && wait_warp(&sh->k_empty[unit_slot], unit_ph); ++u) next_place();
    } else {
        // ================================================================== heads: softmax, output
        // Thread = head, half of the tile's keys (the lane's half of tensor memory) and one of its two quarters; of O, half of the lane's
        // value dims.  A token's output is written after the softmax of the next token's first tile, so that the MMAs run on across tokens.
        const int ln = (warp & 3) * 32 + lane, h = ln & (LP_OWN - 1), half = ln / LP_OWN, ch = warp >> 2, part = 2 * half + ch;
        const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const float neg_inf = __int_as_float(0xff800000);
        const bool out_al32 = (reinterpret_cast<uint64_t>(p.out) & 31u) == 0u;
        uint64_t* x_full = &sh->x_full[warp & 1];          // shared by the four warps of the same heads
        const uint32_t p_row = smem_u32(p_smem) + static_cast<uint32_t>(half * LP_ATOM_BYTES + h * 128);
        uint32_t n_x = 0;                                  // exchanges so far
        auto token = [&](int it) { return cid + it * n_clusters; };
        auto wait_pv = [&](int tile) { return wait_warp(&sh->pv_done[tile & 1], static_cast<uint32_t>(tile >> 1) & 1u); };
        // exchange with the other three quarters: what was left in shared memory before is visible to them after
        auto exchange = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(x_full));
            ok = wait_warp(x_full, n_x++ & 1u);
        };
        // output of token `it` (reference maximum m_ref): normalise, round to bf16.  Its last P.V is complete, its sums are visible.
        auto write_out = [&](int it, float m_ref) {
            const float(&l)[4][LP_OWN] = sh->l[it & 1];
            const float l_sum = (l[0][h] + l[1][h]) + (l[2][h] + l[3][h]);
            const bool have_o = __any_sync(0xffffffffu, l_sum != 0.f);  // some key of one of these heads counts, be it as NaN
            const float inv = l_sum != 0.f ? 1.f / l_sum : 0.f;
            uint16_t* orow = p.out + lp_out_offset(token(it), c, ln) + ch * 128;
            float* mo = reinterpret_cast<float*>(k_smem);               // SPLIT: nothing reads the rings any more
            if (SPLIT && part == 0) { sh->split_m[h] = m_ref; sh->split_l[h] = l_sum; }
#pragma unroll 1
            for (int cc = 0; cc < 4; ++cc) {
                uint32_t o[32];
                if (have_o) {
                    tmem_ld32_wait(lane_addr + LP_COL_O + ch * 128 + cc * 32, o);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) o[j] = 0u;
                }
                if constexpr (SPLIT) {                                  // left for the merge
#pragma unroll
                    for (int v = 0; v < 8; ++v)
                        *reinterpret_cast<uint4*>(mo + ((ch * 32 + cc * 8 + v) * LP_TILE + ln) * 4) = make_uint4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
                } else {
                    if (cc == 3) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) arrive_even(&sh->o_free);
                    }
                    uint32_t w[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) w[j] = lp_pack_bf16x2(__uint_as_float(o[2 * j]) * inv, __uint_as_float(o[2 * j + 1]) * inv);
                    if (out_al32) {      // whole 32-byte sectors per thread: half the store instructions and transactions
                        st_global_v8(orow + cc * 32, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
                        st_global_v8(orow + cc * 32 + 16, w[8], w[9], w[10], w[11], w[12], w[13], w[14], w[15]);
                    } else {
                        uint4* dst = reinterpret_cast<uint4*>(orow + cc * 32);
#pragma unroll
                        for (int v = 0; v < 4; ++v) dst[v] = make_uint4(w[4 * v], w[4 * v + 1], w[4 * v + 2], w[4 * v + 3]);
                    }
                }
            }
            if (!SPLIT && p.lse != nullptr && part == 0)
                p.lse[static_cast<int64_t>(token(it)) * LP_HEADS + LP_OWN * c + h] = l_sum != 0.f ? (m_ref + log2f(l_sum)) * 0.6931471805599453f : neg_inf;
        };
        int gi = 0;                 // tiles done so far, over all tokens
        float m_ref = neg_inf, m_prev = neg_inf;
        for (int it = 0; it < n_my && ok; ++it) {
        m_prev = m_ref;             // the token before, whose output is still to be written
        m_ref = neg_inf;            // reference maximum (scaled, log2 domain) the exponentials are taken against, the same in all four warps
        float l_sum = 0.f;          // over this quarter of the keys
        for (int i = 0; i < n_tiles; ++i, ++gi) {
            const uint32_t ph = static_cast<uint32_t>(gi) & 1u;
            const int slot = gi % LP_RROWS;
            ok = wait_warp(&sh->r_full[slot], static_cast<uint32_t>(gi / LP_RROWS) & 1u) && wait_warp(&sh->s_full, ph);
            if (!ok) break;
            tc_fence_after();
            float2 x[16];                   // logits of keys 2j, 2j+1 of the quarter
            {
                uint32_t r[32];
                tmem_ld32_wait(lane_addr + LP_COL_S + ch * 32, r);
#pragma unroll
                for (int j = 0; j < 16; ++j) x[j] = make_float2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
            }
            const uint32_t vm = sh->vmask[slot][part];
            // the logits are in registers: the next tile's may be computed
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                arrive_even(&sh->s_free);
                mbar_arrive(smem_u32(&sh->r_empty[slot]));
            }
            if (vm != 0xffffffffu) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    x[j].x = ((vm >> (2 * j)) & 1u) ? x[j].x : neg_inf;
                    x[j].y = ((vm >> (2 * j + 1)) & 1u) ? x[j].y : neg_inf;
                }
            }
            float tile_max;
            {
                float mx[4] = {neg_inf, neg_inf, neg_inf, neg_inf};
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                    mx[0] = fmax3(mx[0], x[j].x, x[j].y); mx[1] = fmax3(mx[1], x[j + 1].x, x[j + 1].y);
                    mx[2] = fmax3(mx[2], x[j + 2].x, x[j + 2].y); mx[3] = fmax3(mx[3], x[j + 3].x, x[j + 3].y);
                }
                tile_max = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            }
            // the other quarters' maxima (two places, by parity: the others have read the last ones before they wrote their own)
            float(&shared_max)[4][LP_OWN] = sh->mx[n_x & 1u];
            shared_max[part][h] = tile_max;
            exchange();
            if (!ok) break;
            tile_max = fmaxf(fmaxf(shared_max[0][h], shared_max[1][h]), fmaxf(shared_max[2][h], shared_max[3][h])) * p.scale_log2e;      // softmax_scale > 0
            // move the reference maximum only when this tile exceeds it by more than 2^8 (or on first use)
            float corr = 1.f;
            bool moved = false;
            if (tile_max > m_ref + 8.f) {
                moved = m_ref != neg_inf;
                corr = moved ? lp_exp2(m_ref - tile_max) : 1.f;
                l_sum *= corr;
                m_ref = tile_max;
            }
            if (__any_sync(0xffffffffu, moved)) {
                // rescale this thread's part of O in tensor memory: the previous tile's P.V must have completed first
                ok = wait_pv(gi - 1);
                if (!ok) break;
                tc_fence_after();
#pragma unroll 1
                for (int cc = 0; cc < 4; ++cc) {
                    uint32_t o[32];
                    tmem_ld32_wait(lane_addr + LP_COL_O + ch * 128 + cc * 32, o);
#pragma unroll
                    for (int j = 0; j < 32; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * corr);
                    tmem_st32_wait(lane_addr + LP_COL_O + ch * 128 + cc * 32, o);
                }
            }
            const float neg_m = (m_ref == neg_inf) ? 0.f : -m_ref;
            // P is rounded to bf16 (one pack instruction per pair); the row sum adds the very same rounded values, so the
            // normalisation stays consistent and the log-sum-exp is not biased
            uint32_t pk[16];
            float2 ts[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            const float2 sc2 = make_float2(p.scale_log2e, p.scale_log2e), nm2 = make_float2(neg_m, neg_m);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const float2 e = ffma2(x[j], sc2, nm2);
                pk[j] = lp_pack_bf16x2(lp_exp2(e.x), lp_exp2(e.y));       // low half = bf16(p of key 2j), high half = bf16(p of key 2j+1)
                ts[j & 3] = fadd2(ts[j & 3], make_float2(__uint_as_float(pk[j] << 16), __uint_as_float(pk[j] & 0xffff0000u)));
            }
            const float2 t4 = fadd2(fadd2(ts[0], ts[1]), fadd2(ts[2], ts[3]));
            l_sum += t4.x + t4.y;
            // P has two buffers: the P.V of two tiles ago must have completed
            if (gi > 1) {
                ok = wait_pv(gi - 2);
                if (!ok) break;
                tc_fence_after();
            }
#pragma unroll
            for (int v = 0; v < 4; ++v)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(p_row + ph * LP_P_BYTES + static_cast<uint32_t>(((4 * ch + v) ^ (h & 7)) << 4)), "r"(pk[4 * v]),
                             "r"(pk[4 * v + 1]), "r"(pk[4 * v + 2]), "r"(pk[4 * v + 3])
                             : "memory");
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_even(&sh->p_full[ph]);
            if (i == 0 && it > 0) {                               // (the exchange above made the sums visible)
                ok = wait_pv(gi - 1);
                if (!ok) break;
                tc_fence_after();
                write_out(it - 1, m_prev);
            }
        }
        if (!ok) break;
        sh->l[it & 1][part][h] = l_sum;      // the place was read two tokens ago
        }
        if (ok && n_my > 0) {
            exchange();
            ok = ok && wait_pv(gi - 1);
            tc_fence_after();
            if (ok) write_out(n_my - 1, m_ref);
        }
    }
    if (!ok && lane == 0) report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if constexpr (SPLIT) {
        cluster_sync_all();         // every pair's output lies in its shared memory
        if (!start_abort && n_my > 0) {
            const uint32_t o_addr = smem_u32(k_smem), m_addr = smem_u32(sh->split_m), l_addr = smem_u32(sh->split_l);
            const int sp = static_cast<int>(rank >> 1);
            static_assert(LP_MAX_SPLIT == 8, "cases below");
            switch (n_split) {
                case 2: lp_merge_splits<2>(p, cid, sp, c, o_addr, m_addr, l_addr); break;
                case 3: lp_merge_splits<3>(p, cid, sp, c, o_addr, m_addr, l_addr); break;
                case 4: lp_merge_splits<4>(p, cid, sp, c, o_addr, m_addr, l_addr); break;
                case 5: lp_merge_splits<5>(p, cid, sp, c, o_addr, m_addr, l_addr); break;
                case 6: lp_merge_splits<6>(p, cid, sp, c, o_addr, m_addr, l_addr); break;
                case 7: lp_merge_splits<7>(p, cid, sp, c, o_addr, m_addr, l_addr); break;
                case 8: lp_merge_splits<8>(p, cid, sp, c, o_addr, m_addr, l_addr); break;
            }
        }
    }
    cluster_sync_all();   // no CTA leaves, or gives tensor memory back, while another may still write into its shared memory, arrive on its barriers or use the pair's
    if (warp == LP_QK_WARP) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

bool sparse_attn_latent_tc_supported(int M, int H_q, int d_qk, const void* k_pool, const void* v_pool, int64_t page_stride,
                                     int64_t tok_stride, int n_kv_heads, int d_v, int k) {
    if (H_q != LP_HEADS || d_qk != LP_DQK || d_v != LP_DV || n_kv_heads != 1 || k_pool != v_pool) return false;
    if ((page_stride % 8) != 0 || (tok_stride % 8) != 0 || tok_stride < LP_DQK) return false;
    if (M > (1 << 30) / LP_HEADS || k <= 0) return false;
    return true;
}

static cudaLaunchConfig_t lp_occupancy_config(int cluster_size, int n_clusters, size_t smem, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(cluster_size) * n_clusters);
    cfg.blockDim = dim3(LP_THREADS);
    cfg.dynamicSmemBytes = smem;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = cluster_size;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// n[s] = clusters of 2 s CTAs the device keeps resident at once (one CTA per SM), 0 where it takes none.  A property of the
// device, asked for on its first call; the kernels' attributes are set once in every context.
static int lp_resident_clusters(int dev, size_t smem, int (&n)[LP_MAX_SPLIT + 1]) {
    constexpr int MAX_DEVICES = 64;
    static std::mutex mu;
    static int known[MAX_DEVICES][LP_MAX_SPLIT + 1] = {};
    if (dev < 0 || dev >= MAX_DEVICES) return JANUS_ERR_UNSUPPORTED;
    static once_per_context attributes;
    JANUS_CUDA_CHECK(attributes.run([&] {
        const int bytes = static_cast<int>(smem);
        cudaError_t e = cudaSuccess;
        auto larger = [&](auto kernel) { if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); };
        auto wider = [&](auto kernel) { if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1); };
        larger(sparse_attn_latent_pair_kernel<false, false>);
        larger(sparse_attn_latent_pair_kernel<false, true>);
        larger(sparse_attn_latent_pair_kernel<true, false>);
        larger(sparse_attn_latent_pair_kernel<true, true>);
        wider(sparse_attn_latent_pair_kernel<true, false>);
        wider(sparse_attn_latent_pair_kernel<true, true>);
        return e;
    }));
    std::lock_guard<std::mutex> lock(mu);
    int (&k)[LP_MAX_SPLIT + 1] = known[dev];
    if (k[1] == 0) {
        for (int s = LP_MAX_SPLIT; s >= 1; --s) {
            cudaLaunchAttribute attr;
            const cudaLaunchConfig_t cfg = lp_occupancy_config(2 * s, 148, smem, &attr);
            const cudaError_t e = s > 1 ? cudaOccupancyMaxActiveClusters(&k[s], sparse_attn_latent_pair_kernel<true, true>, &cfg)
                                        : cudaOccupancyMaxActiveClusters(&k[s], sparse_attn_latent_pair_kernel<false, true>, &cfg);
            if (e != cudaSuccess) {
                (void)cudaGetLastError();
                k[s] = 0;
            }
        }
        if (k[1] <= 0) {
            int sms = 0;
            JANUS_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
            k[1] = sms > 2 ? sms / 2 : 1;
        }
    }
    for (int s = 0; s <= LP_MAX_SPLIT; ++s) n[s] = k[s];
    return JANUS_OK;
}

int launch_sparse_attn_latent_tc(const void* q, int M, const void* pool, int64_t page_stride, int64_t tok_stride, const int32_t* idx, int k,
                                 int page_size, const int32_t* page_table, int64_t n_logical_pages, const int64_t* table_offsets,
                                 float softmax_scale, void* out, float* lse, int32_t* dev_status, cudaStream_t stream) {
    LpParams p;
    p.q = static_cast<const uint16_t*>(q);
    p.pool = static_cast<const uint16_t*>(pool);
    p.page_stride = page_stride;
    p.tok_stride = tok_stride;
    p.idx = idx;
    p.k = k;
    p.page_size = page_size;
    p.page_shift = -1;
    if ((page_size & (page_size - 1)) == 0) {
        p.page_shift = 0;
        while ((1 << p.page_shift) < page_size) ++p.page_shift;
    }
    p.page_table = page_table;
    p.n_logical_pages = n_logical_pages;
    p.table_offsets = table_offsets;
    p.scale_log2e = softmax_scale * 1.4426950408889634f;
    p.out = static_cast<uint16_t*>(out);
    p.lse = lse;
    p.M = M;
    p.dev_status = dev_status;
    constexpr size_t smem = LP_SMEM_TILES + 2 * LP_P_BYTES + LP_Q_BYTES + sizeof(LpShared);
    static_assert(smem <= 227 * 1024, "shared memory");
    int dev = 0;
    JANUS_CUDA_CHECK(cudaGetDevice(&dev));
    int n_resident[LP_MAX_SPLIT + 1];
    const int rc = lp_resident_clusters(dev, smem, n_resident);
    if (rc != JANUS_OK) return rc;
    // A pair takes 1.5 us per tile of 128 keys, 8.5 us around them and, with more tokens than pairs, 0.6 us a token.  While the tokens are
    // few, clusters of 2 n CTAs share a token's tiles; start and merge, whose 128 KB per CTA cross the SM-to-SM network, make that
    // 10.2 + 0.66 n us.  The n with the least time is taken.  Measured at 2048 keys: 1 token 32.4 us with one pair, 18.5 with four, 18.6
    // with eight; 19 tokens 32.8, 25.8 and 22.8 with one, two and three (22 clusters of six CTAs are resident at once; four take two
    // waves, 38); 30 tokens 33.2, 25.4; 512 keys: 14.5 with one pair, 14.0 with four; 256 keys 11.5 and, with two, 13.0.
    const int all_tiles = (k + LP_TILE - 1) / LP_TILE;
    int split = 1;
    double best = 0.;
    for (int n = 1; n <= LP_MAX_SPLIT && n <= all_tiles; ++n) {
        if (n_resident[n] <= 0) break;
        const int waves = (M + n_resident[n] - 1) / n_resident[n];
        const double tiles = ((all_tiles + n - 1) / n) * 1.5;
        const double t = n > 1 ? waves * (tiles + 10.2 + 0.66 * n) : 8.5 + waves * (tiles + 0.6);
        if (n == 1 || t < best) { best = t; split = n; }
    }
    const int n_clusters = split > 1 ? M : (M < n_resident[1] ? M : n_resident[1]);     // one pair per cluster: persistent over tokens
    const dim3 grid(static_cast<unsigned>(2 * split) * n_clusters);
    // Rows are gathered by number where the distance of the pages is a multiple of that of the tokens, as it is in any pool without
    // padding between pages (740 x 2048: 322 us; by address 333).
    CUtensorMap map = {}, map_q;
    if (!make_tmap_2d_sw128(&map_q, q, 2, static_cast<uint64_t>(M) * LP_HEADS, LP_DQK, static_cast<uint64_t>(LP_DQK) * 2, LP_OWN, 64)) return JANUS_ERR_CUDA;
    const bool rows = page_stride >= 0 && page_stride % tok_stride == 0 &&
                      make_tmap_2d_sw128(&map, pool, 2, 0x7fffffffu, LP_DQK, static_cast<uint64_t>(tok_stride) * 2, 1, 64);
    const int cluster = 2 * split;
    cudaError_t e;
    if (split > 1) e = rows ? launch_kernel(sparse_attn_latent_pair_kernel<true, true>, grid, LP_THREADS, smem, stream, cluster, map_q, map, p)
                            : launch_kernel(sparse_attn_latent_pair_kernel<true, false>, grid, LP_THREADS, smem, stream, cluster, map_q, map, p);
    else e = rows ? launch_kernel(sparse_attn_latent_pair_kernel<false, true>, grid, LP_THREADS, smem, stream, cluster, map_q, map, p)
                  : launch_kernel(sparse_attn_latent_pair_kernel<false, false>, grid, LP_THREADS, smem, stream, cluster, map_q, map, p);
    JANUS_CUDA_CHECK(e);
    return JANUS_OK;
}

}  // namespace janus
