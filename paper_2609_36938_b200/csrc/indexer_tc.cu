// Tensor-core indexer (Eq. 1, Sec. 2.2, scoring part) for sm_100a:
//     scores[t,s] = k_scale[s] * sum_h (w[t,h]*q_scale[h]) * relu(<q[t,h,:], k[s,:]>) + row_bias[t]*col_bias[s]
//
// Mapping.  The dense contraction is K . Q^T with a reduction depth of only D_I, followed by a ReLU and a
// weighted sum over heads for every accumulator.  Keys go on the MMA M axis (128 keys -> the 128 TMEM lanes)
// and (token, head) pairs on the N axis (256 TMEM columns = 256/H_I tokens x H_I heads), so that after a
// tcgen05.ld every epilogue thread owns one key, holds all heads of a token in its own registers, and reduces
// over heads with no cross-lane traffic; a warp's 32 keys are 32 consecutive floats of one score row.
//
// One CTA keeps NQ query sub-tiles (NQ*256 (token,head) rows, 128 KB) stationary in shared memory and streams
// 128-key tiles past them through a TMA ring; each key tile feeds NQ MMAs (128 x 256 x D_I), whose fp32
// accumulators alternate between the two 256-column halves of tensor memory, so the epilogue of one
// overlaps the MMA of the next.  Warp roles: warp 0 issues TMA, warp 1 issues MMA (one thread each) and owns
// the TMEM allocation, the other warps are two epilogue groups (one per TMEM half) of eight warps (two per TMEM lane
// quadrant, each reducing half of the slot's columns): with four epilogue warps per scheduler one warp's wait for its
// tensor-memory load or its weights is covered by the others.
//
// The launch is persistent: the visible (token group, key tile) pairs, group by group, are cut into as many contiguous ranges of equal
// cost as CTAs are resident, and a CTA walks its range in segments of one group each.  The key ring, the TMEM slots and
// their barriers run on across segments; the queries and weights are replaced, which costs about three quarters of a tile's time,
// once or twice per CTA in a long call.  A grid of fixed chunks left waves unfilled (in loops of this kernel alone): 2048 rows x 34816 keys
// 64 x 128 bf16 901 -> 857 us, 777 x 20788 of 32 heads 121 -> 114, 1024 x 17408 FP8 183 -> 172.  4096 x 135168 FP8, which is on the power limit,
// takes 5.5 ms either way, and where the chunks happened to fill their waves (777 x 66777 bf16) they were 3 % faster.  Small launches give
// every CTA tiles of one group only (MULTI = false).  256 rows x 4352 keys of 4 heads 18.6 -> 8.0 us, with half the sub-tiles per CTA.
// Every wait is bounded; on a timeout the CTA reports JANUS_DEV_WAIT_TIMEOUT and winds down normally.
#include "indexer_tc.cuh"

namespace janus {

constexpr int TC_N = 256;           // (token, head) rows per MMA = MMA N
constexpr int TC_THREADS = 576;     // 1 TMA warp + 1 MMA warp + 16 epilogue warps, two per TMEM lane quadrant and slot, each takes half the columns
constexpr int TC_MAX_STAGES = 6;

struct TcParams {
    const float* w;
    const float* q_scale;
    int64_t q_scale_stride_tok;
    const float* k_scale;
    const float* row_bias;
    const float* col_bias;
    float* scores;
    int64_t ld;
    int64_t n_keys;
    int64_t q_pos0;
    int M, H, causal;
    int n_tiles;          // ceil(n_keys / 128)
    int n_groups;         // token groups
    int tiles_per_cta;    // without MULTI: CTA (x, y) has the tiles x * tiles_per_cta .. of group y
    int nq;               // query sub-tiles per CTA
    int atoms;            // 128-byte swizzle atoms per row (row bytes / 128)
    int stages;           // key ring depth
    int32_t* dev_status;
};

// Candidate mode (fused indexer + top-k): instead of storing scores, every visible score >= thr[t] is appended to row t's
// candidate list; `scores` is unused.  A kernel parameter of its own: the score-matrix kernel's code does not depend on it.
struct TcCandParams {
    const float* thr;     // [M] per-row thresholds
    int32_t* cand_cnt;    // [M] candidates appended so far (may exceed cand_cap: only the first cand_cap are stored)
    int2* cand;           // [M, cand_cap] (score bits, key index)
    int cand_cap;
    // keys are FP4 E2M1, two per byte; the TMA expands 16 of them into the first 8 bytes of every 16-byte shared-memory chunk, which
    // is the layout the f8f6f4 MMA expects for 4-bit operands
    int k_fp4;
};

// Even shares (MULTI): where each CTA's range begins, (token group, key tile).  Made on the host and read from constant memory:
// found by the device it was not known to be uniform, which made the issuing threads' loops up to 8 % slower.  Its 1.2 KB make
// a launch about 0.5 us longer, so small launches do without.
struct TcSchedule {
    int2 first[TC_MAX_CTAS];
    uint16_t less[TC_MAX_CTAS];       // tiles that CTA c's range is shorter than the longest
    int longest;
};
struct TcNoSchedule {};
template <bool TABLE> struct TcScheduleOf { using type = TcSchedule; };
template <> struct TcScheduleOf<false> { using type = TcNoSchedule; };

// Candidate mode stages appends in shared memory: each epilogue warp owns, for each of its (at most TC_CAND_TPW) tokens,
// TC_CAND_SLOTS (score, key) slots, and moves a full set to the row's global list with one counter update.
constexpr int TC_CAND_TPW = 4;
constexpr int TC_CAND_SLOTS = 32;
constexpr int TC_CAND_STAGE_BYTES = 16 * TC_CAND_TPW * TC_CAND_SLOTS * static_cast<int>(sizeof(int2));

struct TcBarriers {
    uint64_t k_full[TC_MAX_STAGES];
    uint64_t k_empty[TC_MAX_STAGES];
    uint64_t tmem_full[2];
    uint64_t tmem_empty[2];
    uint64_t mma_drain;       // abort path only: every MMA issued so far has completed
    uint32_t tmem_base;
    int aborted;
};

// Key tiles visible to some token of group g (tpc tokens per group) under the causal mask.
__host__ __device__ __forceinline__ int tc_causal_tiles(int M, int64_t q_pos0, int n_tiles, int tpc, int g) {
    const int64_t t_hi = (static_cast<int64_t>(g) + 1) * tpc < M ? (static_cast<int64_t>(g) + 1) * tpc - 1 : M - 1;
    const int64_t v = (q_pos0 + t_hi) / TC_KEYS + 1;
    return v < n_tiles ? static_cast<int>(v) : n_tiles;
}
__host__ __device__ __forceinline__ int tc_visible_tiles(const TcParams& p, int tpc, int g) {
    return p.causal ? tc_causal_tiles(p.M, p.q_pos0, p.n_tiles, tpc, g) : p.n_tiles;
}

// Score-matrix mode: the keys in tiles that no token of a row's group may see are -inf.  The rows are shared out over all
// epilogue warps of the launch, before their first accumulators are ready.  (A function of its own: inlined, it cost the
// epilogue spilled registers.)
__device__ __noinline__ void fill_masked_tails(float* scores, int64_t ld, int M, int64_t n_keys, int64_t q_pos0, int n_tiles, int tpc, int first, int end,
                                               int step, int lane) {
    const float neg_inf = __int_as_float(0xff800000);
    const float4 fill = make_float4(neg_inf, neg_inf, neg_inf, neg_inf);
    for (int t = first; t < end; t += step) {
        float* row = scores + static_cast<int64_t>(t) * ld;
        const int64_t from = static_cast<int64_t>(tc_causal_tiles(M, q_pos0, n_tiles, tpc, t / tpc)) * TC_KEYS;
        for (int64_t c = from + 4 * lane; c + 3 < n_keys; c += 128) *reinterpret_cast<float4*>(row + c) = fill;
        const int64_t tail = n_keys & ~int64_t(3);
        if (tail >= from && tail + lane < n_keys) row[tail + lane] = neg_inf;
    }
}

// A CTA's range, one token group at a time: key tiles [tb, te) of group `g`.  Without MULTI there is one.
template <bool MULTI>
struct TcSegments {
    const TcParams& p;
    int tpc, g, tb, te, left;
    bool first;
    __device__ __forceinline__ TcSegments(const TcParams& p_, int tpc_, int g0, int t0, int work)
        : p(p_), tpc(tpc_), g(g0), tb(t0), te(t0), left(work), first(true) {}
    __device__ __forceinline__ bool next() {
        if (left <= 0) return false;
        if constexpr (!MULTI) {
            te = tb + left;
            left = 0;
            return true;
        } else {
            int tiles;
            do {
                if (!first) { ++g; tb = 0; }
                first = false;
                tiles = tc_visible_tiles(p, tpc, g);
            } while (tiles <= tb);
            te = min(tiles, tb + left);
            left -= te - tb;
            return true;
        }
    }
};

template <int H, bool FP8, bool CAND, bool MULTI>
__global__ void __launch_bounds__(TC_THREADS, 1)
indexer_tc_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k, const TcParams p, const TcCandParams cp,
                  const __grid_constant__ typename TcScheduleOf<MULTI>::type sched) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int TPS = TC_N / H;                      // tokens per query sub-tile
    const int atoms = p.atoms, nq = p.nq, stages = p.stages;
    const int q_sub_bytes = atoms * TC_N * 128;        // one query sub-tile
    const int k_stage_bytes = atoms * TC_KEYS * 128;   // one key tile
    unsigned char* q_smem = smem;
    unsigned char* k_smem = smem + nq * q_sub_bytes;
    float* ws = reinterpret_cast<float*>(k_smem + stages * k_stage_bytes);   // [nq*256] w * q_scale, column order
    float* rbs = ws + nq * TC_N;                                             // [nq*TPS] row_bias of the segment's tokens
    float* thrs = rbs + nq * TPS;                                            // [nq*TPS] candidate thresholds of the segment's tokens
    int2* cstage = reinterpret_cast<int2*>(thrs + nq * TPS);                 // candidate staging (candidate mode only)
    TcBarriers* bars = reinterpret_cast<TcBarriers*>(reinterpret_cast<unsigned char*>(cstage) + (CAND ? TC_CAND_STAGE_BYTES : 0));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NEPI = TC_THREADS - 64;                         // epilogue threads
    const int tpc = nq * TPS;                                   // tokens per group

    if ((smem_u32(smem) & 1023u) != 0u) {   // swizzled tiles need 1024-byte alignment
        grid_wait();
        if (threadIdx.x == 0) report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT);
        return;
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) { mbar_init(smem_u32(&bars->k_full[s]), 1); mbar_init(smem_u32(&bars->k_empty[s]), 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(smem_u32(&bars->tmem_full[s]), 1); mbar_init(smem_u32(&bars->tmem_empty[s]), 8); }
        mbar_init(smem_u32(&bars->mma_drain), 1);
        fence_mbar_init();
        prefetch_tensormap(&tmap_q);
        prefetch_tensormap(&tmap_k);
        grid_wait();
        // an earlier CTA of this launch gave up on a wait: this one starts no work on a broken pipeline.  One thread reads the
        // status word and the whole CTA follows that one reading (a second reading could differ and split the roles).
        bars->aborted = (p.dev_status != nullptr && *reinterpret_cast<volatile int32_t*>(p.dev_status) == JANUS_DEV_WAIT_TIMEOUT) ? 1 : 0;
    }
    grid_wait();
    // per-column weights (w * q_scale) and per-token bias factors and thresholds of group g, by threads first, first + step, ..
    auto load_weights = [&](int g, int first, int step) {
        const int t0 = g * tpc;
        for (int n = first; n < nq * TC_N; n += step) {
            const int t = t0 + n / H, h = n % H;
            float v = 0.f;
            if (t < p.M) {
                v = p.w[static_cast<int64_t>(t) * H + h];
                if (FP8) v *= p.q_scale[static_cast<int64_t>(t) * p.q_scale_stride_tok + h];
            }
            ws[n] = 0.5f * v;      // the epilogue forms 2 * relu
        }
        for (int n = first; n < tpc; n += step) {
            rbs[n] = (p.row_bias != nullptr && t0 + n < p.M) ? p.row_bias[t0 + n] : 0.f;
            if constexpr (CAND) thrs[n] = t0 + n < p.M ? cp.thr[t0 + n] : 0.f;
        }
    };
    // ---- this CTA's range: n_work tiles from tile `tile0` of group `g0` on
    int g0, tile0, n_work;
    if constexpr (!MULTI) {
        g0 = blockIdx.y;
        tile0 = blockIdx.x * p.tiles_per_cta;
        load_weights(g0, threadIdx.x, TC_THREADS);
        n_work = min(tc_visible_tiles(p, tpc, g0) - tile0, p.tiles_per_cta);
        if (n_work <= 0) return;
    } else {
        g0 = sched.first[blockIdx.x].x;
        tile0 = sched.first[blockIdx.x].y;
        n_work = sched.longest - sched.less[blockIdx.x];
        load_weights(g0, threadIdx.x, TC_THREADS);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&bars->tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = bars->tmem_base;
    volatile int* aborted = &bars->aborted;
    const bool run = *aborted == 0;       // read once, after the barrier: the same value in every thread

    if (!run) {
        // nothing to do: tensor memory goes back below
    } else if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const int atom_elems = FP8 ? 128 : 64;
            int issued = 0;
            int s = 0;                 // ring stage and its phase bit, advanced per tile
            uint32_t ph = 0;
            bool ok = true;
            // The queries of a segment are counted on the barrier of its first key tile, so the MMA warp needs to know nothing of
            // segments.  They may be replaced when the previous segment's last key tile has been released: every MMA up to it has
            // completed then.
            TcSegments<MULTI> seg(p, tpc, g0, tile0, n_work);
            int left = 0;                               // tiles of this segment still to load
            int q_at = -1;                              // the queries are loaded when `left` has come down to this
            int key_row = 0;
            uint32_t q_bar = 0, free_bar = 0, free_ph = 0;
            auto load_q = [&]() {
                for (int j = 0; j < nq; ++j)
                    for (int a = 0; a < atoms; ++a)
                        tma_load_2d(smem_u32(q_smem + j * q_sub_bytes + a * TC_N * 128), &tmap_q, a * atom_elems, (seg.g * tpc + j * TPS) * H, q_bar);
            };
            const uint32_t tile_bytes = static_cast<uint32_t>((FP8 && cp.k_fp4) ? k_stage_bytes / 2 : k_stage_bytes);   // packed 4-bit keys are counted in the bytes read
            for (int it = 0; it < n_work; ++it, s = (s + 1 == stages ? 0 : s + 1), ph ^= (s == 0 ? 1u : 0u)) {
                const uint32_t kf = smem_u32(&bars->k_full[s]);
                uint32_t bytes = tile_bytes;
                if (left == 0) {
                    if (!seg.next()) break;
                    left = seg.te - seg.tb;
                    key_row = seg.tb * TC_KEYS;
                    bytes += static_cast<uint32_t>(nq * q_sub_bytes);
                    q_bar = kf;
                    q_at = MULTI && it > 0 ? max(0, left - (stages - 1)) : -1;    // later segments: the other stages are filled first
                    const int last = s == 0 ? stages - 1 : s - 1;                 // stage of the previous segment's last tile, and its phase
                    free_bar = smem_u32(&bars->k_empty[last]);
                    free_ph = s == 0 ? ph ^ 1u : ph;
                }
                if (!mbar_wait(smem_u32(&bars->k_empty[s]), ph ^ 1u) || *aborted) { ok = false; break; }
                mbar_expect_tx(kf, bytes);
                if (it == 0) load_q();
                for (int a = 0; a < atoms; ++a)
                    tma_load_2d(smem_u32(k_smem + s * k_stage_bytes + a * TC_KEYS * 128), &tmap_k, a * atom_elems, key_row, kf);
                issued = it + 1;
                key_row += TC_KEYS;
                if (--left == q_at) {
                    q_at = -1;
                    if (!mbar_wait(free_bar, free_ph) || *aborted) { ok = false; break; }
                    load_q();
                }
            }
            if (!ok) {
                *aborted = 1;
                report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT);
            }
            if (*aborted) {   // let the copies already in flight land before the CTA leaves
                for (int it = max(0, issued - stages); it < issued; ++it)
                    mbar_wait(smem_u32(&bars->k_full[it % stages]), static_cast<uint32_t>(it / stages) & 1u);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            // the keys (the A operand) may be E2M1 (format 5) against E4M3 queries
            const uint32_t idesc = umma_idesc(FP8 ? 0u : 1u, TC_KEYS, TC_N) | ((FP8 && cp.k_fp4) ? (5u << 7) : 0u);
            bool ok = true;
            uint32_t cnt = 0;
            // descriptors of the first key stage / first query sub-tile; every other operand is a constant number of 16-byte
            // units further on, so stepping through the tiles is one 64-bit add
            const uint64_t kdesc0 = umma_desc_sw128(smem_u32(k_smem)), qdesc0 = umma_desc_sw128(smem_u32(q_smem));
            int s = 0;
            uint32_t ph = 0;
            for (int it = 0; it < n_work && ok; ++it, s = (s + 1 == stages ? 0 : s + 1), ph ^= (s == 0 ? 1u : 0u)) {
                ok = mbar_wait(smem_u32(&bars->k_full[s]), ph) && !*aborted;
                if (!ok) break;
                const uint64_t kdesc_s = kdesc0 + static_cast<uint64_t>((s * k_stage_bytes) >> 4);
                for (int j = 0; j < nq; ++j, ++cnt) {
                    const uint32_t slot = cnt & 1u, use = cnt >> 1;
                    ok = mbar_wait(smem_u32(&bars->tmem_empty[slot]), (use & 1u) ^ 1u) && !*aborted;
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + slot * TC_N;
                    const uint64_t qdesc_j = qdesc0 + static_cast<uint64_t>((j * q_sub_bytes) >> 4);
                    uint32_t acc = 0;
                    for (int a = 0; a < atoms; ++a) {
                        const uint64_t ka = kdesc_s + static_cast<uint64_t>((a * TC_KEYS * 128) >> 4);
                        const uint64_t qa = qdesc_j + static_cast<uint64_t>((a * TC_N * 128) >> 4);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {   // 32 bytes of K per instruction (16 bf16 or 32 e4m3)
                            umma<FP8>(d_tmem, ka + 2 * ks, qa + 2 * ks, idesc, acc);
                            acc = 1;
                        }
                    }
                    umma_commit(smem_u32(&bars->tmem_full[slot]));
                    if (j == nq - 1) umma_commit(smem_u32(&bars->k_empty[s]));
                }
            }
            if (!ok) {
                *aborted = 1;
                // tensor memory is freed after the barrier below: the instructions already issued finish first
                report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT);
                umma_commit(smem_u32(&bars->mma_drain));
                mbar_wait(smem_u32(&bars->mma_drain), 0);
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue: warps 2 and up
        constexpr int CPW = TC_N / 32 / 2;      // 32-column chunks a warp reduces: half a slot
        constexpr int TPH = TPS / 2;            // tokens of a slot a warp reduces
        static_assert(CPW % 2 == 0, "chunks are processed in pairs");
        const int e = ((warp - 2) >> 2) & 1;    // epilogue group = TMEM half it drains
        const int chalf = (warp - 2) >> 3;   // which half of the slot's columns
        const int quad = warp & 3;              // TMEM lanes 32*quad .. 32*quad+31
        const float neg_inf = __int_as_float(0xff800000);
        bool ok = true;
        // candidate staging of this warp: lane i keeps the fill count of the warp's token slot i
        int2* my_stage = cstage + (warp - 2) * TC_CAND_TPW * TC_CAND_SLOTS;
        int cand_fill = 0;
        auto cand_flush = [&](int slot, int t, int c) {
            __syncwarp();                                        // the staged entries were written by other lanes
            int base = 0;
            if (lane == 0) base = atomicAdd(cp.cand_cnt + t, c);
            base = __shfl_sync(0xffffffffu, base, 0);
            if (lane < c && base + lane < cp.cand_cap) cp.cand[static_cast<int64_t>(t) * cp.cand_cap + base + lane] = my_stage[slot * TC_CAND_SLOTS + lane];
            __syncwarp();                                        // slots are free again
        };
        if constexpr (!CAND) {
            if (p.causal) {
                // the CTAs that work on a group share its rows; with even shares all CTAs share all rows
                constexpr bool own = !MULTI;
                const int sharing = own ? (tc_visible_tiles(p, tpc, g0) + p.tiles_per_cta - 1) / p.tiles_per_cta : static_cast<int>(gridDim.x);
                const int row0 = own ? g0 * tpc : 0;
                fill_masked_tails(p.scores, p.ld, p.M, p.n_keys, p.q_pos0, p.n_tiles, tpc, row0 + (warp - 2) * sharing + static_cast<int>(blockIdx.x),
                                  own ? min(p.M, row0 + tpc) : p.M, (NEPI / 32) * sharing, lane);
            }
        }
        uint32_t it = 0;                        // tiles done so far, over all segments
        bool later = false;
        // every wait is bounded and a warp that gives up keeps to the barriers of the segments that follow
        for (TcSegments<MULTI> seg(p, tpc, g0, tile0, n_work); seg.next(); later = true) {
            if (MULTI && later) {
                epilogue_barrier<NEPI>();       // nobody reads the previous weights any more
                load_weights(seg.g, threadIdx.x - 64, NEPI);
                epilogue_barrier<NEPI>();
            }
            const int t0 = seg.g * tpc;
            for (int tile = seg.tb; tile < seg.te && ok; ++tile, ++it) {
                const int64_t s = static_cast<int64_t>(tile) * TC_KEYS + quad * 32 + lane;
                const bool key_ok = s < p.n_keys;
                const float kscale = (FP8 && key_ok) ? p.k_scale[s] : 1.f;
                const float cb = (p.col_bias != nullptr && key_ok) ? p.col_bias[s] : 0.f;
                // group e drains the sub-tiles j = e, e+2, .. of every key tile (nq is even)
                for (int j = e; j < nq; j += 2) {
                    const int slot = e;
                    const uint32_t use = (it * static_cast<uint32_t>(nq) + static_cast<uint32_t>(j)) >> 1;
                    ok = mbar_wait(smem_u32(&bars->tmem_full[slot]), use & 1u) && !*aborted;
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + slot * TC_N + chalf * CPW * 32;
                    const int tsub0 = t0 + j * TPS + chalf * TPH;
                    const float* wrow = ws + j * TC_N + chalf * CPW * 32;
                    const float* rb = rbs + j * TPS + chalf * TPH;
                    float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                    auto store = [&](int tt, float v) {
                        const int t = tsub0 + tt;
                        if constexpr (!CAND) {
                            if (t < p.M && key_ok) {
                                float out = v * kscale;
                                out = fmaf(rb[tt], cb, out);
                                if (p.causal && s > p.q_pos0 + t) out = neg_inf;
                                p.scores[static_cast<int64_t>(t) * p.ld + s] = out;
                            }
                        } else {
                            // all 32 lanes (32 consecutive keys of one token) get here together
                            float out = v * kscale;
                            out = fmaf(rb[tt], cb, out);
                            const bool masked = p.causal && s > p.q_pos0 + t;
                            const bool pass = t < p.M && key_ok && !masked && out >= thrs[j * TPS + chalf * TPH + tt];
                            const uint32_t m = __ballot_sync(0xffffffffu, pass);
                            if (m != 0u) {
                                const int cs = (j >> 1) * TPH + tt;
                                int c = __shfl_sync(0xffffffffu, cand_fill, cs);
                                const int n = __popc(m);
                                if (c + n > TC_CAND_SLOTS) { cand_flush(cs, t, c); c = 0; }
                                if (pass) my_stage[cs * TC_CAND_SLOTS + c + __popc(m & ((1u << lane) - 1u))] = make_int2(__float_as_int(out), static_cast<int>(s));
                                if (lane == cs) cand_fill = c + n;
                            }
                        }
                    };
                    // two register buffers: the load of the next 32 columns is in flight while this one is reduced
                    uint32_t ra[32], rb32[32];
                    tmem_ld32_issue(taddr, ra);
#pragma unroll
                    for (int c = 0; c < CPW; c += 2) {
                        tmem_ld_wait(ra);
                        tmem_ld32_issue(taddr + (c + 1) * 32, rb32);
                        reduce_chunk<H>(ra, wrow + c * 32, c * 32, acc, store);
                        tmem_ld_wait(rb32);
                        if (c + 2 < CPW) {
                            tmem_ld32_issue(taddr + (c + 2) * 32, ra);
                        } else {
                            // every column of this warp's part is in registers: hand the slot back before the last reduction
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(smem_u32(&bars->tmem_empty[slot]));
                        }
                        reduce_chunk<H>(rb32, wrow + (c + 1) * 32, (c + 1) * 32, acc, store);
                    }
                }
            }
            if (!ok && lane == 0) { *aborted = 1; report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT); }
            if constexpr (CAND) {
                for (int slot = 0; slot < TC_CAND_TPW; ++slot) {
                    const int c = __shfl_sync(0xffffffffu, cand_fill, slot);
                    if (c > 0) cand_flush(slot, t0 + (2 * (slot / TPH) + e) * TPS + chalf * TPH + slot % TPH, c);
                }
                cand_fill = 0;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ---- host side ---------------------------------------------------------------------------------------------
PFN_encodeTiled get_encode_tiled() {
    static std::atomic<PFN_encodeTiled> fn{nullptr};
    if (fn.load() == nullptr) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess && qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_encodeTiled>(p);
    }
    return fn;
}

bool make_tmap_2d_sw128(CUtensorMap* map, const void* base, int elem_bytes, uint64_t rows, uint64_t cols, uint64_t row_pitch_bytes,
                        uint32_t box_rows, uint32_t box_cols) {
    PFN_encodeTiled enc = get_encode_tiled();
    if (enc == nullptr) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {row_pitch_bytes};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    // elem_bytes 0: 4-bit elements, 16 of them expanded to a 16-byte aligned shared-memory chunk (box_cols must be 128)
    const CUtensorMapDataType dt = elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                   : elem_bytes == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_16U4_ALIGN16B;
    // The encoder is a driver call and wants a context on this thread; a thread whose first CUDA call this is has none yet (the runtime's
    // own calls bring one along).
    if (current_context_id() == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess) return false;
    }
    return enc(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool indexer_tc_supported(int M, int H, int D, int64_t n_keys, int64_t q_stride_tok, int64_t /*k_stride_tok*/, int dtype) {
    if (!(H == 4 || H == 8 || H == 16 || H == 32 || H == 64)) return false;
    const int row_bytes = D * (dtype == JANUS_DTYPE_BF16 ? 2 : 1);
    if (row_bytes != 128 && row_bytes != 256) return false;
    if (dtype == JANUS_DTYPE_FP8_Q_FP4_K && D != 128) return false;     // the packed 4-bit TMA box is 128 elements
    if (q_stride_tok != static_cast<int64_t>(H) * D) return false;
    if (static_cast<int64_t>(M) * H >= (int64_t(1) << 31) || n_keys >= (int64_t(1) << 31) - 256) return false;
    return true;
}

// Candidate mode needs every epilogue warp's tokens to fit its staging slots, whatever sub-tile count the launch picks.
bool indexer_tc_candidates_supported(int H, int D, int dtype) {
    const int row_bytes = D * (dtype == JANUS_DTYPE_BF16 ? 2 : 1);
    const int nq_max = row_bytes == 128 ? 4 : 2;
    if (dtype == JANUS_DTYPE_FP8_Q_FP4_K) return false;                 // the sample gather and the exact fallback read 8- and 16-bit keys
    return (H == 32 || H == 64) && (nq_max / 2) * (TC_N / H / 2) <= TC_CAND_TPW;
}

template <int H, bool FP8, bool CAND, bool MULTI>
static int launch_tc(const CUtensorMap& tq, const CUtensorMap& tk, const TcParams& p, const TcCandParams& cp, const TcSchedule& sched, dim3 grid,
                     size_t smem, cudaStream_t stream) {
    static once_per_context attributes;
    JANUS_CUDA_CHECK(attributes.run(
        [] { return cudaFuncSetAttribute(indexer_tc_kernel<H, FP8, CAND, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_BUDGET); }));
    if constexpr (MULTI)
        JANUS_CUDA_CHECK(launch_kernel(indexer_tc_kernel<H, FP8, CAND, MULTI>, grid, TC_THREADS, smem, stream, 1, tq, tk, p, cp, sched));
    else
        JANUS_CUDA_CHECK(launch_kernel(indexer_tc_kernel<H, FP8, CAND, MULTI>, grid, TC_THREADS, smem, stream, 1, tq, tk, p, cp,
                                       TcNoSchedule{}));
    return JANUS_OK;
}

int launch_indexer_tc(const void* q_idx, const void* k_idx, int64_t k_stride_tok, const float* w, const float* q_scale,
                      int64_t q_scale_stride_tok, const float* k_scale, const float* row_bias, const float* col_bias, int M, int H,
                      int D, int64_t n_keys, int64_t q_pos0, int causal, int dtype, float* scores, int64_t ld, int32_t* dev_status,
                      cudaStream_t stream, const float* thr, int32_t* cand_cnt, void* cand, int cand_cap) {
    const bool k_fp4 = dtype == JANUS_DTYPE_FP8_Q_FP4_K;
    const bool fp8 = dtype == JANUS_DTYPE_FP8_E4M3 || k_fp4;
    const int esz = fp8 ? 1 : 2;
    TcParams p;
    p.w = w; p.q_scale = q_scale; p.q_scale_stride_tok = q_scale_stride_tok; p.k_scale = k_scale;
    p.row_bias = row_bias; p.col_bias = col_bias; p.scores = scores; p.ld = ld; p.n_keys = n_keys; p.q_pos0 = q_pos0;
    p.M = M; p.H = H; p.causal = causal; p.dev_status = dev_status;
    const TcCandParams cp{thr, cand_cnt, static_cast<int2*>(cand), cand_cap, k_fp4 ? 1 : 0};
    p.atoms = D * esz / 128;
    p.n_tiles = static_cast<int>((n_keys + TC_KEYS - 1) / TC_KEYS);
    const int tps = TC_N / H;
    auto total_work = [&](int nq) {
        int64_t w = 0;
        const int tpc_ = nq * tps, groups = (M + tpc_ - 1) / tpc_;
        for (int g = 0; g < groups; ++g) w += tc_visible_tiles(p, tpc_, g);
        return w;
    };
    // Query sub-tiles per group: the key tiles are read once per group, so four where 128 KB hold them; two when that leaves SMs
    // idle or the last round of tiles uneven (256 tokens x 34 tiles of 4 heads are 34 CTAs of four sub-tiles or 68 of two).  A tile costs
    // its sub-tiles and about a third of one more (its copy, barriers and the keys' scales), and the longest range decides.  With two
    // and four, us: 256 x 4352 of 4 heads 7.4 and 11.2, 24 x 131096 FP8 34.9 and 42.9, 40 x 20040 13.2 and 16.0; 128 x 131200 166 and 160.5,
    // 128 x 16512 26.2 and 24.8, 777 x 20788 161 and 153.
    p.nq = p.atoms == 1 ? 4 : 2;
    int64_t work = total_work(p.nq);      // visible (token group, key tile) pairs of all groups
    p.tiles_per_cta = 0;
    if (p.nq == 4) {
        const int64_t w2 = total_work(2);
        if (2.35 * static_cast<double>((w2 + TC_MAX_CTAS - 1) / TC_MAX_CTAS) < 4.35 * static_cast<double>((work + TC_MAX_CTAS - 1) / TC_MAX_CTAS)) {
            p.nq = 2;
            work = w2;
        }
    }
    const int q_bytes = p.nq * p.atoms * TC_N * 128;
    const int k_stage = p.atoms * TC_KEYS * 128;
    const bool cand_mode = thr != nullptr;
    if (cand_mode && p.nq / 2 * (tps / 2) > TC_CAND_TPW) return JANUS_ERR_UNSUPPORTED;
    const int tail = static_cast<int>(sizeof(float)) * (p.nq * TC_N + 2 * p.nq * tps) + (cand_mode ? TC_CAND_STAGE_BYTES : 0) +
                     static_cast<int>(sizeof(TcBarriers)) + 16;
    p.stages = (TC_SMEM_BUDGET - q_bytes - tail) / k_stage;
    if (p.stages > TC_MAX_STAGES) p.stages = TC_MAX_STAGES;
    if (p.stages < 2) return JANUS_ERR_UNSUPPORTED;
    const size_t smem = static_cast<size_t>(q_bytes) + static_cast<size_t>(p.stages) * k_stage + tail;
    const int tpc = p.nq * tps;
    // Few tiles: ranges that end with their group, when the longest is no longer for it (a change of group costs most of a
    // tile's time and the table 0.5 us: 19 rows x 9020 keys 9.5 us with even shares, 8.3 without).
    p.n_groups = (M + tpc - 1) / tpc;
    TcSchedule sched;
    bool multi = true;
    dim3 grid(static_cast<unsigned>(work < TC_MAX_CTAS ? work : TC_MAX_CTAS));
    const int64_t longest = (work + TC_MAX_CTAS - 1) / TC_MAX_CTAS;
    if (longest >= (int64_t(1) << 30)) return JANUS_ERR_UNSUPPORTED;
    if (p.n_groups <= TC_MAX_CTAS) {
        int64_t ctas = 0;
        for (int g = 0; g < p.n_groups; ++g) ctas += (tc_visible_tiles(p, tpc, g) + longest - 1) / longest;
        multi = ctas > TC_MAX_CTAS;
    }
    if (multi) {
        // Ranges whose tiles, and the changes of group inside them at three quarters of a tile each, cost at most `budget`: the smallest with
        // which the CTAs get through.  Equal numbers of tiles left the CTAs of a causal call's first groups, which have a tile or two
        // each, far behind: 4096 rows x 4096 keys without history, 64 heads of bf16 167 -> 125 us, FP8 127 -> 96.5; 300 keys of history 150
        // -> 139; from 4 K on unchanged.  (A change at a whole tile: the same there, and calls of three to eight tiles per CTA 9 % slower.)
        const int n_ctas = static_cast<int>(grid.x);
        const int tile_cost = longest < 65536 ? 4 : 1, change_cost = longest < 65536 ? 3 : 0;
        int used = 0;
        int64_t counts[TC_MAX_CTAS];
        auto pack = [&](int64_t budget) {
            int g = 0;
            int64_t done = 0, tile = 0, tiles = tc_visible_tiles(p, tpc, 0);
            for (used = 0; used < n_ctas && done < work; ++used) {
                sched.first[used] = make_int2(g, static_cast<int>(tile));
                int64_t left = budget, count = 0;
                for (;;) {
                    const int64_t fit = left / tile_cost, take = fit < tiles - tile ? fit : tiles - tile;
                    tile += take;
                    count += take;
                    left -= take * tile_cost;
                    if (tile < tiles) break;
                    tile = 0;
                    tiles = ++g < p.n_groups ? tc_visible_tiles(p, tpc, g) : 0;
                    left -= change_cost;
                    if (done + count >= work || left < tile_cost) break;
                }
                done += count;
                counts[used] = count;
            }
            return done >= work;
        };
        const int64_t inside = p.n_groups > n_ctas ? p.n_groups - n_ctas : 0;      // changes that no cut can avoid
        int64_t budget = (work * tile_cost + inside * change_cost + n_ctas - 1) / n_ctas, most = 0;
        if (budget < tile_cost) budget = tile_cost;
        for (int64_t more = 1 + budget / 512; !pack(budget); ++more) budget += more;
        for (int c = 0; c < used; ++c) most = counts[c] > most ? counts[c] : most;
        for (int c = 0; c < used; ++c) sched.less[c] = static_cast<uint16_t>(most - counts[c]);
        sched.longest = static_cast<int>(most);
        grid.x = used;
    } else {
        p.tiles_per_cta = static_cast<int>(longest);
        grid = dim3(static_cast<unsigned>((tc_visible_tiles(p, tpc, p.n_groups - 1) + longest - 1) / longest), p.n_groups);
    }

    CUtensorMap tq, tk;
    const uint32_t box_cols = fp8 ? 128 : 64;
    if (!make_tmap_2d_sw128(&tq, q_idx, esz, static_cast<uint64_t>(M) * H, D, static_cast<uint64_t>(D) * esz, TC_N, box_cols)) return JANUS_ERR_CUDA;
    if (k_fp4) {   // packed 4-bit keys: the copy expands 16 of them into the low halves of a 16-byte chunk
        if (!make_tmap_2d_sw128(&tk, k_idx, 0, static_cast<uint64_t>(n_keys), D, static_cast<uint64_t>(k_stride_tok) / 2, TC_KEYS, 128))
            return JANUS_ERR_CUDA;
    } else if (!make_tmap_2d_sw128(&tk, k_idx, esz, static_cast<uint64_t>(n_keys), D, static_cast<uint64_t>(k_stride_tok) * esz, TC_KEYS, box_cols)) {
        return JANUS_ERR_CUDA;
    }

#define JANUS_TC_CASE(HH, CC)                                                         \
    case HH:                                                                          \
        if (multi) return fp8 ? launch_tc<HH, true, CC, true>(tq, tk, p, cp, sched, grid, smem, stream)          \
                              : launch_tc<HH, false, CC, true>(tq, tk, p, cp, sched, grid, smem, stream);        \
        return fp8 ? launch_tc<HH, true, CC, false>(tq, tk, p, cp, sched, grid, smem, stream)                    \
                   : launch_tc<HH, false, CC, false>(tq, tk, p, cp, sched, grid, smem, stream);
    if (cand_mode) {
        switch (H) {   // head counts whose tokens per epilogue warp fit the staging slots
            JANUS_TC_CASE(32, true)
            JANUS_TC_CASE(64, true)
        }
        return JANUS_ERR_UNSUPPORTED;
    }
    switch (H) {
        JANUS_TC_CASE(4, false)
        JANUS_TC_CASE(8, false)
        JANUS_TC_CASE(16, false)
        JANUS_TC_CASE(32, false)
        JANUS_TC_CASE(64, false)
    }
#undef JANUS_TC_CASE
    return JANUS_ERR_UNSUPPORTED;
}

}  // namespace janus
