// Tensor-core indexer of a decode step over many sessions (Eq. 1, Sec. 2.2): query row b against the keys key_offsets[b] ..
// key_offsets[b + 1] of one concatenated array, no causal mask:
//     scores[s] = k_scale[s] * sum_h (w[b,h]*q_scale[h]) * relu(<q[b,h,:], k[s,:]>) + row_bias[b]*col_bias[s]
//
// Keys on the MMA M axis (128 TMEM lanes), the row's 64 heads on the N axis, as in indexer_tc.cu; but every key is used by one
// row only, so the bound is the keys' bytes, and beside it the threads that issue: a tile is 4 small MMAs, and a copy, a wait or
// a commit costs its issuing thread more than the tensor pipe needs for them.  Hence
//   - the TMA and the MMA warp stay converged and one elected lane issues (in a branch on the lane number the addresses are not
//     known to be uniform: 1300 cycles per 128 keys in the MMA warp, 660 in the TMA warp, whatever the number of MMAs);
//   - a step is 256 keys of 128 one-byte elements: one copy, two accumulators, one commit, whose barrier tells the epilogue that the
//     accumulators are complete and the TMA warp that the stage is free;
//   - eight epilogue warps, one group of four per 128 keys, load the next keys' scales a step ahead;
//   - two CTAs share an SM, three stages of 32 KB each.
// Measured (B200, 64 heads x 128): 64 sessions of 131072 FP4 keys 126 -> 114 us (5.3 TB/s of keys, scales and scores), ragged ones (a
// quarter to all of that) 87.5 -> 72.5, 16 of 131072 38.7 -> 32.8, 64 of 8000 14.3 -> 11.4, 1 of 32768 4.8 -> 4.0; FP8 12 ragged ones of up
// to 50000 14.8 -> 10.6, 64 of 131072 at 6.6 TB/s before and after (173 us); bf16 12 ragged ones 16.1 -> 13.3; against four CTAs per SM
// (bf16 two) with four epilogue warps, steps of 128 keys and two stages (bf16 three) each.
// Every wait is bounded; on a timeout the CTA reports JANUS_DEV_WAIT_TIMEOUT and winds down normally.
#include "indexer_tc.cuh"

namespace janus {

constexpr int TB_HEADS = 64;
constexpr int TB_THREADS = 320;      // 1 TMA warp + 1 MMA warp + 8 epilogue warps
constexpr int TB_NEPI = TB_THREADS - 64;
constexpr int TB_CTAS = 2;           // per SM
constexpr int TB_MAX_STAGES = 6;
// Accumulators of 128 keys x 64 heads per step: a stage holds 32 KB, 256 keys of 128 bytes or 128 keys of 256 (bf16, and E4M3 of 256 dims, of
// which half an SM would hold one stage of 256).
constexpr int tb_subs(int atoms, bool fp8) { return fp8 && atoms == 1 ? 2 : 1; }

struct TbParams {
    const float* w;
    const float* q_scale;
    int64_t q_scale_stride_tok;
    const float* k_scale;
    const float* row_bias;
    const float* col_bias;
    float* scores;
    int64_t n_keys;
    const int64_t* key_offsets;   // [n_sessions + 1], device memory
    int n_sessions;
    int max_tiles;                // key tiles (of 128 or 256) of the longest session
    int tiles_per_cta;            // without MULTI: CTA (x, y) has the tiles x * tiles_per_cta .. of session y
    int atoms;                    // 128-byte swizzle atoms per row
    int stages;
    // keys are FP4 E2M1, two per byte; the TMA expands 16 of them into the first 8 bytes of every 16-byte shared-memory chunk,
    // which is the layout the f8f6f4 MMA expects for 4-bit operands
    int k_fp4;
    int32_t* dev_status;
};

struct TbShared {
    float ws[TB_HEADS];               // half of w * q_scale of the segment's row
    uint64_t k_full[TB_MAX_STAGES];
    uint64_t done[TB_MAX_STAGES];     // the step's MMAs are complete: accumulators readable, stage free
    uint64_t tmem_empty[2];
    uint64_t mma_drain;               // abort path only
    float row_bias;
    uint32_t tmem_base;
    int aborted;
    int first_session, first_tile;    // where this CTA's range begins (even shares)
    int scan[33];
};

// Keys of a session, cut back to the part inside the key array (n_keys rows).
struct TbSession {
    int64_t base, count;
    int tiles;
    bool bad;
};
template <int KEYS>
__device__ __forceinline__ TbSession tb_session(int64_t begin, int64_t end, int64_t n_keys, int max_tiles) {
    TbSession s;
    s.base = begin;
    s.count = end - begin;
    // the offsets come from device memory: neither the per-key scale / bias reads nor the score writes may leave their arrays
    s.bad = s.base < 0 || s.count < 0 || s.base > n_keys || s.count > n_keys - s.base;
    if (s.bad) {
        if (s.base < 0 || s.base > n_keys) { s.base = 0; s.count = 0; }
        if (s.count < 0) s.count = 0;
        if (s.count > n_keys - s.base) s.count = n_keys - s.base;
    }
    s.tiles = static_cast<int>(min((s.count + KEYS - 1) / KEYS, static_cast<int64_t>(max_tiles)));      // max_keys bounds every session
    return s;
}

// A CTA's range, one session at a time: key tiles [tb, te) of session `b`.  Without MULTI there is one.
template <int KEYS, bool MULTI>
struct TbSegments {
    const TbParams& p;
    int b, tb, te, left;
    bool first;
    int64_t key_base, key_count;              // rows key_base .. key_base + key_count of k_idx
    __device__ __forceinline__ TbSegments(const TbParams& p_, int b0, int t0, int work)
        : p(p_), b(b0), tb(t0), te(t0), left(work), first(true), key_base(0), key_count(0) {}
    __device__ __forceinline__ bool next() {
        if (left <= 0) return false;
        int tiles;
        do {
            if (!first) { ++b; tb = 0; }
            first = false;
            if (MULTI && b >= p.n_sessions) { left = 0; return false; }
            const TbSession s = tb_session<KEYS>(ld_input(p.key_offsets + b), ld_input(p.key_offsets + b + 1), p.n_keys, p.max_tiles);
            key_base = s.base;
            key_count = s.count;
            tiles = s.tiles;
        } while (MULTI && tiles <= tb);       // (sessions without keys)
        te = MULTI ? min(tiles, tb + left) : tb + left;
        left -= te - tb;
        return true;
    }
};

template <bool FP8, int SUBS, bool MULTI>
__global__ void __launch_bounds__(TB_THREADS, TB_CTAS)
indexer_tc_batch_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k, const TbParams p) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int KEYS = SUBS * TC_KEYS;                   // keys per step
    constexpr int SLOT_COLS = SUBS * TB_HEADS;             // TMEM columns of a step's accumulators, two sets in turn
    const int atoms = p.atoms, stages = p.stages;
    const int q_bytes = atoms * TB_HEADS * 128, stage_bytes = atoms * KEYS * 128;
    unsigned char* k_smem = smem + q_bytes;
    TbShared* sh = reinterpret_cast<TbShared*>(k_smem + stages * stage_bytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if ((smem_u32(smem) & 1023u) != 0u) {   // swizzled tiles need 1024-byte alignment
        grid_wait();
        if (threadIdx.x == 0) report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT);
        return;
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) { mbar_init(smem_u32(&sh->k_full[s]), 1); mbar_init(smem_u32(&sh->done[s]), 1); }
        for (int s = 0; s < 2; ++s) mbar_init(smem_u32(&sh->tmem_empty[s]), 4 * SUBS);
        mbar_init(smem_u32(&sh->mma_drain), 1);
        fence_mbar_init();
        prefetch_tensormap(&tmap_q);
        prefetch_tensormap(&tmap_k);
        grid_wait();
        // an earlier CTA of this launch gave up on a wait: this one starts no work on a broken pipeline.  One thread reads the
        // status word and the whole CTA follows that one reading (a second reading could differ and split the roles).
        sh->aborted = (p.dev_status != nullptr && *reinterpret_cast<volatile int32_t*>(p.dev_status) == JANUS_DEV_WAIT_TIMEOUT) ? 1 : 0;
    }
    grid_wait();
    auto load_weights = [&](int b, int h) {                // by threads h = 0 .. of those that call
        if (h < TB_HEADS) {
            float v = p.w[static_cast<int64_t>(b) * TB_HEADS + h];
            if (FP8) v *= p.q_scale[static_cast<int64_t>(b) * p.q_scale_stride_tok + h];
            sh->ws[h] = 0.5f * v;                          // the epilogue forms 2 * relu
        }
        if (h == TB_HEADS) sh->row_bias = p.row_bias != nullptr ? p.row_bias[b] : 0.f;
    };
    // ---- this CTA's range: n_work tiles from tile `tile0` of session `b0` on
    int b0, tile0, n_work;
    if constexpr (!MULTI) {
        b0 = blockIdx.y;
        tile0 = blockIdx.x * p.tiles_per_cta;
        const int64_t key_begin = ld_input(p.key_offsets + b0), key_end = ld_input(p.key_offsets + b0 + 1);
        load_weights(b0, threadIdx.x);                     // (while the offsets are on their way)
        const TbSession ses = tb_session<KEYS>(key_begin, key_end, p.n_keys, p.max_tiles);
        if (ses.bad && tile0 == 0 && threadIdx.x == 0) report(p.dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);
        n_work = min(ses.tiles - tile0, p.tiles_per_cta);
        if (n_work <= 0) return;
    } else {
        // the sessions' tile counts are scanned by the block: where this CTA's share of their sum begins
        const bool one_round = p.n_sessions <= TB_THREADS;
        int64_t total = 0, begin = 0, end = 0;
        for (int pass = one_round ? 1 : 0; pass < 2; ++pass) {
            int64_t before = 0;                            // tiles of the sessions of earlier rounds
            if (pass == 1 && threadIdx.x == 0) sh->first_session = p.n_sessions;
            for (int r0 = 0; r0 < p.n_sessions; r0 += TB_THREADS) {
                const int b = r0 + threadIdx.x;
                int tiles = 0;
                if (b < p.n_sessions) {
                    const TbSession ses = tb_session<KEYS>(ld_input(p.key_offsets + b), ld_input(p.key_offsets + b + 1), p.n_keys, p.max_tiles);
                    if (ses.bad && pass == 1 && blockIdx.x == 0) report(p.dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);
                    tiles = ses.tiles;
                }
                int block_total;
                const int mine = block_exclusive_scan<TB_THREADS>(tiles, sh->scan, &block_total);
                if (one_round) total = block_total;
                if (pass == 1) {
                    if (r0 == 0) {
                        const uint32_t each = static_cast<uint32_t>(total) / gridDim.x, more = static_cast<uint32_t>(total) - each * gridDim.x;
                        begin = static_cast<int64_t>(each) * blockIdx.x + min(blockIdx.x, more);
                        end = begin + each + (blockIdx.x < more ? 1 : 0);
                    }
                    const int64_t at = before + mine;
                    if (at <= begin && begin < at + tiles) { sh->first_session = b; sh->first_tile = static_cast<int>(begin - at); }
                }
                before += block_total;
            }
            total = before;
        }
        __syncthreads();
        n_work = static_cast<int>(end - begin);
        b0 = sh->first_session;
        tile0 = sh->first_tile;
        if (n_work <= 0 || b0 >= p.n_sessions) return;
        load_weights(b0, threadIdx.x);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&sh->tmem_base), 2 * SLOT_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;
    volatile int* aborted = &sh->aborted;
    const bool run = *aborted == 0;       // read once, after the barrier: the same value in every thread
    const uint32_t k_full = smem_u32(&sh->k_full[0]), done = smem_u32(&sh->done[0]), t_empty = smem_u32(&sh->tmem_empty[0]);

    if (!run) {
        // nothing to do: tensor memory goes back below
    } else if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        const uint32_t ring = smem_u32(k_smem);
        const uint32_t tile_bytes = static_cast<uint32_t>((FP8 && p.k_fp4) ? stage_bytes / 2 : stage_bytes);   // packed 4-bit keys are counted in the bytes read
        constexpr int ATOM = FP8 ? 128 : 64;
        bool ok = true;
        int issued = 0, s = 0;                          // ring stage and its phase bit, advanced per tile
        uint32_t ph = 0;
        TbSegments<KEYS, MULTI> seg(p, b0, tile0, n_work);
        while (ok && seg.next()) {
            // The queries of a segment are counted on the barrier of its first key tile, so the MMA warp needs to know nothing of
            // segments.  They may be replaced when the previous segment's last key tile has been released: every MMA up to it has
            // completed then; the other stages are filled first.
            const int n = seg.te - seg.tb, last = s == 0 ? stages - 1 : s - 1;
            const uint32_t q_bar = k_full + 8 * s, free_bar = done + 8 * last, free_ph = s == 0 ? ph ^ 1u : ph;
            const int q_after = issued == 0 ? 0 : min(n, stages - 1);       // key tiles before the queries
            int key_row = static_cast<int>(seg.key_base) + seg.tb * KEYS;
            auto load_q = [&]() {
                if (elect_one())
                    for (int a = 0; a < atoms; ++a) tma_load_2d(smem_u32(smem) + a * TB_HEADS * 128, &tmap_q, a * ATOM, seg.b * TB_HEADS, q_bar);
                __syncwarp();
            };
            for (int i = 0; i < n; ++i) {
                if (!__all_sync(0xffffffffu, mbar_test_wait(done + 8 * s, ph ^ 1u))) {
                    ok = mbar_wait(done + 8 * s, ph ^ 1u) && !*aborted;
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                }
                if (elect_one()) {
                    const uint32_t full = k_full + 8 * s, dst = ring + s * stage_bytes;
                    mbar_expect_tx(full, tile_bytes + (i == 0 ? static_cast<uint32_t>(q_bytes) : 0u));
                    tma_load_2d(dst, &tmap_k, 0, key_row, full);
                    if (SUBS == 1 && atoms == 2) tma_load_2d(dst + KEYS * 128, &tmap_k, ATOM, key_row, full);
                }
                __syncwarp();
                if (issued == 0) load_q();
                ++issued;
                key_row += KEYS;
                if (++s == stages) { s = 0; ph ^= 1u; }
                if (i + 1 == q_after) {
                    ok = mbar_wait(free_bar, free_ph) && !*aborted;
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    load_q();
                }
            }
        }
        if (!ok) {
            *aborted = 1;
            if (lane == 0) report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT);
        }
        if (*aborted) {   // let the copies already in flight land before the CTA leaves
            for (int it = max(0, issued - stages); it < issued; ++it) mbar_wait(k_full + 8 * (it % stages), static_cast<uint32_t>(it / stages) & 1u);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t idesc = umma_idesc(FP8 ? 0u : 1u, TC_KEYS, TB_HEADS) | ((FP8 && p.k_fp4) ? (5u << 7) : 0u);     // E2M1 keys (format 5) against E4M3 queries
        const uint64_t kdesc0 = umma_desc_sw128(smem_u32(k_smem)), qdesc = umma_desc_sw128(smem_u32(smem));
        bool ok = true;
        int s = 0;
        uint32_t ph = 0;
        for (int it = 0; it < n_work; ++it) {
            const uint32_t slot = static_cast<uint32_t>(it) & 1u, slot_ph = ((static_cast<uint32_t>(it) >> 1) & 1u) ^ 1u;
            // both probes are under way together; only if one of them fails is there a wait
            const bool slot_free = mbar_test_wait(t_empty + 8 * slot, slot_ph), landed = mbar_test_wait(k_full + 8 * s, ph);
            if (!__all_sync(0xffffffffu, slot_free && landed)) {
                ok = mbar_wait(t_empty + 8 * slot, slot_ph) && mbar_wait(k_full + 8 * s, ph) && !*aborted;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
            tc_fence_after();
            if (elect_one()) {
                const uint64_t kdesc = kdesc0 + static_cast<uint64_t>((s * stage_bytes) >> 4);
#pragma unroll
                for (int sub = 0; sub < SUBS; ++sub) {
                    const uint32_t d = tmem_base + slot * SLOT_COLS + sub * TB_HEADS;
                    const uint64_t ka = kdesc + sub * (TC_KEYS * 128 >> 4);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) umma<FP8>(d, ka + 2 * ks, qdesc + 2 * ks, idesc, ks > 0 ? 1u : 0u);     // 32 bytes of K per instruction
                    if (SUBS == 1 && atoms == 2) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            umma<FP8>(d, ka + (KEYS * 128 >> 4) + 2 * ks, qdesc + (TB_HEADS * 128 >> 4) + 2 * ks, idesc, 1u);
                    }
                }
                umma_commit(done + 8 * s);
            }
            __syncwarp();
            if (++s == stages) { s = 0; ph ^= 1u; }
        }
        if (!ok) {
            *aborted = 1;
            // tensor memory is freed after the barrier below: the instructions already issued finish first
            if (elect_one()) {
                report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT);
                umma_commit(smem_u32(&sh->mma_drain));
            }
            __syncwarp();
            mbar_wait(smem_u32(&sh->mma_drain), 0);
        }
    } else {
        // ------------------------------------------------------------------ epilogue: thread = key
        // Group e of four warps takes the second or first 128 keys of every step, or with one accumulator per step every second step:
        // its next keys are 256 further on either way.
        constexpr int STEP = SUBS == 2 ? 1 : 2;
        const int e = (warp - 2) >> 2, quad = warp & 3;
        const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        bool ok = true, later = false;
        int it = 0;                             // steps of earlier segments
        // every wait is bounded and a warp that gives up keeps to the barriers of the segments that follow
        for (TbSegments<KEYS, MULTI> seg(p, b0, tile0, n_work); seg.next(); later = true) {
            if (MULTI && later) {
                epilogue_barrier<TB_NEPI>();    // nobody reads the previous weights any more
                load_weights(seg.b, threadIdx.x - 64);
                epilogue_barrier<TB_NEPI>();
            }
            const int n = seg.te - seg.tb, skip = SUBS == 2 ? 0 : (it ^ e) & 1;
            int s = (it + skip) % stages;       // ring stage and its phase bit
            uint32_t ph = static_cast<uint32_t>((it + skip) / stages) & 1u;
            int64_t key = static_cast<int64_t>(seg.tb + skip) * KEYS + (SUBS == 2 ? e * TC_KEYS : 0) + quad * 32 + lane;
            float kscale_next = 1.f, cb_next = 0.f;
            auto load_key = [&](int64_t i) {    // scale and bias factor of the session's key i
                if (i < seg.key_count) {
                    if (FP8) kscale_next = p.k_scale[seg.key_base + i];
                    if (p.col_bias != nullptr) cb_next = p.col_bias[seg.key_base + i];
                }
            };
            if (skip < n) load_key(key);
            const float rb = sh->row_bias;
            for (int i = skip; i < n && ok; i += STEP, key += 2 * TC_KEYS) {
                const float kscale = kscale_next, cb = cb_next;
                if (i + STEP < n) load_key(key + 2 * TC_KEYS);
                const int slot = (it + i) & 1;
                ok = mbar_wait(done + 8 * s, ph) && !*aborted;
                if (!ok) break;
                tc_fence_after();
                const uint32_t taddr = lane_addr + slot * SLOT_COLS + (SUBS == 2 ? e * TB_HEADS : 0);
                float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                auto store = [&](int, float v) {
                    if (key < seg.key_count) {
                        float out = v * kscale;
                        out = fmaf(rb, cb, out);
                        p.scores[seg.key_base + key] = out;
                    }
                };
                uint32_t ra[32], rb32[32];
                tmem_ld32_issue(taddr, ra);
                tmem_ld_wait(ra);
                tmem_ld32_issue(taddr + 32, rb32);
                reduce_chunk<TB_HEADS>(ra, sh->ws, 0, acc, store);
                tmem_ld_wait(rb32);
                // every column is in registers: hand the accumulators back before the last reduction
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(t_empty + 8 * slot);
                reduce_chunk<TB_HEADS>(rb32, sh->ws + 32, 32, acc, store);
                s += STEP;
                if (s >= stages) { s -= stages; ph ^= 1u; }
            }
            it += n;
        }
        if (!ok && lane == 0) { *aborted = 1; report(p.dev_status, JANUS_DEV_WAIT_TIMEOUT); }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 2 * SLOT_COLS);
    }
}

template <bool FP8, int SUBS, bool MULTI>
static int launch_tb(const CUtensorMap& tq, const CUtensorMap& tk, const TbParams& p, dim3 grid, size_t smem, cudaStream_t stream) {
    static once_per_context attributes;
    JANUS_CUDA_CHECK(attributes.run(
        [] { return cudaFuncSetAttribute(indexer_tc_batch_kernel<FP8, SUBS, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_BUDGET / TB_CTAS); }));
    JANUS_CUDA_CHECK(launch_kernel(indexer_tc_batch_kernel<FP8, SUBS, MULTI>, grid, TB_THREADS, smem, stream, 1, tq, tk, p));
    return JANUS_OK;
}

bool indexer_tc_batch_supported(int B, int H, int D, int64_t total_keys, int dtype) {
    const int row_bytes = D * (dtype == JANUS_DTYPE_BF16 ? 2 : 1);
    if (dtype == JANUS_DTYPE_FP8_Q_FP4_K && D != 128) return false;      // the packed 4-bit TMA box is 128 elements
    return H == TB_HEADS && (row_bytes == 128 || row_bytes == 256) && static_cast<int64_t>(B) * H < (int64_t(1) << 31) &&
           total_keys < (int64_t(1) << 31) - 256 && B <= 65535;
}

int launch_indexer_tc_batch(const void* q_idx, const void* k_idx, int64_t k_stride_tok, const float* w, const float* q_scale,
                            int64_t q_scale_stride_tok, const float* k_scale, const float* row_bias, const float* col_bias, int B, int H, int D,
                            int64_t total_keys, int64_t max_keys, const int64_t* key_offsets, int dtype, float* scores, int32_t* dev_status,
                            cudaStream_t stream) {
    const bool k_fp4 = dtype == JANUS_DTYPE_FP8_Q_FP4_K;
    const bool fp8 = dtype == JANUS_DTYPE_FP8_E4M3 || k_fp4;
    const int esz = fp8 ? 1 : 2;
    TbParams p;
    p.w = w; p.q_scale = q_scale; p.q_scale_stride_tok = q_scale_stride_tok; p.k_scale = k_scale;
    p.row_bias = row_bias; p.col_bias = col_bias; p.scores = scores; p.n_keys = total_keys;
    p.key_offsets = key_offsets; p.n_sessions = B; p.k_fp4 = k_fp4 ? 1 : 0; p.dev_status = dev_status;
    p.atoms = D * esz / 128;
    const int subs = tb_subs(p.atoms, fp8), keys = subs * TC_KEYS;
    const int q_bytes = p.atoms * TB_HEADS * 128, stage_bytes = p.atoms * keys * 128, tail = static_cast<int>(sizeof(TbShared));
    const int budget = TC_SMEM_BUDGET / TB_CTAS - 1024;      // (the system keeps 1 KB per CTA)
    p.stages = (budget - q_bytes - tail) / stage_bytes;
    if (p.stages > TB_MAX_STAGES) p.stages = TB_MAX_STAGES;
    if (p.stages < 2) return JANUS_ERR_UNSUPPORTED;
    const size_t smem = static_cast<size_t>(q_bytes) + static_cast<size_t>(p.stages) * stage_bytes + tail;
    const int64_t max_tiles = (max_keys + keys - 1) / keys;
    if (max_tiles == 0) return JANUS_OK;
    p.max_tiles = static_cast<int>(max_tiles);
    // Either every CTA gets the same number of one session's tiles (a 2-D grid that is resident at once), or the tiles of all
    // sessions, whose number only the device knows, are shared out evenly.  The second needs a scan of the offsets and changes of
    // session, about the time of 512 keys, so it is taken when the first would leave some CTA that much more than the average, as far
    // as the host can tell from total_keys (1 session of 32768 FP4 keys 4.0 us against 5.4 with even shares, 3 of 20000 5.3 against 7.2;
    // 12 ragged ones of up to 50000 10.7 against 11.9 without, in bf16 13.3 against 16.2).
    const int64_t resident = static_cast<int64_t>(TC_MAX_CTAS) * TB_CTAS;
    const int64_t chunks = resident / B > max_tiles ? max_tiles : resident / B;
    const int64_t per = chunks > 0 ? (max_tiles + chunks - 1) / chunks : 0;
    const bool direct = chunks > 0 && per * keys <= total_keys / resident + 512;
    p.tiles_per_cta = direct ? static_cast<int>(per) : 0;
    const dim3 grid(static_cast<unsigned>(direct ? (max_tiles + per - 1) / per : resident), direct ? B : 1);
    CUtensorMap tq, tk;
    const uint32_t box_cols = fp8 ? 128 : 64;
    if (!make_tmap_2d_sw128(&tq, q_idx, esz, static_cast<uint64_t>(B) * H, D, static_cast<uint64_t>(D) * esz, TB_HEADS, box_cols)) return JANUS_ERR_CUDA;
    if (k_fp4) {
        if (!make_tmap_2d_sw128(&tk, k_idx, 0, static_cast<uint64_t>(total_keys), D, static_cast<uint64_t>(k_stride_tok) / 2, keys, 128))
            return JANUS_ERR_CUDA;
    } else if (!make_tmap_2d_sw128(&tk, k_idx, esz, static_cast<uint64_t>(total_keys), D, static_cast<uint64_t>(k_stride_tok) * esz, keys, box_cols)) {
        return JANUS_ERR_CUDA;
    }
    if (!fp8) return direct ? launch_tb<false, 1, false>(tq, tk, p, grid, smem, stream) : launch_tb<false, 1, true>(tq, tk, p, grid, smem, stream);
    if (subs == 1) return direct ? launch_tb<true, 1, false>(tq, tk, p, grid, smem, stream) : launch_tb<true, 1, true>(tq, tk, p, grid, smem, stream);
    return direct ? launch_tb<true, 2, false>(tq, tk, p, grid, smem, stream) : launch_tb<true, 2, true>(tq, tk, p, grid, smem, stream);
}

}  // namespace janus
