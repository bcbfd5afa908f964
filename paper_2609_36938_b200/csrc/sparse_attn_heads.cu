// Sparse attention for multi-head and grouped layouts (Sec. 2.2, "core attention"): up to eight query heads that share a
// kv head, keys of 64, 128 or 192 dims, values of 64 or 128.
//
// What bounds it: the gather.  A (token, kv head) pair reads its own k rows of 2 (d_qk + d_v) bytes, nothing of which is
// shared between pairs, against 4 flops per byte and head; the pool usually sits in L2.  So rows go from global memory
// straight to the registers of the warp that uses them, and everything else is arranged so that they are already MMA
// fragments there:
//   S^T = K . Q^T   m16n8k16, 16 keys x 8 heads.  Lane (g, t) reads 16 contiguous bytes of the rows g and g + 8 per 32 dims;
//                   the contraction order is permuted to match (the queries are loaded in the same permutation).
//   O^T = V^T . P^T m16n8k16, 16 dims x 8 heads x 16 keys.  Lane (g, t) reads 16 bytes of the rows 2t, 2t+1, 2t+8, 2t+9 per 64
//                   dims; a byte permute pairs the two keys of a dim, which is the A fragment; P^T comes out of the S^T
//                   accumulators with a pack and a movmatrix transpose.
// No shared memory and no block barrier in the key loop: every warp walks its own steps of 32 keys with its own online
// softmax, the next 16 keys' loads are issued before this 16's arithmetic, and the warps merge once at the end.  P is
// carried as three bf16 terms (24 significant bits), so that the tensor cores see what fp32 arithmetic would.  The rounded terms, and the
// rows that stand in for padding, make NaN of an infinite value; a warp whose outputs hold a NaN walks its keys once more with
// terms that are all positive and with zeros in place of padding, which leaves infinities as they are.  (Those terms for every
// warp: 220 -> 242 us at 300 tokens x 8 kv heads x 2048 keys.)
// With few (token, kv head) pairs a cluster of CTAs splits the keys of one pair and merges through distributed shared memory.
//
// Loads are bound by L1's tag stage, one 128-byte line a cycle: with 16-byte loads four lanes touch half a line of each key row
// (347 us at 777 tokens x 4 kv heads x 2048 keys, L1 at 96 %); 32-byte loads touch whole lines.
// Measured (B200, 128 / 128 dims): 777 tokens x 32 heads in 4 groups x 2048 keys 5785 -> 275 us = 11.8 TB/s out of L2 (kernel on
// the fp32 ALUs before; 271 without the check for infinities); 256 tokens x 8 heads x 256 keys 180 -> 34 us.
#include <type_traits>

#include "janus_common.cuh"
#include "sm100_ptx.cuh"

namespace janus {

using namespace ptx;

constexpr int AH_STEP = 32;      // keys a warp resolves at a time (one per lane); two MMA tiles of 16
constexpr int AH_HEADS = 8;      // query heads of a CTA (MMA N)

struct AhParams {
    const uint16_t* q;
    const uint16_t* k_pool;
    const uint16_t* v_pool;
    int64_t page_stride, tok_stride, head_stride;
    int H_q, heads_per_kv, groups_per_kv;
    const int32_t* idx;
    int k, page_size, page_shift;
    const int32_t* page_table;
    int64_t n_logical_pages;
    const int64_t* table_offsets;     // NULL, or [M + 1]: row t uses page_table[table_offsets[t] .. table_offsets[t + 1])
    float scale_log2e;
    uint16_t* out;
    float* lse;
    int32_t* dev_status;
};

__device__ __forceinline__ void ah_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t ah_transpose(uint32_t x) {   // 8x8 b16 matrix held one row per four lanes
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ float ah_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// One load of 16 or 32 bytes; rows are used once and not kept in L1.
__device__ __forceinline__ void ah_load(uint32_t (&v)[4], const uint16_t* p) {
    asm volatile("ld.global.L1::no_allocate.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "l"(p));
}
__device__ __forceinline__ void ah_load(uint32_t (&v)[8], const uint16_t* p) {
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(p));
}
__device__ __forceinline__ float ah_ld_cluster(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

template <int DV, int WARPS>
struct AhShared {
    float o[WARPS][AH_HEADS][DV];      // unnormalised outputs of the warps
    float m[WARPS][AH_HEADS];          // their reference maxima (log2 domain) and row sums
    float l[WARPS][AH_HEADS];
    float co[AH_HEADS][DV];               // the CTA's own merge, read by the other CTAs of a cluster
    float cm[AH_HEADS], cl[AH_HEADS];
};

// CTAs of an SM: twelve warps of up to 168 registers (sixteen of 128 spilled at 128 + 128 dims and were a third slower)
constexpr int ah_ctas_per_sm(int warps) { return 12 / warps; }

template <int DQK, int DV, bool WIDE, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, ah_ctas_per_sm(WARPS))
sparse_attn_heads_kernel(const AhParams p) {
    grid_launch_next();
    grid_wait();
    __shared__ AhShared<DV, WARPS> sh;
    constexpr int KE = WIDE ? 16 : 8;     // elements of a key row per load: four lanes read 128 or 64 contiguous bytes of it
    constexpr int KB = DQK / (4 * KE);
    constexpr int VE = WIDE && DV == 128 ? 16 : 8;      // of a value row: eight lanes read 256 or 128 contiguous bytes
    constexpr int VB = DV / (8 * VE);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
    const float neg_inf = __int_as_float(0xff800000);
    const uint32_t split = cluster_ctarank(), n_split = cluster_nctarank();      // 0 of 1 without a cluster
    const int64_t row = blockIdx.x / n_split;
    const int hk = blockIdx.y / p.groups_per_kv;
    const int h0 = hk * p.heads_per_kv + (blockIdx.y - hk * p.groups_per_kv) * AH_HEADS;
    const int n_heads = min(AH_HEADS, (hk + 1) * p.heads_per_kv - h0);
    const int32_t* table = p.page_table;
    int64_t n_pages = p.n_logical_pages;
    if (p.table_offsets != nullptr) {
        const int64_t tbl = ld_input(p.table_offsets + row);
        n_pages = ld_input(p.table_offsets + row + 1) - tbl;
        if (tbl < 0) n_pages = 0;         // a table that starts before the array: every selected token is reported and skipped
        else table += tbl;
    }

    uint32_t qf[KB][KE / 2];              // queries of head g in the order of the key fragments
    {
        const uint16_t* qrow = p.q + (row * p.H_q + h0 + (g < n_heads ? g : 0)) * DQK + t4 * KE;
#pragma unroll
        for (int c = 0; c < KB; ++c)
#pragma unroll
            for (int v = 0; v < KE / 8; ++v) {
                uint4 u = ld_input(reinterpret_cast<const uint4*>(qrow + c * 4 * KE + v * 8));
                if (g >= n_heads) u = make_uint4(0u, 0u, 0u, 0u);
                qf[c][4 * v] = u.x; qf[c][4 * v + 1] = u.y; qf[c][4 * v + 2] = u.z; qf[c][4 * v + 3] = u.w;
            }
    }

    const int32_t* my_idx = p.idx + row * p.k;
    const int n_steps = (p.k + AH_STEP - 1) / AH_STEP;
    const int stride = WARPS * static_cast<int>(n_split);
    auto load_raw = [&](int s) -> int {
        const int i = s * AH_STEP + lane;
        return i < p.k ? ld_input(my_idx + i) : -1;
    };
    // Element offset of the lane's key row.  A padding slot (or a token without a page) takes the row of the first valid lane, so
    // that no load needs a predicate; its logit is masked, and a row that is attended anyway adds no NaN but those of infinities.
    auto resolve = [&](int tok, uint32_t& mask) -> int64_t {
        int64_t off = 0;
        bool valid = false;
        if (tok >= 0) {
            const int64_t lp = p.page_shift >= 0 ? (tok >> p.page_shift) : (tok / p.page_size);
            const int within = p.page_shift >= 0 ? (tok & (p.page_size - 1)) : (tok % p.page_size);
            const int32_t phys = lp < n_pages ? ld_input(table + lp) : -1;
            if (phys < 0) {
                report(p.dev_status, JANUS_DEV_INDEX_OUT_OF_RANGE);
            } else {
                off = static_cast<int64_t>(phys) * p.page_stride + static_cast<int64_t>(within) * p.tok_stride + static_cast<int64_t>(hk) * p.head_stride;
                valid = true;
            }
        }
        mask = __ballot_sync(0xffffffffu, valid);
        if (mask != 0xffffffffu && mask != 0u) {
            const int64_t first = __shfl_sync(0xffffffffu, off, __ffs(mask) - 1);
            if (!valid) off = first;
        }
        return off;
    };
    uint32_t kf[2][KB][KE / 2];           // rows g and g + 8 of the next 16 keys
    auto load_k = [&](int64_t off, int u) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const uint16_t* src = p.k_pool + __shfl_sync(0xffffffffu, off, 16 * u + 8 * r + g) + t4 * KE;
#pragma unroll
            for (int c = 0; c < KB; ++c) ah_load(kf[r][c], src + c * 4 * KE);
        }
    };

    float o[VB][VE / 2][4];               // [block][dims VE g + 2j, VE g + 2j + 1][heads 2t, 2t+1 of either dim]
    float m_ref[2], l_sum[2];             // heads 2t, 2t + 1 (l: this lane's keys only)
    auto walk = [&](auto keep_infinities) {
        constexpr bool KEEP_INF = decltype(keep_infinities)::value;
#pragma unroll
        for (int b = 0; b < VB; ++b)
#pragma unroll
            for (int j = 0; j < VE / 2; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[b][j][e] = 0.f;
        m_ref[0] = m_ref[1] = neg_inf;
        l_sum[0] = l_sum[1] = 0.f;

        int s = static_cast<int>(split) * WARPS + warp;
        uint32_t mask = 0u;
        int64_t off = resolve(s < n_steps ? load_raw(s) : -1, mask);
        int raw_next = s + stride < n_steps ? load_raw(s + stride) : -1;
        if (mask != 0u) load_k(off, 0);
        for (; s < n_steps; s += stride) {
            uint32_t mask_next;
            const int64_t off_next = resolve(raw_next, mask_next);
            raw_next = s + 2 * stride < n_steps ? load_raw(s + 2 * stride) : -1;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (mask != 0u) {
                    uint32_t vf[4][VB][VE / 2];      // rows 2t, 2t+1, 2t+8, 2t+9 of these 16 keys
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const uint16_t* src = p.v_pool + __shfl_sync(0xffffffffu, off, 16 * u + 2 * t4 + (r & 1) + 8 * (r >> 1)) + g * VE;
#pragma unroll
                        for (int b = 0; b < VB; ++b) ah_load(vf[r][b], src + b * 8 * VE);
                    }
                    float sc[4] = {0.f, 0.f, 0.f, 0.f};      // keys g, g + 8 x heads 2t, 2t+1
#pragma unroll
                    for (int c = 0; c < KB; ++c)
#pragma unroll
                        for (int e = 0; e < KE / 2; e += 2)
                            ah_mma(sc, kf[0][c][e], kf[1][c][e], kf[0][c][e + 1], kf[1][c][e + 1], qf[c][e], qf[c][e + 1]);
                    if (u == 0) load_k(off, 1);
                    else if (mask_next != 0u) load_k(off_next, 0);
#pragma unroll
                    for (int e = 0; e < 4; ++e) sc[e] *= p.scale_log2e;
                    const uint32_t mk = mask >> (16 * u);
                    if ((mk & 0xffffu) != 0xffffu) {
                        if (((mk >> g) & 1u) == 0u) sc[0] = sc[1] = neg_inf;
                        if (((mk >> (g + 8)) & 1u) == 0u) sc[2] = sc[3] = neg_inf;
                        if constexpr (KEEP_INF) {
#pragma unroll
                            for (int r = 0; r < 4; ++r) {
                                if (((mk >> (2 * t4 + (r & 1) + 8 * (r >> 1))) & 1u) != 0u) continue;
#pragma unroll
                                for (int b = 0; b < VB; ++b)
#pragma unroll
                                    for (int j = 0; j < VE / 2; ++j) vf[r][b][j] = 0u;
                            }
                        }
                    }
                    // the reference maximum moves only when a key exceeds it by more than 2^8 (the sums are fp32)
                    const float mx0 = fmaxf(sc[0], sc[2]), mx1 = fmaxf(sc[1], sc[3]);
                    if (__any_sync(0xffffffffu, mx0 > m_ref[0] + 8.f || mx1 > m_ref[1] + 8.f)) {
                        float mx[2] = {mx0, mx1};
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
#pragma unroll
                            for (int d = 4; d < 32; d <<= 1) mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], d));
                            const float m_new = fmaxf(m_ref[h], mx[h]);
                            const float corr = m_ref[h] == neg_inf ? 1.f : ah_exp2(m_ref[h] - m_new);   // nothing accumulated yet: nothing to scale
                            m_ref[h] = m_new;
                            l_sum[h] *= corr;
#pragma unroll
                            for (int b = 0; b < VB; ++b)
#pragma unroll
                                for (int j = 0; j < VE / 2; ++j) { o[b][j][h] *= corr; o[b][j][2 + h] *= corr; }
                        }
                    }
                    const float nm0 = m_ref[0] == neg_inf ? 0.f : m_ref[0], nm1 = m_ref[1] == neg_inf ? 0.f : m_ref[1];
                    float pr[4] = {ah_exp2(sc[0] - nm0), ah_exp2(sc[1] - nm1), ah_exp2(sc[2] - nm0), ah_exp2(sc[3] - nm1)};
                    l_sum[0] += pr[0] + pr[2];
                    l_sum[1] += pr[1] + pr[3];
                    // P = three bf16 terms; each becomes the B fragment (head g, keys 2t, 2t+1 | 2t+8, 2t+9)
                    uint32_t pb[3][2];
#pragma unroll
                    for (int term = 0; term < 3; ++term) {
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            uint32_t bits;
                            if constexpr (KEEP_INF) {      // the largest bf16 below P, the largest below the rest, and what is left: eight bits
                                const int below = term < 2 ? 1 : 0;
                                bits = __byte_perm(max(__float_as_int(pr[2 * r]) - below, 0), max(__float_as_int(pr[2 * r + 1]) - below, 0), 0x7632);
                            } else {
                                const __nv_bfloat162 v = __floats2bfloat162_rn(pr[2 * r], pr[2 * r + 1]);
                                bits = *reinterpret_cast<const uint32_t*>(&v);
                            }
                            pb[term][r] = ah_transpose(bits);
                            pr[2 * r] -= __uint_as_float(bits << 16);
                            pr[2 * r + 1] -= __uint_as_float(bits & 0xffff0000u);
                        }
                    }
#pragma unroll
                    for (int b = 0; b < VB; ++b)
#pragma unroll
                        for (int j = 0; j < VE / 2; ++j) {
                            const uint32_t a0 = __byte_perm(vf[0][b][j], vf[1][b][j], 0x5410), a1 = __byte_perm(vf[0][b][j], vf[1][b][j], 0x7632);
                            const uint32_t a2 = __byte_perm(vf[2][b][j], vf[3][b][j], 0x5410), a3 = __byte_perm(vf[2][b][j], vf[3][b][j], 0x7632);
#pragma unroll
                            for (int term = 2; term >= 0; --term) ah_mma(o[b][j], a0, a1, a2, a3, pb[term][0], pb[term][1]);
                        }
                } else if (u == 1 && mask_next != 0u) {
                    load_k(off_next, 0);
                }
            }
            mask = mask_next;
            off = off_next;
        }
    };
    walk(std::false_type{});
    bool has_nan = false;
#pragma unroll
    for (int b = 0; b < VB; ++b)
#pragma unroll
        for (int j = 0; j < VE / 2; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) has_nan = has_nan || isnan(o[b][j][e]);
    if (__any_sync(0xffffffffu, has_nan)) walk(std::true_type{});

    // ---- merge: the warps of the CTA, then the CTAs of the cluster
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int d = 4; d < 32; d <<= 1) l_sum[h] += __shfl_xor_sync(0xffffffffu, l_sum[h], d);
        if (g == 0) { sh.m[warp][2 * t4 + h] = m_ref[h]; sh.l[warp][2 * t4 + h] = l_sum[h]; }
#pragma unroll
        for (int b = 0; b < VB; ++b) {
            float4* dst = reinterpret_cast<float4*>(&sh.o[warp][2 * t4 + h][b * 8 * VE + g * VE]);
#pragma unroll
            for (int j = 0; j < VE / 2; j += 2) dst[j / 2] = make_float4(o[b][j][h], o[b][j][2 + h], o[b][j + 1][h], o[b][j + 1][2 + h]);
        }
    }
    __syncthreads();
    constexpr int PER = AH_HEADS * DV / (32 * WARPS);     // values of a thread: PER consecutive dims of one head
    const int h = threadIdx.x * PER / DV, d0 = threadIdx.x * PER % DV;
    float m_all = neg_inf, l_all = 0.f, acc[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) acc[e] = 0.f;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) m_all = fmaxf(m_all, sh.m[w][h]);
    const float m_safe = m_all == neg_inf ? 0.f : m_all;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
        const float f = ah_exp2(sh.m[w][h] - m_safe);
        l_all += f * sh.l[w][h];
#pragma unroll
        for (int e = 0; e < PER; ++e) acc[e] += f * sh.o[w][h][d0 + e];
    }
    if (n_split > 1) {
#pragma unroll
        for (int e = 0; e < PER; ++e) sh.co[h][d0 + e] = acc[e];
        if (d0 == 0) { sh.cm[h] = m_all; sh.cl[h] = l_all; }
        cluster_sync_all();
        if (split == 0) {
            for (uint32_t r = 1; r < n_split; ++r) {
                const float m_r = ah_ld_cluster(mapa_shared(smem_u32(&sh.cm[h]), r)), l_r = ah_ld_cluster(mapa_shared(smem_u32(&sh.cl[h]), r));
                const float m_new = fmaxf(m_all, m_r), safe = m_new == neg_inf ? 0.f : m_new;
                const float fa = ah_exp2(m_all - safe), fb = ah_exp2(m_r - safe);
                l_all = fa * l_all + fb * l_r;
                const uint32_t src = mapa_shared(smem_u32(&sh.co[h][d0]), r);
#pragma unroll
                for (int e = 0; e < PER; ++e) acc[e] = fa * acc[e] + fb * ah_ld_cluster(src + 4 * e);
                m_all = m_new;
            }
        }
        cluster_sync_all();               // nobody leaves while its shared memory is read
        if (split != 0) return;
    }
    if (h < n_heads) {
        const float inv = l_all != 0.f ? 1.f / l_all : 0.f;          // (a NaN is a sum)
        uint32_t* dst = reinterpret_cast<uint32_t*>(p.out + (row * p.H_q + h0 + h) * DV + d0);
#pragma unroll
        for (int e = 0; e < PER; e += 2) {
            const __nv_bfloat162 v = __floats2bfloat162_rn(acc[e] * inv, acc[e + 1] * inv);
            dst[e / 2] = *reinterpret_cast<const uint32_t*>(&v);
        }
        if (d0 == 0 && p.lse != nullptr) p.lse[row * p.H_q + h0 + h] = l_all != 0.f ? (m_all + log2f(l_all)) * 0.6931471805599453f : neg_inf;
    }
}

bool sparse_attn_heads_supported(int d_qk, int d_v) { return (d_qk == 64 || d_qk == 128 || d_qk == 192) && (d_v == 64 || d_v == 128); }

template <int DQK, int DV>
static int launch_heads(const AhParams& p, int M, int n_kv_heads, cudaStream_t stream) {
    const int groups = n_kv_heads * p.groups_per_kv;
    if (groups > 65535) return JANUS_ERR_UNSUPPORTED;
    // How many warps share the keys of one (token, kv head) pair.  A warp's step of 32 keys costs the memory latency, 1.3 us, as
    // long as L2 keeps up.  Pairs that fit one CTA per SM take eight warps, and clusters of up to eight CTAs while those still
    // fit (1 token x 4 kv heads x 2048 keys: 43.9 us with two warps a pair, 17.2 with eight, 8.5 with eight CTAs of eight; 16
    // tokens: 17.6 and, with two CTAs, 12.6; two waves of clusters are slower than one of CTAs: 18.2 against 23.7 at 32 tokens).
    // Beyond that, CTAs of four warps (1024 pairs x 2048 keys: 109 us, 134 with two, 124 with eight), or of two when a warp
    // would be left with fewer than four steps (2048 pairs x 256 keys: 33.7 us against 37.3).
    const int64_t pairs = static_cast<int64_t>(M) * groups;
    const int steps = (p.k + AH_STEP - 1) / AH_STEP;
    int warps = 8, split = 1;
    if (pairs <= 148) {
        while (split < 8 && pairs * split * 2 <= 148 && steps >= 16 * split) split *= 2;
    } else {
        warps = steps >= 16 ? 4 : 2;
    }
    const dim3 grid(static_cast<unsigned>(M) * split, groups);
    // 32-byte loads where every row starts on 32 bytes
    const bool wide = ((reinterpret_cast<uintptr_t>(p.k_pool) | reinterpret_cast<uintptr_t>(p.v_pool)) & 31u) == 0 &&
                      ((p.page_stride | p.tok_stride | p.head_stride) & 15) == 0;
#define JANUS_AH_CASE(WIDE)                                                                                       \
    if (warps == 2) JANUS_CUDA_CHECK(launch_kernel(sparse_attn_heads_kernel<DQK, DV, WIDE, 2>, grid, 32 * warps, 0, stream, split, p));    \
    else if (warps == 4) JANUS_CUDA_CHECK(launch_kernel(sparse_attn_heads_kernel<DQK, DV, WIDE, 4>, grid, 32 * warps, 0, stream, split, p)); \
    else JANUS_CUDA_CHECK(launch_kernel(sparse_attn_heads_kernel<DQK, DV, WIDE, 8>, grid, 32 * warps, 0, stream, split, p));
    if (wide) {
        JANUS_AH_CASE(true)
    } else {
        JANUS_AH_CASE(false)
    }
#undef JANUS_AH_CASE
    return JANUS_OK;
}

int launch_sparse_attn_heads(const void* q, int M, int H_q, int d_qk, const void* k_pool, const void* v_pool, int64_t page_stride,
                             int64_t tok_stride, int64_t head_stride, int n_kv_heads, int d_v, const int32_t* idx, int k, int page_size,
                             const int32_t* page_table, int64_t n_logical_pages, const int64_t* table_offsets, float softmax_scale, void* out,
                             float* lse, int32_t* dev_status, cudaStream_t stream) {
    AhParams p;
    p.q = static_cast<const uint16_t*>(q);
    p.k_pool = static_cast<const uint16_t*>(k_pool);
    p.v_pool = static_cast<const uint16_t*>(v_pool);
    p.page_stride = page_stride; p.tok_stride = tok_stride; p.head_stride = head_stride;
    p.H_q = H_q;
    p.heads_per_kv = H_q / n_kv_heads;
    p.groups_per_kv = (p.heads_per_kv + AH_HEADS - 1) / AH_HEADS;
    p.idx = idx; p.k = k; p.page_size = page_size;
    p.page_shift = -1;
    if ((page_size & (page_size - 1)) == 0) {
        p.page_shift = 0;
        while ((1 << p.page_shift) < page_size) ++p.page_shift;
    }
    p.page_table = page_table; p.n_logical_pages = n_logical_pages; p.table_offsets = table_offsets;
    p.scale_log2e = softmax_scale * 1.4426950408889634f;
    p.out = static_cast<uint16_t*>(out);
    p.lse = lse; p.dev_status = dev_status;
    if (d_v == 64) {
        if (d_qk == 64) return launch_heads<64, 64>(p, M, n_kv_heads, stream);
        if (d_qk == 128) return launch_heads<128, 64>(p, M, n_kv_heads, stream);
        return launch_heads<192, 64>(p, M, n_kv_heads, stream);
    }
    if (d_qk == 64) return launch_heads<64, 128>(p, M, n_kv_heads, stream);
    if (d_qk == 128) return launch_heads<128, 128>(p, M, n_kv_heads, stream);
    return launch_heads<192, 128>(p, M, n_kv_heads, stream);
}

}  // namespace janus
