"""The multi-head / grouped attention kernel at the edges of its dispatch: every key / value dim it takes, head groups of 1 to 16,
selections around its 16- and 32-key tiles, few and many (token, kv head) pairs (clusters, 8-, 4- and 2-warp CTAs), padding anywhere,
rows that start on 16 but not 32 bytes.  Reference: the oracle; tolerance as in helpers.assert_attention_close (bf16 outputs)."""
import numpy as np
import pytest
import torch

import helpers as Hp
from oracle import janus_oracle as O
from paper_2609_36938_b200 import binding as B
from paper_2609_36938_b200 import build
from paper_2609_36938_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()
    yield
    B.check_dev_status()


@pytest.mark.parametrize("M,n_kv,group,d_qk,d_v,k,shift", [
    (1, 4, 8, 128, 128, 2048, 0),     # clusters of eight CTAs
    (9, 4, 3, 64, 64, 1037, 0),       # clusters of four, ragged tail
    (40, 2, 16, 192, 128, 513, 0),    # two head groups per kv head; one CTA per pair
    (75, 2, 1, 128, 64, 16, 0),       # 150 pairs: two warps, one of them without keys
    (300, 1, 8, 64, 128, 511, 0),     # four warps
    (160, 1, 5, 192, 64, 33, 8),      # rows on 16-byte boundaries
    (3, 8, 2, 128, 128, 17, 8),
])
def test_heads_kernel_matches_oracle(M, n_kv, group, d_qk, d_v, k, shift):
    rng = np.random.default_rng(M * 1000 + k)
    H_q, page, S = n_kv * group, 64, 3000
    n_log = (S + page - 1) // page
    table = rng.permutation(n_log).astype(np.int32)
    d_row = max(d_qk, d_v)
    pools = [W.to_bf16_bits((rng.standard_normal((n_log, page, n_kv, d_row)) / 4).astype(np.float32)) for _ in range(2)]
    Q = W.to_bf16_bits(rng.standard_normal((M, H_q, d_qk)).astype(np.float32))
    idx = np.full((M, k), -1, np.int32)
    for t in range(M):
        m = k if t % 3 else int(rng.integers(0, k + 1))
        idx[t, np.sort(rng.permutation(k)[:m])] = rng.choice(S, size=m, replace=False)
    dev = []
    for x in pools:
        flat = torch.empty((x.size + 16,), dtype=torch.bfloat16, device="cuda")
        view = flat[shift:shift + x.size].view(x.shape)
        view.copy_(B.to_device(x, "bf16"))
        dev.append(view)
    scale = float(1.0 / np.sqrt(d_qk))
    out, lse = B.janus_sparse_attn_prefill(B.to_device(Q, "bf16"), dev[0], dev[1], B.to_device(idx, "i32"), page_table=B.to_device(table, "i32"),
                                           page_size=page, softmax_scale=scale, d_v=d_v)
    B.check_dev_status()
    rows = sorted({0, 1 % M, M // 2, M - 1})
    ref_o, ref_l = O.sparse_attention(Q, pools[0], pools[1], table, idx[rows], page_size=page, softmax_scale=scale, d_qk=d_qk, d_v=d_v, rows=rows)
    Hp.assert_attention_close(Hp.bf16_tensor_to_f64(out)[rows], ref_o, "heads")
    got, fin = lse.cpu().numpy().astype(np.float64)[rows], np.isfinite(ref_l)
    assert np.array_equal(np.isfinite(got), fin)
    # logits are fp32 sums of d_qk exact products (relative error d_qk 2^-24 of their absolute sum, below 1e-4 here)
    assert np.all(np.abs(got[fin] - ref_l[fin]) <= 1e-4 * (1 + np.abs(ref_l[fin])))


@pytest.mark.parametrize("M,n_kv,group,d_qk,d_v,k", [(3, 2, 4, 128, 128, 1), (5, 4, 8, 64, 64, 37), (2, 1, 8, 192, 128, 2048), (300, 1, 1, 128, 64, 45)])
def test_infinite_values_come_out_as_they_are(M, n_kv, group, d_qk, d_v, k):
    """Every token's value is +Inf in one dim, -Inf in another and finite elsewhere: so are the outputs, whatever padding is near."""
    rng = np.random.default_rng(M + k)
    H_q, page, S = n_kv * group, 16, 2500
    n_log = (S + page - 1) // page
    table = np.arange(n_log, dtype=np.int32)
    kp, v = rng.standard_normal((n_log, page, n_kv, max(d_qk, d_v))).astype(np.float32) / 4, rng.standard_normal((n_log, page, n_kv, max(d_qk, d_v))).astype(np.float32)
    v[..., 5], v[..., d_v - 2] = np.inf, -np.inf
    Q = W.to_bf16_bits(rng.standard_normal((M, H_q, d_qk)).astype(np.float32))
    idx = np.stack([rng.permutation(S)[:k] for _ in range(M)]).astype(np.int32)
    idx[(rng.random(idx.shape) < 0.3) & (np.arange(k) > 0)] = -1
    out, _ = B.janus_sparse_attn_prefill(B.to_device(Q, "bf16"), B.to_device(W.to_bf16_bits(kp), "bf16"), B.to_device(W.to_bf16_bits(v), "bf16"), B.to_device(idx, "i32"),
                                         page_table=B.to_device(table, "i32"), page_size=page, softmax_scale=d_qk ** -0.5, d_v=d_v)
    B.check_dev_status()
    got = Hp.bf16_tensor_to_f64(out)
    want = np.zeros(d_v)
    want[5], want[d_v - 2] = np.inf, -np.inf
    assert np.array_equal(np.where(np.isfinite(got), 0, got), np.broadcast_to(want, got.shape))


@pytest.mark.parametrize("n,n_kv,group,d_qk,d_v,k", [(1, 4, 8, 128, 128, 700), (6, 2, 4, 64, 64, 129), (200, 1, 1, 192, 128, 33)])
def test_decode_rows_have_tables_of_their_own(n, n_kv, group, d_qk, d_v, k):
    """One query row per session, each with its own page table and history; a table that starts before the array has no pages (reported)."""
    rng = np.random.default_rng(n + k)
    H_q, page = n_kv * group, 32
    lengths = rng.integers(k, 3 * k, n)
    pages = (lengths + page - 1) // page
    off = np.concatenate([[0], np.cumsum(pages)]).astype(np.int64)
    n_phys = int(off[-1])
    tables = rng.permutation(n_phys).astype(np.int32)
    pools = [W.to_bf16_bits((rng.standard_normal((n_phys, page, n_kv, max(d_qk, d_v))) / 4).astype(np.float32)) for _ in range(2)]
    Q = W.to_bf16_bits(rng.standard_normal((n, H_q, d_qk)).astype(np.float32))
    idx = np.stack([rng.permutation(int(m))[:k] for m in lengths]).astype(np.int32)
    idx[rng.random(idx.shape) < 0.1] = -1
    scale = float(d_qk ** -0.5)
    args = (B.to_device(Q, "bf16"), B.to_device(pools[0], "bf16"), B.to_device(pools[1], "bf16"), B.to_device(idx, "i32"))
    out, lse = B.janus_sparse_attn_decode(*args, page_tables=B.to_device(tables, "i32"), table_offsets=torch.from_numpy(off).cuda(), page_size=page,
                                          softmax_scale=scale, d_v=d_v)
    B.check_dev_status()
    for b in sorted({0, n // 2, n - 1}):
        ref_o, ref_l = O.sparse_attention(Q[b:b + 1], pools[0], pools[1], tables[off[b]:off[b + 1]], idx[b:b + 1], page_size=page, softmax_scale=scale,
                                          d_qk=d_qk, d_v=d_v)
        Hp.assert_attention_close(Hp.bf16_tensor_to_f64(out)[b:b + 1], ref_o, f"session {b}")
        assert np.all(np.abs(lse.cpu().numpy().astype(np.float64)[b] - ref_l[0]) <= 1e-4 * (1 + np.abs(ref_l[0])))
    bad = off.copy()
    bad[0] = -1
    out2, lse2 = B.janus_sparse_attn_decode(*args, page_tables=B.to_device(tables, "i32"), table_offsets=torch.from_numpy(bad).cuda(), page_size=page,
                                            softmax_scale=scale, d_v=d_v)
    assert bool((out2[0] == 0).all()) and bool(torch.isneginf(lse2[0]).all()) and torch.equal(out2[1:], out[1:])
    with pytest.raises(B.JanusError, match="OUT_OF_RANGE"):
        B.check_dev_status()
