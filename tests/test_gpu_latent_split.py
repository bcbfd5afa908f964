"""Latent attention of few tokens, whose keys a cluster of CTA pairs splits and merges: cluster sizes from two to eight pairs, ragged last
tiles, pairs without a single valid key, rows without any, logits whose maximum sits in one pair only, pools whose rows are gathered by
number and, where pages are padded, by address; one page table for all rows, and one for each.  Reference: the oracle."""
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


def draw(M, k, gain, page, S):
    rng = np.random.default_rng(M * 5000 + k)
    n_log = (S + page - 1) // page
    Q = W.to_bf16_bits((gain * rng.standard_normal((M, 128, 576))).astype(np.float32))
    idx = np.stack([rng.permutation(S)[:k] for _ in range(M)]).astype(np.int32)
    if M > 1:
        idx[1, :k // 2] = -1            # the first pairs of the cluster have no key
        idx[0, k // 3:] = -1            # the last ones
    if M > 2:
        idx[2] = -1
    return rng, n_log, Q, idx


def check(out, lse, ref_o, ref_l):
    Hp.assert_attention_close(Hp.bf16_tensor_to_f64(out), ref_o, "split")
    got, fin = lse.cpu().numpy().astype(np.float64), np.isfinite(ref_l)
    assert np.array_equal(np.isfinite(got), fin)
    # the sum adds probabilities rounded to bf16 (2^-9 each); the logits are fp32 sums of 576 exact products
    assert np.all(np.abs(got[fin] - ref_l[fin]) <= 2.0 ** -8 + 1e-5 * np.abs(ref_l[fin]))


# 577 keys are five tiles, the last of one key, which three tokens split; 65 are one tile, which nothing splits
@pytest.mark.parametrize("tok_pad,page_pad", [(0, 0), (0, 8), (64, 72)])
@pytest.mark.parametrize("M,k,gain", [(1, 2048, 1.0), (1, 2048, 12.0), (2, 1985, 1.0), (7, 1500, 4.0), (10, 2048, 1.0), (19, 2001, 12.0), (30, 1089, 1.0),
                                      (3, 577, 1.0), (3, 65, 1.0)])
def test_split_latent_attention_matches_oracle(M, k, gain, tok_pad, page_pad):
    page, S = 64, 6000
    rng, n_log, Q, idx = draw(M, k, gain, page, S)
    table = rng.permutation(n_log).astype(np.int32)
    pool = W.to_bf16_bits((rng.standard_normal((n_log, page, 1, 576)) / 4).astype(np.float32))
    scale = 1.0 / 24.0
    kd, td = Hp.strided_pool(pool, tok_pad, page_pad), B.to_device(table, "i32")
    out, lse = B.janus_sparse_attn_prefill(B.to_device(Q, "bf16"), kd, kd, B.to_device(idx, "i32"), page_table=td, page_size=page,
                                           softmax_scale=scale, d_v=512)
    B.check_dev_status()
    check(out, lse, *O.sparse_attention(Q, pool, pool, table, idx, page_size=page, softmax_scale=scale, d_qk=576, d_v=512))


@pytest.mark.parametrize("tok_pad,page_pad", [(0, 0), (0, 8)])
@pytest.mark.parametrize("M,k", [(5, 2048), (12, 1100)])
def test_split_decode_takes_every_rows_own_table(M, k, tok_pad, page_pad):
    page, S, scale = 16, 3000, 1.0 / 24.0
    rng, n_log, Q, idx = draw(M, k, 2.0, page, S)
    tables = rng.permutation(M * n_log).astype(np.int32)
    offsets = torch.arange(M + 1, dtype=torch.int64, device="cuda") * n_log
    pool = W.to_bf16_bits((rng.standard_normal((M * n_log, page, 1, 576)) / 4).astype(np.float32))
    kd = Hp.strided_pool(pool, tok_pad, page_pad)
    out, lse = B.janus_sparse_attn_decode(B.to_device(Q, "bf16"), kd, kd, B.to_device(idx, "i32"), page_tables=B.to_device(tables, "i32"), table_offsets=offsets,
                                          page_size=page, softmax_scale=scale, d_v=512)
    B.check_dev_status()
    refs = [O.sparse_attention(Q[t:t + 1], pool, pool, tables[t * n_log:(t + 1) * n_log], idx[t:t + 1], page_size=page, softmax_scale=scale, d_qk=576, d_v=512)
            for t in range(M)]
    check(out, lse, np.concatenate([o for o, _ in refs]), np.concatenate([l for _, l in refs]))


@pytest.mark.parametrize("M", [1, 5, 200])
def test_a_call_on_a_broken_pipeline_does_nothing(M):
    """The status word says that a wait has given up: no CTA starts, all of a cluster agree on it, and the outputs stay as they were."""
    q, pool = torch.zeros((M, 128, 576), dtype=torch.bfloat16, device="cuda"), torch.zeros((8, 64, 1, 576), dtype=torch.bfloat16, device="cuda")
    idx, table = torch.arange(512, dtype=torch.int32, device="cuda").repeat(M, 1), torch.arange(8, dtype=torch.int32, device="cuda")
    out, lse = torch.full((M, 128, 512), 7.0, dtype=torch.bfloat16, device="cuda"), torch.full((M, 128), 7.0, device="cuda")
    status = torch.full((1,), 103, dtype=torch.int32, device="cuda")
    rc = B.load().janus_sparse_attn_prefill(q.data_ptr(), M, 128, 576, pool.data_ptr(), pool.data_ptr(), pool.stride(0), pool.stride(1), pool.stride(2), 1, 512,
                                            idx.data_ptr(), 512, 64, table.data_ptr(), 8, 1.0, out.data_ptr(), lse.data_ptr(), None, 0, status.data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
    assert rc == B.JANUS_OK
    assert bool((out == 7).all()) and bool((lse == 7).all()) and int(status.item()) == 103
