"""Latent attention by CTA pairs: tokens that follow one another on a pair with one to three tiles each, ragged last tiles, pools whose
rows lie at whole multiples of the token stride (gathered by number) and pools with padded pages (gathered by address), rows that were
not selected and must not be touched.  Reference: the oracle."""
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


@pytest.mark.parametrize("tok_pad,page_pad", [(0, 0), (64, 0), (0, 576), (0, 8), (64, 72)])
@pytest.mark.parametrize("M,k,page", [(1, 1, 64), (3, 300, 16), (160, 128, 64), (160, 129, 64), (230, 37, 48), (230, 383, 16)])
def test_tokens_strides_and_tails(M, k, page, tok_pad, page_pad):
    rng = np.random.default_rng(M * 1000 + k)
    S = 1500
    n_log = (S + page - 1) // page
    table = rng.permutation(n_log + 3)[:n_log].astype(np.int32)
    pool = W.to_bf16_bits((rng.standard_normal((n_log + 3, page, 1, 576)) / 4).astype(np.float32))
    Q = W.to_bf16_bits((2.0 * rng.standard_normal((M, 128, 576))).astype(np.float32))
    idx = np.stack([rng.permutation(S)[:k] for _ in range(M)]).astype(np.int32)
    idx[M // 2, k // 2:] = -1
    if M > 1:
        idx[M - 1] = -1
    # rows that no token selects, among them the first of every page that is not in the table, hold NaN
    used = np.zeros((n_log + 3, page), bool)
    sel = idx[idx >= 0]
    used[table[sel // page], sel % page] = True
    pool[~used] = 0x7fc0
    kd = Hp.strided_pool(pool, tok_pad, page_pad)
    scale = 1.0 / 24.0
    out, lse = B.janus_sparse_attn_prefill(B.to_device(Q, "bf16"), kd, kd, B.to_device(idx, "i32"), page_table=B.to_device(table, "i32"), page_size=page,
                                           softmax_scale=scale, d_v=512)
    B.check_dev_status()
    rows = sorted({0, M // 2, M - 1, *rng.integers(0, M, 12).tolist()})       # (the first and the later tokens of a pair)
    pool[~used] = 0
    ref_o, ref_l = O.sparse_attention(Q[rows], pool, pool, table, idx[rows], page_size=page, softmax_scale=scale, d_qk=576, d_v=512)
    Hp.assert_attention_close(Hp.bf16_tensor_to_f64(out[rows]), ref_o, "pair")
    assert bool(torch.isfinite(out).all())
    got, fin = lse[rows].cpu().numpy().astype(np.float64), np.isfinite(ref_l)
    assert np.array_equal(np.isfinite(got), fin)
    # the sum adds probabilities rounded to bf16 (2^-9 each); the logits are fp32 sums of 576 exact products
    assert np.all(np.abs(got[fin] - ref_l[fin]) <= 2.0 ** -8 + 1e-5 * np.abs(ref_l[fin]))
