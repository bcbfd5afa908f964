"""Latent attention of few tokens, whose keys a cluster of CTA pairs splits and merges: cluster sizes from two to eight pairs, ragged last
tiles, pairs without a single valid key, rows without any, logits whose maximum sits in one pair only.  Reference: the oracle."""
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


@pytest.mark.parametrize("M,k,gain", [(1, 2048, 1.0), (1, 2048, 12.0), (2, 1985, 1.0), (7, 1500, 4.0), (10, 2048, 1.0), (19, 2001, 12.0), (30, 1089, 1.0),
                                      (3, 65, 1.0)])
def test_split_latent_attention_matches_oracle(M, k, gain):
    rng = np.random.default_rng(M * 5000 + k)
    page, S = 64, 6000
    n_log = (S + page - 1) // page
    table = rng.permutation(n_log).astype(np.int32)
    pool = W.to_bf16_bits((rng.standard_normal((n_log, page, 1, 576)) / 4).astype(np.float32))
    Q = W.to_bf16_bits((gain * rng.standard_normal((M, 128, 576))).astype(np.float32))
    idx = np.stack([rng.permutation(S)[:k] for _ in range(M)]).astype(np.int32)
    if M > 1:
        idx[1, :k // 2] = -1            # the first pairs of the cluster have no key
        idx[0, k // 3:] = -1            # the last ones
    if M > 2:
        idx[2] = -1
    scale = 1.0 / 24.0
    kd, td = B.to_device(pool, "bf16"), B.to_device(table, "i32")
    out, lse = B.janus_sparse_attn_prefill(B.to_device(Q, "bf16"), kd, kd, B.to_device(idx, "i32"), page_table=td, page_size=page,
                                           softmax_scale=scale, d_v=512)
    B.check_dev_status()
    ref_o, ref_l = O.sparse_attention(Q, pool, pool, table, idx, page_size=page, softmax_scale=scale, d_qk=576, d_v=512)
    Hp.assert_attention_close(Hp.bf16_tensor_to_f64(out), ref_o, "split")
    got, fin = lse.cpu().numpy().astype(np.float64), np.isfinite(ref_l)
    assert np.array_equal(np.isfinite(got), fin)
    # partial logits cross between the two SMs as fp16: 2^-11 of a partial logit (up to 40 here), and P is bf16
    assert np.all(np.abs(got[fin] - ref_l[fin]) <= 2e-2 + 1e-3 * np.abs(ref_l[fin]))


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
