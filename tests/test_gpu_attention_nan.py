"""A query that is not a number: its heads come out as NaN, with a log-sum-exp of NaN, in every attention kernel and whether the NaN is in one
head or in all of them; the other heads and rows are what they are without it.  (Zeros and -inf mean an empty selection.)"""
import pytest
import torch

from paper_2609_36938_b200 import binding as B
from paper_2609_36938_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()
    yield
    B.check_dev_status()


@pytest.mark.parametrize("M,k", [(3, 700), (5, 2000), (200, 130)])
@pytest.mark.parametrize("h_q,n_kv,d_qk,d_v", [(128, 1, 576, 512), (8, 8, 128, 128), (32, 4, 128, 128), (16, 2, 96, 96)])
def test_a_nan_query_comes_out_as_nan(M, k, h_q, n_kv, d_qk, d_v):
    g = torch.Generator(device="cuda").manual_seed(M + k + d_qk)
    pages, page = 40, 64
    normal = lambda *s: torch.randn(s, device="cuda", generator=g).bfloat16()  # noqa: E731
    k_pool = normal(pages, page, n_kv, d_qk)
    v_pool = k_pool if d_qk == 576 else normal(pages, page, n_kv, d_v)
    q, table = normal(M, h_q, d_qk), torch.randperm(pages, device="cuda", generator=g).int()
    idx = torch.stack([torch.randperm(pages * page, device="cuda", generator=g)[:k] for _ in range(M)]).int()
    idx[M - 1] = -1

    def attend(x):
        out, lse = B.janus_sparse_attn_prefill(x, k_pool, v_pool, idx, page_table=table, page_size=page, softmax_scale=d_qk ** -0.5, d_v=d_v)
        B.check_dev_status()
        return out.float(), lse

    want, want_l = attend(q)
    bad = torch.zeros((M, h_q), dtype=torch.bool, device="cuda")
    bad[0] = True                       # every head of a row
    bad[1, h_q // 2] = True             # one head
    nan = q.clone()
    nan[:, :, 7][bad] = float("nan")
    got, got_l = attend(nan)
    assert bool(got[bad].isnan().all()) and bool(got_l[bad].isnan().all())
    assert bool((got[M - 1] == 0).all()) and bool(torch.isneginf(got_l[M - 1]).all())
    # the same sums of probabilities, which a warp that meets a NaN may split into other bf16 terms
    torch.testing.assert_close(got[~bad], want[~bad], rtol=2.0 ** -7, atol=2.0 ** -9)
    torch.testing.assert_close(got_l[~bad], want_l[~bad], rtol=0, atol=2.0 ** -12)
