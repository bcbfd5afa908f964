"""How the tensor-core indexer shares its tiles out: ranges inside one token group and across several or many of one tile, one and many tiles per CTA, both sub-tile
counts, masked tails of rows (ragged ends included), and batches of sessions on either side of the even-share rule, more sessions than
the block that scans them, empty ones and one-tile ones among them.  Against the oracle; tolerance as in test_gpu_parity.py (fp32 sums of
exact products)."""
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


def operands(rng, n_q, n_k, H, D, dtype):
    q, k = rng.standard_normal((n_q, H, D)).astype(np.float32), rng.standard_normal((n_k, D)).astype(np.float32)
    w = (rng.uniform(-0.2, 1, (n_q, H)) / 8).astype(np.float32)
    if dtype == "bf16":
        return W.to_bf16_bits(q), W.to_bf16_bits(k), w, None, None
    return W.to_e4m3_bits(q), W.to_e4m3_bits(k), w, np.exp2(rng.uniform(-1, 1, H)).astype(np.float32), np.exp2(rng.uniform(-1, 1, n_k)).astype(np.float32)


@pytest.mark.parametrize("M,L,n_keys,H,D,dtype,causal", [
    (1, 0, 1, 64, 128, "bf16", True), (1, 200, 201, 64, 128, "fp8", True), (8, 4000, 4008, 64, 128, "bf16", True),
    (9, 4000, 4009, 64, 128, "bf16", True), (700, 0, 700, 64, 128, "fp8", True), (1300, 129, 1429, 32, 128, "bf16", True),
    (33, 5000, 4777, 64, 128, "fp8", False), (513, 3, 515, 4, 64, "bf16", True), (100, 5000, 5100, 8, 128, "fp8", True),
    (2500, 130, 2630, 64, 64, "bf16", True), (300, 1000, 1203, 16, 128, "bf16", True),
    (3001, 0, 3001, 64, 128, "bf16", True), (1192, 0, 100, 64, 128, "bf16", True), (2400, 0, 2400, 64, 128, "fp8", True),
])
def test_scores_of_every_range(M, L, n_keys, H, D, dtype, causal):
    rng = np.random.default_rng(M + n_keys)
    q, k, w, qs, ks = operands(rng, M, n_keys, H, D, dtype)
    dev = lambda x, kind: B.to_device(x, kind)  # noqa: E731
    sc = torch.full((M, (n_keys + 3) // 4 * 4), float("nan"), device="cuda")
    B.janus_indexer_scores(dev(q, dtype), dev(k, dtype), dev(w, "f32"), q_scale=dev(qs, "f32"), k_scale=dev(ks, "f32"), q_pos0=L, causal=causal, scores=sc)
    B.check_dev_status()
    assert bool(torch.isnan(sc[:, n_keys:]).all())                        # columns past the keys are left alone
    got = sc[:, :n_keys].cpu().numpy()
    rows = np.unique(np.concatenate([rng.integers(0, M, 24), [0, M - 1, M // 2, max(0, M // 2 - 1)]]))
    ref = O.indexer_scores(q, k, w, dtype=dtype, q_scale=qs, k_scale=ks, q_pos0=L, causal=causal, rows=rows)
    Hp.assert_scores_close(got[rows], ref, 1e-4, f"{M} rows x {n_keys}")
    pos = np.arange(n_keys)[None, :] > L + np.arange(M)[:, None]
    assert np.array_equal(np.isneginf(got), pos if causal else np.zeros_like(pos)) and not np.isnan(got).any()


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("lengths", [[1], [130, 0, 0, 5], [90000] + [129] * 30, [60, 128, 300, 1000] * 64, [5000] * 33, [7] * 700])
def test_batch_scores_of_every_session(lengths, dtype):
    rng = np.random.default_rng(len(lengths))
    n = len(lengths)
    off = np.concatenate([[0], np.cumsum([(x + 3) // 4 * 4 for x in lengths])]).astype(np.int64)
    total = int(off[-1])
    q, k, w, qs, ks = operands(rng, n, total, 64, 128, dtype)
    dev = lambda x, kind: B.to_device(x, kind)  # noqa: E731
    sc = torch.full((total + 4,), float("nan"), device="cuda")
    B.janus_indexer_scores_batch(dev(q, dtype), dev(k, dtype), dev(w, "f32"), torch.from_numpy(off).cuda(), int(np.diff(off).max()),
                                 q_scale=dev(qs, "f32"), k_scale=dev(ks, "f32"), scores=sc)
    B.check_dev_status()
    got = sc.cpu().numpy()
    assert np.isnan(got[total:]).all() and not np.isnan(got[:total]).any()
    for b in {0, 1 % n, n // 2, n - 1, *rng.integers(0, n, 8).tolist()}:
        a, e = int(off[b]), int(off[b]) + lengths[b]
        if e == a:
            continue
        ref = O.indexer_scores(q[b:b + 1], k[a:e], w[b:b + 1], dtype=dtype, q_scale=qs, k_scale=None if ks is None else ks[a:e], q_pos0=0, causal=False)
        Hp.assert_scores_close(got[None, a:e], ref, 1e-4, f"session {b} of {n}")
