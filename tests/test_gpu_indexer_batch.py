"""The batch indexer's steps: sessions that end on either side of 128 and 256 keys, some of them empty, with one, a few and many steps per
session and ranges that cross sessions more often than the key ring is deep; every key format, both biases.  Against the oracle; tolerance as
in test_gpu_parity.py (fp32 sums of exact products)."""
import numpy as np
import pytest
import torch

import helpers as Hp
from oracle import janus_oracle as O
from paper_2609_36938_b200 import binding as B
from paper_2609_36938_b200 import build
from paper_2609_36938_b200 import workloads as W

pytestmark = pytest.mark.gpu

EDGES = [1, 127, 128, 129, 0, 255, 256, 257, 383, 385, 511, 513, 769, 1025]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()
    yield
    B.check_dev_status()


@pytest.mark.parametrize("lengths", [EDGES, EDGES * 30, [40000] + EDGES, [20000, 1, 20001, 129, 19999, 257] * 8])
@pytest.mark.parametrize("dtype,D", [("bf16", 128), ("bf16", 64), ("fp8", 128), ("fp8", 256), ("fp4", 128)])
def test_steps_of_every_session(lengths, dtype, D):
    rng = np.random.default_rng(len(lengths) + D)
    n, total = len(lengths), sum(lengths)
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    q, w = rng.standard_normal((n, 64, D)).astype(np.float32), (rng.uniform(-0.2, 1, (n, 64)) / 8).astype(np.float32)
    rb, cb = rng.standard_normal(n).astype(np.float32), rng.standard_normal(total).astype(np.float32)
    qs = ks = None
    if dtype == "bf16":
        q, k = W.to_bf16_bits(q), W.to_bf16_bits(rng.standard_normal((total, D)).astype(np.float32))
    else:
        q, qs, ks = W.to_e4m3_bits(q), np.exp2(rng.uniform(-1, 1, (n, 64))).astype(np.float32), np.exp2(rng.uniform(-1, 1, total)).astype(np.float32)
        k = rng.integers(0, 256, (total, D // 2), dtype=np.uint8) if dtype == "fp4" else W.to_e4m3_bits(rng.standard_normal((total, D)).astype(np.float32))
    dev = lambda x, kind: B.to_device(x, kind)  # noqa: E731
    sc = torch.full((total + 300,), float("nan"), device="cuda")
    B.janus_indexer_scores_batch(dev(q, "bf16" if dtype == "bf16" else "fp8"), dev(k, "bf16" if dtype == "bf16" else "fp8"), dev(w, "f32"), torch.from_numpy(off).cuda(),
                                 max(lengths), q_scale=dev(qs, "f32"), k_scale=dev(ks, "f32"), row_bias=dev(rb, "f32"), col_bias=dev(cb, "f32"),
                                 scores=sc, keys_fp4=dtype == "fp4")
    B.check_dev_status()
    got = sc.cpu().numpy()
    assert np.isnan(got[total:]).all() and not np.isnan(got[:total]).any()
    for b in {*range(min(n, len(EDGES) + 1)), n - 1, *rng.integers(0, n, 6).tolist()}:
        s = slice(int(off[b]), int(off[b + 1]))
        if s.start == s.stop:
            continue
        ref = O.indexer_scores(q[b:b + 1], k[s], w[b:b + 1], dtype="fp8+fp4k" if dtype == "fp4" else dtype, q_scale=None if qs is None else qs[b:b + 1],
                               k_scale=None if ks is None else ks[s], row_bias=rb[b:b + 1], col_bias=cb[s], q_pos0=0, causal=False)
        Hp.assert_scores_close(got[None, s], ref, 1e-4, f"session {b} of {n}")
