"""Pooled entry scores: every entry size with a kernel of its own and some without, rows that end inside a 16-byte load, inside an entry and
inside a strip of 1024 scores, unaligned rows.  A maximum of fp32 values is exact: compared with the oracle bit for bit."""
import numpy as np
import pytest
import torch

from oracle import janus_oracle as O
from paper_2609_36938_b200 import binding as B
from paper_2609_36938_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()


@pytest.mark.parametrize("entry", [1, 4, 8, 16, 20, 32, 64, 100, 128, 256])
@pytest.mark.parametrize("M,n_keys,pad,shift", [(5, 1, 0, 0), (3, 1023, 1, 0), (40, 1025, 3, 0), (7, 9001, 3, 0), (70, 2050, 6, 0), (4, 700, 0, 0), (4, 5000, 0, 1)])
def test_pooled_scores(entry, M, n_keys, pad, shift):
    rng = np.random.default_rng(entry + n_keys)
    sc = rng.standard_normal((M, n_keys + pad)).astype(np.float32)
    flat = torch.zeros(sc.size + 4, device="cuda")
    dev = flat[shift:shift + sc.size].view(sc.shape)
    dev.copy_(torch.from_numpy(sc))
    n_entries = (n_keys + entry - 1) // entry
    for causal, pos in ((True, max(0, n_keys - M)), (True, 0), (False, 0)):
        got = B.janus_entry_pool_scores(dev, n_keys, entry_size=entry, q_pos0=pos, causal=causal)[:, :n_entries].cpu().numpy()
        want = O.entry_pool_scores(sc[:, :n_keys], entry_size=entry, q_pos0=pos, causal=causal)
        assert np.array_equal(got.astype(np.float64), want), f"entry {entry}, {M} x {n_keys}, causal {causal} from {pos}"
