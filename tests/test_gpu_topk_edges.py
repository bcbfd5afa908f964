"""Top-k where its routes change: rows around the candidate buffers (3840, 5632 and 8192 elements), the cluster sizes with their shares of a row,
ragged rows of very different lengths in one launch, and score distributions the sample or the buckets cannot settle (ties by the thousand,
one value, scores cut off at zero, two far-apart levels, -0 and +0, an outlier that stretches the key range, a row whose large scores hide from the sample).
A selection is checked against a full sort: the values above the k-th are all there, ties at it are free."""
import numpy as np
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


def check_row(idx, count, kth, row, k, tag):
    want = min(k, len(row))
    sel = idx[:want]
    assert count == want and np.all(idx[want:] == -1), tag
    assert len(np.unique(sel)) == want and (want == 0 or (sel.min() >= 0 and sel.max() < len(row))), tag
    if want == 0:
        assert np.isneginf(kth), tag
        return
    t = np.partition(row, len(row) - want)[len(row) - want]
    assert kth == t, f"{tag}: k-th {kth} instead of {t}"
    vals = row[sel]
    assert np.all(vals >= t) and np.sum(vals > t) == np.sum(row > t), tag


def draw(kind, n, rng):
    x = rng.standard_normal(n).astype(np.float32)
    if kind == "ties":
        x = np.round(x * 2) / 2
    elif kind == "constant":
        x[:] = 1.25
    elif kind == "levels":
        x = np.where(rng.random(n) < 0.02, np.float32(1e30), np.float32(-1e-30)) * (1 + rng.random(n).astype(np.float32) / 8)
    elif kind == "cut":                          # nothing below 1.5 counts: most of the row is one value, as often as not the threshold
        x = np.maximum(x - np.float32(1.5), np.float32(0))
    elif kind == "zeros":
        x = np.where(rng.random(n) < 0.5, np.float32(-0.0), np.float32(0.0))
    elif kind == "outlier" and n:
        x[rng.integers(0, n)] = 3e38
    elif kind == "hidden":                       # a dense block of large scores between sampled groups
        x[n // 2:n // 2 + min(9000, n // 3)] += 50
    return x.astype(np.float32)


@pytest.mark.parametrize("kind", ["normal", "ties", "constant", "cut", "levels", "zeros", "outlier", "hidden"])
@pytest.mark.parametrize("rows,n", [(3, 5640), (90, 8193), (5, 40009), (20, 99991), (70, 65003), (80, 66001)])
def test_topk_rows(kind, rows, n):
    rng = np.random.default_rng(n + rows)
    sc = np.stack([draw(kind, n, rng) for _ in range(rows)])
    ld = (n + 3) // 4 * 4
    dev = torch.full((rows, ld), float("nan"), device="cuda")
    dev[:, :n] = torch.from_numpy(sc)
    for k in (1, 2048):
        idx, cnt, kth = B.janus_topk(dev, n, k, q_pos0=n - rows, causal=True)
        B.check_dev_status()
        idx, cnt, kth = idx.cpu().numpy(), cnt.cpu().numpy(), kth.cpu().numpy()
        for t in {0, 1, rows // 2, rows - 1}:
            check_row(idx[t], cnt[t], kth[t], sc[t, :n - rows + t + 1], k, f"{kind} row {t} of {rows} x {n}, k {k}")


@pytest.mark.parametrize("kind", ["normal", "ties", "cut", "zeros", "outlier", "hidden"])
@pytest.mark.parametrize("rows,n,k", [(148, 8192, 64), (149, 3840, 64), (149, 3841, 64), (300, 4090, 1000), (160, 4500, 2048), (149, 5633, 700),
                                      (149, 8192, 2048), (149, 8193, 2176), (149, 8193, 2177), (700, 20003, 2048), (160, 20003, 3500),
                                      (8, 22004, 2048), (14, 36003, 2048), (15, 36003, 2048), (30, 112007, 2048), (37, 32009, 1000),
                                      (14, 45003, 2048), (30, 32009, 1000), (33, 112007, 2048), (34, 112007, 2048)])
def test_topk_rows_that_share_an_sm(kind, rows, n, k):
    """Around the slots of the three forms and the rules between them: more rows than SMs and not; rows a little longer than the smallest form
    (sampled groups overlap there); the longest k of the smallest form and one more; rows of which half is on the list; the lines between cluster sizes."""
    rng = np.random.default_rng(n + rows + k)
    sc = np.stack([draw(kind, n, rng) for _ in range(rows)])
    dev = torch.full((rows, (n + 3) // 4 * 4), float("nan"), device="cuda")
    dev[:, :n] = torch.from_numpy(sc)
    for causal in (False, True):
        idx, cnt, kth = B.janus_topk(dev, n, k, q_pos0=n - rows, causal=causal)
        B.check_dev_status()
        idx, cnt, kth = idx.cpu().numpy(), cnt.cpu().numpy(), kth.cpu().numpy()
        for t in {0, 1, rows // 2, rows - 2, rows - 1}:
            check_row(idx[t], cnt[t], kth[t], sc[t, :n - rows + t + 1 if causal else n], k, f"{kind} row {t} of {rows} x {n}, k {k}")


@pytest.mark.parametrize("kind", ["normal", "ties", "cut", "zeros", "hidden"])
@pytest.mark.parametrize("lengths", [[131072], [0, 1, 2047, 2048, 2049, 8192, 8196, 70001], [100003] + [9001] * 11, [17999, 18000, 18004, 30001], [23999, 24000, 24004, 9000, 60001, 300, 8193, 40000, 24001], [23999, 24001] * 10, [300 * i + 5 for i in range(64)],
                                     [12001] * 80])
def test_topk_batch(kind, lengths):
    rng = np.random.default_rng(len(lengths))
    off = np.concatenate([[0], np.cumsum([(n + 3) // 4 * 4 for n in lengths])])
    flat = torch.full((int(off[-1]) + 4,), float("nan"), device="cuda")
    rows = [draw(kind, n, rng) for n in lengths]
    for o, r in zip(off, rows):
        flat[o:o + len(r)] = torch.from_numpy(r)
    k = 2048
    idx, cnt, kth = B.janus_topk_batch(flat, torch.from_numpy(off).cuda(), k, row_lengths=torch.tensor(lengths, dtype=torch.int64, device="cuda"))
    B.check_dev_status()
    idx, cnt, kth = idx.cpu().numpy(), cnt.cpu().numpy(), kth.cpu().numpy()
    for b, r in enumerate(rows):
        check_row(idx[b], cnt[b], kth[b], r, k, f"{kind} row {b}")


@pytest.mark.parametrize("rows,n,k", [(2048, 8000, 512), (1024, 6000, 2048)])
def test_a_threshold_with_many_copies_costs_no_second_selection(rows, n, k):
    """Where the k-th score is one value of thousands the row is still read once: it takes no longer than twice what distinct scores do (2.6 to
    three times as long when the copies overflowed the list and the row was selected from memory all over)."""
    x = torch.randn((rows, n), device="cuda", generator=torch.Generator(device="cuda").manual_seed(rows))
    took = {}
    for name, sc in (("distinct", x), ("cut", torch.relu(x - 1.5))):
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                B.janus_topk(sc, n, k, q_pos0=n, causal=False, want_count=False, want_kth=False)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        took[name] = min(times)
    assert took["cut"] < 2 * took["distinct"], took


@pytest.mark.parametrize("rows", [12, 20])
def test_short_rows_of_a_batch_are_not_split(rows):
    """A batch whose lengths only the device knows takes 9000 elements a row about as fast as a call that knows them (10 % more than one CTA
    allows for the start of a cluster; split, such rows took 24 and 15 % more)."""
    n, k = 9000, 2048
    x = torch.randn((rows, n), device="cuda", generator=torch.Generator(device="cuda").manual_seed(rows))
    off, length = torch.arange(rows + 1, dtype=torch.int64, device="cuda") * n, torch.full((rows,), n, dtype=torch.int64, device="cuda")
    calls = {"rows": lambda: B.janus_topk(x, n, k, q_pos0=n, causal=False), "batch": lambda: B.janus_topk_batch(x.flatten(), off, k, row_lengths=length)}
    took = {}
    for name, call in calls.items():
        call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(20):
                call()
        times = []
        for _ in range(25):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            graph.replay()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        took[name] = min(times)
    assert took["batch"] < 1.1 * took["rows"], took
