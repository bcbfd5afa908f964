"""The chain indexer -> top-k -> page demand -> attention, and a decode step, where overlapped launches and state kept between calls would
show: two streams at once, two threads, a captured graph whose inputs change between replays.  Compared with the same chain run alone, with
a synchronisation after every call: page sets and counts exactly, attention within bf16 rounding (the order of a selection is free)."""
import threading

import pytest
import torch

from paper_2609_36938_b200 import binding as B
from paper_2609_36938_b200 import build

pytestmark = pytest.mark.gpu

LATENT, HEADS = (128, 1, 576, 512), (16, 2, 128, 128)      # query heads, kv heads, key dims, value dims


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()
    B.check_dev_status()
    yield
    B.check_dev_status()


class Chain:
    """A prefill of M tokens on a history of L (one session) with buffers of its own."""

    def __init__(self, seed, M, L, layout, k=512):
        g = torch.Generator(device="cuda").manual_seed(seed)
        self.M, self.L, self.S, self.k, self.page = M, L, L + M, k, 64
        self.h_q, self.n_kv, self.d_qk, self.d_v = layout
        self.n_pages = (self.S + 63) // 64
        self.q, self.keys, self.w = (torch.empty(s, dtype=t, device="cuda") for s, t in (
            ((M, 64, 128), torch.bfloat16), ((self.S, 128), torch.bfloat16), ((M, 64), torch.float32)))
        self.Q = torch.empty((M, self.h_q, self.d_qk), dtype=torch.bfloat16, device="cuda")
        self.k_pool = torch.empty((self.n_pages, 64, self.n_kv, self.d_qk), dtype=torch.bfloat16, device="cuda")
        self.v_pool = self.k_pool if layout is LATENT else torch.empty_like(self.k_pool)
        self.table = torch.randperm(self.n_pages, device="cuda", generator=g).int()
        self.scores = torch.empty((M, (self.S + 31) // 32 * 32), device="cuda")
        self.idx = torch.empty((M, k), dtype=torch.int32, device="cuda")
        self.pages = B.page_demand_buffers(self.n_pages)
        self.out = torch.empty((M, self.h_q, self.d_v), dtype=torch.bfloat16, device="cuda")
        self.fill(g)

    def fill(self, g):
        for t in (self.q, self.keys, self.Q, self.k_pool, self.v_pool):
            t.copy_(torch.randn(t.shape, device="cuda", generator=g))
        self.w.copy_(torch.rand(self.w.shape, device="cuda", generator=g))

    def calls(self):
        yield lambda: B.janus_indexer_scores(self.q, self.keys, self.w, q_pos0=self.L, scores=self.scores)
        yield lambda: B.janus_topk(self.scores, self.S, self.k, q_pos0=self.L, want_count=False, want_kth=False, idx=self.idx)
        yield lambda: B.janus_page_demand(self.idx, demand_limit=self.L, page_size=64, page_table=self.table, n_phys_pages=self.n_pages, out=self.pages)
        yield lambda: B.janus_sparse_attn_prefill(self.Q, self.k_pool, self.v_pool, self.idx, page_table=self.table, page_size=64,
                                                  softmax_scale=self.d_qk ** -0.5, d_v=self.d_v, want_lse=False, out=self.out)

    def run(self, alone=False):
        for call in self.calls():
            call()
            if alone:
                torch.cuda.synchronize()

    def results(self):
        n, n_runs = self.pages["counts"][:2].tolist()
        return self.pages["bitmap"].clone(), self.pages["pages"][:n].clone(), self.pages["runs"][:n_runs].clone(), self.out.float().clone()

    def wipe(self):
        for t in (self.scores, self.out):
            t.fill_(float("nan"))
        for t in (self.idx, self.pages["bitmap"], self.pages["pages"], self.pages["runs"], self.pages["counts"]):
            t.fill_(0x7fffffff if t is self.idx else -1)


def same(got, want):
    for a, b in zip(got[:3], want[:3]):
        assert torch.equal(a, b)
    err = (got[3] - want[3]).abs()
    assert float(err.norm() / want[3].norm()) < 1e-2 and float(err.max()) < 0.1      # bf16 outputs, P in bf16, sums in another order


def reference(chain):
    chain.run(alone=True)
    want = chain.results()
    chain.wipe()
    torch.cuda.synchronize()
    return want


def test_two_streams_at_once():
    chains = [Chain(1, 24, 20000, LATENT), Chain(2, 40, 9001, HEADS)]
    wants = [reference(c) for c in chains]
    streams = [torch.cuda.Stream() for _ in chains]
    for _ in range(30):
        for c, s in zip(chains, streams):
            with torch.cuda.stream(s):
                c.run()
    torch.cuda.synchronize()
    for c, want in zip(chains, wants):
        same(c.results(), want)


def test_two_threads():
    """Calls of other shapes go through the same kernels at the same time; the general attention kernel's shared memory differs by call."""
    chains = [Chain(3, 8, 30000, LATENT), Chain(4, 200, 700, HEADS), Chain(5, 30, 4000, (6, 2, 96, 80)), Chain(6, 30, 4000, (16, 2, 256, 160))]
    for c in chains[2:]:
        c.v_pool = c.k_pool                                    # an aliased value row is a prefix of the key row
    wants = [reference(c) for c in chains]
    errors = []

    def work(c):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(60):
                    c.run()
        except Exception as e:      # noqa: BLE001 (reported below, in the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in chains]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    for c, want in zip(chains, wants):
        same(c.results(), want)


@pytest.mark.parametrize("M,L,layout", [(3, 40000, LATENT), (100, 6000, HEADS)])
def test_a_captured_graph_follows_its_inputs(M, L, layout):
    c = Chain(7, M, L, layout)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(2):                                     # a launch whose predecessor is the chain's own last kernel
            c.run()
    for seed in (11, 12):
        c.fill(torch.Generator(device="cuda").manual_seed(seed))
        want = reference(c)
        graph.replay()
        torch.cuda.synchronize()
        same(c.results(), want)


def test_decode_steps_overlap_on_one_stream():
    """Step after step through the same buffers without a synchronisation: a call overwrites what the step before still reads, if it may."""
    n, L, k, n_steps = 5, 6000, 256, 12
    g = torch.Generator(device="cuda").manual_seed(9)
    rows = (L + 1 + 3) // 4 * 4
    off, lens = torch.arange(n + 1, device="cuda") * rows, torch.full((n,), L + 1, device="cuda")
    per = (L + 64) // 64
    tables, tab_off = torch.randperm(n * per, device="cuda", generator=g).int(), torch.arange(n + 1, device="cuda") * per
    keys, w = torch.randn((n * rows, 128), device="cuda", generator=g).bfloat16(), torch.rand((n, 64), device="cuda", generator=g)
    pool = torch.randn((n * per, 64, 1, 576), device="cuda", generator=g).bfloat16()
    q, Q = (torch.randn((n_steps, n, h, d), device="cuda", generator=g).bfloat16() for h, d in ((64, 128), (128, 576)))
    scores, pages = torch.empty((n * rows,), device="cuda"), B.page_demand_buffers(n * per)
    out = torch.empty((n, 128, 512), dtype=torch.bfloat16, device="cuda")

    def steps(alone):
        seen = []
        pause = torch.cuda.synchronize if alone else lambda: None
        for i in range(n_steps):
            B.janus_indexer_scores_batch(q[i], keys, w, off, rows, scores=scores)
            pause()
            idx, count, kth = B.janus_topk_batch(scores, off, k, row_lengths=lens)
            pause()
            B.janus_page_demand_batch(idx, demand_limits=lens - 1, page_size=64, page_tables=tables, table_offsets=tab_off, n_phys_pages=n * per, out=pages)
            pause()
            B.janus_sparse_attn_decode(Q[i], pool, pool, idx, page_tables=tables, table_offsets=tab_off, page_size=64, softmax_scale=1 / 24, d_v=512, out=out)
            pause()
            seen.append((pages["bitmap"].clone(), count, kth, out.float()))
        torch.cuda.synchronize()
        return seen

    for got, want in zip(steps(False), steps(True)):
        same(got, want)
