"""Page demand where its dispatch changes: bitmaps around one word, one chunk of 1024 words, the slices of 4, 8 and 16 CTAs, and past what a
CTA keeps in shared memory; index counts on either side of the one-launch limit; runs that cross words, slices and CTAs; lists that exceed
their capacity; rows with their own tables.  Exact against the oracle."""
import numpy as np
import pytest
import torch

import helpers as Hp
from oracle import janus_oracle as O
from paper_2609_36938_b200 import binding as B
from paper_2609_36938_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()
    yield
    B.check_dev_status()


def dev32(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.int32)).cuda()


def bitmap_of(pages, n_phys):
    bits = np.zeros((n_phys + 31) // 32 * 32, np.uint8)
    bits[pages] = 1
    return np.packbits(bits, bitorder="little").view(np.int32)


@pytest.mark.parametrize("n_rows,k,n_phys,page", [
    (1, 7, 31, 64), (3, 700, 33, 16), (2, 2048, 32768, 1), (5, 1000, 32800, 64), (40, 1639, 262144, 1), (33, 2048, 262176, 1),
    (64, 2048, 2049, 48), (65, 2048, 2049, 64), (70, 2000, 300000, 1), (3, 2048, 600000, 1), (90, 2048, 900000, 1),
])
def test_page_demand_edges(n_rows, k, n_phys, page):
    rng = np.random.default_rng(n_rows * 7 + n_phys)
    n_log = n_phys
    L = n_log * page - page // 2
    lo = rng.integers(0, L, (n_rows, k))
    run = (rng.integers(0, max(1, L - 40 * k), (n_rows, 1)) + np.arange(k) * max(1, page // 2)) % L       # neighbouring pages: long runs
    idx = np.where(rng.random((n_rows, 1)) < 0.5, lo, run).astype(np.int32)
    idx[rng.random(idx.shape) < 0.05] = -1
    table = np.arange(n_log, dtype=np.int32) if n_rows % 2 else rng.permutation(n_log).astype(np.int32)
    limit = L - L // 10
    ref = O.page_demand(idx, limit, page, table)
    predicted = np.array(sorted(rng.permutation(ref["pages"])[: len(ref["pages"]) // 2]), np.int64)
    pd = B.janus_page_demand(dev32(idx), demand_limit=limit, page_size=page, page_table=dev32(table), n_phys_pages=n_phys,
                             predicted_bitmap=torch.from_numpy(bitmap_of(predicted, n_phys)).cuda())
    B.check_dev_status()
    got = Hp.page_lists_from_device(pd)
    miss = sorted(set(ref["pages"]) - set(predicted.tolist()))
    assert Hp.bitmap_to_pages(pd["bitmap"], n_phys) == list(ref["pages"])
    assert got["pages"] == list(ref["pages"]) and got["runs"] == [tuple(r) for r in ref["runs"]]
    assert got["miss"] == miss and got["miss_runs"] == [tuple(r) for r in O.maximal_runs(miss)]
    # lists shorter than the set: the first entries, true counts, and the status word
    cap = max(1, len(ref["runs"]) // 3)
    small = B.janus_page_demand(dev32(idx), demand_limit=limit, page_size=page, page_table=dev32(table), n_phys_pages=n_phys, capacity=cap, want_miss=False)
    assert small["counts"][:2].tolist() == [len(ref["pages"]), len(ref["runs"])]
    assert small["pages"].tolist() == list(ref["pages"])[:cap] and [tuple(r) for r in small["runs"].tolist()] == [tuple(r) for r in ref["runs"]][:cap]
    if len(ref["pages"]) > cap:
        with pytest.raises(B.JanusError, match="CAPACITY"):
            B.check_dev_status()


@pytest.mark.parametrize("n_rows,k", [(1, 2048), (20, 2048), (70, 2048)])
def test_page_demand_batch_edges(n_rows, k):
    rng = np.random.default_rng(n_rows)
    page = 64
    n_pages = rng.integers(1, 900, n_rows)
    off = np.concatenate([[0], np.cumsum(n_pages)]).astype(np.int64)
    n_phys = int(off[-1]) + 5
    tables = rng.permutation(n_phys)[:off[-1]].astype(np.int32)
    limits = n_pages * page - rng.integers(0, page, n_rows)
    idx = (rng.random((n_rows, k)) * n_pages[:, None] * page).astype(np.int32)
    pd = B.janus_page_demand_batch(dev32(idx), demand_limits=torch.from_numpy(limits.astype(np.int64)).cuda(), page_size=page, page_tables=dev32(tables),
                                   table_offsets=torch.from_numpy(off).cuda(), n_phys_pages=n_phys)
    B.check_dev_status()
    want = sorted(set().union(*[O.page_demand(idx[r:r + 1], int(limits[r]), page, tables[off[r]:off[r + 1]])["pages"] for r in range(n_rows)]))
    got = Hp.page_lists_from_device(pd)
    assert got["pages"] == want and got["runs"] == [tuple(r) for r in O.maximal_runs(want)] and got["miss"] == want


def test_runs_across_the_clusters_of_a_large_pool():
    """Lists of a pool that several clusters share (four, of 16 x 831 words each): runs that cross from one cluster into the next, that end
    or begin on the boundary, and a miss set with other runs."""
    n_phys, step = 1_700_000, 16 * 831 * 32
    here = np.ones(n_phys, bool)
    here[[5, 2 * step, 3 * step - 1, n_phys - 40]] = False
    here[n_phys - 1000:n_phys - 900] = False
    known = np.zeros(n_phys, bool)
    known[[step - 70, 2 * step - 1, n_phys - 1]] = True
    known[3 * step:3 * step + 500] = True
    idx = np.flatnonzero(here).astype(np.int32)
    idx = np.concatenate([idx, np.full(-len(idx) % 2048, -1, np.int32)]).reshape(-1, 2048)
    pd = B.janus_page_demand(dev32(idx), demand_limit=n_phys, page_size=1, page_table=dev32(np.arange(n_phys)), n_phys_pages=n_phys,
                             predicted_bitmap=torch.from_numpy(bitmap_of(np.flatnonzero(known), n_phys)).cuda())
    B.check_dev_status()
    for want, n, n_runs, ids, runs in ((here, 0, 1, "pages", "runs"), (here & ~known, 2, 3, "miss_pages", "miss_runs")):
        pages = np.flatnonzero(want)
        cut = np.flatnonzero(np.diff(pages) > 1)
        first, last = np.concatenate([[0], cut + 1]), np.concatenate([cut, [len(pages) - 1]])
        counts = pd["counts"].cpu().numpy()
        assert counts[n] == len(pages) and counts[n_runs] == len(first)
        assert np.array_equal(pd[ids][:len(pages)].cpu().numpy(), pages)
        assert np.array_equal(pd[runs][:len(first)].cpu().numpy(), np.stack([pages[first], pages[last] - pages[first] + 1], 1))


def test_a_pool_beyond_one_chunk_per_cta():
    """40 million pages: the clusters' CTAs take their words in several chunks; one run across every cluster boundary and single pages between."""
    n_phys, words = 40_000_000, 1_250_000
    step = 16 * -(-words // (64 * 16)) * 32            # pages of a cluster
    here = np.concatenate([np.arange(i * step - 40, i * step + 40) for i in range(1, -(-n_phys // step))] + [np.arange(0, n_phys, 99_991), [n_phys - 1]])
    want = np.unique(here)
    idx = np.random.default_rng(0).permutation(here).astype(np.int32)
    idx = np.concatenate([idx, np.full(-len(idx) % 64, -1, np.int32)]).reshape(-1, 64)
    known = want[::7]
    bits = torch.zeros((words,), dtype=torch.int64, device="cuda").index_add_(0, torch.from_numpy(known // 32).cuda(), torch.from_numpy(1 << (known % 32)).cuda())
    pd = B.janus_page_demand(dev32(idx), demand_limit=n_phys, page_size=1, page_table=torch.arange(n_phys, dtype=torch.int32, device="cuda"), n_phys_pages=n_phys,
                             predicted_bitmap=bits.to(torch.int32), capacity=20_000)
    B.check_dev_status()
    got = Hp.page_lists_from_device(pd)
    miss = np.setdiff1d(want, known)
    for pages, ids, runs in ((want, "pages", "runs"), (miss, "miss", "miss_runs")):
        cut = np.flatnonzero(np.diff(pages) > 1)
        first, last = np.concatenate([[0], cut + 1]), np.concatenate([cut, [len(pages) - 1]])
        assert got[ids] == pages.tolist() and got[runs] == list(zip(pages[first].tolist(), (pages[last] - pages[first] + 1).tolist()))


@pytest.mark.parametrize("n_phys", [1, 32, 250, 8160, 8191, 8192, 8193])
@pytest.mark.parametrize("which", ["all", "every other", "blocks", "none"])
def test_pools_of_few_words(n_phys, which):
    """Around the largest pool whose lists one CTA makes: as many runs as there can be, one run over all words, no page at all; a predicted
    set and none."""
    rng = np.random.default_rng(n_phys)
    pages = {"all": np.arange(n_phys), "every other": np.arange(0, n_phys, 2), "none": np.arange(0),
             "blocks": np.flatnonzero(np.arange(n_phys) // 37 % 3 > 0)}[which]
    k = max(4, (len(pages) + 7) // 8 * 4)                       # two rows and more
    idx = np.full((3, k), -1, np.int32)
    idx.flat[: len(pages)] = rng.permutation(pages)
    table = np.arange(n_phys, dtype=np.int32)
    ref = O.page_demand(idx, n_phys, 1, table)
    predicted = pages[rng.random(len(pages)) < 0.3]
    for bits in (torch.from_numpy(bitmap_of(predicted, n_phys)).cuda(), None):
        pd = B.janus_page_demand(dev32(idx), demand_limit=n_phys, page_size=1, page_table=dev32(table), n_phys_pages=n_phys, predicted_bitmap=bits)
        B.check_dev_status()
        got = Hp.page_lists_from_device(pd)
        assert Hp.bitmap_to_pages(pd["bitmap"], n_phys) == list(ref["pages"]) == pages.tolist()
        assert got["pages"] == list(ref["pages"]) and got["runs"] == [tuple(r) for r in ref["runs"]]
        if bits is not None:
            miss = sorted(set(pages.tolist()) - set(predicted.tolist()))
            assert got["miss"] == miss and got["miss_runs"] == [tuple(r) for r in O.maximal_runs(miss)]


@pytest.mark.parametrize("n_phys", [1, 250, 8192, 8193])
def test_large_blocks_over_few_words(n_phys):
    """More indices than one cluster marks, around the largest pool whose lists one CTA makes; buffers that still hold another block's set."""
    rng = np.random.default_rng(n_phys)
    out = B.page_demand_buffers(n_phys)
    table = rng.permutation(n_phys).astype(np.int32)
    for rows, k, share in ((65, 2048, 1.0), (800, 168, 0.2), (130, 1024, 0.0)):
        some = np.flatnonzero(rng.random(n_phys) < share)
        idx = (rng.choice(some, (rows, k)) * 16 + 5 if len(some) else np.full((rows, k), -1)).astype(np.int32)
        ref = O.page_demand(idx, n_phys * 16, 16, table)
        predicted = np.flatnonzero(rng.random(n_phys) < 0.3)
        B.janus_page_demand(dev32(idx), demand_limit=n_phys * 16, page_size=16, page_table=dev32(table), n_phys_pages=n_phys,
                            predicted_bitmap=torch.from_numpy(bitmap_of(predicted, n_phys)).cuda(), out=out)
        B.check_dev_status()
        got = Hp.page_lists_from_device(out)
        miss = sorted(set(ref["pages"]) - set(predicted.tolist()))
        assert Hp.bitmap_to_pages(out["bitmap"], n_phys) == list(ref["pages"])
        assert got["pages"] == list(ref["pages"]) and got["runs"] == [tuple(r) for r in ref["runs"]]
        assert got["miss"] == miss and got["miss_runs"] == [tuple(r) for r in O.maximal_runs(miss)]
