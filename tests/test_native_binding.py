"""The native half of the binding: loads next to the library, and refuses what the Python signatures promise to refuse."""
import pytest
import torch

from paper_2609_36938_b200 import binding as B
from paper_2609_36938_b200 import build


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def test_loads_and_counts_its_arguments():
    native = B._native()
    for name in ("indexer_scores", "topk", "indexer_topk", "page_demand", "page_demand_batch", "page_union", "sparse_attn", "topk_entries",
                 "entry_pool_scores", "entry_expand", "indexer_scores_batch", "topk_batch"):
        with pytest.raises(TypeError, match="arguments"):
            getattr(native, name)()


def test_another_torch_makes_the_build_stale(monkeypatch):
    assert not build._stale()
    monkeypatch.setattr(build.importlib.metadata, "version", lambda name: "2.0.0")
    assert build._stale()


def test_sizes_are_whole_numbers_and_errors_keep_their_types():
    """Where a size shapes an output, only a whole number is taken; a missing dimension and a failed allocation raise what torch raises."""
    sc, e = torch.zeros(4, 8), torch.zeros(4, 2, dtype=torch.int32)
    with pytest.raises(TypeError):
        B.janus_topk(sc, 8, 2.5)
    with pytest.raises(TypeError):
        B.janus_topk_entries(sc, 8, 2.0, q_pos0=0, entry_size=4)
    with pytest.raises(TypeError):
        B.janus_topk_batch(sc, torch.zeros(3, dtype=torch.int64), 2.0)
    with pytest.raises(TypeError):
        B.janus_entry_expand(e, q_pos0=0, entry_size=4.0)
    with pytest.raises(TypeError):
        B.janus_entry_pool_scores(sc, 8, entry_size=4.0)
    with pytest.raises(IndexError):
        B.janus_topk(torch.zeros(()), 8, 2)


@pytest.mark.gpu
def test_out_of_memory_is_torch_s_own_error():
    off = torch.arange(65, device="cuda") * 4
    with pytest.raises(torch.OutOfMemoryError):
        B.janus_topk_batch(torch.zeros(256, device="cuda"), off, 1 << 30)      # 256 GB of indices
    torch.cuda.empty_cache()


@pytest.mark.gpu
def test_bad_tensors_raise():
    q, k, w = torch.zeros(4, 64, 128).bfloat16(), torch.zeros(32, 128).bfloat16(), torch.zeros(4, 64)
    with pytest.raises(B.JanusError, match="CUDA tensor"):
        B.janus_indexer_scores(q, k, w)
    with pytest.raises(B.JanusError, match="share a dtype"):
        B.janus_indexer_scores(q.cuda(), k.cuda().to(torch.float8_e4m3fn), w.cuda())
    with pytest.raises(B.JanusError, match="must be bfloat16 or E4M3"):
        B.janus_indexer_scores(q.cuda().float(), k.cuda().float(), w.cuda())
    with pytest.raises(B.JanusError, match="JANUS_ERR_INVALID_ARG"):
        B.janus_topk(torch.zeros(2, 8, device="cuda"), 8, 0)
    with pytest.raises(B.JanusError, match="contiguous"):
        B.janus_indexer_topk(q.cuda(), k.cuda(), w.cuda(), 8, idx=torch.zeros(4, 9, dtype=torch.int32, device="cuda"))
    B.check_dev_status()
