"""The work that users of this library have it do, as cases that can be timed and whose outputs can be compared.

Five kinds of pass, each through the public calls of ``paper_2609_36938_b200.binding`` / ``.prediction``:

  prefill   one sparse layer of an append prefill: indexer scores -> top-k -> page demand against a predicted page set ->
            sparse attention, on one session
  onecall   the same layer with ``janus_indexer_topk`` in place of the first two calls (no score matrix in memory)
  decode    one decode step over a batch of sessions with ragged histories
  predict   the sharded lookahead prediction pass: page sets of N history shards and their union
  entries   selection by entries of E tokens pooled from token scores, then page demand and attention

Inputs are drawn on the device from the seed.  Output buffers that a serving loop keeps (scores, selections, page lists,
workspace) are made once in ``prepare``.  The order of a selection's indices and the winner of a tie at the k-th score are
unspecified by the library, so a selection itself is not among the outputs: what is computed from it is (page sets, runs and
counts, attention outputs with their log-sum-exp, and counts and k-th scores where the pass asks for them).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_36938_b200 import binding as B
from paper_2609_36938_b200 import prediction as P

#: attention layouts: query heads, key/value heads, key dim, value dim, values alias the keys
LAYOUTS = {
    "latent": (128, 1, 576, 512, True),     # one shared 512 + 64 latent row per token
    "mha": (8, 8, 128, 128, False),         # one query head per key/value head
    "gqa": (32, 4, 128, 128, False),        # eight query heads per key/value head
}


# ---- the cases ------------------------------------------------------------------------------------------------------------
def listed():
    def prefill(name, L, M, dtype, layout="latent", heads=64, dim=128, k=2048, table="shuffled", page=64):
        return {"name": name, "kind": "prefill", "L": L, "M": M, "dtype": dtype, "heads": heads, "dim": dim, "k": k, "layout": layout,
                "page": page, "table": table}

    return [
        # the tiny configuration: a few heads of indexer, multi-head attention; latency and launches count
        prefill("prefill_tiny_mha", 4096, 256, "bf16", layout="mha", heads=4, dim=64, k=256, table="identity"),
        # a short user message after a short history: few query rows, all of the chip idle but a few SMs
        prefill("prefill_short_message", 9001, 19, "bf16"),
        # an ordinary append on a bf16 indexer (32K history)
        prefill("prefill_bf16_32k", 32768, 2048, "bf16"),
        # the headline: a long append on a 128K history, FP8 indexer
        prefill("prefill_fp8_128k", 131072, 4096, "fp8"),
        # a ragged session of a shared, fragmented pool, grouped-query attention
        prefill("prefill_ragged_gqa", 20011, 777, "bf16", layout="gqa", heads=32, table="fragmented"),
        # a tool result appended to a long agentic history, one call for indexer and selection
        {"name": "onecall_fp8_append", "kind": "onecall", "L": 131072, "M": 128, "dtype": "fp8", "k": 2048, "clustered": False},
        # the longest session: clustered keys, recency bias; the score matrix would be 8.9 GB
        {"name": "onecall_fp8_256k", "kind": "onecall", "L": 262144, "M": 8192, "dtype": "fp8", "k": 2048, "clustered": True},
        # one user decoding: the smallest step there is
        {"name": "decode_1_fp8", "kind": "decode", "sessions": 1, "L": 32768, "dtype": "fp8", "k": 2048},
        # a small serving batch of ragged sessions, bf16 indexer
        {"name": "decode_12_bf16", "kind": "decode", "sessions": 12, "L": 50021, "dtype": "bf16", "k": 2048},
        # a full batch of long sessions, 4-bit indexer keys
        {"name": "decode_64_fp4", "kind": "decode", "sessions": 64, "L": 131072, "dtype": "fp4", "k": 2048},
        # lookahead prediction over eight history shards
        {"name": "predict_8_shards", "kind": "predict", "L": 131072, "M": 1024, "dtype": "fp8", "k": 2048, "shards": 8},
        # selection by entries of 128 tokens
        {"name": "entries_128", "kind": "entries", "L": 40000, "M": 512, "dtype": "bf16", "entry": 128, "k": 16},
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "prefill", "prefill", "onecall", "onecall", "decode", "decode", "decode", "predict", "entries"])
    if kind == "prefill":
        layout = rng.choice(["latent", "latent", "latent", "mha", "gqa"])
        if layout == "latent":
            heads, dim, dtype = 64, 128, rng.choice(["bf16", "fp8", "fp8", "fp4"])
        else:
            heads, dim = rng.choice([(4, 64), (16, 64), (32, 128), (64, 128)])
            dtype = "fp8" if dim == 128 and rng.random() < 0.4 else "bf16"
        return {"kind": kind, "L": _spread(rng, 512, 131072), "M": _spread(rng, 1, 4096), "dtype": dtype, "heads": heads, "dim": dim,
                "k": rng.choice([256, 512, 1024, 2048, 2048]), "layout": layout, "page": rng.choice([16, 64, 64, 128]),
                "table": rng.choice(["shuffled", "fragmented"])}
    if kind == "onecall":
        return {"kind": kind, "L": _spread(rng, 8192, 262144), "M": _spread(rng, 16, 4096), "dtype": rng.choice(["bf16", "fp8", "fp8"]),
                "k": rng.choice([1024, 2048]), "clustered": rng.random() < 0.5}
    if kind == "decode":
        return {"kind": kind, "sessions": _spread(rng, 1, 64), "L": _spread(rng, 1024, 131072), "dtype": rng.choice(["bf16", "fp8", "fp4"]),
                "k": rng.choice([1024, 2048, 2048])}
    if kind == "predict":
        return {"kind": kind, "L": _spread(rng, 16384, 131072), "M": _spread(rng, 64, 2048), "dtype": rng.choice(["bf16", "fp8"]), "k": 2048,
                "shards": rng.choice([1, 2, 4, 8])}
    entry = rng.choice([16, 32, 64, 128])
    return {"kind": kind, "L": _spread(rng, 4096, 131072), "M": _spread(rng, 16, 2048), "dtype": rng.choice(["bf16", "fp8"]), "entry": entry,
            "k": 2048 // entry}


# ---- inputs -----------------------------------------------------------------------------------------------------------------
def _indexer_operands(g, n_q, n_k, heads, dim, dtype):
    """Standard-normal queries and keys in their storage format, per-head / per-key scales for the 8- and 4-bit formats, head weights."""
    q = torch.randn((n_q, heads, dim), device="cuda", generator=g)
    w = torch.rand((n_q, heads), device="cuda", generator=g) / 8
    if dtype == "bf16":
        return {"q": q.bfloat16(), "k": torch.randn((n_k, dim), device="cuda", generator=g).bfloat16(), "w": w, "q_scale": None, "k_scale": None}
    out = {"q": q.to(torch.float8_e4m3fn).view(torch.uint8), "w": w,
           "q_scale": torch.exp2(torch.rand((heads,), device="cuda", generator=g) * 4 - 2),
           "k_scale": torch.exp2(torch.rand((n_k,), device="cuda", generator=g) * 8 - 4)}
    if dtype == "fp4":      # any byte is two E2M1 values
        out["k"] = torch.randint(0, 256, (n_k, dim // 2), dtype=torch.uint8, device="cuda", generator=g)
    else:
        out["k"] = torch.randn((n_k, dim), device="cuda", generator=g).to(torch.float8_e4m3fn).view(torch.uint8)
    return out


def _clustered_operands(g, rng, L, M, heads, dim, dtype):
    """Keys in topical segments around 32 centroids, four large-norm sink keys, queries leaning toward the centroid of their
    256-token stretch, a recency bias 2 exp(-(distance) / 4096) as a rank-1 product."""
    S = L + M
    seg = np.repeat(rng.integers(0, 32, S // 256 + 1), rng.integers(256, 4097, S // 256 + 1))[:S]
    centroid = torch.randn((32, dim), device="cuda", generator=g)
    key = centroid[torch.from_numpy(seg).cuda()] + 0.5 * torch.randn((S, dim), device="cuda", generator=g)
    key[:4] = 8.0 * torch.randn((4, dim), device="cuda", generator=g)
    gain = 0.5 + torch.rand((1, heads, 1), device="cuda", generator=g)
    lean = torch.from_numpy(np.repeat(rng.integers(0, 32, (M + 255) // 256), 256)[:M]).cuda()
    q = gain * centroid[lean][:, None, :] + torch.randn((M, heads, dim), device="cuda", generator=g)
    out = {"w": torch.rand((M, heads), device="cuda", generator=g) / 8, "q_scale": None, "k_scale": None}
    if dtype == "bf16":
        out["q"], out["k"] = q.bfloat16(), key.bfloat16()
    else:
        out["k_scale"] = key.abs().amax(1) / 448.0
        out["q_scale"] = q.abs().amax((0, 2)) / 448.0
        out["k"] = (key / out["k_scale"][:, None]).to(torch.float8_e4m3fn).view(torch.uint8)
        out["q"] = (q / out["q_scale"][None, :, None]).to(torch.float8_e4m3fn).view(torch.uint8)
    out["row_bias"] = 2.0 * torch.exp(-(L + torch.arange(M, device="cuda", dtype=torch.float32)) / 4096.0)
    out["col_bias"] = torch.exp(torch.arange(S, device="cuda", dtype=torch.float32) / 4096.0)
    return out


def _page_table(rng, n_pages, table):
    """Logical -> physical pages: in order, shuffled, or chunks of 1 to 8 neighbours out of a pool shared with other sessions."""
    if table == "identity":
        return np.arange(n_pages), n_pages
    if table == "shuffled":
        return rng.permutation(n_pages), n_pages
    chunk = rng.integers(1, 9, n_pages)
    logical = np.arange(n_pages)
    ends = np.cumsum(chunk)
    owner = np.searchsorted(ends, logical, side="right")       # chunk of each page; before it lies as large a chunk of another session
    return logical + ends[owner], 2 * n_pages + 8


def _attention_operands(g, n_q, n_phys, page, layout):
    h_q, n_kv, d_qk, d_v, alias = LAYOUTS[layout]
    std = 1.0 / math.sqrt(d_qk)
    normal = lambda shape: torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=g)  # noqa: E731
    k_pool = normal((n_phys, page, n_kv, d_qk))
    return {"Q": normal((n_q, h_q, d_qk)), "k_pool": k_pool, "v_pool": k_pool if alias else normal((n_phys, page, n_kv, d_v)),
            "out": torch.empty((n_q, h_q, d_v), dtype=torch.bfloat16, device="cuda"), "scale": std, "d_v": d_v}


def _page_buffers(n_phys, want_miss=True):
    bufs = B.page_demand_buffers(n_phys, want_miss=want_miss)
    for t in bufs.values():      # what lies past the counts is never written
        t.zero_()
    return bufs


def _resident(g, n_phys, share):
    """A page bitmap in which about `share` of the pages are set."""
    bits = torch.rand(((n_phys + 31) // 32, 32), device="cuda", generator=g) < share
    return (bits.long() << torch.arange(32, device="cuda")).sum(1).to(torch.int32)


def _score_rows(n_rows, n_keys):
    return torch.empty((n_rows, (n_keys + 31) // 32 * 32), dtype=torch.float32, device="cuda")


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    st = dict(case, k_top=case["k"])
    if kind == "decode":
        return _prepare_decode(st, g, rng)
    L, M, k = case["L"], case["M"], case["k"]
    S = L + M
    page, table, layout = case.get("page", 64), case.get("table", "shuffled"), case.get("layout", "latent")
    st.update(page=page, S=S)
    if kind == "onecall" and case["clustered"]:
        st.update(_clustered_operands(g, rng, L, M, 64, 128, case["dtype"]))
    else:
        st.update(_indexer_operands(g, M, L if kind == "predict" else S, case.get("heads", 64), case.get("dim", 128), case["dtype"]))
    n_pages = (S + page - 1) // page
    tab, n_phys = _page_table(rng, n_pages, table)
    st["page_table"], st["n_phys"] = torch.from_numpy(tab.astype(np.int32)).cuda(), n_phys
    if kind == "predict":
        return st
    st["pages"] = _page_buffers(n_phys)
    st["predicted"] = _resident(g, n_phys, 0.96)
    st.update(_attention_operands(g, M, n_phys, page, layout))
    if kind == "onecall":
        code = B.DTYPE_BF16 if case["dtype"] == "bf16" else B.DTYPE_FP8_E4M3
        need = int(B.load().janus_indexer_topk_workspace_size(M, 64, 128, S, L, 1, code, k))
        st["workspace"] = torch.empty((max(need, 16),), dtype=torch.uint8, device="cuda")
    else:
        st["scores"] = _score_rows(M, S)
    if kind != "entries":
        st["idx"] = torch.empty((M, k), dtype=torch.int32, device="cuda")
    return st


def _prepare_decode(st, g, rng):
    n, page = st["sessions"], 64
    sizes = np.random.default_rng([n, st["L"]])                             # the lengths belong to the case, not to the seed
    length = sizes.integers(max(1, st["L"] // 4), st["L"] + 1, n)           # cached tokens of each session; the longest is as named
    length[sizes.integers(0, n)] = st["L"]
    rows = (length + 1 + 3) // 4 * 4
    key_off = np.concatenate([[0], np.cumsum(rows)])
    st.update(_indexer_operands(g, n, int(key_off[-1]), 64, 128, st["dtype"]))
    pages = (length + 1 + page - 1) // page
    tab_off = np.concatenate([[0], np.cumsum(pages)])
    n_phys = int(tab_off[-1])
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    st.update(page=page, n_phys=n_phys, max_keys=int(rows.max()), key_off=dev(key_off), row_len=dev(length + 1), limits=dev(length),
              tables=dev(rng.permutation(n_phys).astype(np.int32)), tab_off=dev(tab_off))
    st["scores"] = torch.empty((int(key_off[-1]),), dtype=torch.float32, device="cuda")
    st["pages"] = _page_buffers(n_phys)
    st["predicted"] = _resident(g, n_phys, 0.99)                          # pages already on the device
    st.update(_attention_operands(g, n, n_phys, page, "latent"))
    return st


# ---- one pass -----------------------------------------------------------------------------------------------------------------
def _demand_and_attention(st, idx):
    pd = B.janus_page_demand(idx, demand_limit=st["L"], page_size=st["page"], page_table=st["page_table"], n_phys_pages=st["n_phys"],
                             predicted_bitmap=st["predicted"], out=st["pages"])
    out, lse = B.janus_sparse_attn_prefill(st["Q"], st["k_pool"], st["v_pool"], idx, page_table=st["page_table"], page_size=st["page"],
                                           softmax_scale=st["scale"], d_v=st["d_v"], out=st["out"])
    return {"pages": pd, "out": out, "lse": lse}


def run(st):
    kind = st["kind"]
    scales = {"q_scale": st["q_scale"], "k_scale": st["k_scale"]}
    if kind == "prefill":
        B.janus_indexer_scores(st["q"], st["k"], st["w"], q_pos0=st["L"], scores=st["scores"], keys_fp4=st["dtype"] == "fp4", **scales)
        B.janus_topk(st["scores"], st["S"], st["k_top"], q_pos0=st["L"], want_count=False, want_kth=False,
                     idx=st["idx"])
        return _demand_and_attention(st, st["idx"])
    if kind == "onecall":
        _, count, kth = B.janus_indexer_topk(st["q"], st["k"], st["w"], st["k_top"], q_pos0=st["L"], row_bias=st.get("row_bias"),
                                             col_bias=st.get("col_bias"), workspace=st["workspace"], idx=st["idx"], **scales)
        return {"count": count, "kth": kth, **_demand_and_attention(st, st["idx"])}
    if kind == "decode":
        B.janus_indexer_scores_batch(st["q"], st["k"], st["w"], st["key_off"], st["max_keys"], scores=st["scores"], keys_fp4=st["dtype"] == "fp4",
                                     **scales)
        idx, count, kth = B.janus_topk_batch(st["scores"], st["key_off"], st["k_top"], row_lengths=st["row_len"])
        pd = B.janus_page_demand_batch(idx, demand_limits=st["limits"], page_size=st["page"], page_tables=st["tables"], table_offsets=st["tab_off"],
                                       n_phys_pages=st["n_phys"], predicted_bitmap=st["predicted"], out=st["pages"])
        out, lse = B.janus_sparse_attn_decode(st["Q"], st["k_pool"], st["v_pool"], idx, page_tables=st["tables"], table_offsets=st["tab_off"],
                                              page_size=st["page"], softmax_scale=st["scale"], d_v=st["d_v"], out=st["out"])
        return {"count": count, "kth": kth, "pages": pd, "out": out, "lse": lse}
    if kind == "predict":
        union, shards, _ = P.sharded_predicted_pages(st["q"], st["k"], st["w"], L=st["L"], k=st["k_top"], n_shards=st["shards"], page_size=st["page"],
                                                     page_table=st["page_table"], n_phys_pages=st["n_phys"], **scales)
        return {"union": union, "shards": shards}
    B.janus_indexer_scores(st["q"], st["k"], st["w"], q_pos0=st["L"], scores=st["scores"], **scales)
    pooled = B.janus_entry_pool_scores(st["scores"], st["S"], entry_size=st["entry"], q_pos0=st["L"])
    n_entries = (st["S"] + st["entry"] - 1) // st["entry"]
    entries, count, kth = B.janus_topk_entries(pooled, n_entries, st["k_top"], q_pos0=st["L"], entry_size=st["entry"])
    idx = B.janus_entry_expand(entries, q_pos0=st["L"], entry_size=st["entry"])
    return {"pooled": pooled[:, :n_entries], "count": count, "kth": kth, **_demand_and_attention(st, idx)}


# ---- what a pass cannot do without ------------------------------------------------------------------------------------------------
def work(case):
    kind, k = case["kind"], case["k"]
    heads, dim = case.get("heads", 64), case.get("dim", 128)
    page = case.get("page", 64)
    elem = {"bf16": 2.0, "fp8": 1.0, "fp4": 0.5}[case["dtype"]]
    scale = 0 if case["dtype"] == "bf16" else 4
    h_q, n_kv, d_qk, d_v, alias = LAYOUTS[case.get("layout", "latent")]
    row_bytes = 2 * n_kv * (d_qk + (0 if alias else d_v))
    if kind == "decode":
        n = case["sessions"]
        S = case["L"] * (1 + (n - 1) * 5 / 8) / n + 1           # the longest history, the others 1/4 to 1 of it
        pairs, keys, n_q, n_sel = n * S, n * S, n, n * min(k, S)
        gathered = n_sel
    else:
        n_q, L = case["M"], case["L"]
        S = L if kind == "predict" else L + n_q
        pairs = float(n_q) * L if kind == "predict" else float(n_q) * L + n_q * (n_q + 1) / 2
        keys = S
        n_sel = n_q * min(k * case.get("entry", 1), S)
        gathered = min(n_sel, S)
    q_elem = 2 if case["dtype"] == "bf16" else 1
    n_bytes = keys * (dim * elem + scale) + n_q * heads * (dim * q_elem + 4)
    flops = 2.0 * heads * dim * pairs
    n_bytes += (S if kind != "decode" else keys) / page * (4 + 1 / 8 + 12)      # page table, bitmaps, lists
    if kind != "predict":
        n_bytes += gathered * row_bytes + n_q * h_q * (2 * d_qk + 2 * d_v + 4)
        flops += 2.0 * h_q * (d_qk + d_v) * n_sel
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "predict":
        return "exact"                     # bitmaps only
    # attention outputs are bf16 and P is rounded to bf16; the order of a selection, and with it the order of the sums, is free:
    # two runs on the same inputs differ by 2.2e-3.  Over thousands of rows a few have a tie at the k-th score, where either key
    # may be taken: one of 2048 equally weighted values replaced is up to 0.1 of the outputs' root mean square
    return {"rel": 1e-2, "max": 0.3}
