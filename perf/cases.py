"""Workloads of the decode-attention library at the sizes it is used at, through its public calls.

A case is a dict of plain values.  `listed()` names the standing ones, `draw(rng)` gives one more
of the same ranges, `prepare(case, seed)` builds what a serving program holds before the call
(paged cache, index, queries, workspace), `run(state)` makes one call, `work(case)` and
`tolerance(case)` say what that call has to move and how far two correct results may be apart.

Kinds of call:
  decode   pqhsa_decode, one attention layer of one decode step
  update   pqhsa_index_update, the periodic encoding of a layer's newest tokens
  build    pqhsa_index_build, the index of a layer after its prompt was read
  dense    pqhsa_dense_decode, the whole cache attended (contexts below the break-even length)
"""
from __future__ import annotations

import math

import torch

from paper_2609_33746_b200 import pqhsa
from paper_2609_33746_b200.index_builder import build_index, seed_positions
from paper_2609_33746_b200.runner import DecodeOp
from paper_2609_33746_b200.workload import DecodeConfig, generate, named_config

K = 1024
DEFAULTS = dict(kind="decode", dtype="bf16", q_heads=32, kv_heads=8, n_list=1024, pq_m=32, pq_ncode=256,
                budget_ppm=10000, layout="split", page_size=16, n_sink=0, n_local=0, page_rounded=False,
                window="", tables="fp32", outlier_scale=8.0, n_new=0, coarse_iters=1, pq_iters=2)


def _lens(*lens) -> str:
    return ",".join(str(n) for n in lens)


def _named(name: str) -> dict:
    """Shape of one of the repository's named workloads."""
    c = named_config(name)
    return dict(lens=_lens(*c.seq_lens), dtype=c.dtype, q_heads=c.n_q_heads, kv_heads=c.n_kv_heads,
                n_list=c.n_list, pq_m=c.pq_m, pq_ncode=c.pq_ncode, budget_ppm=c.budget_ppm,
                n_sink=c.n_sink, n_local=c.n_local, page_rounded=c.exact_set_multiple > 1,
                outlier_scale=c.outlier_scale)


def listed():
    return [
        # one KV head's share of a short conversation: nothing but latency
        dict(_named("c1"), name="decode_4k"),
        # a single request at 32K, 2 % budget: the short end of where the method is used
        dict(_named("c2"), name="decode_32k"),
        # a single request at 128K: interactive use
        dict(_named("c3_b1_r1"), name="decode_128k"),
        # eight requests at 128K: the throughput setting, and the repository's benchmark
        dict(_named("c3_b8_r1"), name="decode_128k_b8"),
        # sixteen requests of different lengths, eight query heads per KV head, strong outliers
        dict(_named("c4"), name="decode_ragged_g8_b16"),
        # one very long request
        dict(_named("c5_n512_b1"), name="decode_512k"),
        # eight requests with the paper's own index (4-bit codes, sinks, window, whole pages)
        dict(_named("c3p_b8_r1"), name="decode_4bit_b8"),
        # four requests of odd lengths between two index updates (a window of its own each), fp16,
        # interleaved cache, two query heads per KV head, shorter codes
        dict(lens=_lens(20011, 33333, 7777, 48001), dtype="fp16", q_heads=16, kv_heads=8, n_list=250, pq_m=16,
             budget_ppm=20000, layout="interleaved", n_sink=4, window=_lens(37, 255, 1, 128),
             name="decode_windows_fp16"),
        # the throughput setting with fp16 tables and the fp32 re-score
        dict(_named("c3_b8_r1"), tables="rescore", name="decode_rescore_b8"),
        # every 256 steps: the newest 256 tokens of eight requests enter the lists
        dict(_named("c3_b8_r1"), kind="update", n_new=256, name="update_b8"),
        # after a 128K prompt: the index of one layer (one coarse, two codebook iterations)
        dict(_named("c3_b1_r1"), kind="build", name="build_128k"),
        # eight requests too short for the method: attention over the whole cache
        dict(lens=_lens(*(32 * K,) * 8), kind="dense", name="dense_32k_b8"),
    ]


MAX_TOKENS = 64 * 128 * K                        # tokens x KV heads of the largest decode
MAX_BUILD = 8 * 128 * K * 1024                   # tokens x KV heads x lists of the largest build
MAX_DENSE = 64 * 32 * K


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("decode", "update", "build", "dense"), (64, 12, 12, 12))[0]
    c = dict(kind=kind, dtype=rng.choice(("bf16", "bf16", "fp16")), layout=rng.choice(("split", "interleaved")),
             page_size=rng.choice((16, 16, 32)))
    c["kv_heads"] = rng.choice((1, 2, 4, 8, 8))
    group = rng.choice((1, 2, 4, 4, 4, 8))
    n = _log_int(rng, 2 * K, 512 * K)
    c["q_heads"] = c["kv_heads"] * group
    four_bit = n >= 8 * K and rng.random() < 0.25
    c["pq_ncode"] = 16 if four_bit else 256
    c["pq_m"] = 8 if four_bit else rng.choice((16, 32, 32, 32))
    c["budget_ppm"] = _log_int(rng, 5000, 40000)
    most = MAX_DENSE if kind == "dense" else MAX_TOKENS
    batch = max(1, min(_log_int(rng, 1, 32), most // (n * c["kv_heads"])))
    n = min(n, most // c["kv_heads"])
    # about 128 tokens a list, as the context sweep has it; any whole number is allowed.  Codes of
    # four bits resolve little by themselves: they go with hundreds of lists (the paper's 512)
    n_list = max(16, min(4096, int(n / 128 * rng.uniform(0.5, 2.0))))
    if four_bit:
        n_list = _log_int(rng, 256, 1024)
    if kind == "build":
        batch = max(1, min(batch, MAX_BUILD // (n * c["kv_heads"] * n_list)))
        n = min(n, MAX_BUILD // (c["kv_heads"] * n_list))
        c["coarse_iters"] = rng.choice((1, 1, 2))
        c["pq_iters"] = rng.choice((1, 2, 2))
    c["n_list"] = n_list
    ragged = rng.random() < 0.5
    lens = [rng.randint(max(1, n * 3 // 4), n) if ragged else n for _ in range(batch)]
    c["lens"] = _lens(*lens)
    if kind in ("decode", "build"):
        part = rng.choice(("none", "fixed", "own"))
        if part != "none":
            c["n_sink"] = 4
        if part == "fixed":
            c["n_local"] = 128
            c["page_rounded"] = True
        if part == "own":
            c["window"] = _lens(*(rng.randint(0, 256) for _ in lens))
    if kind == "decode" and group >= 4 and c["pq_m"] == 32:
        c["tables"] = rng.choice(("fp32", "fp32", "fp32", "rescore"))
    if kind == "update":
        c["n_new"] = _log_int(rng, 1, 1024)
    return c


def _config(case, seed: int) -> DecodeConfig:
    c = {**DEFAULTS, **case}
    lens = tuple(int(x) for x in c["lens"].split(","))
    indexed = None
    if c["window"]:
        indexed = tuple(max(0, n - int(w)) for n, w in zip(lens, c["window"].split(",")))
    if c["kind"] == "update":                    # the newest tokens are in no list yet
        indexed = tuple(max(0, n - c["n_new"]) for n in lens)
    return DecodeConfig(c["kind"], len(lens), c["q_heads"], c["kv_heads"], lens, c["dtype"], c["n_list"],
                        c["pq_m"], c["budget_ppm"], pq_ncode=c["pq_ncode"], page_size=c["page_size"],
                        outlier_scale=c["outlier_scale"], kmeans_iters=1,
                        pq_iters=2 if c["pq_ncode"] == 16 else 0, seed=seed,
                        kv_layout=c["layout"], n_sink=c["n_sink"], n_local=c["n_local"],
                        exact_set_multiple=c["page_size"] if c["page_rounded"] else 0, indexed_lens=indexed)


def _params(cfg: DecodeConfig, inp, n_max: int):
    return pqhsa.make_params(batch=cfg.batch, n_q_heads=cfg.n_q_heads, n_kv_heads=cfg.n_kv_heads,
                             n_list=cfg.n_list, pq_m=cfg.pq_m, pq_ncode=cfg.pq_ncode, max_seq_len=n_max,
                             max_pages_per_seq=inp.max_pages_per_seq, budget_ppm=cfg.budget_ppm,
                             dtype=cfg.dtype, page_size=cfg.page_size, n_sink=cfg.n_sink,
                             n_local=cfg.n_local, exact_set_multiple=cfg.exact_set_multiple)


def _paged(cfg: DecodeConfig, inp):
    v = inp.k_cache.view(-1)[cfg.head_dim:] if cfg.kv_layout == "interleaved" else inp.v_cache
    return pqhsa.make_paged_kv(inp.k_cache, v, inp.stride_page, inp.stride_token, inp.stride_head,
                               inp.block_table)


def prepare(case, seed):
    c = {**DEFAULTS, **case}
    cfg = _config(case, seed)
    inp = generate(cfg, device="cuda")
    n_max = (cfg.max_seq_len + 15) // 16 * 16
    if c["kind"] == "dense":
        params = _params(cfg, inp, n_max)
        ws = torch.empty(pqhsa.dense_workspace_bytes(params), dtype=torch.uint8, device="cuda")
        return dict(kind="dense", inp=inp, params=params, kv=_paged(cfg, inp), ws=ws, out=torch.empty_like(inp.q))
    if c["kind"] == "build":
        units, dev = (cfg.batch, cfg.n_kv_heads), "cuda"
        params = _params(cfg, inp, n_max)
        indexed = None
        if cfg.indexed_lens is not None:
            indexed = torch.tensor(cfg.indexed_lens, dtype=torch.int32, device=dev)
            params.indexed_lens = indexed.data_ptr()
        code_bytes = cfg.pq_m // 2 if cfg.pq_ncode == 16 else cfg.pq_m
        out = (torch.zeros((*units, cfg.n_list, 128), device=dev),
               torch.zeros((*units, cfg.pq_m, cfg.pq_ncode, cfg.pq_dsub), device=dev),
               torch.zeros((*units, n_max, code_bytes), dtype=torch.uint8, device=dev),
               torch.zeros((*units, n_max), dtype=torch.int16, device=dev),
               torch.zeros((*units, n_max), device=dev),
               torch.zeros((*units, cfg.n_list, 128), device=dev),
               torch.zeros((*units, cfg.n_list), dtype=torch.int32, device=dev))
        lists, words = seed_positions(inp)
        ws = torch.empty(pqhsa.index_build_workspace_bytes(params), dtype=torch.uint8, device=dev)
        return dict(kind="build", inp=inp, params=params, kv=_paged(cfg, inp), lists=lists, words=words,
                    iters=(c["coarse_iters"], c["pq_iters"]), out=out, ws=ws, indexed=indexed)
    idx = build_index(inp)
    if c["kind"] == "update":
        n_new = [min(n, c["n_new"]) for n in cfg.seq_lens]
        first = torch.tensor([n - k for n, k in zip(cfg.seq_lens, n_new)], dtype=torch.int32, device="cuda")
        rw = pqhsa.make_index_rw(idx.centroids, idx.codebooks, idx.codes, idx.list_ids, idx.key_norms,
                                 idx.list_vmeans, idx.list_counts)
        return dict(kind="update", inp=inp, params=_params(cfg, inp, idx.codes.shape[2]), kv=_paged(cfg, inp),
                    rw=rw, idx=idx, first=first, max_new=max(n_new),
                    n_new=torch.tensor(n_new, dtype=torch.int32, device="cuda"))
    tables = {"fp32": False, "rescore": "rescore"}[c["tables"]]
    return dict(kind="decode", op=DecodeOp(inp, idx, fp16_tables=tables))


def run(state):
    kind = state["kind"]
    if kind == "decode":
        return state["op"].decode()
    if kind == "update":
        i = state["idx"]
        pqhsa.index_update(state["params"], state["rw"], state["kv"], state["first"], state["n_new"],
                           state["max_new"])
        return [i.codes, i.list_ids, i.key_norms, i.list_vmeans, i.list_counts]
    if kind == "build":
        pqhsa.index_build(state["params"], state["kv"], state["inp"].seq_lens, state["lists"], state["words"],
                          *state["iters"], *state["out"], state["ws"])
        return list(state["out"])
    pqhsa.dense_decode(state["params"], state["inp"].q, state["kv"], state["inp"].seq_lens, state["out"],
                       state["ws"])
    return state["out"]


def _exact_tokens(c, n: int, window: int) -> int:
    """Tokens of one sequence that are attended exactly (sinks, window, selected)."""
    fixed = min(n, c["n_sink"]) + min(n, window)
    k = -(-max(0, n - fixed) * c["budget_ppm"] // 1000000)
    if c["page_rounded"]:
        k = -(-(fixed + k) // c["page_size"]) * c["page_size"] - fixed
    return min(n, fixed + k)


def work(case):
    c = {**DEFAULTS, **case}
    lens = [int(x) for x in c["lens"].split(",")]
    windows = [int(x) for x in c["window"].split(",")] if c["window"] else [c["n_local"]] * len(lens)
    kv, hq, tokens = c["kv_heads"], c["q_heads"], sum(lens) * c["kv_heads"]
    code = c["pq_m"] // 2 if c["pq_ncode"] == 16 else c["pq_m"]
    units = len(lens) * kv
    tables = units * (c["n_list"] * 512 + c["pq_ncode"] * 512)       # centroids and codebooks
    io = 2 * len(lens) * hq * 256                                    # queries in, outputs out
    if c["kind"] == "dense":
        return dict(bytes=tokens * 512 + io, flops=4 * 128 * sum(lens) * hq)
    if c["kind"] == "build":
        passes = c["coarse_iters"] + 1, c["pq_iters"] + 1
        flops = tokens * 2 * 128 * (passes[0] * c["n_list"] + passes[1] * c["pq_ncode"])
        return dict(bytes=tokens * (512 + code + 6) + tables + units * c["n_list"] * 516, flops=flops)
    if c["kind"] == "update":
        new = sum(min(n, c["n_new"]) for n in lens) * kv
        touched = units * min(c["n_list"], c["n_new"]) * 2 * 516     # means and counts, read and written
        return dict(bytes=new * (512 + code + 6) + tables + touched,
                    flops=new * 2 * 128 * (c["n_list"] + c["pq_ncode"]))
    exact = sum(_exact_tokens(c, n, w) for n, w in zip(lens, windows)) * hq
    # codes, norm and list id of every token; K and V rows of the exact set of every query head;
    # list means; the flops are the table sums and the dot products of the exact part
    return dict(bytes=tokens * (code + 6) + exact * 512 + tables + units * c["n_list"] * 512 + io,
                flops=sum(lens) * hq * (c["pq_m"] + 2) + exact * 512)


def tolerance(case):
    """Decode and dense: half an ulp of the output type (measured against float64: 1.6e-3 of the
    2-norm in bf16, 2e-4 in fp16) and, with 4-bit codes, what the order of the fp32 list sums
    leaves after the selected tokens were taken out (up to 5e-4).  Build and update: a token whose
    two nearest centres tie in fp32 changes lists and moves two means by a part in their size."""
    c = {**DEFAULTS, **case}
    if c["kind"] == "build":
        return dict(rel=5e-3, max=0.5, differ=2e-3)
    if c["kind"] == "update":
        return dict(rel=1e-3, max=0.5, differ=1e-5)
    if c["dtype"] == "bf16" or c["pq_ncode"] == 16:
        return dict(rel=6e-3, max=0.05)
    return dict(rel=1e-3, max=0.02)
