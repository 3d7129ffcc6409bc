"""The forms of a call that reach the top-k from the tiles' maxima (-m gpu), against the staged calls on the same
inputs, which use the other top-k: code widths and subspaces (every shape of the scans' maxima), groups of one to
sixteen heads, sinks, windows, rounded exact sets, fp16 tables with and without the re-score, the variants.

Both top-k are exact and both scans form the same scores: selection and k-th score are equal.  Output: half an ulp of
the output type on either side, and what the order of the fp32 list sums leaves (5e-4 of the row's size)."""
import pytest
import torch

from paper_2609_33746_b200 import pqhsa
from paper_2609_33746_b200.runner import DecodeOp
from paper_2609_33746_b200.workload import DecodeConfig, generate
from paper_2609_33746_b200.index_builder import build_index

pytestmark = pytest.mark.gpu

BASE = dict(batch=2, n_q_heads=64, n_kv_heads=16, seq_lens=(20001, 17003), dtype="bf16", n_list=64, pq_m=32, budget_ppm=10000,
            kmeans_iters=1, seed=11)
ROUTES = {
    "m8": dict(pq_m=8), "m16": dict(pq_m=16), "m8_one_head": dict(pq_m=8, n_kv_heads=64),
    "m64_two_heads": dict(pq_m=64, n_kv_heads=32), "m64_one_head": dict(pq_m=64, n_kv_heads=64), "group_16": dict(n_kv_heads=4), "group_3": dict(n_q_heads=60, n_kv_heads=20),
    "four_bit_m16": dict(pq_m=16, pq_ncode=16), "four_bit_m16_one_head": dict(pq_m=16, pq_ncode=16, n_kv_heads=64),
    "four_bit_m8_two_heads": dict(pq_m=8, pq_ncode=16, n_kv_heads=32), "four_bit_lists": dict(pq_m=8, pq_ncode=16, n_list=1500),
    "fp16_interleaved": dict(dtype="fp16", kv_layout="interleaved"),
    "sinks_window_pages": dict(n_sink=4, n_local=128, exact_set_multiple=16),
    "own_windows": dict(n_sink=4, indexed_lens=(20001 - 37, 17003 - 255)),
    "nothing_indexed": dict(n_sink=4, indexed_lens=(20001, 2)),
    "rounded_to_512": dict(seq_lens=(90000, 300), exact_set_multiple=512),         # (rows of 300: all, with no bound)
    "empty_row": dict(seq_lens=(30000, 0)),
    "fp16_tables": dict(tables=True), "fp16_tables_g8": dict(tables=True, n_kv_heads=8),
    "rescore": dict(tables="rescore", seq_lens=(60000, 41000)), "rescore_g8": dict(tables="rescore", n_kv_heads=8, seq_lens=(60000, 41000)),
    # the large scores of a row stand at its end: the list is cut and the re-score reads the row
    "rescore_rising": dict(tables="rescore", seq_lens=(131071, 100001), rising=True),
    "rising": dict(seq_lens=(131071, 100001), rising=True),
    **{"variant_" + v: dict(variant=v) for v in ("T", "Bx", "C", "C2", "C2b")},
}


@pytest.mark.parametrize("route", list(ROUTES))
def test_fused_call_selects_what_the_stages_select(route):
    given = {**BASE, **ROUTES[route]}
    tables, rising = given.pop("tables", False), given.pop("rising", False)
    cfg = DecodeConfig(route, pq_iters=2 if given.get("pq_ncode") == 16 else None, **given)
    inp = generate(cfg, device="cuda")
    inp.q.mul_(1.0 / 32)                                 # (logits of a few units: no token's mass is all of its list's)
    idx = build_index(inp)
    if rising:
        idx.key_norms.mul_(torch.linspace(0.7, 1.4, idx.key_norms.shape[-1], device="cuda"))
    op = DecodeOp(inp, idx, fp16_tables=tables)
    last = pqhsa.decode_buffer_offset(op.params, pqhsa.BUF_OUT_F32) + 4 * pqhsa.buffer_elems(op.params, pqhsa.BUF_OUT_F32)
    assert pqhsa.workspace_bytes(op.params) > last + 255           # (the maxima have their place: this route is taken)
    op.alloc_stage_buffers()
    op.build_lut(), op.scan(), op.select(), op.hybrid_attend()
    assert op.device_status() == pqhsa.OK
    staged = op.out.clone()
    op.ws.fill_(0xAB)                                              # (nothing of the staged calls is left)
    op.out.fill_(9.0)
    op.decode()
    assert op.device_status() == pqhsa.OK
    rows, k_max = cfg.batch * cfg.n_q_heads, op.params.k_max
    count = op.decode_buffer(pqhsa.BUF_SEL_COUNT, torch.int32)
    assert torch.equal(count, op.sel_count)
    listed = torch.arange(k_max, device="cuda") < count[:, None]
    sets = [torch.where(listed, s.view(rows, k_max), -1).sort(dim=1).values
            for s in (op.decode_buffer(pqhsa.BUF_SEL_IDX, torch.int32), op.sel_idx)]
    assert torch.equal(*sets)
    some = count > 0
    assert torch.equal(op.decode_buffer(pqhsa.BUF_KTH)[some], op.kth[some])
    ulp = 2.0 ** -7 if cfg.dtype == "bf16" else 2.0 ** -10
    size = staged.double().norm(dim=-1, keepdim=True) / 128 ** 0.5
    diff = (op.out.double() - staged.double()).abs()
    assert bool((diff <= ulp * staged.double().abs() + 5e-4 * size).all()), float((diff / size).max())
