"""Scores that are not numbers (a cached key with a NaN): they rank below every number, -inf
included, on both top-k paths, and a decode leaves such a token out (-m gpu).  Exact."""
import pytest
import torch

from paper_2609_33746_b200 import pqhsa
from paper_2609_33746_b200.runner import DecodeOp
from paper_2609_33746_b200.workload import DecodeConfig

from helpers import make_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("heads,n,ppm", [
    (4, 4096, 10000), (32, 32769, 10000), (1, 5000, 300000), (8, 450011, 5000), (300, 16383, 20000),
    (256, 65536, 10000), (32, 524288, 10000)])
def test_nan_scores_rank_last(heads, n, ppm, sign):
    n_max = (n + 15) // 16 * 16
    p = pqhsa.make_params(batch=1, n_q_heads=heads, n_kv_heads=heads, n_list=16, pq_m=8, max_seq_len=n_max,
                          max_pages_per_seq=n_max // 16, budget_ppm=ppm, dtype="bf16")
    g = torch.Generator(device="cuda").manual_seed(n)
    scores = torch.randn((heads, n_max), generator=g, device="cuda")
    scores[:, 7::1013] = float("nan")
    scores[:, 100:140] = float("nan")
    scores *= sign                                       # (both signs of NaN)
    scores[:, :4] = -float("inf")
    seq = torch.tensor([n], dtype=torch.int32, device="cuda")
    sel = torch.full((heads, p.k_max), -7, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(heads, dtype=torch.int32, device="cuda")
    kth = torch.zeros(heads, device="cuda")
    ws = torch.zeros(pqhsa.workspace_bytes(p), dtype=torch.uint8, device="cuda")
    pqhsa.select(p, scores, seq, sel, cnt, kth, ws)
    assert pqhsa.last_device_status(p, ws) == pqhsa.OK
    k = (n * ppm + 999999) // 1000000
    numbers = torch.where(scores[:, :n].isnan(), -float("inf"), scores[:, :n])     # (fewer than n - k are not)
    want = torch.sort(numbers, dim=1, descending=True, stable=True)
    assert cnt.tolist() == [k] * heads
    assert torch.equal(kth, want.values[:, k - 1])
    assert torch.equal(sel[:, :k].long().sort(dim=1).values, want.indices[:, :k].sort(dim=1).values)


@pytest.mark.parametrize("lens", [(5000,), (3000,) * 40])
def test_decode_leaves_a_token_without_a_number_out(lens):
    cfg = DecodeConfig(name="nan", batch=len(lens), n_q_heads=8, n_kv_heads=2, seq_lens=lens, dtype="bf16", n_list=64,
                       pq_m=32, budget_ppm=20000, seed=5, kmeans_iters=1)
    inp, idx = make_case(cfg, device="cuda")
    for i in (17, 1234):                                 # cache rows and norms of these tokens
        idx.key_norms[:, :, i] = float("nan")
        for b in range(cfg.batch):
            page, slot = int(inp.block_table[b, i // cfg.page_size]), i % cfg.page_size
            inp.k_cache[page, slot] = float("nan")
            inp.v_cache[page, slot] = float("nan")
    op = DecodeOp(inp, idx)
    out = op.decode()
    torch.cuda.synchronize()
    assert op.device_status() == pqhsa.OK
    assert bool(out.isfinite().all())
