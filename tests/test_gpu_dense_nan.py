"""Dense decode attention over a cache with a key that is not a number (-m gpu): the softmax of such a
row is not a number either, so every query head of that KV head says so, and no other head changes."""
import pytest
import torch

from paper_2609_33746_b200 import pqhsa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group", [1, 2, 3, 8])
@pytest.mark.parametrize("n,at", [(1, 0), (40, 39), (700, 333)])
def test_a_nan_key_shows_in_the_output(n, at, group):
    kv_heads, page, d = 2, 16, 128
    pages = (n + page - 1) // page
    g = torch.Generator(device="cuda").manual_seed(n + group)
    k, v = (torch.randn((pages, page, kv_heads, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn((1, kv_heads * group, d), generator=g, device="cuda").bfloat16()
    table = torch.arange(pages, dtype=torch.int32, device="cuda").view(1, pages)
    seq = torch.tensor([n], dtype=torch.int32, device="cuda")
    p = pqhsa.make_params(batch=1, n_q_heads=kv_heads * group, n_kv_heads=kv_heads, n_list=16, pq_m=8,
                          max_seq_len=pages * page, max_pages_per_seq=pages, budget_ppm=10000, dtype="bf16")
    kv = pqhsa.make_paged_kv(k, v, page * kv_heads * d, kv_heads * d, d, table)
    ws = torch.empty(pqhsa.dense_workspace_bytes(p), dtype=torch.uint8, device="cuda")

    def run():
        out = torch.zeros_like(q)
        pqhsa.dense_decode(p, q, kv, seq, out, ws)
        return out.view(kv_heads, group, d)

    clean = run()
    k[at // page, at % page, 0, 17] = float("nan")
    out = run()
    assert bool(out[0].isnan().all()) and torch.equal(out[1], clean[1]) and bool(clean.isfinite().all())
