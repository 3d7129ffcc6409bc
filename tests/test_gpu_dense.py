"""Dense decode attention at the edges of its windows, stages and head groups (-m gpu), against
softmax attention in float64 on the same cache values.  Tolerance: half an ulp of the output type
(2^-8 of the value in bf16, 2^-11 in fp16) plus 1e-4 for the fp32 sums of at most 2,000 terms."""
import math

import pytest
import torch

from paper_2609_33746_b200 import pqhsa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,half_ulp", [("bf16", 2.0 ** -8), ("fp16", 2.0 ** -11)])
@pytest.mark.parametrize("group", [1, 2, 3, 5, 8, 12, 16])
@pytest.mark.parametrize("lens,page", [((1, 7, 8), 16), ((9, 31, 32), 1), ((33, 255, 257), 32), ((1000, 0, 2003), 16)])
def test_dense_at_the_edges(lens, page, group, dtype, half_ulp):
    kv_heads, d, B = 2, 128, len(lens)
    tdt = {"bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    n_max = (max(lens) + 15) // 16 * 16
    pages = (n_max + page - 1) // page
    g = torch.Generator(device="cuda").manual_seed(group * 1000 + lens[2])
    cache = [torch.randn((B * pages, page, kv_heads, d), generator=g, device="cuda").to(tdt) for _ in range(2)]
    q = (2 * torch.randn((B, kv_heads * group, d), generator=g, device="cuda")).to(tdt)
    table = torch.randperm(B * pages, generator=g, device="cuda").int().view(B, pages)
    for b, n in enumerate(lens):            # what lies past the end of a sequence must not matter
        for i in range(n, pages * page):
            cache[1][table[b, i // page], i % page] = float("nan")
    p = pqhsa.make_params(batch=B, n_q_heads=kv_heads * group, n_kv_heads=kv_heads, n_list=16, pq_m=8,
                          max_seq_len=n_max, max_pages_per_seq=pages, budget_ppm=10000, dtype=dtype, page_size=page)
    kv = pqhsa.make_paged_kv(cache[0], cache[1], page * kv_heads * d, kv_heads * d, d, table)
    out = torch.full_like(q, 3.0)
    ws = torch.empty(pqhsa.dense_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    pqhsa.dense_decode(p, q, kv, torch.tensor(lens, dtype=torch.int32, device="cuda"), out, ws)
    for b, n in enumerate(lens):
        if n == 0:
            assert bool((out[b] == 0).all())
            continue
        pos = torch.arange(n, device="cuda")
        K, V = (c[table[b, pos // page].long(), pos % page].double().transpose(0, 1) for c in cache)
        s = torch.einsum("hgd,hnd->hgn", q[b].double().view(kv_heads, group, d), K) / math.sqrt(d)
        want = torch.einsum("hgn,hnd->hgd", s.softmax(-1), V).reshape(-1, d)
        assert bool(((out[b].double() - want).abs() <= half_ulp * want.abs() + 1e-4).all())
