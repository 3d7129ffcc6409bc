"""Dense decode attention on the tensor cores (-m gpu): weights over many binary orders, scores far apart, values that
are not finite, caches whose K and V interleave; against softmax attention in float64.

Tolerance: half an ulp of the output type, plus for the fp32 sums 2^-24 per addition over a warp's tokens and a
score's rounding (2^-24 of its size, some ten of them), relative to the sum of the weighted magnitudes."""
import math

import pytest
import torch

from paper_2609_33746_b200 import pqhsa

pytestmark = pytest.mark.gpu

D, PAGE = 128, 16


def run(q, k, v, n, dtype, kv_heads, interleaved=False):
    """q [heads, D]; k, v [kv_heads, n, D], laid out in pages in reverse order."""
    pages = (n + PAGE - 1) // PAGE
    table = torch.arange(pages - 1, -1, -1, dtype=torch.int32, device="cuda").view(1, pages)
    cache = torch.zeros((2, pages * PAGE, kv_heads, D), dtype=dtype, device="cuda")
    cache[0, :n], cache[1, :n] = k.transpose(0, 1), v.transpose(0, 1)
    cache = cache.view(2, pages, PAGE, kv_heads, D).flip(1)
    if interleaved:
        both = torch.cat([cache[0], cache[1]], dim=-1).contiguous()
        kv = pqhsa.make_paged_kv(both, both.view(-1)[D:], PAGE * kv_heads * 2 * D, kv_heads * 2 * D, 2 * D, table)
    else:
        kc, vc = cache[0].contiguous(), cache[1].contiguous()
        kv = pqhsa.make_paged_kv(kc, vc, PAGE * kv_heads * D, kv_heads * D, D, table)
    p = pqhsa.make_params(batch=1, n_q_heads=q.shape[0], n_kv_heads=kv_heads, n_list=16, pq_m=8, max_seq_len=pages * PAGE,
                          max_pages_per_seq=pages, budget_ppm=10000, dtype="bf16" if dtype == torch.bfloat16 else "fp16",
                          page_size=PAGE)
    ws = torch.empty(pqhsa.dense_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    out = torch.zeros_like(q).view(1, *q.shape)
    pqhsa.dense_decode(p, q, kv, torch.tensor([n], dtype=torch.int32, device="cuda"), out, ws)
    torch.cuda.synchronize()
    return out[0]


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("group,n", [(4, 1), (4, 15), (8, 17), (4, 4099), (8, 9001), (16, 2050), (1, 20000)])
@pytest.mark.parametrize("spread", [0.05, 1.0, 6.0])
def test_weights_of_every_size(group, n, spread, dtype):
    g = torch.Generator(device="cuda").manual_seed(n + group)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
    q, k, v = (spread * rnd(2 * group, D)).to(dtype), rnd(2, n, D).to(dtype), (rnd(2, n, D) + 3).to(dtype)
    out = run(q, k, v, n, dtype, 2, interleaved=n % 2 == 1).double()
    qs = q.double().view(2, group, D) / math.sqrt(D)
    s = qs @ k.double().transpose(1, 2)
    w = s.softmax(-1)
    want = (w @ v.double()).view(-1, D)
    size = (w @ v.double().abs()).view(-1, D)
    score = float((qs.abs() @ k.double().abs().transpose(1, 2)).max())
    bound = (10 * score + n / 64 + 40) * 2.0 ** -24 * size
    ulp = 2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -11
    assert bool(((out - want).abs() <= ulp * want.abs() + bound).all())


def cancelling(group, n, head, dtype, seed, device="cuda"):
    """Queries and keys of one dim, so that dot products are exact; values whose sum weighted for one head of each
    KV head is next to nothing: the last three take back what the others leave."""
    g = torch.Generator().manual_seed(seed)
    q, k = torch.zeros(2, group, D), torch.zeros(2, n, D)
    q[..., 0], k[..., 0] = 1 + 3 * torch.rand(2, group, generator=g), 6 * torch.rand(2, n, generator=g)
    q, k, v = q.to(dtype).view(-1, D), k.to(dtype), torch.randn(2, n, D, generator=g).to(dtype)
    w = (q.double().view(2, group, D)[:, head:head + 1] / math.sqrt(D) @ k.double().transpose(1, 2)).softmax(-1)[:, 0, :, None]
    left = (w * v.double())[:, :-3].sum(1)
    for j in (-3, -2, -1):
        v[:, j] = (-left / w[:, j]).to(dtype)
        left = left + w[:, j] * v[:, j].double()
    return [x.to(device) for x in (q, k, v, left, (w * v.double().abs()).sum(1))]


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("group", [1, 4, 8, 16])
@pytest.mark.parametrize("n", [5, 8, 16, 21])
def test_sums_that_cancel(group, n, dtype):
    """What is left of values that cancel shows the bits of the weights, not the output's rounding.  Tolerance, of the
    weighted magnitudes: exponentials to 2 ulp (2^-22), their argument of at most 3 rounded once (2^-22.5 times ln 2), a few
    fp32 additions (2^-24 each): 2^-20.  (Without the third bf16 number of a weight the errors reach 2^-18.9 and more in
    every case, without the second fp16 one 2^-12.5; the third fp16 number is below the exponential's error.)"""
    for seed in range(4):
        head = seed % group
        q, k, v, want, size = cancelling(group, n, head, dtype, 100 * n + seed)
        out = run(q, k, v, n, dtype, 2).double().view(2, group, D)[:, head]
        assert bool(((out - want).abs() <= 2.0 ** -20 * size + 2.0 ** -11 * want.abs()).all()), float(((out - want).abs() / size).max())


@pytest.mark.parametrize("dtype,half_ulp", [(torch.bfloat16, 2.0 ** -9), (torch.float16, 2.0 ** -12)])
@pytest.mark.parametrize("group", [4, 8])
@pytest.mark.parametrize("log2_weight", [24, 41, 48])
def test_many_small_weights_beside_a_large_one(log2_weight, group, dtype, half_ulp):
    """60 thousand weights far below that of a token whose values are zero: the output is theirs alone."""
    n = 60001
    q, k, v = torch.zeros((2 * group, D)), torch.zeros((2, n, D)), torch.full((2, n, D), 60000.0)
    q[:, 0], k[:, n // 2, 0], v[:, n // 2] = 16.0, log2_weight * math.log(2) * math.sqrt(D) / 16, 0.0
    q, k, v = (x.cuda().to(dtype) for x in (q, k, v))
    out = run(q, k, v, n, dtype, 2).double()
    w = (q.double().view(2, group, D) / math.sqrt(D) @ k.double().transpose(1, 2)).softmax(-1)
    want = (w @ v.double()).view(-1, D)
    # (fp32: 2^-24 of the exponent's argument, 48, and of some ten thousand additions in a chain; fp16 below 2^-14: 2^-25)
    assert bool(((out - want).abs() <= (half_ulp + 2.0 ** -11) * want + 2.0 ** -25).all()), (float(out[0, 0]), float(want[0, 0]))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("group", [2, 8])
def test_an_infinite_value_stays_one(group, dtype):
    """An infinite value makes its dim infinite and leaves the others as they are, as a weighted sum does."""
    g = torch.Generator(device="cuda").manual_seed(group)
    q, k, v = (torch.randn(s, generator=g, device="cuda").to(dtype) for s in ((2 * group, D), (2, 300, D), (2, 300, D)))
    clean = run(q, k, v, 300, dtype, 2)
    v[0, 133, 5], v[0, 7, 90] = float("inf"), -float("inf")
    out = run(q, k, v, 300, dtype, 2)
    assert bool((out[:group, 5] == float("inf")).all()) and bool((out[:group, 90] == -float("inf")).all())
    keep = torch.ones(D, dtype=torch.bool, device="cuda")
    keep[5] = keep[90] = False
    torch.testing.assert_close(out[:group, keep], clean[:group, keep], rtol=2.0 ** -7, atol=2.0 ** -12)
    assert torch.equal(out[group:], clean[group:])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("group,n", [(1, 31), (4, 700), (8, 700), (16, 3000)])
def test_infinite_values_in_many_places(group, n, dtype):
    """Infinite values of either sign and values that are no numbers, several in a dim and in a stage of 16 tokens:
    infinite, no number and finite where the weighted sum in float64 is."""
    g = torch.Generator(device="cuda").manual_seed(group)
    q, k, v = (torch.randn(s, generator=g, device="cuda").to(dtype) for s in ((2 * group, D), (2, n, D), (2, n, D)))
    bad = torch.tensor([float("inf"), -float("inf"), float("nan")], device="cuda", dtype=dtype)
    at, dim, what = (torch.randint(0, m, (40,), generator=g, device="cuda") for m in (n, 100, 3))
    v[0, at, dim] = bad[what]
    v[0, :, 127] = float("inf")
    out = run(q, k, v, n, dtype, 2).double()
    w = (q.double().view(2, group, D) / math.sqrt(D) @ k.double().transpose(1, 2)).softmax(-1)
    want = (w @ v.double()).view(-1, D)
    assert torch.equal(out.isnan(), want.isnan()) and torch.equal(out.isinf(), want.isinf())
    assert torch.equal(out[want.isinf()], want[want.isinf()])
    size = (w @ v.double().abs()).view(-1, D)
    fine = want.isfinite()
    assert bool(((out - want).abs() <= 2.0 ** -7 * want.abs() + 2.0 ** -12 * size)[fine].all())


@pytest.mark.parametrize("group", [4, 8])
def test_an_infinite_value_costs_no_time(group):
    """The 16 tokens around it are taken again, nothing else (13 times the call when a warp repeated all of its tokens)."""
    n, kv_heads = 65536, 4
    g = torch.Generator(device="cuda").manual_seed(group)
    q, k, v = (torch.randn(s, generator=g, device="cuda").bfloat16() for s in ((kv_heads * group, D), (kv_heads, n, D), (kv_heads, n, D)))
    pages = n // PAGE
    table = torch.arange(pages, dtype=torch.int32, device="cuda").view(1, pages)
    kc, vc = (x.transpose(0, 1).contiguous() for x in (k, v))
    kv = pqhsa.make_paged_kv(kc, vc, PAGE * kv_heads * D, kv_heads * D, D, table)
    p = pqhsa.make_params(batch=1, n_q_heads=q.shape[0], n_kv_heads=kv_heads, n_list=16, pq_m=8, max_seq_len=n,
                          max_pages_per_seq=pages, budget_ppm=10000, dtype="bf16", page_size=PAGE)
    ws = torch.empty(pqhsa.dense_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    out, seq = torch.zeros_like(q), torch.tensor([n], dtype=torch.int32, device="cuda")

    def time_of():
        best = float("inf")
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                pqhsa.dense_decode(p, q, kv, seq, out, ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    clean = time_of()
    vc.view(-1)[n * kv_heads * D // 2 + 77] = float("inf")
    assert time_of() <= 1.5 * clean
