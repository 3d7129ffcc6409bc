"""Top-k by one thread-block cluster per score row (few or short rows), against a stable sort (-m gpu).

Exact: positions of the k largest scores, equal scores by position, for rows in random order, rows
that pile up on few values, rows sorted so that neighbours are all selected, and rows whose range
is stretched by outliers; at the edges of the kernel's slices and on both sides of the size at
which a slice leaves shared memory."""
import pytest
import torch

from paper_2609_33746_b200 import pqhsa

pytestmark = pytest.mark.gpu

PATTERNS = ("normal", "equal", "two_values", "sorted", "outliers", "narrow", "minus_inf",
            "tiny_or_zero")


def rows_of(pattern, rows, n, g):
    x = torch.randn((rows, n), generator=g, device="cuda") * 7 + 20
    if pattern == "equal":
        x.fill_(1.25)
    elif pattern == "two_values":
        x = torch.where(x > 20, 3.0, -0.0)
        x[:, ::3] *= -1.0                                # -0 and +0 compare equal
    elif pattern == "sorted":
        x = x.sort(dim=1, descending=bool(n % 2)).values
    elif pattern == "outliers":
        x[:, n // 2] = 1e30
        x[:, n // 3] = -1e30
        x[:, 0] = 65000.0
    elif pattern == "narrow":                            # neighbouring floats: few bits differ
        x = 50.0 + torch.randint(0, 3000, (rows, n), generator=g, device="cuda") * 2.0 ** -18
    elif pattern == "minus_inf":                         # sinks and window hold -inf
        x[:, :4] = -float("inf")
        x[:, n - min(n // 2, 128):] = -float("inf")
    elif pattern == "tiny_or_zero":                      # -0, +0 at a range's edge
        x = torch.where(x > 35, 1e-30, torch.where(x > 20, -0.0, 0.0))
    return x


@pytest.mark.parametrize("pattern", PATTERNS)
@pytest.mark.parametrize("heads,n,ppm", [
    (1, 5, 200000), (4, 1023, 20000), (32, 4100, 40000), (4, 32769, 10000), (32, 131071, 10000),
    (1, 70001, 300000), (3, 20000, 1000000), (8, 450011, 5000), (128, 9001, 20000),
    (64, 48001, 20000), (300, 16383, 20000)])
def test_cluster_select_is_the_stable_top_k(heads, n, ppm, pattern):
    n_max = (n + 15) // 16 * 16
    p = pqhsa.make_params(batch=1, n_q_heads=heads, n_kv_heads=heads, n_list=16, pq_m=8,
                          max_seq_len=n_max, max_pages_per_seq=n_max // 16, budget_ppm=ppm, dtype="bf16")
    g = torch.Generator(device="cuda").manual_seed(n + heads)
    scores = torch.full((heads, n_max), 1e38, device="cuda")      # past the row's end: never read as a score
    scores[:, :n] = rows_of(pattern, heads, n, g)
    seq = torch.tensor([n], dtype=torch.int32, device="cuda")
    sel = torch.full((heads, p.k_max), -7, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(heads, dtype=torch.int32, device="cuda")
    kth = torch.zeros(heads, device="cuda")
    ws = torch.zeros(pqhsa.workspace_bytes(p), dtype=torch.uint8, device="cuda")
    pqhsa.select(p, scores, seq, sel, cnt, kth, ws)
    assert pqhsa.last_device_status(p, ws) == pqhsa.OK
    k = (n * ppm + 999999) // 1000000
    order = torch.sort(scores[:, :n] + 0.0, dim=1, descending=True, stable=True)
    assert cnt.tolist() == [k] * heads
    assert torch.equal(kth, order.values[:, k - 1])
    assert torch.equal(sel[:, :k].long().sort(dim=1).values, order.indices[:, :k].sort(dim=1).values)
    assert bool((sel[:, k:] == -7).all())
