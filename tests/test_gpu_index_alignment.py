"""Index build and update with arrays that start at any element (-m gpu): a cache view that begins in the
middle of a buffer, codes at an odd byte, codebooks at any float.  Same outputs as on aligned arrays."""
import pytest
import torch

from paper_2609_33746_b200 import pqhsa

pytestmark = pytest.mark.gpu


def run(shift, m, ncode, dtype):
    n, n_list, heads, page = 1100, 65, 2, 16
    pages = (n + page - 1) // page
    n_max, tdt = pages * page, {"bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    g = torch.Generator(device="cuda").manual_seed(m)

    def at(shape, dtype, off, fill=None):                # a contiguous tensor `off` elements into a buffer
        size = 1
        for s in shape:
            size *= s
        buf = torch.zeros(size + 64, dtype=dtype, device="cuda")
        assert buf.data_ptr() % 64 == 0
        t = buf[off:off + size].view(shape)
        if fill is not None:
            t.copy_(fill)
        return t

    k, v = (at((pages, page, heads, 128), tdt, shift, torch.randn((pages, page, heads, 128), generator=g, device="cuda").to(tdt))
            for _ in range(2))
    table = torch.randperm(pages, generator=g, device="cuda").int().view(1, pages)
    p = pqhsa.make_params(batch=1, n_q_heads=heads, n_kv_heads=heads, n_list=n_list, pq_m=m, pq_ncode=ncode, max_seq_len=n_max,
                          max_pages_per_seq=pages, budget_ppm=10000, dtype=dtype)
    kv = pqhsa.make_paged_kv(k, v, page * heads * 128, heads * 128, 128, table)
    seeds = [torch.randint(0, n, (heads, c), generator=g, device="cuda").int() for c in (n_list, ncode)]
    seq = torch.tensor([n], dtype=torch.int32, device="cuda")
    code_bytes = m if ncode == 256 else m // 2
    cen = torch.zeros((heads, n_list, 128), device="cuda")
    books = at((heads, m, ncode, 128 // m), torch.float32, shift)
    codes = at((heads, n_max, code_bytes), torch.uint8, shift)
    ids, norms = at((heads, n_max), torch.int16, shift), at((heads, n_max), torch.float32, shift)
    means, counts = torch.zeros((heads, n_list, 128), device="cuda"), at((heads, n_list), torch.int32, shift)
    ws = torch.empty(pqhsa.index_build_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    pqhsa.index_build(p, kv, seq, *seeds, 1, 1, cen, books, codes, ids, norms, means, counts, ws)
    out = [t.clone() for t in (cen, books, codes, ids, norms, means, counts)]
    books = books.clone()                                # (the update has always wanted whole vectors here)
    rw = pqhsa.make_index_rw(cen, books, codes, ids, norms, means, counts)
    first = torch.full((1,), 900, dtype=torch.int32, device="cuda")
    pqhsa.index_update(p, rw, kv, first, torch.full((1,), 200, dtype=torch.int32, device="cuda"), 200)
    torch.cuda.synchronize()
    return out + [codes, ids, norms, means, counts]


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
@pytest.mark.parametrize("m,ncode", [(64, 256), (32, 256), (16, 256), (8, 256), (16, 16), (8, 16)])
def test_any_alignment(m, ncode, dtype):
    want = run(0, m, ncode, dtype)
    for shift in (1, 2, 3):
        for a, b in zip(run(shift, m, ncode, dtype), want):
            assert torch.equal(a, b), shift
