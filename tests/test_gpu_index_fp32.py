"""Lists and codes of the index build and update are those of a plain fp32 search over all centres
(-m gpu), lower index on ties, whatever arithmetic the search itself runs in: with centres that are
close to one another, equal, far outside the unit ball, not numbers, or residuals near zero.

Exact: the fp32 chains (one per sum, over the dims in order, fused multiply-adds) are formed here step
by step in float64 and rounded after each."""
import pytest
import torch

from paper_2609_33746_b200 import pqhsa

pytestmark = pytest.mark.gpu


def fma(a, b, c):
    return (a.double() * b.double() + c.double()).float()


def chain(terms, shape):
    acc = torch.zeros(shape, device="cuda")
    for a, b in terms:
        acc = fma(a, b, acc)
    return acc


def first_argmin(d):                                     # not a number: never the nearest; none: 0
    d = torch.where(d.isnan(), float("inf"), d)
    low = d.min(dim=-1, keepdim=True).values
    return torch.where(d == low, 1, 0).argmax(dim=-1) * (low[..., 0] < float("inf"))


def nearest_lists(u, c, with_x2):
    n, L = u.shape[0], c.shape[0]
    dot = chain(((u[:, None, k], c[None, :, k]) for k in range(128)), (n, L))
    cc = chain(((c[:, k], c[:, k]) for k in range(128)), (L,))
    if not with_x2:
        return first_argmin(fma(torch.full_like(dot, -2.0), dot, cc.expand(n, L)))
    xx = chain(((u[:, k], u[:, k]) for k in range(128)), (n,))
    return first_argmin(fma(torch.full_like(dot, -2.0), dot, xx[:, None].expand(n, L)) + cc)


def nearest_codes(e, books, expanded):
    n, (m, z, ds) = e.shape[0], books.shape
    out = []
    for j in range(m):
        x, p = e[:, None, j * ds:(j + 1) * ds], books[None, j]
        if expanded:
            dot = chain(((x[..., t], p[..., t]) for t in range(ds)), (n, z))
            xx = chain(((x[..., t], x[..., t]) for t in range(ds)), (n, 1))
            pp = chain(((p[..., t], p[..., t]) for t in range(ds)), (1, z))
            d = fma(torch.full_like(dot, -2.0), dot, xx.expand(n, z)) + pp
        else:
            d = chain(((x[..., t] - p[..., t], x[..., t] - p[..., t]) for t in range(ds)), (n, z))
        out.append(first_argmin(d))
    return torch.stack(out, dim=1)


def keys_of(kind, n, g):
    k = torch.randn((n, 128), generator=g, device="cuda")
    if kind == "mean":                                   # a large common part: centroids close to one another
        k = 5 * torch.randn((1, 128), generator=g, device="cuda") + k
    elif kind == "tight":                                # residuals near zero
        k = torch.randn((50, 128), generator=g, device="cuda")[torch.randint(0, 50, (n,), generator=g, device="cuda")]
        k = k + 2e-3 * torch.randn((n, 128), generator=g, device="cuda")
    elif kind == "repeats":                              # equal keys: equal seeds, equal centroids
        k = k[torch.randint(0, 97, (n,), generator=g, device="cuda")]
    elif kind == "zeros":
        k[::3] = 0
    elif kind == "nan":                                  # (list 0, and its centroid is no direction any more)
        k[5::501] = float("nan")
        k[11::777, 3] = float("inf")
    return k.bfloat16()


class Index:
    def __init__(self, kind, n, n_list, m, ncode, seed, heads=1):
        g = torch.Generator(device="cuda").manual_seed(seed)
        self.n, self.n_list, self.m, self.ncode, self.heads = n, n_list, m, ncode, heads
        self.n_max = nm = (n + 15) // 16 * 16
        self.k = torch.zeros((nm, heads, 128), dtype=torch.bfloat16, device="cuda")
        for h in range(heads):
            self.k[:n, h] = keys_of(kind, n, g)
        self.v = torch.randn((nm, heads, 128), generator=g, device="cuda").bfloat16()
        self.table = torch.arange(nm // 16, dtype=torch.int32, device="cuda").view(1, -1)
        self.params = pqhsa.make_params(batch=1, n_q_heads=heads, n_kv_heads=heads, n_list=n_list, pq_m=m, pq_ncode=ncode,
                                        max_seq_len=nm, max_pages_per_seq=nm // 16, budget_ppm=10000, dtype="bf16")
        self.kv = pqhsa.make_paged_kv(self.k, self.v, 16 * heads * 128, heads * 128, 128, self.table)
        self.centroids = torch.zeros((heads, n_list, 128), device="cuda")
        self.books = torch.zeros((heads, m, ncode, 128 // m), device="cuda")
        self.seq = torch.tensor([n], dtype=torch.int32, device="cuda")
        self.seeds = [torch.randint(0, n, (heads, c), generator=g, device="cuda").int() for c in (n_list, ncode)]
        self.clear()

    def clear(self):
        z = lambda *s, dtype=torch.float32: torch.zeros((self.heads, *s), dtype=dtype, device="cuda")
        self.codes = z(self.n_max, self.m if self.ncode == 256 else self.m // 2, dtype=torch.uint8)
        self.ids, self.norms = z(self.n_max, dtype=torch.int16), z(self.n_max)
        self.vmeans, self.counts = z(self.n_list, 128), z(self.n_list, dtype=torch.int32)

    def build(self, coarse_iters, pq_iters):
        ws = torch.empty(pqhsa.index_build_workspace_bytes(self.params), dtype=torch.uint8, device="cuda")
        pqhsa.index_build(self.params, self.kv, self.seq, *self.seeds, coarse_iters, pq_iters, self.centroids,
                          self.books, self.codes, self.ids, self.norms, self.vmeans, self.counts, ws)

    def update(self, n_new):
        self.clear()
        rw = pqhsa.make_index_rw(self.centroids, self.books, self.codes, self.ids, self.norms, self.vmeans, self.counts)
        first = torch.zeros(1, dtype=torch.int32, device="cuda")
        pqhsa.index_update(self.params, rw, self.kv, first, torch.tensor([n_new], dtype=torch.int32, device="cuda"), n_new)
        torch.cuda.synchronize()

    def check(self, n, build):
        for h in {0, self.heads - 1}:
            r = self.norms[h, :n]
            u = self.k[:n, h].float() * torch.where(r > 0, 1.0 / r, 0.0)[:, None]
            a = self.ids[h, :n].long() & 0xffff
            assert torch.equal(a, nearest_lists(u, self.centroids[h], build)), "lists"
            z = self.codes[h, :n].long()
            if self.ncode == 16:
                z = torch.stack((z & 15, z >> 4), dim=2).view(n, self.m)
            assert torch.equal(z, nearest_codes(u - self.centroids[h, a], self.books[h], build)), "codes"


# update: of one unit the small fp32 kernel up to some 460 lists; of twelve the tensor cores
HEADS = [1, 12]
SHAPES = [(193, 32, 256), (600, 16, 256), (40, 8, 16), (129, 64, 256), (1000, 8, 256), (65, 16, 16)]


@pytest.mark.parametrize("heads", HEADS)
@pytest.mark.parametrize("n_list,m,ncode", SHAPES)
@pytest.mark.parametrize("kind", ["normal", "mean", "tight", "repeats", "zeros", "nan"])
def test_lists_and_codes_are_those_of_an_fp32_search(kind, n_list, m, ncode, heads):
    ix = Index(kind, 3001, n_list, m, ncode, n_list + m, heads)
    ix.build(1, 1)
    ix.check(ix.n, build=True)
    ix.update(700)
    ix.check(700, build=False)


@pytest.mark.parametrize("heads", HEADS)
@pytest.mark.parametrize("n_list,m,ncode", SHAPES[:3])
@pytest.mark.parametrize("centroids,books", [(1e-3, 1.0), (20.0, 1.0), (300.0, 1.0), (1.0, 1e-3), (1.0, 20.0), (1.0, 3000.0)])
def test_update_takes_any_centroids_and_codebooks(centroids, books, n_list, m, ncode, heads):
    ix = Index("normal", 1500, n_list, m, ncode, 3, heads)
    ix.build(1, 1)
    ix.centroids *= centroids
    ix.books *= books
    ix.update(600)
    ix.check(600, build=False)
    ix.centroids[:, 5, 7], ix.centroids[:, 17, 3] = float("nan"), float("inf")
    ix.books[:, :, 3, 0], ix.books[:, :, 9, 1] = float("nan"), -float("inf")
    ix.update(600)
    ix.check(600, build=False)


@pytest.mark.parametrize("heads,n_new", [(1, 1), (1, 7), (1, 8), (1, 9), (3, 17), (40, 4), (40, 129)])
def test_update_of_a_few_tokens(heads, n_new):
    ix = Index("normal", 400, 100, 32, 256, n_new, heads)
    ix.build(1, 1)
    ix.update(n_new)
    ix.check(n_new, build=False)
    assert not ix.codes[:, n_new:].any() and not ix.norms[:, n_new:].any()
    assert ix.counts.sum(dim=1).tolist() == [n_new] * heads


@pytest.mark.parametrize("heads", [1, 40])
def test_the_lowest_of_equal_centroids(heads):
    ix = Index("normal", 512, 193, 32, 256, 9, heads)
    ix.seeds[0][ix.seeds[0] < 4] = 100
    for token, columns in ((0, (3, 7, 9)), (1, (40, 75, 130)), (2, (20, 21, 22, 150)), (3, (190, 191, 192))):
        ix.seeds[0][:, list(columns)] = token            # in one block of columns and across blocks
    ix.build(0, 0)
    assert ix.ids[:, :4].tolist() == [[3, 40, 20, 190]] * heads
    ix.update(400)
    assert ix.ids[:, :4].tolist() == [[3, 40, 20, 190]] * heads


@pytest.mark.parametrize("n,n_list", [(500, 40), (1025, 256), (40, 64)])
def test_a_cache_without_a_number(n, n_list):
    """Every key is NaN: no distance is a number, and there are empty lists to re-seed."""
    ix = Index("normal", n, n_list, 16, 256, seed=4)
    ix.k[:n] = float("nan")
    ix.build(2, 1)
    ids, codes, norms, counts = (t[0, :n] for t in (ix.ids, ix.codes, ix.norms, ix.counts))
    assert bool((ids == 0).all()) and bool((codes == 0).all()) and bool(norms.isnan().all())
    assert counts[0] == n and counts.sum() == n


@pytest.mark.parametrize("n_nan", [2, 3])
@pytest.mark.parametrize("m,ncode", [(32, 256), (64, 256), (16, 256), (8, 16)])
def test_codewords_are_the_fixed_point_means_of_their_members(m, ncode, n_nan):
    """One training pass from known codewords.  A component that is not a number enters the 64-bit sums
    as the conversion to integers has it (-2^63), and no other codeword changes."""
    n, n_list, ds = 1700, 40, 128 // m
    ix = Index("normal", n, n_list, m, ncode, seed=m)
    ix.k[[1600, 77, 1699][:n_nan]] = float("nan")
    ix.seeds = [torch.arange(100, 100 + n_list, device="cuda").int(), torch.arange(200, 200 + ncode, device="cuda").int()]
    ix.build(0, 0)
    r = ix.norms[0, :n]
    u = ix.k[:n, 0].float() * torch.where(r > 0, 1.0 / r, 0.0)[:, None]
    e = u - ix.centroids[0, ix.ids[0, :n].long() & 0xffff]
    z = ix.codes[0, :n].long()
    if ncode == 16:
        z = torch.stack((z & 15, z >> 4), dim=2).view(n, m)
    before = ix.books[0].clone()
    ix.build(0, 1)
    fixed = torch.round((e * 2.0 ** 40).double()).nan_to_num(0).long()
    fixed = torch.where(e.isnan(), torch.iinfo(torch.int64).min, fixed).view(n, m, ds)
    for j in range(m):
        sums = torch.zeros((ncode, ds), dtype=torch.int64, device="cuda").index_add_(0, z[:, j], fixed[:, j])
        count = torch.bincount(z[:, j], minlength=ncode)
        mean = (sums.double() / 2.0 ** 40 / count.clamp(min=1)[:, None]).float()
        assert torch.equal(ix.books[0, j], torch.where(count[:, None] > 0, mean, before[j])), j
