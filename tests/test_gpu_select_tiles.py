"""Top-k from the tiles' maxima (fused call, many long rows), against a stable sort of the call's scores (-m gpu).

All tokens share one list and one code, so a score is the token's norm times a factor of the query head: the
norms put any pattern into the score rows.  Exact: the positions of the k largest scores, equal scores by
position; rows in random order, that pile up on few values, sorted (all large scores in few tiles: the list
overflows), stretched by outliers, with scores that are not numbers; at the edges of tiles and groups."""
import pytest
import torch

from paper_2609_33746_b200 import pqhsa
from paper_2609_33746_b200.runner import DecodeOp
from paper_2609_33746_b200.workload import DecodeConfig, generate
from paper_2609_33746_b200.index_builder import build_index

pytestmark = pytest.mark.gpu

PATTERNS = ("normal", "equal", "two_values", "sorted", "runs", "outliers", "narrow", "infinite", "nan", "negative", "tiny")


def norms_of(pattern, n, g):
    x = torch.randn(n, generator=g, device="cuda") * 7 + 20
    if pattern == "equal":
        x.fill_(1.25)
    elif pattern == "two_values":
        x = torch.where(x > 35, 3.0, -0.0)
        x[::3] *= -1.0                                   # -0 and +0 compare equal
    elif pattern == "sorted":
        x = x.sort().values
    elif pattern == "runs":                              # 40 neighbours at a time
        x[:n // 40 * 40] = x[:n // 40].repeat_interleave(40) + torch.rand(n // 40 * 40, generator=g, device="cuda")
    elif pattern == "outliers":
        x[n // 2], x[n // 3], x[0] = 1e30, -1e30, 65000.0
    elif pattern == "narrow":                            # neighbouring floats
        x = 50.0 + torch.randint(0, 3000, (n,), generator=g, device="cuda") * 2.0 ** -18
    elif pattern == "infinite":
        x[5::1000] = float("inf")
        x[7::3] = -float("inf")
    elif pattern == "nan":
        x[11::50] = float("nan")
        x[64:128] = float("nan")
    elif pattern == "negative":
        x -= 100.0
    elif pattern == "tiny":                              # 512 over the range of the scores is no number
        x = torch.rand(n, generator=g, device="cuda") * 6e-38
    return x


@pytest.mark.parametrize("pattern", PATTERNS)
@pytest.mark.parametrize("lens,ppm,sinks", [((16385, 20001), 10000, 0), ((40000, 33), 23000, 4), ((131071, 70016), 5000, 0),
                                            ((17000, 31999), 0, 0)])
@pytest.mark.parametrize("codes,tables", [(256, False), (16, False), (256, "rescore")])
def test_tiles_select_is_the_stable_top_k(lens, ppm, sinks, codes, tables, pattern):
    if tables and pattern != "normal":
        pytest.skip("the re-score decides from the tables: see the fp16 table tests")
    m = 8 if codes == 16 else 32
    cfg = DecodeConfig("tiles", len(lens), 64, 8, lens, "bf16", 16, m, ppm, pq_ncode=codes, n_sink=sinks, kmeans_iters=0, seed=5)
    inp = generate(cfg, device="cuda")
    idx = build_index(inp)
    if not tables:
        g = torch.Generator(device="cuda").manual_seed(len(pattern) + sum(lens))
        idx.codes.zero_()
        idx.list_ids.zero_()
        for b, n in enumerate(lens):
            idx.key_norms[b, :, :n] = norms_of(pattern, n, g)
    op = DecodeOp(inp, idx, fp16_tables=tables)
    op.decode()
    assert op.device_status() == pqhsa.OK
    rows, n_max = cfg.batch * cfg.n_q_heads, op.params.max_seq_len
    scores = op.decode_buffer(pqhsa.BUF_SCORES).view(rows, n_max)
    sel = op.decode_buffer(pqhsa.BUF_SEL_IDX, torch.int32).view(rows, op.params.k_max)
    count = op.decode_buffer(pqhsa.BUF_SEL_COUNT, torch.int32).tolist()
    kth = op.decode_buffer(pqhsa.BUF_KTH)
    for row in range(rows):
        n = lens[row // cfg.n_q_heads]
        k = ((n - min(n, sinks)) * ppm + 999999) // 1000000
        assert count[row] == k
        if k == 0 or tables:
            continue
        s = scores[row, :n] + 0.0
        # numbers first, then -inf, then what is no number; a stable sort keeps the lower position first
        order = torch.argsort(torch.where(s.isnan(), -float("inf"), s), descending=True, stable=True)
        order = torch.cat([order[~s[order].isnan()], order[s[order].isnan()]])
        assert torch.equal(sel[row, :k].long().sort().values, order[:k].sort().values), (row, pattern)
        want = s[order[k - 1]]
        assert kth[row] == want or bool(want.isnan())
