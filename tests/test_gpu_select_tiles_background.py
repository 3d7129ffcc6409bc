"""What the top-k from the tiles' maxima leaves besides the selection (-m gpu): the background's mass per list, out of
which the selected tokens are taken, and the output of the fused call beside that of the staged calls, which use
another top-k.  Rows whose scores overflow the CTA's list or tie at the threshold among them.

Tolerance of the mass, relative to the list's whole mass: exponentials to 2 ulp, and half an ulp for each of the fp32
additions in a chain; all tokens are in one list, so a chain is as long as what one SM scans.  Output: both calls
round the same sums, half an ulp of bf16 each, and the masses differ as above."""
import pytest
import torch

from paper_2609_33746_b200 import pqhsa
from paper_2609_33746_b200.runner import DecodeOp
from paper_2609_33746_b200.workload import DecodeConfig, generate
from paper_2609_33746_b200.index_builder import build_index

from test_gpu_select_tiles import norms_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pattern", ["normal", "equal", "two_values", "sorted", "runs", "narrow", "negative"])
@pytest.mark.parametrize("lens,ppm", [((16385, 20001), 10000), ((131071, 70016), 5000)])
@pytest.mark.parametrize("q_heads,kv_heads,codes", [(64, 8, 256), (64, 32, 16), (64, 64, 16)])
def test_selected_tokens_leave_the_background(q_heads, kv_heads, codes, lens, ppm, pattern):
    m = 8 if codes == 16 else 32
    cfg = DecodeConfig("tiles", len(lens), q_heads, kv_heads, lens, "bf16", 16, m, ppm, pq_ncode=codes, kmeans_iters=0, seed=9)
    inp = generate(cfg, device="cuda")
    inp.q.mul_(1.0 / 64)                                 # (exact logits of a few units: the background weighs as much)
    idx = build_index(inp)
    g = torch.Generator(device="cuda").manual_seed(len(pattern) + sum(lens))
    idx.codes.zero_()
    idx.list_ids.zero_()
    for b, n in enumerate(lens):
        idx.key_norms[b, :, :n] = norms_of(pattern, n, g)
    op = DecodeOp(inp, idx)
    op.alloc_stage_buffers()
    op.build_lut(), op.scan()
    top = max(float(op.scores.view(cfg.batch, q_heads, -1)[b, :, :n].abs().max()) for b, n in enumerate(lens))
    op.key_norms.mul_(4.0 / top)                         # scores of up to 4
    op.scan(), op.select(), op.hybrid_attend()
    staged = op.out.clone()
    op.decode()
    assert op.device_status() == pqhsa.OK
    rows, n_max = cfg.batch * cfg.n_q_heads, op.params.max_seq_len
    scores = op.decode_buffer(pqhsa.BUF_SCORES).view(rows, n_max)
    assert torch.equal(scores[0, :lens[0]], op.scores.view(rows, n_max)[0, :lens[0]])
    sel = op.decode_buffer(pqhsa.BUF_SEL_IDX, torch.int32).view(rows, op.params.k_max)
    count = op.decode_buffer(pqhsa.BUF_SEL_COUNT, torch.int32).tolist()
    assert count == op.sel_count.tolist()
    for row in range(rows):
        assert torch.equal(sel[row, :count[row]].sort().values, op.sel_idx.view(rows, -1)[row, :count[row]].sort().values), row
    mass = op.decode_buffer(pqhsa.BUF_BG_MASS).view(rows, cfg.n_list).double()
    top = op.decode_buffer(pqhsa.BUF_BG_MAX)
    passes = 2 if q_heads // kv_heads == 8 else 1        # (of up to four heads)
    chain = sum(lens) * kv_heads * passes / torch.cuda.get_device_properties(0).multi_processor_count
    for row in range(rows):
        n = lens[row // q_heads]
        e = (scores[row, :n].double() - scores[row, :n].double().max()).exp()
        chosen = sel[row, :count[row]].long()
        assert top[row] == scores[row, :n].max()
        left = e.sum() - e[chosen].sum()
        assert abs(mass[row, 0] - left) <= (chain * 2.0 ** -25 + 2.0 ** -20) * e.sum(), (row, float(mass[row, 0]), float(left))
        assert bool((mass[row, 1:] == 0).all())
    diff = (op.out.double() - staged.double()).abs()
    assert bool((diff <= 2.0 ** -7 * staged.double().abs() + 2.0 ** -11).all())


@pytest.mark.parametrize("pattern", ["equal", "sorted", "runs"])
def test_rows_that_crowd_are_not_walked(pattern):
    """Scores that tie or crowd in few tiles cost a few cuts of the list (1.4 times the call on scattered ones here, and
    4.9 times when such rows were walked by one CTA each); the bound is twice."""
    n, batch = 131072, 8
    cfg = DecodeConfig("tiles", batch, 32, 8, (n,) * batch, "bf16", 512, 32, 10000, kmeans_iters=0, seed=3)
    inp = generate(cfg, device="cuda")
    idx = build_index(inp)
    idx.codes.zero_()
    g = torch.Generator(device="cuda").manual_seed(1)

    def time_of(norms):
        idx.key_norms[:] = norms
        op = DecodeOp(inp, idx)
        best = float("inf")
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            op.decode()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        assert op.device_status() == pqhsa.OK
        return best

    idx.list_ids.copy_(torch.randint(0, 512, idx.list_ids.shape, generator=g, device="cuda"))
    scattered = time_of(norms_of("normal", n, g))
    crowded = time_of(0.0 if pattern == "equal" else norms_of(pattern, n, g))
    assert crowded <= 2 * scattered, (crowded, scattered)
