"""Nearest-centre searches of the index on the tensor cores, at the edges of their tiles (-m gpu).

Build and update assign tokens to 128 centroids and 128 tokens at a time and codewords per group
of 8.  Every list and every code has to be a nearest one: its distance, in float64 and to the
centres that the library itself returned, is within the rounding of an fp32 squared distance of
unit-scale vectors (2e-6: 128 products of 2^-24 relative error each, two sums) of the smallest."""
import numpy as np
import pytest
import torch

from paper_2609_33746_b200 import pqhsa
from paper_2609_33746_b200.index_builder import build_index_batched
from paper_2609_33746_b200.runner import DecodeOp
from paper_2609_33746_b200.workload import DecodeConfig, generate

from helpers import unpacked_codes

pytestmark = pytest.mark.gpu

DIST_TOL = 2e-6


def check_nearest(inp, idx, cfg):
    for b, n in enumerate(cfg.seq_lens):
        codes = unpacked_codes(idx.codes[b].cpu().numpy(), cfg).astype(np.int64)
        for g in range(cfg.n_kv_heads):
            k = inp.gather_kv(b, g)[0].double()
            u = k / k.norm(dim=1, keepdim=True)
            c = idx.centroids[b, g].double()
            a = idx.list_ids[b, g, :n].long() & 0xffff
            d = torch.cdist(u, c, compute_mode="donot_use_mm_for_euclid_dist") ** 2
            assert float((d.gather(1, a[:, None])[:, 0] - d.min(dim=1).values).max()) <= DIST_TOL, (b, g)
            e = (u - c[a]).view(n, cfg.pq_m, 1, -1)
            dq = ((e - idx.codebooks[b, g].double()[None]) ** 2).sum(-1)         # [n, m, codewords]
            z = torch.from_numpy(codes[g, :n]).cuda()
            assert float((dq.gather(2, z[..., None])[..., 0] - dq.min(dim=2).values).max()) <= DIST_TOL, (b, g)


@pytest.mark.parametrize("lens,n_list,m,ncode,dtype", [
    ((128, 127), 64, 32, 256, "bf16"), ((129, 255), 63, 16, 256, "fp16"), ((256, 257), 65, 64, 256, "bf16"),
    ((511, 400), 127, 8, 256, "bf16"), ((513, 512), 128, 8, 16, "bf16"), ((640, 385), 129, 16, 16, "fp16"),
    ((1000, 769), 193, 32, 256, "bf16"), ((900, 600), 257, 16, 16, "bf16")])
def test_lists_and_codes_are_nearest(lens, n_list, m, ncode, dtype):
    cfg = DecodeConfig(name="edges", batch=2, n_q_heads=4, n_kv_heads=2, seq_lens=lens, dtype=dtype, n_list=n_list,
                       pq_m=m, pq_ncode=ncode, budget_ppm=20000, seed=n_list + m, kmeans_iters=1, pq_iters=1)
    inp = generate(cfg, device="cuda")
    idx = build_index_batched(inp)
    check_nearest(inp, idx, cfg)
    # the same tokens again, all of them encoded by the update
    op = DecodeOp(inp, idx)
    counts = torch.zeros_like(idx.list_counts)
    for t in (idx.codes, idx.list_ids, idx.key_norms, idx.list_vmeans):
        t.zero_()
    rw = pqhsa.make_index_rw(idx.centroids, idx.codebooks, idx.codes, idx.list_ids, idx.key_norms, idx.list_vmeans,
                             counts)
    first = torch.zeros(2, dtype=torch.int32, device="cuda")
    pqhsa.index_update(op.params, rw, op.kv, first, torch.tensor(lens, dtype=torch.int32, device="cuda"), max(lens))
    torch.cuda.synchronize()
    check_nearest(inp, idx, cfg)
    assert counts.sum(dim=-1).tolist() == [[n, n] for n in lens]
