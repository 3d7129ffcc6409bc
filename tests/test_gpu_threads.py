"""Host threads that call the library at the same time, each on its own stream and workspace and with a
shape of its own (-m gpu): every call succeeds and gives what it gives alone."""
import threading

import pytest
import torch

from paper_2609_33746_b200 import pqhsa
from paper_2609_33746_b200.runner import DecodeOp
from paper_2609_33746_b200.workload import DecodeConfig

from helpers import make_case

pytestmark = pytest.mark.gpu


def together(works):
    errors = []

    def run(work):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                work()
            stream.synchronize()
        except Exception as e:                           # noqa: BLE001 (a thread's error belongs to the test)
            errors.append(repr(e))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=run, args=(w,)) for w in works]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[:2]


def test_top_k_of_different_row_lengths():
    def work(rows, n, calls):
        p = pqhsa.make_params(batch=1, n_q_heads=rows, n_kv_heads=rows, n_list=16, pq_m=8, max_seq_len=n,
                              max_pages_per_seq=n // 16, budget_ppm=10000, dtype="bf16")
        g = torch.Generator(device="cuda").manual_seed(n)
        scores = torch.randn((rows, n), generator=g, device="cuda")
        seq = torch.tensor([n], dtype=torch.int32, device="cuda")
        sel = torch.zeros((rows, p.k_max), dtype=torch.int32, device="cuda")
        cnt, kth = torch.zeros(rows, dtype=torch.int32, device="cuda"), torch.zeros(rows, device="cuda")
        ws = torch.zeros(pqhsa.workspace_bytes(p), dtype=torch.uint8, device="cuda")
        want = torch.topk(scores, p.k_max, dim=1).values[:, -1]
        torch.cuda.synchronize()

        def run():
            for _ in range(calls):
                pqhsa.select(p, scores, seq, sel, cnt, kth, ws)
            assert torch.equal(kth, want)
        return run
    together([work(1, 4096, 3000), work(8, 49152, 1500), work(1, 4096, 3000), work(2, 49152, 1500)])


@pytest.mark.parametrize("kw", [dict(pq_m=32), dict(pq_m=8, pq_ncode=16)])
def test_decodes_of_different_index_sizes(kw):
    def work(n_list, seed):
        cfg = DecodeConfig(name="t", batch=1, n_q_heads=8, n_kv_heads=2, seq_lens=(3000,), dtype="bf16", n_list=n_list,
                           budget_ppm=20000, seed=seed, kmeans_iters=1, **kw)
        inp, idx = make_case(cfg, device="cuda")
        op = DecodeOp(inp, idx)
        want = op.decode().clone()
        torch.cuda.synchronize()

        def run():
            for _ in range(1500):
                op.decode()
            assert float((op.out.float() - want.float()).abs().max()) <= 2.0 ** -6      # (order of the atomics)
            assert op.device_status() == pqhsa.OK
        return run
    together([work(16, 1), work(1024, 2), work(64, 3), work(512, 4)])
