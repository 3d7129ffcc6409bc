"""Which fused calls keep the tiles' maxima in their workspace (behind the last buffer), by the most that a row may
select: where the exact set is rounded up to a large multiple that is more than the budget."""
import pytest

from paper_2609_33746_b200 import pqhsa


@pytest.mark.parametrize("n,batch,multiple,used", [(131072, 8, 0, True), (131072, 8, 16, True), (131072, 8, 1024, True),
                                                   (131072, 8, 4096, False), (32768, 8, 0, True), (32768, 8, 1024, False),
                                                   (131072, 1, 0, False)])
def test_rounding_of_the_exact_set_counts(n, batch, multiple, used):
    p = pqhsa.make_params(batch=batch, n_q_heads=32, n_kv_heads=8, n_list=512, pq_m=32, max_seq_len=n,
                          max_pages_per_seq=n // 16, budget_ppm=10000, dtype="bf16", exact_set_multiple=multiple)
    last = pqhsa.decode_buffer_offset(p, pqhsa.BUF_OUT_F32) + 4 * pqhsa.buffer_elems(p, pqhsa.BUF_OUT_F32)
    maxima = 4 * batch * 32 * (n // 32)
    assert (pqhsa.workspace_bytes(p) - last >= maxima) == used
