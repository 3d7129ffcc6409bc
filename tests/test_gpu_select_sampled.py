"""Top-k with the bracket from a sample (many or long rows), against a stable sort (-m gpu).

Exact, as for the cluster kernel: at the edges of the filter's chunks, with more candidates than
the finishing block stages in shared memory (a bracket of 512K scores; a large budget), with more
hits per warp than are written out together, and for rows whose order or values defeat the sample."""
import pytest

from test_gpu_select_cluster import PATTERNS, test_cluster_select_is_the_stable_top_k as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pattern", PATTERNS)
@pytest.mark.parametrize("heads,n,ppm", [
    (32, 524288, 10000), (64, 300003, 60000), (256, 65536, 10000), (512, 32769, 100000), (600, 24577, 300000)])
def test_sampled_select_is_the_stable_top_k(heads, n, ppm, pattern):
    check(heads, n, ppm, pattern)
