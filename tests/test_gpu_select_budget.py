"""Top-k at the lines between its two paths, against a stable sort (-m gpu): budgets at which a CTA's list
overflows, the largest budget of the cluster kernel and the next one, the most clusters of eight, at once and in turns, and
a last wave that is nearly empty or not."""
import pytest

from test_gpu_select_cluster import PATTERNS, test_cluster_select_is_the_stable_top_k as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pattern", PATTERNS)
@pytest.mark.parametrize("heads,n,ppm", [
    (32, 32001, 400000), (32, 32001, 400001), (512, 8191, 390000), (64, 16400, 125000), (64, 16400, 130000),
    (14, 200003, 10000), (15, 200003, 10000), (19, 200003, 10000), (160, 32001, 10000), (256, 32001, 10000),
    (74, 60003, 10000), (75, 60003, 10000)])
def test_select_at_the_lines_of_its_dispatch(heads, n, ppm, pattern):
    check(heads, n, ppm, pattern)
