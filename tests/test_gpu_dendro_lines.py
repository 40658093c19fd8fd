"""The dendrogram at the lines between its forms, by the exact number of forest
edges: the one-CTA rounds take over at 4,096 live edges, the middle rounds at
524,288, and from 152 x 512 on the middle rounds have one CTA an SM. A relay of
n + 1 edges has a forest of n edges; random gaps give many rounds, so edges are
left to hand over at every line."""
import numpy as np
import pytest

from gpu_helpers import compare_all

pytestmark = pytest.mark.gpu

LINES = [4_096, 152 * 512, 524_288]


@pytest.mark.parametrize("n", [x + d for x in LINES for d in (-1, 0, 1)] + [1_048_577])
@pytest.mark.parametrize("ties", [False, True])
def test_forest_sizes_at_the_lines(n, ties):
    rng = np.random.default_rng(n)
    gaps = rng.integers(1, max(2, n // 50), n) if ties else 1 + rng.permutation(n)
    t = np.concatenate([[0], np.cumsum(gaps)])
    p = rng.permutation(n + 1)
    a = np.arange(n + 1, dtype=np.int32)
    q = np.arange(0, n, n // 50).astype(np.int32)
    g, _ = compare_all(a[p], a[p] + 1, t[p], n + 2, 4, 5, knn_query=q)
    assert len(g["mst_u"]) == n
