"""Dendrogram rounds over every form they take: the last rounds in one CTA (at
most 4,096 live edges), the middle rounds in one cooperative kernel, large
rounds (above 524,288) as separate launches, and in each both group sizes (up
to 128 accepted edges an edge scans its group, above they are sorted). The
exact lines between the forms are in test_gpu_dendro_lines.py."""
import numpy as np
import pytest

from gpu_helpers import compare_all

pytestmark = pytest.mark.gpu


def _stars(sizes, seed):
    """One vertex a star: its in-edges at distinct times, then one out-edge.
    The skeleton joins every in-edge to the out-edge, all weights distinct
    within the star, so a star is one group of one round."""
    rng = np.random.default_rng(seed)
    src, dst, t = [], [], []
    v = 0
    for n in sizes:
        hub = v
        src.append(np.append(np.arange(v + 1, v + 1 + n), hub))
        dst.append(np.append(np.full(n, hub), v + n + 1))
        gaps = rng.choice(4 * n + 8, n, replace=False) + 1
        start = int(rng.integers(0, 1 << 20))
        t.append(np.append(start + (4 * n + 10) - gaps, start + 4 * n + 10))
        v += n + 2
    src, dst, t = np.concatenate(src), np.concatenate(dst), np.concatenate(t)
    o = rng.permutation(len(src))
    return src[o].astype(np.int32), dst[o].astype(np.int32), t[o].astype(np.int64), v


@pytest.mark.parametrize("reps", [1, 30, 900])
def test_stars_around_the_group_limit(reps):
    sizes = np.tile([1, 2, 3, 31, 127, 128, 129, 130, 300], reps)
    if reps > 1:
        sizes = np.append(sizes, [4095, 4096, 5000, 9000])
    src, dst, t, V = _stars(sizes, reps)
    q = np.arange(0, len(src), max(1, len(src) // 500)).astype(np.int32)
    compare_all(src, dst, t, V, 4, 5, knn_query=q)


@pytest.mark.parametrize("E", [8_190, 8_200, 530_000, 1_100_000])
def test_random_graphs_around_the_round_forms(E):
    rng = np.random.default_rng(E)
    V = E // 4
    src = rng.integers(0, V, E).astype(np.int32)
    dst = ((src + 1 + rng.integers(0, V - 1, E)) % V).astype(np.int32)
    t = rng.integers(0, 1 << 22, E).astype(np.int64)
    q = np.arange(0, E, E // 300).astype(np.int32)
    compare_all(src, dst, t, V, 4, 5, knn_query=q)
