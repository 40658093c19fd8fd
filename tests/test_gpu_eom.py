"""Excess of mass on cluster trees of every shape the pass treats apart: deep
spines (far above the height its first walk covers and above the 64 steps of a
shortcut walk), several spines under one another, and bushy trees."""
import numpy as np
import pytest

from gpu_helpers import compare_all

pytestmark = pytest.mark.gpu


def _relay(gaps, burst=5):
    """A relay chain of len(gaps) + 1 bursts of `burst` edges a second apart,
    gaps[b] seconds after burst b."""
    d = []
    for g in list(gaps) + [1]:
        d += [1] * (burst - 1) + [int(g)]
    t = np.concatenate([[0], np.cumsum(d)[:-1]]).astype(np.int64)
    m = len(t)
    return np.arange(m, dtype=np.int32), np.arange(1, m + 1, dtype=np.int32), t, m + 1


@pytest.mark.parametrize("name", ["short", "spine", "deep", "down_up", "nested", "bushy"])
def test_cluster_tree_shapes(name):
    rng = np.random.default_rng(7)
    if name == "short":
        gaps = 2 + np.arange(23)  # heights around the first walk's limit
    elif name == "spine":
        gaps = 2 + np.arange(700)
    elif name == "deep":
        gaps = 2 + np.arange(5000)
    elif name == "down_up":
        gaps = np.concatenate([2 + np.arange(900)[::-1], 5000 + np.arange(900)])
    elif name == "nested":  # spines that join as subtrees of longer spines
        gaps = np.concatenate([np.append(2 + np.arange(40 + 7 * i), 10_000 + i) for i in range(30)])
    else:
        gaps = rng.permutation(4000) + 2
    src, dst, t, V = _relay(gaps)
    g, _ = compare_all(src, dst, t, V, 2, 5)
    if name in ("spine", "deep"):
        assert len(g["cl_id"]) > 2 * len(gaps)  # every merge of two bursts splits
