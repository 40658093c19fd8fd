"""The search for each member's hyperedge (a warp finds its first member's,
its lanes look a few offsets on) where it can go wrong: hyperedge counts at
the steps of the search (32, 1,024), one hyperedge holding several warps'
members, and runs of empty hyperedges longer than the lanes look ahead."""
import numpy as np
import pytest

from paper_2311_10337_gb300 import synth
from test_gpu_hyper import compare_hyper

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [1, 2, 31, 32, 33, 34, 1023, 1024, 1025, 2500])
@pytest.mark.parametrize("shape", ["dense", "gaps", "ends", "one"])
def test_offsets(E, shape):
    rng = np.random.default_rng(E)
    V = 200
    size = rng.integers(0, 4, E)
    if shape == "gaps":      # members in a few places, 40 and more empty hyperedges between
        size[:] = 0
        size[rng.integers(0, E)] = 3
        size[::77] = 2
    elif shape == "ends":    # only the first and the last hyperedge have members
        size[:] = 0
        size[0] = size[-1] = 40
    elif shape == "one":     # one hyperedge over five warps' members
        size[E // 2] = 150
    off = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    vert = np.concatenate([rng.permutation(V)[:n] for n in size] + [np.zeros(0, np.int64)]).astype(np.int32)
    t = rng.integers(0, 50, E).astype(np.int64)
    compare_hyper(synth.HyperWorkload("offsets", t, off, vert, None, None, V, 2, ""))
