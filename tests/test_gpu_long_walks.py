"""Inputs on which one address or one chain holds everything up: pointer
walks on the longest chains, whose walkers meet only pointers as short as their
own, and edges of one weight at one vertex, whose bids meet at one slot.
Each test compares a stage with another of the same call or of a call on as
many edges without long chains, on the device's own clock."""
import numpy as np
import pytest

from gpu_helpers import compare_all, ctx

pytestmark = pytest.mark.gpu


def _stages(call, runs=3):
    """Smallest device time of every stage over some calls, after one more."""
    call()
    best = {}
    for _ in range(runs):
        call()
        for name, ms in ctx().stage_timing():
            best[name] = min(ms, best.get(name, ms))
    return best


def test_one_run_of_equal_weights():
    """One threshold: almost every merge has the same weight, so one run of
    tens of millions of merges collapses into its last. The collapse takes a
    few passes over the merges, as building the incidence lists does."""
    import torch
    E, V = 60_000_000, 3_000_000
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    src = torch.randint(0, V, (E,), generator=g, device="cuda")
    dst = (src + torch.randint(1, V, (E,), generator=g, device="cuda")) % V
    t = torch.randint(0, 30 * 86400, (E,), generator=g, device="cuda")
    src, dst = src.int(), dst.int()
    s = _stages(lambda: ctx().run_levels(src, dst, t, V, [1 << 20], 5))
    ctx().ws = None  # tens of GB: not kept for the tests after
    assert s["D2 condense and labels"] < 5 * s["A incidence lists"]


def _path(n, rising):
    """A relay of n + 1 edges whose gaps rise or fall, so that in the first
    round every edge points to its neighbour on one side: one chain. Edge ids
    in random order."""
    gaps = 2 + np.arange(n, dtype=np.int64)
    t = np.concatenate([[0], np.cumsum(gaps if rising else gaps[::-1])])
    p = np.random.default_rng(n).permutation(n + 1)
    a = np.arange(n + 1, dtype=np.int32)
    return a[p], a[p] + 1, t[p], n + 2


def _path_stages(n, rising):
    import torch
    src, dst, t, V = _path(n, rising)
    e = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (src, dst, t)]
    return _stages(lambda: ctx().run(*e, V, 2, 2))


@pytest.mark.parametrize("n", [400_000, 2_000_000])  # middle rounds; a large round
def test_dendrogram_of_a_path(n):
    fall, rise = _path_stages(n, False), _path_stages(n, True)
    assert fall["D1 dendrogram"] < 8 * rise["D1 dendrogram"]


@pytest.mark.parametrize("n", [400_000, 2_000_000])
def test_forest_of_a_path(n):
    fall, rise = _path_stages(n, False), _path_stages(n, True)
    assert fall["C spanning forest"] < 8 * rise["C spanning forest"]


@pytest.mark.parametrize("n", [1_000_000, 5_000_000])  # cooperative rounds alone; a large round first
def test_long_paths_merge_from_the_last(n):
    import torch
    src, dst, t, V = _path(n, False)
    out = ctx().run(*(torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (src, dst, t)), V, 2, 2)
    assert np.array_equal(out.numpy("mst_w"), 2 + np.arange(n))
    assert np.array_equal(out.numpy("link_size"), 2 + np.arange(n))
    assert out.n_mst == n


def _chain_of_chains(m):
    """m relay chains of falling gaps, joined end to end by longer ones that
    fall too: after the first round a long chain of components is left."""
    gaps = np.concatenate([np.append(2 + np.arange(8)[::-1], 1000 + m - i) for i in range(m)])[:-1]
    t = np.concatenate([[0], np.cumsum(gaps)])
    p = np.random.default_rng(m).permutation(len(t))
    a = np.arange(len(t), dtype=np.int32)
    return a[p], a[p] + 1, t[p], len(t) + 1


@pytest.mark.parametrize("shift", [0, 27])  # with and without labels in the bids
def test_walks_cut_in_a_later_round(shift):
    src, dst, t, V = _chain_of_chains(240_000)
    t = t << shift
    assert (int(t.max()).bit_length() + 3 * (len(t) - 1).bit_length() > 127) == (shift > 0)
    q = np.arange(0, len(t), 50_000).astype(np.int32)
    compare_all(src, dst, t, V, 2, 2, knn_query=q)


@pytest.mark.parametrize("n", [100_000, 600_000])
def test_paths_equal_the_oracle(n):
    src, dst, t, V = _path(n, False)
    q = np.arange(0, n, n // 100).astype(np.int32)
    compare_all(src, dst, t, V, 2, 2, knn_query=q)


def test_bids_of_one_weight_at_one_vertex():
    """A vertex that millions of edges reach at one time before it sends: all
    of them bid the same weight there. The forest of as many edges at distinct
    times has the same edges and more digits to sort."""
    import torch
    m = 3_000_000
    src = torch.arange(1, m + 2, dtype=torch.int32, device="cuda")
    src[m] = 0
    dst = torch.zeros(m + 1, dtype=torch.int32, device="cuda")
    dst[m] = m + 1
    one = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    many = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    many[:m] = torch.randperm(m, generator=g, device="cuda")
    one[m] = many[m] = m + 5
    a, b = (_stages(lambda: ctx().run(src, dst, t, m + 2, 4, 5), 6)["C spanning forest"] for t in (one, many))
    assert a < b
