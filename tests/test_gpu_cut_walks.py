"""Every pointer walk cut after one or two steps, so that the passes behind the
walks do the work: the jumping rounds of the forest (and its restart), of the
dendrogram and of the condensing, and the repeated rounds of the selected
ancestors. Results do not depend on where a walk is cut."""
import numpy as np
import pytest

from gpu_helpers import compare_all, ctx
from paper_2311_10337_gb300 import synth
from test_gpu_dendro import _stars
from test_gpu_eom import _relay

pytestmark = pytest.mark.gpu


@pytest.fixture(params=[1, 2, 5])
def cut(request):
    ctx().set_limits(walk_steps=request.param)
    yield
    ctx().set_limits()


def _random(E, V, span, seed):
    rng = np.random.default_rng(seed)
    src = rng.integers(0, V, E).astype(np.int32)
    dst = ((src + 1 + rng.integers(0, V - 1, E)) % V).astype(np.int32)
    return src, dst, rng.integers(0, span, E).astype(np.int64), V


def _compare(src, dst, t, V, k=4, M=5):
    n = len(src)
    compare_all(src, dst, t, V, k, M, knn_query=np.arange(0, n, max(1, n // 200)).astype(np.int32))


@pytest.mark.parametrize("name", ["rising", "falling", "down_up", "nested", "equal"])
def test_relays(cut, name):
    gaps = {"rising": 2 + np.arange(3000), "falling": 2 + np.arange(3000)[::-1],
            "down_up": np.concatenate([2 + np.arange(900)[::-1], 5000 + np.arange(900)]),
            "nested": np.concatenate([np.append(2 + np.arange(40 + 7 * i), 10_000 + i) for i in range(30)]),
            "equal": np.full(3000, 7)}[name]
    for burst in (1, 5):
        _compare(*_relay(gaps, burst), 2, 5 if burst > 1 else 2)


@pytest.mark.parametrize("E,V,span,shift", [(3_000, 300, 50, 0), (60_000, 6_000, 1, 0), (60_000, 6_000, 1 << 20, 0),
                                            (700_000, 80_000, 4_000, 0), (2_200_000, 300_000, 1 << 20, 42)])
def test_random_graphs(cut, E, V, span, shift):
    src, dst, t, V = _random(E, V, span, E)
    _compare(src, dst, t << shift, V)


def test_large_forest_rounds(cut):
    src, dst, t, V = _random(4_400_000, 500_000, 100_000, 9)  # above 4M links
    _compare(src, dst, t, V)


def test_stars(cut):
    _compare(*_stars([1, 2, 3, 127, 128, 129, 130, 300, 4095, 9000], 1))


def test_batch_and_levels(cut):
    import torch
    from oracle import oracle as O
    rng = np.random.default_rng(3)
    graphs = [synth.random_small(E, max(4, E // 8), max(5, E // 10), 50 + E) for E in (40, 900, 7_000, 15_000)]
    off = np.concatenate([[0], np.cumsum([len(g.src) for g in graphs])]).astype(np.int64)
    e = [torch.from_numpy(np.concatenate([getattr(g, f) for g in graphs])).cuda() for f in ("src", "dst", "t")]
    nv = np.array([g.n_vertices for g in graphs], np.int32)
    k, M = np.full(4, 4, np.int32), np.full(4, 5, np.int32)
    labels = ctx().run_batch(*e, off, nv, k, M).numpy("labels").copy()
    for i, g in enumerate(graphs):
        r = O.run(g.src, g.dst, g.t, g.n_vertices, 4, 5)
        assert np.array_equal(labels[off[i]:off[i + 1]], r["condensed"]["labels"])
    src, dst, t, V = _random(50_000, 5_000, 1 << 18, 4)
    e = [torch.from_numpy(x).cuda() for x in (src, dst, t)]
    omega = [1 << i for i in range(0, 19, 3)]
    got = ctx().run_levels(*e, V, omega, 5).numpy("labels").copy()
    ctx().set_limits()
    assert np.array_equal(got, ctx().run_levels(*e, V, omega, 5).numpy("labels"))
