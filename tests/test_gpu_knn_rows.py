"""kNN rows against the oracle where a row's write can go wrong: every padded
width and k on both sides of it (rows written as whole 32- or 16-byte words
when k fills the width and the row is aligned, id by id otherwise), duplicate
candidates (an edge reached through both of its vertices), short rows, and
batches whose row offsets are odd multiples of 4 bytes."""
import numpy as np
import pytest

from gpu_helpers import ctx, run_gpu
from oracle import oracle as O
from paper_2311_10337_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [0, 1, 2])
@pytest.mark.parametrize("k", [1, 3, 4, 5, 7, 8, 9, 15, 16])
def test_rows_of_every_width(form, k):
    c = ctx()
    default = c.launch_config()
    try:
        c.set_launch_config(default[0], default[1], form)
        # few vertices and times: reciprocal pairs and repeated triples give duplicates and tie groups
        for E, V, T, cut in ((1, 2, 1, None), (33, 2, 3, None), (257, 3, 5, None), (600, 9, 40, 3), (1500, 40, 90, None)):
            g = synth.random_small(E, V, T, 40 + E + k)
            out = run_gpu(g.src, g.dst, g.t, g.n_vertices, k, 3, cut)
            ids, core = O.knn(g.src, g.dst, g.t, g.n_vertices, k, None, cut)
            assert np.array_equal(out["knn_id"].reshape(-1), ids.reshape(-1)), (E, V)
            assert np.array_equal(out["core"], core), (E, V)
    finally:
        c.set_launch_config(*default)


@pytest.mark.parametrize("form", [0, 1, 2])
def test_unaligned_rows_of_a_batch(form):
    import torch
    c = ctx()
    default = c.launch_config()
    ks = [8, 3, 8, 16, 1, 8, 4, 16, 8]  # E * k of the odd ones leaves the next graph's rows unaligned
    gs = [synth.random_small(61 + 2 * i, 5 + i, 9, 900 + i) for i in range(len(ks))]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    eoff = np.concatenate([[0], np.cumsum([len(g.src) for g in gs])]).astype(np.int64)
    try:
        c.set_launch_config(default[0], default[1], form)
        out = c.run_batch(dev(np.concatenate([g.src for g in gs]).astype(np.int32)),
                          dev(np.concatenate([g.dst for g in gs]).astype(np.int32)),
                          dev(np.concatenate([g.t for g in gs]).astype(np.int64)), eoff,
                          np.array([g.n_vertices for g in gs], np.int32), np.array(ks, np.int32),
                          np.array([3] * len(gs), np.int32))
        for i, (g, k) in enumerate(zip(gs, ks)):
            ids, core = O.knn(g.src, g.dst, g.t, g.n_vertices, k)
            got = out.graph(i)
            assert np.array_equal(got["knn_id"].reshape(-1), ids.reshape(-1)), (i, k)
            assert np.array_equal(got["core"], core), (i, k)
    finally:
        c.set_launch_config(*default)
