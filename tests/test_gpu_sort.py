"""The radix sort at the sizes where its forms change, through the entry
points that use it: one CTA's tile (4,096 keys), one tile a CTA, few and many
CTAs (64 count their neighbours themselves), several tiles a CTA, and times
whose digits are skewed or all equal. Every output equals the oracle's."""
import numpy as np
import pytest

from gpu_helpers import compare_all
from paper_2311_10337_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [2047, 2048, 2049, 4095, 4096, 4097, 8192, 131_073, 266_241])
def test_sort_form_edges(E):
    # incidence items are 2E: 2,048 / 4,096 edges cross one tile, 131,073 edges
    # 64 CTAs of one tile
    w = synth.random_small(E, max(40, E // 20), max(50, E // 3), 900 + E % 97)
    rng = np.random.default_rng(E)
    q = np.sort(rng.choice(E, min(E, 500), replace=False)).astype(np.int32)
    compare_all(w.src, w.dst, w.t, w.n_vertices, 4, 5, knn_query=q)


def test_incidence_lists_of_several_tiles_a_cta():
    """3M edges: 6M incidence items are more tiles than the device holds CTAs
    of the sort; the lists and positions are fixed by their definition."""
    import torch
    from gpu_helpers import ctx
    E, V = 3_000_017, 70_001
    rng = np.random.default_rng(5)
    src = (rng.random(E) ** 3 * V).astype(np.int32)  # skewed digits
    dst = ((src + 1 + rng.integers(0, V - 1, E)) % V).astype(np.int32)
    t = (rng.integers(0, 5000, E) * 60).astype(np.int64)
    out = ctx().run(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), V, 4, 5)
    for lst, off, pos, end in (("out_id", "out_off", "pos_out", src), ("in_id", "in_off", "pos_in", dst)):
        want = np.lexsort((np.arange(E), t, end)).astype(np.int32)
        assert np.array_equal(out.numpy(lst), want), lst
        assert np.array_equal(out.numpy(off), np.searchsorted(end[want], np.arange(V + 1))), off
        inv = np.empty(E, np.int32)
        inv[want] = np.arange(E, dtype=np.int32)
        assert np.array_equal(out.numpy(pos), inv), pos
