"""The forest's cooperative rounds in both forms of their bids: with the label
of the other end packed beside (w, u, v), and -- when time span and ids need
more than 127 bits together -- without it. The forest is fixed by its order,
so it equals the oracle's."""
import numpy as np
import pytest

from gpu_helpers import ctx, sorted_skeleton
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,shift", [(70_000, 0), (70_000, 42), (2_200_000, 42)])
def test_forest_with_and_without_labels_in_the_bids(E, shift):
    import torch
    rng = np.random.default_rng(E + shift)
    V = E // 8
    src = rng.integers(0, V, E).astype(np.int32)
    dst = ((src + 1 + rng.integers(0, V - 1, E)) % V).astype(np.int32)
    t = rng.integers(0, 1 << 20, E).astype(np.int64) << shift
    span, ids = int(t.max() - t.min()).bit_length(), (E - 1).bit_length()
    assert (span + 3 * ids > 127) == (E > 2_000_000)
    out = ctx().run(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), V, 4, 5)
    r = O.run(src, dst, t, V, 4, 5, np.arange(0, E, E // 50, dtype=np.int32))
    g = sorted_skeleton(out.numpy("sk_u"), out.numpy("sk_v"), out.numpy("sk_w"))
    for a, b in zip(g, r["skeleton"]):
        assert np.array_equal(a, b)
    for a, b in zip(("mst_u", "mst_v", "mst_w"), r["mst"]):
        assert np.array_equal(out.numpy(a), b), a
    for a, b in zip(("link_a", "link_b", "link_size"), r["linkage"]):
        assert np.array_equal(out.numpy(a), b), a
    assert np.array_equal(out.numpy("labels"), r["condensed"]["labels"])
