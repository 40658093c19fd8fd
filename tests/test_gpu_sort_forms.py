"""The radix sort at the lines between its forms for large inputs: tiles dealt
out from 8 a CTA on (9,961,472 keys in 304 CTAs of 4,096), and narrow digits
above 2^24 pairs and keys. The incidence lists sort two pairs an edge and are
fixed by their definition; the forest's order sorts pairs, then keys."""
import pytest

from gpu_helpers import ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [4_980_736, 4_980_737, 8_388_608, 8_388_609, 17_000_001])
def test_incidence_lists_at_the_lines(E):
    import torch
    V = 70_001
    g = torch.Generator(device="cuda")
    g.manual_seed(E)
    src = (torch.rand(E, generator=g, device="cuda", dtype=torch.float64) ** 4 * V).long()  # skewed digits
    dst = (src + torch.randint(1, V, (E,), generator=g, device="cuda")) % V
    t = torch.randint(0, 500_000, (E,), generator=g, device="cuda") * 5
    out = ctx().run(src.int(), dst.int(), t, V, 4, 5)
    t_order = torch.sort(t, stable=True).indices
    at = torch.arange(E, device="cuda", dtype=torch.int32)
    for lst, times, off, pos, end in (("out_id", "out_t", "out_off", "pos_out", src), ("in_id", "in_t", "in_off", "pos_in", dst)):
        want = t_order[torch.sort(end[t_order], stable=True).indices]
        assert torch.equal(out.tensor(lst).long(), want), lst
        assert torch.equal(out.tensor(times), t[want]), times
        assert torch.equal(out.tensor(off)[1:], torch.cumsum(torch.bincount(end, minlength=V), 0)), off
        assert torch.equal(out.tensor(pos)[want], at), pos
    w = out.tensor("mst_w")
    key = out.tensor("mst_u").long() * E + out.tensor("mst_v").long()
    same = w[1:] == w[:-1]
    assert bool((w[1:] >= w[:-1]).all()) and bool((key[1:][same] > key[:-1][same]).all())
    size = out.tensor("link_size")  # of the merges in that order: a child's is smaller
    child = torch.maximum(out.tensor("link_a"), out.tensor("link_b")).long() - E
    inner = child >= 0
    assert bool((size[inner] > size[child[inner]]).all()) and int(size.max()) <= E
    ctx().ws = None  # tens of GB: not kept for the tests after
