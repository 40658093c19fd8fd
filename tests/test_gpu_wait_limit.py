"""A grid barrier that gives up ends its call with DGEC_ERR_TIMEOUT, wherever
in the call that is: the kernels behind follow nothing that was left half made,
and the context and its workspace serve the next call. The bound 0 gives up at
every barrier without a poll; from the n-th cooperative launch of a call on, for
every n until the call ends well."""
import numpy as np
import pytest

from gpu_helpers import ctx

pytestmark = pytest.mark.gpu

TIMEOUT = 7


def _edges(E, V, span, seed, shift=0):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    src = torch.randint(0, V, (E,), generator=g, device="cuda")
    dst = (src + torch.randint(1, V, (E,), generator=g, device="cuda")) % V
    t = torch.randint(0, span, (E,), generator=g, device="cuda")
    return src.int(), dst.int(), t << shift


def _path(n):
    import torch
    t = torch.cumsum(torch.arange(n, 0, -1, device="cuda"), 0)
    p = torch.randperm(n, device="cuda")
    a = torch.arange(n, dtype=torch.int32, device="cuda")
    return a[p], a[p] + 1, t[p]


def _rows(E, V, most, seed):
    import torch
    r = np.random.default_rng(seed)
    size = r.integers(0, most, E)
    off = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    at = np.arange(off[-1]) - np.repeat(off[:-1], size)
    hub = np.where(r.random(E) < 0.3, 0, r.integers(0, V // 2, E))  # vertex 0: a list of thousands
    vert = (np.repeat(hub, size) + at) % (V // 2)
    return torch.from_numpy(off).cuda(), torch.from_numpy(vert.astype(np.int32)).cuda()


def _calls():
    import torch
    c = ctx()
    names = ["labels", "link_a", "link_b", "link_size", "mst_u", "mst_w"]

    def run(e, V, k=4, M=5, **kw):
        return lambda: [c.run(*e, V, k, M, **kw).tensor(n) for n in names]

    e = _edges(20_000, 2_000, 100_000, 1)
    yield "run", run(e, 2_000)
    yield "wide span", run(_edges(20_000, 2_000, 1 << 20, 2, 30), 2_000, 16)
    yield "large rounds", run(_edges(2_600_000, 300_000, 1 << 20, 3), 300_000)
    yield "path", run(_path(400_000), 400_002, 2, 2)
    yield "mutual reachability", run(e, 2_000, mrd=True)
    yield "nearly causal", run(e, 2_000, delta_nc=50)
    sizes = np.array([3_000, 0, 9_000, 50, 8_000])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    nv = np.full(5, 400, np.int32)
    kk, MM = np.array([4, 4, 8, 4, 16], np.int32), np.full(5, 3, np.int32)
    b = _edges(int(off[-1]), 400, 5_000, 4)
    yield "batch", lambda: [c.run_batch(*b, off, nv, kk, MM).t[n] for n in names[:4]]
    lv = _edges(200_000, 8_000, 1 << 20, 5)
    for dense in (False, True):
        def levels(dense=dense):
            o = c.run_levels(*lv, 8_000, [1 << i for i in range(20)], 5, dense)
            return [o.tensor(n) for n in ("labels", "merge_level", "merge_parent")]
        yield f"levels {dense}", levels
    E, V = 60_000, 3_000
    t = torch.randint(0, 1 << 20, (E,), device="cuda")
    (so, sv), (do, dv) = _rows(E, V, 5, 6), _rows(E, V, 4, 7)
    dv = dv + V // 2
    for kw in ({}, {"d_off": do, "d_vert": dv}):
        def hyper(kw=kw):
            o = c.run_hyper(t, so, sv, V, 5, **kw)
            return [o.tensor(n) for n in names]
        yield f"hypergraph {len(kw)}", hyper


@pytest.mark.parametrize("name", ["run", "wide span", "large rounds", "path", "mutual reachability", "nearly causal", "batch",
                                  "levels False", "levels True", "hypergraph 0", "hypergraph 2"])
def test_every_barrier_can_give_up(name):
    import torch
    from paper_2311_10337_gb300 import dgec
    c = ctx()
    call = dict(_calls())[name]
    want = [x.clone() for x in call()]
    try:
        n = 0
        while True:
            c.set_limits(barrier_polls=0, barrier_from=n)
            try:
                got = call()
                break
            except dgec.DgecError as e:
                assert e.status == TIMEOUT, e
            if n % 4 == 0:  # the context as it was
                c.set_limits()
                assert all(torch.equal(a, b) for a, b in zip(want, call()))
            n += 1
            assert n < 400
        assert n >= 5
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    finally:
        c.set_limits()


def test_bad_limits_are_rejected():
    from paper_2311_10337_gb300 import dgec
    for polls, first, steps in ((-1, 0, 1), (1, -1, 1), (1, 0, 0), (1, 0, -5)):
        with pytest.raises(dgec.DgecError) as e:
            ctx().set_limits(polls, first, steps)
        assert e.value.status == 1
