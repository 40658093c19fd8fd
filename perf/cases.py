"""What the library's users have it do, as measurable cases: single graphs
from the smallest to half of the largest benchmark graph, batches, the
serving loop, the discrete dendrogram, hypergraphs and the option switches,
each through the Python binding's public calls.

Inputs are drawn on the GPU from the seed alone. Their shapes are those of
the package's synth module (whose NumPy generators take minutes at these
sizes): "uniform" is its tiny graph (rank-Zipf(2.1) endpoints, uniform
times), "mid" its 70 % planted conversations with 30 % Zipf(2.1) background
over 30 days, "hub" its Zipf(1.8) background on a 60 s grid with 40 %
conversations and 10 % pairs replayed on an hourly grid, "mail" its
broadcast hypergraph. No self loops; a repeated (i, j, t) triple is moved a
second on, as synth does.

Every output is whole numbers (ids, times, counts, exact 128-bit sums).
"""
import math

import torch

from paper_2311_10337_gb300 import dgec

DAY = 86400
SPAN = 30 * DAY
MAX_GRAPH = 100_000_000

_CTX = None


def _context():
    """The one context a program keeps: its workspace grows to the largest
    call made and is reused by the others."""
    global _CTX
    if _CTX is None:
        _CTX = dgec.Context(0)
    return _CTX


# ------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest graph of the batching workload on its own: all latency
        {"name": "run_1k", "kind": "run", "shape": "uniform", "E": 1_000, "V": 100, "k": 4},
        # the tiny benchmark graph: still latency and launches
        {"name": "run_20k", "kind": "run", "shape": "uniform", "E": 20_000, "V": 2_000, "k": 4},
        # one window of a time-ordered stream, the median served job, odd size
        {"name": "run_window_317k", "kind": "run", "shape": "mid", "E": 316_229, "V": 6_007, "k": 8,
         "sorted": True},
        # nanosecond stamps: spans that fit no 64-bit (t, id) key, and k at its most
        {"name": "run_ns_3m", "kind": "run", "shape": "mid", "E": 3_000_001, "V": 60_000, "k": 16, "ns": True},
        # the 50M-edge benchmark graph
        {"name": "run_mid_50m", "kind": "run", "shape": "mid", "E": 50_000_000, "V": 1_000_000, "k": 8},
        # half of the headline 200M-edge hub graph
        {"name": "run_hub_100m", "kind": "run", "shape": "hub", "E": MAX_GRAPH, "V": 5_000_000, "k": 8},
        # edges from pinned host memory, labels back to it
        {"name": "host_10m", "kind": "host", "shape": "mid", "E": 10_000_000, "V": 200_000, "k": 8},
        # many independent graphs in one call (10^3 to 10^6 edges, k of 4, 8 or 16)
        {"name": "batch_128", "kind": "batch", "G": 128, "lo": 3.0, "hi": 6.0},
        # a burst of windowed jobs through the serving loop
        {"name": "serve_24", "kind": "serve", "E": 20_000_000, "V": 400_000, "jobs": 24, "lo": 4.0, "hi": 6.3},
        # the discrete dendrogram at 1 s to 2^28 s with condensing on it
        {"name": "levels_20m", "kind": "levels", "shape": "mid", "E": 20_000_000, "V": 400_000, "q": 29, "M": 5,
         "dense": False},
        # broadcast messages: one sender, several receivers
        {"name": "hyper_5m", "kind": "hyper", "E": 5_000_000, "V": 250_000, "directed": True},
        # tolerance for clock skew: the nearly-causal line graph
        {"name": "causal60_5m", "kind": "run", "shape": "mid", "E": 5_000_000, "V": 100_000, "k": 8, "dnc": 60},
    ]


def _log(rng, lo, hi):
    return int(round(10.0 ** rng.uniform(math.log10(lo), math.log10(hi))))


def draw(rng):
    """One more case: any kind, sizes log-uniform over its range."""
    kind = rng.choice(["run"] * 6 + ["host", "batch", "batch", "serve", "levels", "hyper", "hyper"])
    if kind == "run":
        c = {"kind": "run", "shape": rng.choice(["uniform", "mid", "hub"]), "k": rng.choice([4, 5, 8, 8, 16])}
        option = rng.choice(["", "", "", "", "sorted", "ns", "dmax", "dnc", "mrd"])
        c["E"] = _log(rng, 1_000, {"": 60e6, "sorted": 30e6, "ns": 10e6, "dnc": 10e6, "mrd": 4e6, "dmax": 30e6}[option])
        c["V"] = max(16, int(c["E"] / rng.uniform(10, 50)))
        if option in ("sorted", "ns", "mrd"):
            c[option] = True
        elif option == "dmax":
            c["dmax"] = _log(rng, 60, 10 * DAY)
        elif option == "dnc":
            c["dnc"] = rng.randint(1, 600)
        return c
    if kind == "host":
        E = _log(rng, 10_000, 20e6)
        return {"kind": "host", "shape": rng.choice(["uniform", "mid", "hub"]), "E": E, "V": max(16, E // 40), "k": 8}
    if kind == "batch":
        lo = rng.uniform(2.0, 4.5)
        return {"kind": "batch", "G": _log(rng, 3, 300), "lo": lo, "hi": rng.uniform(lo, 6.0)}
    if kind == "serve":
        E = _log(rng, 3e6, 30e6)
        lo = rng.uniform(3.0, 5.0)
        return {"kind": "serve", "E": E, "V": E // 50, "jobs": rng.randint(2, 40), "lo": lo, "hi": rng.uniform(lo, 6.3)}
    if kind == "levels":
        E = _log(rng, 3_000, 25e6)
        return {"kind": "levels", "shape": rng.choice(["mid", "hub"]), "E": E, "V": max(16, E // 40),
                "q": rng.randint(4, 29), "M": rng.choice([0, 5, 5]), "dense": E < 3_000_000 and rng.random() < 0.5}
    E = _log(rng, 3_000, 8e6)
    return {"kind": "hyper", "E": E, "V": max(256, E // rng.randint(15, 40)), "directed": rng.random() < 0.5}


# ------------------------------------------------------------------- inputs

class _Draw:
    def __init__(self, seed):
        self.dev = torch.device("cuda:0")
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(seed)

    def uniform(self, n):
        return torch.rand(n, generator=self.g, device=self.dev, dtype=torch.float64)

    def integers(self, lo, hi, n):
        return torch.randint(lo, hi, (n,) if isinstance(n, int) else n, generator=self.g, device=self.dev)

    def perm(self, n):
        return torch.randperm(n, generator=self.g, device=self.dev)

    def geometric(self, n):  # 0, 1, 2, ... with P(x) = 2^-(x + 1)
        return torch.floor(torch.log1p(-self.uniform(n)) / math.log(0.5)).long()

    def zipf_cdf(self, V, s):
        c = torch.cumsum(torch.arange(1, V + 1, device=self.dev, dtype=torch.float64) ** (-s), 0)
        return c

    def ranks(self, n, cdf, cap=None):
        """Rank-Zipf draws; cap: the mass of each draw's own ranks."""
        u = self.uniform(n) * (cdf[-1] if cap is None else cap)
        return torch.searchsorted(cdf, u, right=True).clamp_(max=cdf.shape[0] - 1)


def _zipf_pairs(d, n, V, s, perm):
    cdf = d.zipf_cdf(V, s)
    src = perm[d.ranks(n, cdf)]
    dst = perm[d.ranks(n, cdf)]
    bad = torch.nonzero(src == dst).flatten()
    for _ in range(64):
        if bad.numel() == 0:
            break
        dst[bad] = perm[d.ranks(bad.numel(), cdf)]
        bad = bad[src[bad] == dst[bad]]
    dst[bad] = (src[bad] + 1) % V
    return src, dst


def _conversations(d, n, V, span):
    """Groups of U{3..20} vertices, bursts of U{5..200} records with
    floor(Exp(60 s)) gaps; the sender is the previous receiver w.p. 0.75."""
    out = [[], [], []]
    left = n
    while left > 0:
        nb = left // 100 + 8
        g, length = d.integers(3, 21, nb), d.integers(5, 201, nb)
        base, start = d.integers(0, 1 << 40, nb), d.integers(0, span, nb)
        stride = d.integers(1, max(2, V // 20), nb)
        steps = 200
        gap = torch.floor(-60.0 * torch.log1p(-d.uniform(steps * nb))).long().view(steps, nb)
        gap[0] = 0
        t = torch.cumsum(gap, 0) + start
        del gap
        keep = (d.uniform(steps * nb) < 0.75).view(steps, nb)
        ps, pr = d.integers(0, 1 << 30, (steps, nb)), d.integers(0, 1 << 30, (steps, nb))
        prev = torch.zeros_like(g)
        for x in range(steps):
            s = ps[x] % g
            if x:
                s = torch.where(keep[x], prev, s)
            r = pr[x] % (g - 1)
            prev = r + (r >= s)
            ps[x], pr[x] = s, prev
        live = (torch.arange(steps, device=d.dev)[:, None] < length[None, :])
        # members: base + j * stride (mod V), distinct while 20 strides fit in V
        for o, x in zip(out, ((base + ps * stride) % V, (base + pr * stride) % V, t)):
            o.append(x[live][:left])
        left -= out[0][-1].numel()
    src, dst, t = (torch.cat(o) for o in out)
    dst = torch.where(src == dst, (dst + 1) % V, dst)
    return src, dst, t


def _distinct_triples(src, dst, t, V):
    """A repeat of (i, j, t) moves to a second after its predecessor."""
    pair = src * V + dst
    by_t = torch.sort(t, stable=True).indices
    o = by_t[torch.sort(pair[by_t], stable=True).indices]
    del by_t
    pk, tt = pair[o], t[o]
    head = torch.ones(o.numel(), dtype=torch.bool, device=t.device)
    head[1:] = pk[1:] != pk[:-1]
    del pair, pk
    at = torch.arange(o.numel(), device=t.device)
    gid = torch.cumsum(head, 0) - 1
    r = at - torch.cummax(torch.where(head, at, 0), 0).values
    lo = int(tt.min())
    v = torch.cummax(tt - lo - r + (gid << 33), 0).values - (gid << 33) + r + lo
    out = torch.empty_like(t)
    out[o] = v
    return out


def _graph(d, shape, E, V, in_order=False, ns=False):
    perm = d.perm(V)
    if shape == "uniform":
        src, dst = _zipf_pairs(d, E, V, 2.1, perm)
        t = d.integers(0, 1_000_000, E)
    else:
        hub = shape == "hub"
        n_conv = int(round((0.4 if hub else 0.7) * E))
        n_bg = E // 2 if hub else E - n_conv
        parts = [_conversations(d, n_conv, V, SPAN)]
        b = _zipf_pairs(d, n_bg, V, 1.8 if hub else 2.1, perm)
        parts.append(b + (d.integers(0, SPAN // 60, n_bg) * 60 if hub else d.integers(0, SPAN, n_bg),))
        n_rep = E - n_conv - n_bg
        if n_rep:
            ps, pd = _zipf_pairs(d, max(1, n_rep // 50), V, 1.8, perm)
            which = d.integers(0, ps.numel(), n_rep)
            parts.append((ps[which], pd[which], d.integers(0, SPAN // 3600, n_rep) * 3600))
        src, dst, t = (torch.cat(x) for x in zip(*parts))
        del parts, b
        order = d.perm(E)
        src, dst, t = src[order], dst[order], t[order]
        del order
    t = _distinct_triples(src, dst, t, V)
    if ns:
        t = t * 1_000_000_000 + d.integers(0, 1_000_000_000, E)
    src, dst = src.int(), dst.int()
    if in_order:
        o = torch.sort(t, stable=True).indices
        src, dst, t = src[o], dst[o], t[o]
    return src.contiguous(), dst.contiguous(), t.contiguous()


def _batch(d, G, lo, hi):
    """Graphs of 10^U(lo, hi) edges, a tenth as many vertices, k in {4, 8, 16}."""
    place = d.perm(G)  # the seed orders the graphs; their sizes are the law's G quantiles
    sizes = torch.round(10.0 ** (lo + (hi - lo) * (place + 0.5) / G)).long()
    nv = (sizes // 10).clamp(min=2)
    k = torch.tensor([4, 8, 16], device=d.dev)[place % 3]
    n = int(sizes.sum())
    gid = torch.repeat_interleave(torch.arange(G, device=d.dev), sizes)
    cdf = d.zipf_cdf(int(nv.max()), 2.1)
    cap, top = cdf[nv - 1][gid], nv[gid] - 1
    src = torch.minimum(d.ranks(n, cdf, cap), top)
    dst = torch.minimum(d.ranks(n, cdf, cap), top)
    bad = torch.nonzero(src == dst).flatten()
    for _ in range(64):
        if bad.numel() == 0:
            break
        dst[bad] = torch.minimum(d.ranks(bad.numel(), cdf, cap[bad]), top[bad])
        bad = bad[src[bad] == dst[bad]]
    dst[bad] = (src[bad] + 1) % nv[gid[bad]]
    voff = torch.cumsum(nv, 0) - nv
    V = int(nv.sum())
    t = _distinct_triples(src + voff[gid], dst + voff[gid], d.integers(0, 1_000_000, n), V)
    off = torch.zeros(G + 1, dtype=torch.int64)
    off[1:] = torch.cumsum(sizes, 0).cpu()
    tables = (off.numpy(), nv.int().cpu().numpy(), k.int().cpu().numpy(), torch.full((G,), 5, dtype=torch.int32).numpy())
    return (src.int(), dst.int(), t), tables


def _mail(d, E, V, directed):
    """70 % messages in groups of U{3..12} (a member to the next 1 + Geom(1/2)
    members, bursts of U{5..100} with Exp(60 s) gaps), 30 % background with
    Zipf(2.1) senders and receivers. The receiver counts come from a fixed
    draw (so every seed has as many members), the rest from the seed."""
    n_conv = int(round(0.7 * E))
    n_bg = E - n_conv
    nb = n_conv // 50 + 8
    f = _Draw(5)
    length = f.integers(5, 101, nb)
    live = torch.arange(100, device=d.dev)[:, None] < length[None, :]
    gap = torch.floor(-60.0 * torch.log1p(-d.uniform(100 * nb))).long().view(100, nb)
    gap[0] = 0
    t = (torch.cumsum(gap, 0) + d.integers(0, SPAN, nb))[live][:n_conv]
    while t.numel() < n_conv:  # (the bursts fell short: repeat from the front, a day on)
        t = torch.cat([t, t[:n_conv - t.numel()] + DAY])
    conv = torch.arange(nb, device=d.dev).expand(100, nb)[live]
    conv = conv.repeat(1 + n_conv // max(1, conv.numel()))[:n_conv]
    g, base, stride = f.integers(3, 13, nb), d.integers(0, V, nb), d.integers(1, max(2, V // 12), nb)
    gg = g[conv]
    s = d.integers(0, 1 << 30, n_conv) % gg
    nr = torch.minimum(1 + f.geometric(n_conv), gg - 1)
    row = torch.repeat_interleave(torch.arange(n_conv, device=d.dev), nr)
    x = torch.arange(row.numel(), device=d.dev) - (torch.cumsum(nr, 0) - nr)[row]
    cr = conv[row]
    member = (s[row] + 1 + x) % gg[row]
    rcv = (base[cr] + member * stride[cr]) % V
    snd = (base[conv] + s * stride[conv]) % V
    # background: distinct members, the sender stays
    perm, cdf = d.perm(V), d.zipf_cdf(V, 2.1)
    bn = torch.clamp(1 + f.geometric(n_bg), max=8)
    bs = perm[d.ranks(n_bg, cdf)]
    brow = torch.repeat_interleave(torch.arange(n_bg, device=d.dev), bn)
    br = perm[d.ranks(brow.numel(), cdf)]
    for _ in range(64):
        o = torch.sort(brow * V + br, stable=True).indices
        dup = br == bs[brow]
        dup[o[1:]] |= (brow[o[1:]] == brow[o[:-1]]) & (br[o[1:]] == br[o[:-1]])
        bad = torch.nonzero(dup).flatten()
        if bad.numel() == 0:
            break
        br[bad] = d.integers(0, V, bad.numel())
    snd, nr, rcv = torch.cat([snd, bs]), torch.cat([nr, bn]), torch.cat([rcv, br])
    t = torch.cat([t, d.integers(0, SPAN, n_bg)])
    order = d.perm(E)
    first, cnt = (torch.cumsum(nr, 0) - nr)[order], nr[order]
    snd, t = snd[order], t[order].contiguous()
    off = torch.zeros(E + 1, dtype=torch.int64, device=d.dev)
    off[1:] = torch.cumsum(cnt, 0)
    row = torch.repeat_interleave(torch.arange(E, device=d.dev), cnt)
    at = torch.arange(row.numel(), device=d.dev) - off[:-1][row]
    rcv = rcv[first[row] + at].int()
    if directed:
        return t, torch.arange(E + 1, device=d.dev), snd.int(), off, rcv
    m_off = off + torch.arange(E + 1, device=d.dev)
    mv = torch.empty(int(m_off[-1]), dtype=torch.int32, device=d.dev)
    mv[m_off[:-1]] = snd.int()
    mv[m_off[:-1][row] + 1 + at] = rcv
    return t, m_off, mv, None, None


# Result arrays whose length depends on the data; a program that keeps them
# past the next call copies them out of the workspace, here end to end into
# one buffer per type (-1 beyond the last).
_VAR32 = ("sk_u", "sk_v", "mst_u", "mst_v", "link_a", "link_b", "cl_id", "cl_parent", "cl_selected")
_VAR64 = ("sk_w", "mst_w", "link_size", "cl_size", "cl_birth", "cl_death", "cl_stab_hi", "cl_stab_lo")


def _room(links, edges, clusters=0):
    return tuple(torch.full((n,), -1, dtype=dt, device="cuda:0")
                 for n, dt in ((2 * links + 4 * edges + 3 * clusters, torch.int32),
                               (links + 2 * edges + 5 * clusters, torch.int64)))


def _keep(room, get, names32=_VAR32, names64=_VAR64):
    for buf, names in zip(room, (names32, names64)):
        parts = [get(n) for n in names]
        torch.cat(parts, out=buf[:sum(x.numel() for x in parts)])
    return room


def prepare(case, seed):
    d = _Draw(seed)
    kind = case["kind"]
    st = {"case": case, "ctx": _context()}
    if kind == "batch":
        st["edges"], st["tables"] = _batch(d, case["G"], case["lo"], case["hi"])
        st["room"] = _room(0, int(st["tables"][0][-1]))
    elif kind == "hyper":
        st["hyper"] = _mail(d, case["E"], case["V"], case["directed"])
        st["room"] = _room(sum(x.numel() for x in (st["hyper"][2], st["hyper"][4]) if x is not None), case["E"])
    elif kind == "serve":
        st["edges"] = _graph(d, "mid", case["E"], case["V"], in_order=True)
        N = case["jobs"]  # sizes: the law's N quantiles, in the seed's order
        st["jobs"] = []
        for a, b in zip(d.perm(N).tolist(), d.uniform(N).tolist()):
            n = min(case["E"], int(round(10.0 ** (case["lo"] + (case["hi"] - case["lo"]) * (a + 0.5) / N))))
            st["jobs"].append((int(b * (case["E"] - n + 1)), n))
        st["labels"] = torch.empty(sum(n for _, n in st["jobs"]), dtype=torch.int32, device="cuda:0")
        st["server"] = dgec.Server(pool_bytes=18 << 30, n_lanes=3, vertex_bound=case["V"])
    else:
        src, dst, t = _graph(d, case["shape"], case["E"], case["V"], case.get("sorted", False), case.get("ns", False))
        if kind == "host":
            pinned = [x.cpu().pin_memory() for x in (src, dst, t)]
            pinned.append(torch.empty(case["E"], dtype=torch.int32).pin_memory())
            st["pinned"] = pinned  # the numpy views below share their memory
            st["host"] = [x.numpy() for x in pinned]
        else:
            st["edges"] = (src, dst, t)
        if kind == "run":
            E = case["E"]
            links = (4 if "dnc" in case else 2 + case["k"] if case.get("mrd") else 2) * E
            st["room"] = _room(links, E, E // 2 + 1)  # (a cluster holds 5 edges or more)
        if kind == "levels":
            st["omega"] = [1 << i for i in range(case["q"])]
            st["room"] = _room(2 * case["E"], 0)
    return st


_GRAPH_OUT = ("out_off", "in_off", "out_t", "in_t", "out_id", "in_id", "pos_out", "pos_in", "knn_id", "core",
              "fall_cluster", "fall_lambda", "labels")


def run(st):
    c, ctx = st["case"], st["ctx"]
    kind = c["kind"]
    if kind == "run":
        o = ctx.run(*st["edges"], c["V"], c["k"], 5, delta_max=c.get("dmax"), mrd=c.get("mrd", False),
                    delta_nc=c.get("dnc"))
        return {**{n: o.tensor(n) for n in _GRAPH_OUT}, "sized": _keep(st["room"], o.tensor),
                "counts": [o.n_skeleton, o.n_mst, o.n_condensed, o.n_clusters]}
    if kind == "host":
        src, dst, t, labels = st["host"]
        labels, n = ctx.run_host(src, dst, t, c["V"], c["k"], 5, labels_out=labels)
        return {"labels": labels, "n_clusters": n}
    if kind == "batch":
        o = ctx.run_batch(*st["edges"], *st["tables"])
        names = ["labels", "knn_id", "core", "n_clusters", "mst_off", "knn_off"]
        return {**{n: o.t[n] for n in names}, "sized": _keep(st["room"], o.t.get, _VAR32[2:6], _VAR64[1:3])}
    if kind == "serve":
        srv, (src, dst, t) = st["server"], st["edges"]
        tickets = [srv.submit(src[a:a + n], dst[a:a + n], t[a:a + n], 8, 5, lab)
                   for (a, n), lab in zip(st["jobs"], st["labels"].split([n for _, n in st["jobs"]]))]
        done = [srv.wait(x) for x in tickets]
        return {"status": torch.tensor([x[0] for x in done]), "n_clusters": torch.tensor([x[1] for x in done]),
                "labels": st["labels"]}
    if kind == "levels":
        o = ctx.run_levels(*st["edges"], c["V"], st["omega"], c["M"], c["dense"])
        names = ["merge_level", "merge_parent", "n_components", "level_labels", "labels"]
        return {**{n: o.tensor(n) for n in names}, "sized": _keep(st["room"], o.tensor, _VAR32[:2], _VAR64[:1]),
                "counts": [o.n_skeleton, o.n_merges, o.n_clusters]}
    t, s_off, s_vert, d_off, d_vert = st["hyper"]
    o = ctx.run_hyper(t, s_off, s_vert, c["V"], 5, d_off, d_vert)
    names = ["src_voff", "src_list", "dst_voff", "dst_list", "labels"]
    return {**{n: o.tensor(n) for n in names}, "sized": _keep(st["room"], o.tensor, _VAR32[:6], _VAR64[:3]),
            "counts": [o.n_skeleton, o.n_mst, o.n_clusters]}


# ------------------------------------------------------------------- the work

def work(case):
    """Bytes of the inputs read once and of the outputs written once (no
    floating-point work). A graph's edge: 16 B in; lists 32, skeleton 16 per
    link at about 1.9 links, core 8, kNN 4k, forest 16, rows 16, condensed
    12, label 4 out; 16 B of offsets a vertex."""
    kind = case["kind"]
    lists_to_labels = 32 + 30 + 8 + 16 + 16 + 12 + 4
    if kind == "run":
        b = case["E"] * (16 + lists_to_labels + 4 * case["k"]) + 16 * case["V"]
    elif kind == "host":
        b = 20 * case["E"]
    elif kind == "batch":
        lo, hi = case["lo"] * math.log(10.0), case["hi"] * math.log(10.0)
        mean = (math.exp(hi) - math.exp(lo)) / (hi - lo) if hi > lo else math.exp(lo)
        b = case["G"] * mean * (16 + 8 + 4 * 28 / 3 + 16 + 16 + 4)
    elif kind == "serve":
        lo, hi = case["lo"] * math.log(10.0), case["hi"] * math.log(10.0)
        mean = (math.exp(hi) - math.exp(lo)) / (hi - lo) if hi > lo else math.exp(lo)
        b = case["jobs"] * mean * 20
    elif kind == "levels":
        b = case["E"] * (16 + 30 + 8 + (4 if case["M"] else 0) + (4 * case["q"] if case["dense"] else 0))
    else:
        members = 2.85 * case["E"]
        b = 8 * case["E"] + 4 * members + members * (4 + 16 * 0.8) + case["E"] * (16 + 16 + 4) + 16 * case["V"]
    return {"bytes": float(b), "flops": 0.0}


def exact(case, seed):
    """No output is a rounded number: all are whole numbers, exact already."""
    return None
