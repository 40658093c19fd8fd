// Stage D2: condensed tree with minimum cluster size M (Alg. 1, condensing),
// excess-of-mass selection (Alg. 1, clusters chosen by their volume in the
// dendrogram)
// and the edge-cluster labels of Alg. 4.
//
// The paper defines these steps by citation to HDBSCAN. Readings kept
// here, identical to the oracle's:
//   - merges of equal weight are one multi-way merge (only the top merge of
//     an equal-weight run is kept), so labels depend only on the weighted
//     connectivity that Thm. 3 preserves;
//   - lambda(w) = floor((2^64 - 1) / (w + 1)); a virtual root of weight
//     infinity (lambda 0) has the components as children;
//   - top-down: a kept merge X of cluster K with >= 2 children of size >= M
//     ends K and starts one cluster per such child; with exactly one such
//     child, that child continues K; every point under a smaller child
//     leaves K at lambda(X);
//   - stabilities are exact 128-bit integers; EOM keeps a cluster when its
//     stability is >= the best total of its children; the root is never
//     kept; clusters are numbered by their smallest member id.
//
// Everything is computed by data-parallel passes: pointer jumping for the
// equal-weight runs and for "which cluster does this merge belong to",
// short upward walks (< M steps) for where a point leaves, 128-bit atomics
// for stabilities, and upward walks plus a rake-and-compress contraction of
// what they leave for the EOM maximisation, whose per-node update
// S = max(stab, sum of children) composes along unary chains as
// x -> max(a, c + x).
#include "coop.cuh"
#include "stages.cuh"

namespace dgec {

typedef unsigned __int128 u128;

// Node ids: leaves [0, E), merges E + s, and one virtual root per graph at
// R0 + g (R0 = E + number of merges).
struct Gview {
    int64_t E, n, R0;
    int G;
    const int32_t *egraph;  // graph of each leaf
    const int32_t *mu;      // original lower end of each merge's forest edge
    const int64_t *eoff;    // [G+1]
    const int32_t *gM;      // [G] min cluster size per graph
};

__device__ __forceinline__ int graph_of(const Gview &g, int64_t x) {
    if (g.G == 1) return 0;  // one graph: no lookup (a merge's lookup is a random read)
    return x < g.E ? g.egraph[x] : (x < g.R0 ? g.egraph[g.mu[x - g.E]] : (int)(x - g.R0));
}

__device__ __forceinline__ unsigned long long lam_node(int64_t X, const Gview &g, const int64_t *w) {
    return X >= g.R0 ? 0ull : lambda_of(w[X - g.E]);
}

__device__ __forceinline__ int64_t node_size(int64_t X, const Gview &g, const int64_t *size) {
    if (X < g.E) return 1;
    if (X < g.R0) return size[X - g.E];
    int gr = (int)(X - g.R0);
    return g.eoff[gr + 1] - g.eoff[gr];
}

__global__ void k_c_up(int64_t E, int64_t n, const int32_t *parent, const int64_t *w, int32_t *up,
                       int *isrep) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        int P = parent[E + s];
        bool rep = P < 0 || w[P - E] != w[s];
        isrep[s] = rep;
        up[s] = rep ? (int32_t)s : (int32_t)(P - E);
    }
}

struct SelAll {
    __device__ bool operator()(int64_t) const { return true; }
};
struct SelBigRep {  // big kept merges (the nodes whose cluster link is set)
    Gview gv;
    const int *isrep;
    const int64_t *size;
    __device__ bool operator()(int64_t s) const {
        return isrep[s] && size[s] >= gv.gM[graph_of(gv, gv.E + s)];
    }
};
// One pass of start-compressing walks, in descending index order: parents
// have larger ids than their children, so ancestors tend to be resolved
// first and later walks stop after a few steps. A walk that exceeds
// kTopWalk steps stores the ancestor it reached and goes to the list of cut
// walks (*cut: their number). The limit bounds what a long run of equal weights
// costs, whose first walkers meet only pointers as short as their own: this
// stage on 60M edges at one threshold, walks of up to 4,096 / 256 / 128 / 64 steps:
// 190 / 16.8 / 10.7 / 8.9 ms; 60M edges with times in whole days 92.6 / 14.3 / 11.5 /
// 10.2. 200M hub edges, whose few long walks the rounds finish in 0.05 ms, 51.4 ms
// at 4,096 and 51.3 at 64.
constexpr int kTopWalk = 64;
// OWN: the limit is kTopWalk, known when the loop is compiled (read from the
// arguments, the walks of 20M edges take 0.63 ms instead of 0.32).
template <bool OWN, class Sel>
__global__ void k_c_top(const unsigned *stop, int64_t n, int64_t off, Sel sel, int32_t *ptr, int steps, int32_t *list,
                        unsigned long long *cut) {
    if (stopped(stop)) return;
    const int limit = OWN ? kTopWalk : steps;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = n - 1 - t;
        if (!sel(s)) continue;
        const int64_t x = off + s;
        int r = ptr[x];
        int it = 0;
        for (; it < limit; it++) {
            const int rr = ptr[r];
            if (rr == r) break;
            r = rr;
            atomicExch(ptr + x, r);  // not a store: other CTAs read these lines meanwhile
        }
        if (it == limit) list_cut(list, cut, (int)x);
    }
}

// The cut walks' pointers to their fixed points. cut[1 .. 3]: the rounds'
// flags, zero at the start.
__global__ void __launch_bounds__(kBlock) k_c_jump(const int32_t *list, int32_t *ptr, unsigned long long *cut, BarRef ref) {
    const int64_t n = (int64_t)cut[0];
    if (n == 0) return;  // the same for every CTA: written before this launch
    GridBar bar(ref);
    if (bar.stopped()) return;
    const JumpEnd e = jump_rounds(bar, n, ListItem{list}, ptr, cut + 1);
    if (e == kJumpBarrier) return;
    if (e == kJumpBound && threadIdx.x == 0) bar.stop(kStopJump);
    bar.finish();
}

// Every selected pointer to its fixed point: one walk pass, then the jumping
// rounds, which return at once unless some walk was cut short. (Asking the
// host whether to launch them cost a call two waits; with the memsets that
// k_c_zero took over, this stage took 0.20 ms instead of 0.16 at 1,000 edges.)
template <class Sel>
static dgec_status jump_to_fixed(Ctx *c, int64_t n, int64_t off, Sel sel, int32_t *ptr, int32_t *list,
                                 unsigned long long *cut) {
    if (n <= 0) return DGEC_OK;
    const int g = grid_for(n, kBlock, kStreamCap);
    if (c->own_walk(kTopWalk))
        TK(c, "k_c_top", k_c_top<true, Sel><<<g, kBlock, 0, c->stream>>>(c->stop(), n, off, sel, ptr, kTopWalk, list, cut));
    else
        TK(c, "k_c_top", k_c_top<false, Sel><<<g, kBlock, 0, c->stream>>>(c->stop(), n, off, sel, ptr, c->walk_steps, list, cut));
    int grid = 1;
    DG_TRY(coop_grid(c, kCoopCJump, (const void *)k_c_jump, kBlock, 0, &grid));
    BarRef ref = c->next_bar();
    void *args[] = {&list, &ptr, &cut, &ref};
    cudaError_t e;
    TK(c, "k_c_jump", e = cudaLaunchCooperativeKernel((const void *)k_c_jump, dim3((unsigned)(g < grid ? g : grid)),
                                                      dim3(kBlock), args, 0, c->stream));
    if (e != cudaSuccess) return set_err(c, DGEC_ERR_CUDA, "k_c_jump launch: %s", cudaGetErrorString(e));
    return DGEC_OK;
}


// Collapsed parent of every leaf and kept merge. nbs[X - E] of a kept merge
// or virtual root X sums (1 << 32) + size over its big children: the high
// word counts them, the low word totals their sizes (below 2^31, as every
// child count and size is), so the points that leave a big X's cluster at X
// number size(X) minus the low word.
__global__ void k_c_cpar(Gview gv, const int32_t *__restrict__ parent, const int32_t *__restrict__ up,
                         const int *__restrict__ isrep, const int64_t *__restrict__ size,
                         int32_t *__restrict__ cpar, unsigned long long *__restrict__ nbs) {
    const int64_t E = gv.E, total = E + gv.n;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < total;
         base += stride) {  // warp-uniform
        const int64_t x = base + lane_id();
        bool big = false;
        int64_t cp = E;
        unsigned sz = 0;
        if (x < total && (x < E || isrep[x - E])) {
            const int P = parent[x];
            cp = P < 0 ? gv.R0 + graph_of(gv, x) : E + up[P - E];
            cpar[x] = (int32_t)cp;
            if (x >= E) {
                sz = (unsigned)size[x - E];
                big = (int64_t)sz >= gv.gM[graph_of(gv, x)];
            }
        }
        // (merges of equal weight collapse: a parent can have very many big
        // children; one atomic a child took 7.5 ms at 100M hub edges, 3.8 by key)
        warp_add_count_size(big, (int)(cp - E), sz, nbs);
    }
}

// link: a big kept merge continues its parent's cluster when it is the
// parent's only big child, else it starts a cluster (link to itself);
// virtual roots link to themselves.
__global__ void k_c_link(const unsigned *stop, Gview gv, const int *isrep, const int64_t *size, const int32_t *cpar,
                         const unsigned long long *nbs, int32_t *link) {
    if (stopped(stop)) return;
    const int64_t E = gv.E, n = gv.n;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n + gv.G;
         s += (int64_t)gridDim.x * blockDim.x) {
        if (s >= n) {
            link[E + s] = (int32_t)(E + s);
            continue;
        }
        if (!isrep[s] || size[s] < gv.gM[graph_of(gv, E + s)]) continue;
        int64_t X = cpar[E + s];
        link[E + s] = (nbs[X - E] >> 32) >= 2 ? (int32_t)(E + s) : (int32_t)X;
    }
}


// cluster records, indexed by node id
__global__ void k_c_clusters(const unsigned *stop, Gview gv, const int *isrep, const int64_t *size, const int64_t *w,
                             const int32_t *cpar, const unsigned long long *nbs, const int32_t *link, int *isc,
                             unsigned long long *cbirth, unsigned long long *cdeath,
                             int32_t *cparent) {
    if (stopped(stop)) return;
    const int64_t E = gv.E, n = gv.n;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n + gv.G;
         s += (int64_t)gridDim.x * blockDim.x) {
        int64_t X = E + s;
        bool big = s >= n || (isrep[s] && size[s] >= gv.gM[graph_of(gv, X)]);
        if (!big) continue;
        int K = link[X];
        if ((nbs[s] >> 32) >= 2) cdeath[K] = lam_node(X, gv, w);
        if (K == (int)X) {
            isc[X] = 1;
            if (X >= gv.R0) {
                cbirth[X] = 0;
                cparent[X] = -1;
            } else {
                int64_t P = cpar[X];
                cbirth[X] = lam_node(P, gv, w);
                cparent[X] = link[P];
            }
        }
    }
}

// Per node a point can land on or walk through (kept merges, virtual
// roots): its collapsed parent, its cluster when it is big (else -1), its
// lambda and, when big, the stability share of a point leaving its cluster
// there (lambda - the cluster's birth), in one 32-byte record: each step of
// a point's walk reads one sector, and the landing needs no other lookup.
struct __align__(32) NodeRec {
    int32_t cpar;
    int32_t link;
    unsigned long long lam;
    unsigned long long share;
    unsigned long long pad;
};

// The records, and the stability the points leaving at each node give its
// cluster. Every point that leaves cluster K at the big node X does so at
// lambda(X), so together they add nf(X) * (lambda(X) - birth(K)), with nf(X)
// = size(X) minus the sizes of X's big children (the points under its small
// children, which walk up to X): one exact 128-bit add per node, summed per
// warp and cluster, instead of one per point.
__global__ void k_c_nrec(const unsigned *stop, Gview gv, const int *isrep, const int64_t *size, const int64_t *w,
                         const int32_t *cpar, const int32_t *link, const unsigned long long *cbirth,
                         const unsigned long long *__restrict__ nbs, NodeRec *rec, unsigned long long *st_hi,
                         unsigned long long *st_lo) {
    if (stopped(stop)) return;
    const int64_t E = gv.E, n = gv.n, total = n + gv.G;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < total;
         base += stride) {  // warp-uniform
        const int64_t s = base + lane_id();
        bool has = false;
        int K = 0;
        unsigned __int128 val = 0;
        if (s < total) {
            const int64_t X = E + s;
            NodeRec r;
            r.pad = 0;
            bool write = true;
            if (s >= n) {
                r.cpar = (int32_t)X;
                r.link = link[X];
                r.lam = 0ull;
                r.share = 0ull;  // a virtual root: lambda 0, birth 0
            } else if (!isrep[s]) {
                write = false;  // never a collapsed parent
            } else {
                const int64_t sz = size[s];
                const bool big = sz >= gv.gM[graph_of(gv, X)];
                r.cpar = cpar[X];
                r.link = big ? link[X] : -1;
                r.lam = lambda_of(w[s]);
                r.share = big ? r.lam - cbirth[r.link] : 0ull;
                if (big && r.share != 0ull) {
                    const int64_t nf = sz - (int64_t)(nbs[s] & 0xffffffffull);
                    if (nf > 0) {
                        has = true;
                        K = r.link;
                        val = (unsigned __int128)(unsigned long long)nf * r.share;  // below 2^95
                    }
                }
            }
            if (write) rec[s] = r;
        }
        warp_add_u96(has, K, val, st_hi, st_lo);
    }
}

// where each point leaves: the lowest kept ancestor of size >= M (its
// stability share is counted per node above)
__global__ void k_c_points(const unsigned *stop, Gview gv, const int32_t *__restrict__ cpar, const NodeRec *__restrict__ rec,
                           int32_t *__restrict__ fall_cluster, uint64_t *__restrict__ fall_lambda) {
    if (stopped(stop)) return;
    const int64_t E = gv.E;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < E;
         p += (int64_t)gridDim.x * blockDim.x) {
        NodeRec r = rec[cpar[p] - E];
        for (int it = 0; it < kMaxWalk && r.link < 0; it++) r = rec[r.cpar - E];
        fall_cluster[p] = r.link;
        fall_lambda[p] = r.lam;
    }
}

// Every cluster's parent as a cluster index, and per parent the number of its
// child clusters and their total size, (count << 32) + size: the child
// clusters' points leave the parent P at P's death, so P gains (death - birth)
// * (that size), a product taken when the stabilities are gathered.
__global__ void k_c_kids(int64_t ncl, Gview gv, const int32_t *__restrict__ clist,
                         const int32_t *__restrict__ cparent, const int32_t *__restrict__ cidx,
                         const int64_t *__restrict__ size, int32_t *__restrict__ par, unsigned long long *kids) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < ncl;
         base += stride) {  // warp-uniform
        const int64_t c = base + lane_id();
        int p = -1;
        unsigned sz = 0;
        bool add = false;
        if (c < ncl) {
            const int K = clist[c];
            if (K < gv.R0) {
                p = cidx[cparent[K]];
                sz = (unsigned)size[K - gv.E];
                add = true;
            }
            par[c] = p;
        }
        warp_add_count_size(add, p, sz, kids);
    }
}

// compact cluster list (ascending node id) and per-cluster arrays; only
// merges and virtual roots (node ids E + i) can be clusters, so the flags
// and their prefix sums cover those alone
__global__ void k_c_compact(int64_t E, int64_t m, int64_t ncl, const int *isc, const long long *cpos,
                            int32_t *clist, int32_t *cidx, unsigned long long *csz, int *minmem) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        csz[ncl] = 0;
        minmem[ncl] = INT_MAX;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!isc[i]) continue;
        const long long at = cpos[i];
        clist[at] = (int32_t)(E + i);
        cidx[E + i] = (int32_t)at;
        csz[at] = 0;
        minmem[at] = INT_MAX;
    }
}

struct Eom {
    int64_t ncl;
    int64_t root0;  // clusters [root0, ncl) are the virtual roots (never selected, nothing reads their sums)
    int64_t R0;     // node ids >= R0 are virtual roots
    const int32_t *clist, *cparent;  // cparent by node id
    const int32_t *par;                      // compact parent, -1 root
    int *pending, *done, *fin;
    u128 *stab, *S, *Fa, *Fc, *Fa2, *Fc2;
    const unsigned long long *kids;       // (child clusters << 32) + their total size (0: none)
    unsigned long long *acc_hi, *acc_lo;  // sum of the children's S
    int32_t *ucand, *nxt, *nxt2, *al, *al2;
    unsigned long long *slot;  // (next ancestor << 32) | highest selected on the way there
    int32_t *H;                // highest selected ancestor-or-self, -1
    unsigned long long *cnt;   // [0], [1] open clusters, [2..4] flags; zeroed before the kernel
    int walk;                  // limit of a walk
    BarRef bar;
};

__global__ void k_e_init(Eom e, const unsigned long long *st_hi, const unsigned long long *st_lo,
                         const unsigned long long *cbirth, const unsigned long long *cdeath) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < e.ncl;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int node = e.clist[c];
        const unsigned long long kids = e.kids[c];
        const u128 from_kids = kids ? (u128)(cdeath[node] - cbirth[node]) * (kids & 0xffffffffull) : (u128)0;
        e.stab[c] = (((u128)st_hi[node] << 64) | st_lo[node]) + from_kids;
        e.pending[c] = (int)(kids >> 32);
        e.done[c] = 0;
        e.acc_hi[c] = 0;
        e.acc_lo[c] = 0;
    }
}

__device__ __forceinline__ u128 acc_of(const Eom &e, int64_t c) {
    return ((u128)e.acc_hi[c] << 64) | e.acc_lo[c];
}

__device__ __forceinline__ void acc_add(const Eom &e, int p, u128 s) {
    atomic_add_u128(&e.acc_hi[p], &e.acc_lo[p], (unsigned long long)(s >> 64), (unsigned long long)s);
}

// From a cluster c whose children have all reported, up while this thread is
// the last child to report: S = max(stab, sum of the children's S) is added
// to the parent's sum, and the last report makes the parent ready. At most
// kEomWalk clusters; the one reached then stays open (ready, not done).
constexpr int kEomWalk = 24;
__device__ __forceinline__ void e_walk(const Eom &e, int c) {
    for (int step = 0; step < kEomWalk; step++) {
        const u128 acc = ((u128) * (volatile unsigned long long *)&e.acc_hi[c] << 64) |
                         *(volatile unsigned long long *)&e.acc_lo[c];
        const u128 st = e.stab[c];
        const int p = e.par[c];
        e.done[c] = 1;
        if (p < 0 || p >= e.root0) return;
        acc_add(e, p, st > acc ? st : acc);
        __threadfence();
        if (atomicSub(&e.pending[p], 1) != 1) return;
        __threadfence();
        c = p;
    }
}

// Excess of mass over the cluster tree in one cooperative kernel: every
// cluster's sum of its children's S = max(stab, that sum), then for every
// cluster its highest selected ancestor-or-self (selected: stab >= the sum,
// ties to the parent; a virtual root never).
//   1. Every leaf cluster walks up (e_walk): all subtrees of height up to
//      kEomWalk, which is nearly every cluster, are done in this one pass.
//   2. What stays open are the long spines. Contraction over the open list
//      only: runs of clusters with one open child compose x -> max(a, c + x)
//      by doubling; runs that end in a ready cluster resolve and report to
//      the parent above, whose last report walks on. Repeated until nothing
//      is open; a phase at least halves the spines' branchings.
//   3. Walks toward the root that leave a (next, highest selected) shortcut
//      in their slot, in descending order, so the clusters near the root
//      finish first and later walks are short; a walk cut at e.walk steps
//      is taken up again in another round.
// What bounds it: the random 8 and 16-byte accesses of the walks' reports at
// large trees, the barriers (about 2 us each) of the contraction at small ones.
// Against a contraction of the whole tree phase by phase (up to 160 launches
// and a host read every other one; a serial sweep up to 4,096 clusters): 0.06 ms
// for 0.55 at 20,000 edges, 0.63 for 2.7 at 10M, 4.7 for about 15 at 100M hub
// edges.
__global__ void __launch_bounds__(256, 4) k_e_tree(Eom e) {
    GridBar bar(e.bar);
    if (bar.stopped()) return;
    const int64_t gsize = (int64_t)gridDim.x * blockDim.x, g0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    for (int64_t c = g0; c < e.root0; c += gsize)
        if (e.kids[c] == 0) e_walk(e, (int)c);  // no child cluster
    if (!bar.sync()) return;
    int32_t *al = e.al, *al2 = e.al2;
    int64_t nact = e.root0;
    for (int phase = 0;; phase++) {
        if (phase > 4096) {
            if (lead) bar.stop(kStopEom);
            return;
        }
        // the open clusters; each tells a parent that waits for it alone
        for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nact; base += gsize) {  // CTA-uniform
            const int64_t ix = base + threadIdx.x;
            bool open = false;
            int c = 0;
            if (ix < nact) {
                c = phase == 0 ? (int)ix : al[ix];
                open = !e.done[c];
                if (open) {
                    const int p = e.par[c];
                    if (p >= 0 && p < e.root0 && e.pending[p] == 1) e.ucand[p] = c;
                }
            }
            const long long at = cta_reserve(open, e.cnt + (phase & 1));
            if (open) al2[at] = c;
        }
        if (!bar.sync()) return;
        nact = (int64_t) * (volatile unsigned long long *)(e.cnt + (phase & 1));
        if (nact == 0) break;
        {
            int32_t *t = al;
            al = al2;
            al2 = t;
        }
        for (int64_t ix = g0; ix < nact; ix += gsize) {
            const int c = al[ix];
            const int pd = e.pending[c];
            const u128 acc = acc_of(e, c), st = e.stab[c];
            if (pd == 0) e.S[c] = st > acc ? st : acc;
            e.nxt[c] = pd == 1 ? e.ucand[c] : -1;
            e.Fa[c] = st;
            e.Fc[c] = acc;
        }
        if (lead) e.cnt[(phase & 1) ^ 1] = 0;
        if (!bar.sync()) return;
        int32_t *ni = e.nxt, *no = e.nxt2;
        u128 *ai = e.Fa, *ao = e.Fa2, *ci = e.Fc, *co = e.Fc2;
        for (int it = 0;; it++) {  // at most 32: chains are shorter than 2^31
            bool moved = false;
            for (int64_t ix = g0; ix < nact; ix += gsize) {
                const int c = al[ix];
                int x = ni[c];
                u128 a = ai[c], cc = ci[c];
                if (x >= 0) {
                    const int nx = ni[x];
                    if (nx >= 0) {  // x is unary: compose (x's function applies first)
                        const u128 t = cc + ai[x];
                        a = a > t ? a : t;
                        cc = cc + ci[x];
                        x = nx;
                        moved = true;
                    }
                }
                no[c] = x;
                ao[c] = a;
                co[c] = cc;
            }
            if (__syncthreads_or(moved) && threadIdx.x == 0) *(volatile unsigned long long *)(e.cnt + 2 + it % 3) = 1;
            if (lead) e.cnt[2 + (it + 1) % 3] = 0;
            if (!bar.sync()) return;
            {
                int32_t *t = ni;
                ni = no;
                no = t;
                u128 *u = ai;
                ai = ao;
                ao = u;
                u = ci;
                ci = co;
                co = u;
            }
            if (*(volatile unsigned long long *)(e.cnt + 2 + it % 3) == 0) break;
        }
        for (int64_t ix = g0; ix < nact; ix += gsize) {
            const int c = al[ix];
            const int pd = e.pending[c];
            int f = pd == 0;
            if (pd == 1) {
                const int x = ni[c];
                if (e.pending[x] == 0) {
                    const u128 t = ci[c] + e.S[x];
                    e.S[c] = ai[c] > t ? ai[c] : t;
                    f = 1;
                }
            }
            e.fin[c] = f;
        }
        if (lead) e.cnt[2] = e.cnt[3] = e.cnt[4] = 0;
        if (!bar.sync()) return;
        for (int64_t ix = g0; ix < nact; ix += gsize) {
            const int c = al[ix];
            if (!e.fin[c]) continue;
            e.done[c] = 1;
            const int p = e.par[c];
            if (p < 0 || p >= e.root0) continue;
            acc_add(e, p, e.S[c]);
            if (e.fin[p]) continue;  // resolved in this phase too
            __threadfence();
            if (atomicSub(&e.pending[p], 1) == 1) {
                __threadfence();
                e_walk(e, p);
            }
        }
        if (!bar.sync()) return;
    }
    // highest selected ancestor-or-self
    for (int64_t c = g0; c < e.ncl; c += gsize) {
        const bool sel = c < e.root0 && e.stab[c] >= acc_of(e, c);
        e.slot[c] = ((unsigned long long)(unsigned)e.par[c] << 32) | (unsigned)(sel ? (int)c : -1);
        e.fin[c] = 0;
    }
    if (lead) e.cnt[2] = 0;
    if (!bar.sync()) return;
    for (int round = 0;; round++) {
        if (round > 4096) {
            if (lead) bar.stop(kStopEom);
            return;
        }
        bool cut = false;
        for (int64_t t = g0; t < e.ncl; t += gsize) {
            const int64_t c = e.ncl - 1 - t;
            if (e.fin[c]) continue;
            unsigned long long v = e.slot[c];
            int it = 0;
            while ((int)(v >> 32) >= 0 && it < e.walk) {
                const unsigned long long u = *(volatile unsigned long long *)(e.slot + (v >> 32));
                v = (u & 0xffffffff00000000ull) | ((int)(unsigned)u >= 0 ? (unsigned)u : (unsigned)v);
                atomicExch(e.slot + c, v);  // not a store: other CTAs read these lines meanwhile
                it++;
            }
            if ((int)(v >> 32) >= 0) {
                cut = true;
            } else {
                e.H[c] = (int)(unsigned)v;
                e.fin[c] = 1;
            }
        }
        if (__syncthreads_or(cut) && threadIdx.x == 0) *(volatile unsigned long long *)(e.cnt + 2 + round % 3) = 1;
        if (lead) e.cnt[2 + (round + 1) % 3] = 0;
        if (!bar.sync()) return;
        if (*(volatile unsigned long long *)(e.cnt + 2 + round % 3) == 0) break;
    }
    bar.finish();
}

__global__ void k_e_labels(const unsigned *stop, int64_t E, const int32_t *fall_cluster, const int32_t *cidx,
                           const int32_t *H, int32_t *lab, int *minmem) {
    if (stopped(stop)) return;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < E;
         p += (int64_t)gridDim.x * blockDim.x) {
        int L = H[cidx[fall_cluster[p]]];
        lab[p] = L;
        if (L >= 0 && (int)p < minmem[L]) atomicMin(&minmem[L], (int)p);
    }
}

__global__ void k_e_final_keys(int64_t ncl, const int32_t *H, int *flag) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c <= ncl;
         c += (int64_t)gridDim.x * blockDim.x)
        flag[c] = (c < ncl && H[c] == (int32_t)c) ? 1 : 0;
}

__global__ void k_e_final_emit(int64_t ncl, const int *flag, const long long *pos, const int *minmem,
                               unsigned long long *k, unsigned long long *v) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < ncl;
         c += (int64_t)gridDim.x * blockDim.x) {
        if (!flag[c]) continue;
        k[pos[c]] = (unsigned long long)minmem[c];
        v[pos[c]] = (unsigned long long)c;
    }
}

// Final clusters sorted by smallest member (a global edge id, so graphs
// come in order); a cluster's label is its position within its graph.
__global__ void k_e_gstart(const unsigned *stop, int64_t nf, const unsigned long long *key, const int32_t *egraph,
                           int64_t *gstart, int32_t *gcount) {
    if (stopped(stop)) return;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nf;
         x += (int64_t)gridDim.x * blockDim.x) {
        int g = egraph[key[x]];
        if (x == 0 || egraph[key[x - 1]] != g) gstart[g] = x;
        if (x == nf - 1 || egraph[key[x + 1]] != g) gcount[g] = (int32_t)(x + 1);  // end, fixed below
    }
}
__global__ void k_e_gcount(int G, const int64_t *gstart, int32_t *gcount) {
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x)
        if (gcount[g] > 0) gcount[g] -= (int32_t)gstart[g];
}
__global__ void k_e_rank(const unsigned *stop, int64_t nf, const unsigned long long *key, const unsigned long long *v,
                         const int32_t *egraph, const int64_t *gstart, int32_t *rank) {
    if (stopped(stop)) return;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nf;
         x += (int64_t)gridDim.x * blockDim.x)
        rank[v[x]] = (int32_t)(x - gstart[egraph[key[x]]]);
}

__global__ void k_e_relabel(int64_t E, const int32_t *rank, int32_t *lab) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < E;
         p += (int64_t)gridDim.x * blockDim.x) {
        int L = lab[p];
        lab[p] = L < 0 ? -1 : rank[L];
    }
}

__global__ void k_e_out(Eom e, Gview gv, const int64_t *size, const unsigned long long *cbirth,
                        const unsigned long long *cdeath, const int32_t *H, int32_t *cl_id,
                        int32_t *cl_parent, uint64_t *cl_birth, uint64_t *cl_death, int64_t *cl_size,
                        uint64_t *cl_hi, uint64_t *cl_lo, int32_t *cl_sel) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < e.ncl;
         c += (int64_t)gridDim.x * blockDim.x) {
        int node = e.clist[c];
        cl_id[c] = node;
        cl_parent[c] = e.cparent[node];
        cl_birth[c] = cbirth[node];
        cl_death[c] = cdeath[node];
        cl_size[c] = node_size(node, gv, size);
        cl_hi[c] = (uint64_t)(e.stab[c] >> 64);
        cl_lo[c] = (uint64_t)e.stab[c];
        bool sel = (node < e.R0) && e.stab[c] >= acc_of(e, c);
        cl_sel[c] = !sel ? 0 : (H[c] == (int32_t)c ? 2 : 1);
    }
}

void plan_condensed(Arena &ws, const Problem &p, Condensed &o) {
    int64_t E = p.E;
    o.fall_cluster = ws.take<int32_t>(E);
    o.fall_lambda = ws.take<uint64_t>(E);
    const int64_t C = E + p.G;  // clusters: at most one per merge plus the virtual roots
    o.cl_id = ws.take<int32_t>(C);
    o.cl_parent = ws.take<int32_t>(C);
    o.cl_birth = ws.take<uint64_t>(C);
    o.cl_death = ws.take<uint64_t>(C);
    o.cl_stab_hi = ws.take<uint64_t>(C);
    o.cl_stab_lo = ws.take<uint64_t>(C);
    o.cl_size = ws.take<int64_t>(C);
    o.cl_selected = ws.take<int32_t>(C);
    o.labels = ws.take<int32_t>(E);
    o.gclusters = ws.take<int32_t>(p.G);
}

struct CScratch {
    int32_t *up, *cpar, *link, *cparent, *clist, *cidx, *par, *ucand, *nxt, *nxt2, *H,
        *rank, *al1, *al2;
    int *isrep, *isc, *pending, *done, *fin, *minmem, *flag;
    unsigned long long *cbirth, *cdeath, *st_hi, *st_lo, *acc_hi, *acc_lo, *csz, *cnt, *k1, *k2, *v1, *v2, *jflag;
    long long *cpos, *scan_tmp;
    int64_t *gstart;
    u128 *stab, *S, *Fa, *Fc, *Fa2, *Fc2;
    void *radix;
};
static CScratch carve_condense(Arena &a, const Problem &p) {
    CScratch s;
    int64_t E = p.E, N = 2 * E + p.G + 1;  // nodes: leaves, merges, virtual roots
    s.up = a.take<int32_t>(E);
    s.isrep = a.take<int>(E);
    s.cpar = a.take<int32_t>(N);
    s.link = a.take<int32_t>(N);
    s.isc = a.take<int>(N + 1);
    s.cbirth = a.take<unsigned long long>(N);
    s.cdeath = a.take<unsigned long long>(N);
    s.cparent = a.take<int32_t>(N);
    s.st_hi = a.take<unsigned long long>(N);
    s.st_lo = a.take<unsigned long long>(N);
    s.cpos = a.take<long long>(N + 1);
    s.scan_tmp = a.take<long long>(scan_scratch_elems(N + 1));
    s.clist = a.take<int32_t>(E + p.G + 1);
    s.cidx = a.take<int32_t>(N);
    s.par = a.take<int32_t>(E + p.G + 1);
    s.pending = a.take<int>(E + p.G + 1);
    s.done = a.take<int>(E + p.G + 1);
    s.fin = a.take<int>(E + p.G + 1);
    s.ucand = a.take<int32_t>(E + p.G + 1);
    s.nxt = a.take<int32_t>(E + p.G + 1);
    s.nxt2 = a.take<int32_t>(E + p.G + 1);
    s.stab = a.take<u128>(E + p.G + 1);
    s.S = a.take<u128>(E + p.G + 1);
    s.Fa = a.take<u128>(2 * (E + p.G + 1));  // Fa and Fc adjacent: the node records span both
    s.Fc = s.Fa + (E + p.G + 1);
    s.Fa2 = a.take<u128>(E + p.G + 1);
    s.Fc2 = a.take<u128>(E + p.G + 1);
    s.acc_hi = a.take<unsigned long long>(E + p.G + 1);
    s.acc_lo = a.take<unsigned long long>(E + p.G + 1);
    s.csz = a.take<unsigned long long>(E + p.G + 1);
    s.H = a.take<int32_t>(E + p.G + 1);
    s.minmem = a.take<int>(E + p.G + 1);
    s.flag = a.take<int>(E + p.G + 2);
    s.rank = a.take<int32_t>(E + p.G + 1);
    s.gstart = a.take<int64_t>(p.G + 1);
    s.al1 = a.take<int32_t>(E + p.G + 1);
    s.al2 = a.take<int32_t>(E + p.G + 1);
    s.cnt = a.take<unsigned long long>(8);
    s.jflag = a.take<unsigned long long>(8);
    s.k1 = a.take<unsigned long long>(E + p.G + 1);
    s.k2 = a.take<unsigned long long>(E + p.G + 1);
    s.v1 = a.take<unsigned long long>(E + p.G + 1);
    s.v2 = a.take<unsigned long long>(E + p.G + 1);
    s.radix = a.take<char>(radix_scratch_bytes(E + p.G + 1));
    return s;
}
size_t condense_scratch_bytes(const Problem &p) {
    Arena a(nullptr, 0);
    carve_condense(a, p);
    return a.off;
}

// What the stage counts up from zero, in one pass: per merge or virtual root
// (m of them), per graph, and the counters.
__global__ void k_c_zero(int64_t m, int G, unsigned long long *nbs, int *isc, unsigned long long *cdeath,
                         unsigned long long *st_hi, unsigned long long *st_lo, int32_t *gclusters,
                         unsigned long long *cnt, unsigned long long *jflag) {
    const int64_t x0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = x0; i < m; i += stride) {
        nbs[i] = 0;
        isc[i] = 0;
        cdeath[i] = 0;  // (a cluster is a merge or a virtual root, never a leaf)
        st_hi[i] = 0;
        st_lo[i] = 0;
    }
    for (int64_t g = x0; g < G; g += stride) gclusters[g] = 0;
    if (x0 < 8) cnt[x0] = jflag[x0] = 0;
    if (x0 == 0) isc[m] = 0;
}

dgec_status stage_condense(Ctx *c, const Problem &p, const Msf &m, const Dendro &d, Condensed &o,
                           void *scratch) {
    cudaStream_t st = c->stream;
    int64_t E = p.E, n = m.n, N = E + n + p.G;
    o.n_cl = 0;
    o.n_clusters = 0;
    if (E == 0) {
        CU_TRY(c, cudaMemsetAsync(o.gclusters, 0, sizeof(int32_t) * p.G, st));
        return DGEC_OK;
    }
    Gview gv{E, n, E + n, p.G, p.egraph, m.u, p.eoff, p.gM};
    Arena a(scratch, SIZE_MAX);
    CScratch s = carve_condense(a, p);
    const int gN = grid_for(N, kBlock, kStreamCap), gE = grid_for(E, kBlock, kStreamCap),
              gn = grid_for(n + p.G, kBlock, kStreamCap);
    // big-child counts and sizes of node ids E .. N: in cpos, unused until the cluster scan
    unsigned long long *nbs = reinterpret_cast<unsigned long long *>(s.cpos);
    TK(c, "k_c_zero", k_c_zero<<<gn, kBlock, 0, st>>>(n + p.G, p.G, nbs, s.isc + E, s.cdeath + E, s.st_hi + E, s.st_lo + E,
                                                     o.gclusters, s.cnt, s.jflag));
    // (the lists of cut walks lie in al1, which the EOM pass takes later)
    if (n > 0) {
        TK(c, "k_c_up", k_c_up<<<gn, kBlock, 0, st>>>(E, n, d.parent, m.w, s.up, s.isrep));
        DG_TRY(jump_to_fixed(c, n, 0, SelAll{}, s.up, s.al1, s.jflag));
    }
    TK(c, "k_c_cpar", k_c_cpar<<<gN, kBlock, 0, st>>>(gv, d.parent, s.up, s.isrep, d.size, s.cpar, nbs));
    TK(c, "k_c_link", k_c_link<<<gn, kBlock, 0, st>>>(c->stop(), gv, s.isrep, d.size, s.cpar, nbs, s.link));
    DG_TRY(jump_to_fixed(c, n, E, SelBigRep{gv, s.isrep, d.size}, s.link, s.al1, s.jflag + 4));
    TK(c, "k_c_clusters", k_c_clusters<<<gn, kBlock, 0, st>>>(c->stop(), gv, s.isrep, d.size, m.w, s.cpar, nbs, s.link,
                                                             s.isc, s.cbirth, s.cdeath, s.cparent));
    // the node records live in the EOM phase's Fa and Fc arrays (adjacent, not in use yet)
    NodeRec *nrec = reinterpret_cast<NodeRec *>(s.Fa);
    TK(c, "k_c_nrec", k_c_nrec<<<gn, kBlock, 0, st>>>(c->stop(), gv, s.isrep, d.size, m.w, s.cpar, s.link, s.cbirth, nbs,
                                                     nrec, s.st_hi, s.st_lo));
    TK(c, "k_c_points", k_c_points<<<gE, kBlock, 0, st>>>(c->stop(), gv, s.cpar, nrec, o.fall_cluster, o.fall_lambda));
    // cluster flags of node ids E .. N (the last one a zero sentinel)
    DG_TRY(exclusive_scan_i32(c, s.isc + E, s.cpos, n + p.G + 1, s.scan_tmp));
    int64_t ncl;
    DG_TRY(read_counters(c, (const int64_t *)(s.cpos + n + p.G), 1, &ncl));
    TK(c, "k_c_compact", k_c_compact<<<gn, kBlock, 0, st>>>(E, n + p.G, ncl, s.isc + E, s.cpos, s.clist, s.cidx,
                                                           s.csz, s.minmem));
    o.n_cl = ncl;
    TK(c, "k_c_kids", k_c_kids<<<grid_for(ncl, kBlock, kStreamCap), kBlock, 0, st>>>(ncl, gv, s.clist, s.cparent, s.cidx,
                                                                                d.size, s.par, s.csz));
    // ---- excess of mass over the cluster tree
    Eom e;
    e.ncl = ncl;
    e.root0 = ncl - p.G;  // every virtual root is a cluster, and their node ids are the last
    e.R0 = E + n;
    e.clist = s.clist;
    e.cparent = s.cparent;
    e.par = s.par;
    e.pending = s.pending;
    e.done = s.done;
    e.fin = s.fin;
    e.stab = s.stab;
    e.S = s.S;
    e.Fa = s.Fa;
    e.Fc = s.Fc;
    e.Fa2 = s.Fa2;
    e.Fc2 = s.Fc2;
    e.kids = s.csz;
    e.acc_hi = s.acc_hi;
    e.acc_lo = s.acc_lo;
    e.ucand = s.ucand;
    e.nxt = s.nxt;
    e.nxt2 = s.nxt2;
    e.al = s.al1;
    e.al2 = s.al2;
    e.slot = s.k1;
    e.H = s.H;
    e.cnt = s.cnt;
    const int gc = grid_for(ncl + 1, kBlock, kStreamCap);
    TK(c, "k_e_init", k_e_init<<<gc, kBlock, 0, st>>>(e, s.st_hi, s.st_lo, s.cbirth, s.cdeath));
    {
        int grid = 1;
        e.bar = c->next_bar();
        e.walk = c->walk(kTopWalk);
        DG_TRY(coop_grid(c, kCoopEom, (const void *)k_e_tree, kBlock, 0, &grid));
        const int64_t want = cdiv(ncl, kBlock);  // (two clusters a thread: 0.070 ms instead of 0.058 at 20,000 edges)
        DG_TRY(coop_launch(c, "k_e_tree", (const void *)k_e_tree, want < grid ? (int)want : grid, kBlock, 0, e));
    }
    TK(c, "k_e_labels", k_e_labels<<<gE, kBlock, 0, st>>>(c->stop(), E, o.fall_cluster, s.cidx, s.H, o.labels, s.minmem));
    TK(c, "k_e_final_keys", k_e_final_keys<<<gc, kBlock, 0, st>>>(ncl, s.H, s.flag));
    DG_TRY(exclusive_scan_i32(c, s.flag, s.cpos, ncl + 1, s.scan_tmp));
    int64_t nf;
    DG_TRY(read_counters(c, (const int64_t *)(s.cpos + ncl), 1, &nf));
    o.n_clusters = (int32_t)nf;
    if (nf > 0) {
        TK(c, "k_e_final_emit", k_e_final_emit<<<gc, kBlock, 0, st>>>(ncl, s.flag, s.cpos, s.minmem, s.k1, s.v1));
        bool in_b;
        DG_TRY(radix_sort(c, RadixBuffers{s.k1, s.k2, s.v1, s.v2}, nf, 0, p.idbits > 0 ? p.idbits : 1,
                          s.radix, &in_b));
        unsigned long long *kk = in_b ? s.k2 : s.k1, *vv = in_b ? s.v2 : s.v1;
        const int gf = grid_for(nf, kBlock, kStreamCap);
        TK(c, "k_e_gstart", k_e_gstart<<<gf, kBlock, 0, st>>>(c->stop(), nf, kk, p.egraph, s.gstart, o.gclusters));
        TK(c, "k_e_gcount", k_e_gcount<<<grid_for(p.G), kBlock, 0, st>>>(p.G, s.gstart, o.gclusters));
        TK(c, "k_e_rank", k_e_rank<<<gf, kBlock, 0, st>>>(c->stop(), nf, kk, vv, p.egraph, s.gstart, s.rank));
        TK(c, "k_e_relabel", k_e_relabel<<<gE, kBlock, 0, st>>>(E, s.rank, o.labels));
    }
    TK(c, "k_e_out", k_e_out<<<gc, kBlock, 0, st>>>(e, gv, d.size, s.cbirth, s.cdeath, s.H, o.cl_id, o.cl_parent,
                                   o.cl_birth, o.cl_death, o.cl_size, o.cl_stab_hi, o.cl_stab_lo,
                                   o.cl_selected));
    return DGEC_OK;
}

}  // namespace dgec
