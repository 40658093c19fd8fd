// Stage C: minimum spanning forest of the undirected skeleton (Alg. 1)
// by Borůvka rounds, then sorted by (w, u, v) as Alg. 1 orders it.
//
// The order (w, min id, max id) is strict (a pair appears once in L*), so
// the forest is unique. Each round: every live edge between two components
// bids its key into both, each component hooks along its winning edge, a
// mutual pair keeps the smaller label as root, labels are pointer-jumped to
// their roots, and edges inside one component are dropped while the survivors
// are compacted for the next round. The pipeline's forms are the k_m_*
// rounds while many edges live and k_m_forest after that; the kernels before
// them serve dgec_msf_static.
#include <algorithm>
#include <utility>

#include "coop.cuh"
#include "stages.cuh"

namespace dgec {

constexpr unsigned long long kMax64 = 0xFFFFFFFFFFFFFFFFull;

// A forest edge as the rounds append it: original ends (u < v), internal
// ends, weight. One 32-byte record, so that it is written and gathered (by
// sorted index, after the rounds) as one sector.
struct __align__(32) FEdge {
    int32_t u, v, ru, rv;
    int64_t w, pad;
};
__device__ __forceinline__ void put_fedge(FEdge *p, int u, int v, int ru, int rv, int64_t w) {
    store_sector(p, pack_i32(u, v), pack_i32(ru, rv), (unsigned long long)w, 0ull);
}

// Drop edges inside one component; compact the rest; bid w. In the first
// round every node is its own component, so the label reads are skipped.
template <bool FIRST>
__device__ __forceinline__ void filter_bid(const int32_t *u, const int32_t *v, const int64_t *w,
                                           int64_t n, const int32_t *comp, int32_t *u2, int32_t *v2,
                                           int64_t *w2, unsigned long long *cnt,
                                           unsigned long long *bw) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t wb = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; wb < n;
         wb += stride) {
        int64_t x = wb + lane_id();
        bool keep = false;
        int a = 0, b = 0, ca = 0, cb = 0;
        int64_t ww = 0;
        if (x < n) {
            a = u[x];
            b = v[x];
            ww = w[x];
            ca = FIRST ? a : comp[a];
            cb = FIRST ? b : comp[b];
            keep = ca != cb;
        }
        unsigned m = __ballot_sync(0xffffffffu, keep);
        if (m == 0) continue;
        int leader = __ffs(m) - 1;
        unsigned long long base = 0;
        if ((int)lane_id() == leader) base = atomicAdd(cnt, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (keep) {
            int64_t at = (int64_t)base + __popc(m & ((1u << lane_id()) - 1u));
            u2[at] = a;
            v2[at] = b;
            w2[at] = ww;
            // read first: most bids into a large component cannot win, and
            // skipping them keeps one hot slot from serialising the grid
            // (the slot only decreases, so a stale read never skips a winner)
            unsigned long long uw = (unsigned long long)ww;
            if (uw < bw[ca]) atomicMin(&bw[ca], uw);
            if (uw < bw[cb]) atomicMin(&bw[cb], uw);
        }
    }
}

__global__ void k_filter_bid(const int32_t *u, const int32_t *v, const int64_t *w, int64_t n,
                             const int32_t *comp, int32_t *u2, int32_t *v2, int64_t *w2,
                             unsigned long long *cnt, unsigned long long *bw) {
    filter_bid<false>(u, v, w, n, comp, u2, v2, w2, cnt, bw);
}
__global__ void k_bid_uv(const int32_t *u, const int32_t *v, const int64_t *w, int64_t n,
                         const int32_t *comp, const unsigned long long *bw,
                         unsigned long long *buv) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        int a = u[x], b = v[x];
        unsigned long long ww = (unsigned long long)w[x];
        int ca = comp[a], cb = comp[b];
        unsigned long long key = ((unsigned long long)(unsigned)a << 32) | (unsigned)b;
        if (ww == bw[ca] && key < buv[ca]) atomicMin(&buv[ca], key);
        if (ww == bw[cb] && key < buv[cb]) atomicMin(&buv[cb], key);
    }
}

// Each component root with a winning edge hooks to the other side and, once
// per forest edge, appends it to the output.
__global__ void k_hook(int64_t E, const int32_t *comp, const unsigned long long *bw,
                       const unsigned long long *buv, int32_t *par, int32_t *mu, int32_t *mv,
                       int64_t *mw, unsigned long long *n_out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < E;
         base += stride) {
        int64_t x = base + lane_id();
        bool emit = false;
        int a = 0, b = 0;
        unsigned long long ww = 0;
        if (x < E && comp[x] == (int32_t)x) {
            if (bw[x] == kMax64) {
                par[x] = (int32_t)x;
            } else {
                unsigned long long key = buv[x];
                a = (int)(key >> 32);
                b = (int)(key & 0xffffffffu);
                int ca = comp[a], cb = comp[b];
                int partner = ca == (int)x ? cb : ca;
                bool mutual = buv[partner] == key;
                par[x] = (mutual && (int)x < partner) ? (int32_t)x : partner;
                emit = !mutual || (int)x < partner;
                ww = bw[x];
            }
        }
        // one counter update per warp for the forest edges it appends
        unsigned m = __ballot_sync(0xffffffffu, emit);
        if (!m) continue;
        int leader = __ffs(m) - 1;
        unsigned long long at = 0;
        if ((int)lane_id() == leader) at = atomicAdd(n_out, (unsigned long long)__popc(m));
        at = __shfl_sync(0xffffffffu, at, leader);
        if (emit) {
            at += __popc(m & ((1u << lane_id()) - 1u));
            mu[at] = a;
            mv[at] = b;
            mw[at] = (int64_t)ww;
        }
    }
}

// Pointer jumping: every root walks to its new root, compressing its own
// pointer as it goes (pointers only ever move toward a root).
__global__ void k_jump(int64_t E, const int32_t *comp, int32_t *par) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < E;
         x += (int64_t)gridDim.x * blockDim.x) {
        if (comp[x] != (int32_t)x) continue;
        int r = par[x];
        for (int it = 0; it < kMaxWalk; it++) {  // bounded: pointers form a forest
            int rr = par[r];
            if (rr == r) break;
            r = rr;
            par[x] = r;
        }
    }
}

__global__ void k_relabel(int64_t E, int32_t *comp, const int32_t *par, unsigned long long *bw,
                          unsigned long long *buv) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < E;
         x += (int64_t)gridDim.x * blockDim.x) {
        int c = comp[x];
        comp[x] = par[c];
    }
}

__global__ void k_reset_best(int64_t E, unsigned long long *bw, unsigned long long *buv) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < E;
         x += (int64_t)gridDim.x * blockDim.x) {
        bw[x] = kMax64;
        buv[x] = kMax64;
    }
}

__global__ void k_iota(int64_t E, int32_t *comp) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < E;
         x += (int64_t)gridDim.x * blockDim.x)
        comp[x] = (int32_t)x;
}

// ----- the pipeline's forest stage: nodes are internal ids r; each edge
// carries its original ends (u < v) for the (w, u, v) tie-break key.

// ---- large rounds: one kernel a step (more threads resident than the
// cooperative kernel below allows, which the random accesses need here)

// Edges carry the labels (cu, cv) of the components at their ends; the
// labels move one hop per round (par of the old root), so no per-node
// label array is swept. Live edges: (cu, cv) labels, (u, v) original ends
// (the tie-break key), w.

// Bid w into both ends (round 1: every node is a root and nothing is
// filtered yet).
__global__ void k_m_bid(const int32_t *cu, const int32_t *cv, const int64_t *w, int64_t n,
                        unsigned long long *bw) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        int a = cu[x], b = cv[x];
        unsigned long long uw = (unsigned long long)w[x];
        if (uw < bw[a]) atomicMin(&bw[a], uw);
        if (uw < bw[b]) atomicMin(&bw[b], uw);
    }
}

// Items per thread between two slot reservations of the compacting
// kernels below (one atomic on the shared counter per 2,048 items).
constexpr int kRes8 = 8;

// Move labels one hop to the merged roots, drop edges inside one
// component, compact the rest and bid w.
__global__ void k_m_filter_bid(const int32_t *cu, const int32_t *cv, const int32_t *u, const int32_t *v,
                               const int64_t *w, int64_t n, const int32_t *par, int32_t *cu2,
                               int32_t *cv2, int32_t *u2, int32_t *v2, int64_t *w2,
                               unsigned long long *cnt, unsigned long long *bw) {
    const int64_t tile = (int64_t)blockDim.x * kRes8;
    for (int64_t base = (int64_t)blockIdx.x * tile; base < n; base += (int64_t)gridDim.x * tile) {  // CTA-uniform
        int a[kRes8], b[kRes8];
        unsigned keep = 0;
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            const int64_t x = base + (int64_t)q * blockDim.x + threadIdx.x;
            a[q] = b[q] = 0;
            if (x < n) {
                a[q] = par[cu[x]];
                b[q] = par[cv[x]];
                if (a[q] != b[q]) keep |= 1u << q;
            }
        }
        long long at = cta_reserve_count(__popc(keep), cnt);
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            if (!((keep >> q) & 1u)) continue;
            const int64_t x = base + (int64_t)q * blockDim.x + threadIdx.x;
            const unsigned long long uw = (unsigned long long)w[x];
            cu2[at] = a[q];
            cv2[at] = b[q];
            u2[at] = u[x];
            v2[at] = v[x];
            w2[at] = (int64_t)uw;
            at++;
            if (uw < bw[a[q]]) atomicMin(&bw[a[q]], uw);
            if (uw < bw[b[q]]) atomicMin(&bw[b[q]], uw);
        }
    }
}

__global__ void k_m_bid_uv(const int32_t *cu, const int32_t *cv, const int32_t *u, const int32_t *v,
                           const int64_t *w, int64_t n, const unsigned long long *bw,
                           unsigned long long *buv) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long ww = (unsigned long long)w[x];
        int a = cu[x], b = cv[x];
        bool wa = ww == bw[a], wb = ww == bw[b];
        if (!wa && !wb) continue;
        unsigned long long key = ((unsigned long long)(unsigned)u[x] << 32) | (unsigned)v[x];
        if (wa && key < buv[a]) atomicMin(&buv[a], key);
        if (wb && key < buv[b]) atomicMin(&buv[b], key);
    }
}

// The edge that won a root's bid records itself there (one writer: keys
// are unique), with the label on its other end.
__global__ void k_m_claim(const int32_t *cu, const int32_t *cv, const int32_t *u, const int32_t *v,
                          int64_t n, const unsigned long long *buv, int32_t *bp, int32_t *win) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        int a = cu[x], b = cv[x];
        unsigned long long key = ((unsigned long long)(unsigned)u[x] << 32) | (unsigned)v[x];
        if (buv[a] == key) {
            bp[a] = b;
            win[a] = (int32_t)x;
        }
        if (buv[b] == key) {
            bp[b] = a;
            win[b] = (int32_t)x;
        }
    }
}

// Over the current roots: hook along the winner (a mutual pair keeps the
// smaller label), append each forest edge once. Each thread first issues
// all its loads (8 roots), then writes: the loads of one tile are in flight
// together. In the first round (orig_of given) every label is a node, so the
// root and its partner are the edge's internal ids, and orig_of, read in
// order, says which is which; later rounds read both from rank_of at random
// (the first one too: 5.5 ms of hooks instead of 4.7 at 100M edges).
__global__ void k_m_hook(const int32_t *__restrict__ roots, int64_t nr, const unsigned long long *__restrict__ bw,
                         const unsigned long long *__restrict__ buv, const int32_t *__restrict__ bp,
                         const int32_t *__restrict__ win, const int32_t *__restrict__ u,
                         const int32_t *__restrict__ v, const int64_t *__restrict__ w,
                         const int32_t *__restrict__ rank_of, const int32_t *__restrict__ orig_of,
                         int32_t *__restrict__ par, FEdge *__restrict__ fe, unsigned long long *n_out) {
    const int64_t tile = (int64_t)blockDim.x * kRes8;
    for (int64_t base = (int64_t)blockIdx.x * tile; base < nr; base += (int64_t)gridDim.x * tile) {  // CTA-uniform
        int xs[kRes8], ps[kRes8], wx[kRes8];
        unsigned live = 0, mutual = 0;
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            const int64_t ix = base + (int64_t)q * blockDim.x + threadIdx.x;
            xs[q] = ix < nr ? roots[ix] : -1;
        }
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            ps[q] = wx[q] = 0;
            if (xs[q] < 0) continue;
            if (bw[xs[q]] != kMax64) {
                live |= 1u << q;
                ps[q] = bp[xs[q]];
                wx[q] = win[xs[q]];
            }
        }
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            if (!((live >> q) & 1u)) continue;
            const int x = xs[q], p = ps[q];
            if (bp[p] == x && buv[p] == buv[x]) mutual |= 1u << q;
        }
        unsigned emit = 0;
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            if (xs[q] < 0) continue;
            const int x = xs[q];
            if (!((live >> q) & 1u)) {
                par[x] = x;
                continue;
            }
            const bool mu = (mutual >> q) & 1u;
            par[x] = (mu && x < ps[q]) ? x : ps[q];
            if (!mu || x < ps[q]) emit |= 1u << q;
        }
        long long at = cta_reserve_count(__popc(emit), n_out);
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            if (!((emit >> q) & 1u)) continue;
            const int a = u[wx[q]], b = v[wx[q]];
            int ra, rb;
            if (orig_of) {
                const bool own = orig_of[xs[q]] == a;
                ra = own ? xs[q] : ps[q];
                rb = own ? ps[q] : xs[q];
            } else {
                ra = rank_of[a];
                rb = rank_of[b];
            }
            put_fedge(fe + at++, a, b, ra, rb, w[wx[q]]);
        }
    }
}

// Roots walk to their new root (own pointer compressed on the way). Walks are
// cut after kMWalk steps and left to k_m_settle: on a long chain the threads
// running meet only pointers as short as their own, and the last of them walks
// all of it (3M roots: 2.3 s). The few cut walks of 200M hub edges settle in
// 0.06 ms, 9 launches included.
constexpr int kMWalk = 64;
// OWN: the limit is kMWalk, known when the loop is compiled.
template <bool OWN>
__global__ void k_m_jump(const int32_t *roots, int64_t nr, int32_t *par, int steps, int32_t *list, unsigned long long *cut) {
    const int limit = OWN ? kMWalk : steps;
    for (int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; ix < nr;
         ix += (int64_t)gridDim.x * blockDim.x) {
        int x = roots[ix];
        int r = par[x];
        int it = 0;
        for (; it < limit; it++) {
            int rr = par[r];
            if (rr == r) break;
            r = rr;
            atomicExch(par + x, r);  // not a store: other CTAs read these lines meanwhile
        }
        if (it == limit) list_cut(list, cut, x);
    }
}
// Jumping rounds for the walks that were cut (cut[1 .. 3]: their flags): nothing
// to do unless some were.
__global__ void __launch_bounds__(kBlock) k_m_settle(const int32_t *list, int32_t *par, unsigned long long *cut, BarRef ref) {
    const int64_t n = (int64_t)cut[0];
    if (n == 0) return;  // the same for every CTA: written before this launch
    GridBar bar(ref);
    if (bar.stopped()) return;
    const JumpEnd e = jump_rounds(bar, n, ListItem{list}, par, cut + 1);
    if (e == kJumpBarrier) return;
    if (e == kJumpBound && threadIdx.x == 0) bar.stop(kStopJump);
    bar.finish();
}

// Next round's roots (old roots that stayed roots); every old root's bid
// slots are cleared. Loads first, then stores (see k_m_hook).
__global__ void k_m_next_roots(const int32_t *__restrict__ roots, int64_t nr, const int32_t *__restrict__ par,
                               unsigned long long *__restrict__ bw, unsigned long long *__restrict__ buv,
                               int32_t *__restrict__ roots2, unsigned long long *cnt) {
    const int64_t tile = (int64_t)blockDim.x * kRes8;
    for (int64_t base = (int64_t)blockIdx.x * tile; base < nr; base += (int64_t)gridDim.x * tile) {  // CTA-uniform
        int xs[kRes8];
        unsigned keep = 0;
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            const int64_t ix = base + (int64_t)q * blockDim.x + threadIdx.x;
            xs[q] = ix < nr ? roots[ix] : -1;
        }
#pragma unroll
        for (int q = 0; q < kRes8; q++)
            if (xs[q] >= 0 && par[xs[q]] == xs[q] && bw[xs[q]] != kMax64) keep |= 1u << q;
#pragma unroll
        for (int q = 0; q < kRes8; q++) {
            if (xs[q] < 0) continue;
            bw[xs[q]] = kMax64;
            buv[xs[q]] = kMax64;
        }
        long long at = cta_reserve_count(__popc(keep), cnt);
#pragma unroll
        for (int q = 0; q < kRes8; q++)
            if ((keep >> q) & 1u) roots2[at++] = xs[q];
    }
}

__global__ void k_m_init(int64_t E, int32_t *par, int32_t *roots, unsigned long long *bw,
                         unsigned long long *buv) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < E;
         x += (int64_t)gridDim.x * blockDim.x) {
        par[x] = (int32_t)x;
        roots[x] = (int32_t)x;
        bw[x] = kMax64;
        buv[x] = kMax64;
    }
}

// ---- the other rounds, in one cooperative kernel

typedef unsigned __int128 u128;

struct MsfArgs {
    int64_t nr0, n0;
    const int32_t *roots0;           // the roots to begin with (null: 0 .. nr0-1)
    const int32_t *ru, *rv, *u, *v;  // the edges to begin with: labels of the ends, original ends
    const int64_t *w;
    const int32_t *rank_of;
    int32_t *par, *roots, *roots2, *bp;
    ulonglong2 *slot, *slot2;  // best key bid at each root (all ones: none), one for each round parity
    int2 *la, *lb;          // live edges: labels
    ulonglong2 *ka, *kb;    // live edges: keys without the label
    FEdge *fe;
    unsigned long long *cnt;  // [0], [1] live edges, [2], [3] (next roots << 32) | forest edges of the round,
                              // [4] forest edges, [5] error, [6] a walk was cut; if so [7] rounds begun, [8] the
                              // last one's live edges, [9] next roots; all but [4] zeroed before
    int ib, lbits;            // bits of an original id, of the label in a key (0: none)
    int walk;                 // limit of a walk
    BarRef bar;
};

__device__ __forceinline__ u128 as_u128(ulonglong2 x) { return ((u128)x.y << 64) | x.x; }
__device__ __forceinline__ ulonglong2 as_pair(u128 x) {
    return make_ulonglong2((unsigned long long)x, (unsigned long long)(x >> 64));
}
__device__ __forceinline__ u128 cas_u128(ulonglong2 *p, u128 cmp, u128 val) {
    unsigned long long lo, hi;
    asm volatile(
        "{\n\t.reg .b128 c, v, o;\n\t"
        "mov.b128 c, {%2, %3};\n\t"
        "mov.b128 v, {%4, %5};\n\t"
        "atom.relaxed.gpu.global.cas.b128 o, [%6], c, v;\n\t"
        "mov.b128 {%0, %1}, o;\n\t}"
        : "=l"(lo), "=l"(hi)
        : "l"((unsigned long long)cmp), "l"((unsigned long long)(cmp >> 64)), "l"((unsigned long long)val),
          "l"((unsigned long long)(val >> 64)), "l"(p)
        : "memory");
    return ((u128)hi << 64) | lo;
}
// A slot as one value (a plain 16-byte read may mix words of two writes).
__device__ __forceinline__ u128 whole_u128(const ulonglong2 *p) {
    unsigned long long lo, hi;
    asm volatile(
        "{\n\t.reg .b128 o;\n\t"
        "ld.relaxed.gpu.global.b128 o, [%2];\n\t"
        "mov.b128 {%0, %1}, o;\n\t}"
        : "=l"(lo), "=l"(hi)
        : "l"(p)
        : "memory");
    return ((u128)hi << 64) | lo;
}
// Minima of two keys into two slots, their reads and their swaps in flight
// together. The read before skips bids that cannot win (most, at a large
// component). It trusts the high word alone, which only falls: the two words
// of the read need not belong together, so where the high words tie, a swap
// of the value for itself reads it whole. FIRST: every label is a node, and
// very many edges of one weight can meet at one of them, whose swaps would wait
// for one another; there a bid that seems lost reads the slot whole instead
// (3M in-edges of one time: k_m_forest 1.28 ms with swaps alone, 0.43 so;
// in every round 0.40, but 2M mixed edges then 1.02 ms instead of 0.99).
template <bool FIRST>
__device__ __forceinline__ void bid_u128(ulonglong2 *sa, u128 ka, ulonglong2 *sb, u128 kb) {
    const ulonglong2 pa = *sa, pb = *sb;
    bool ga = (unsigned long long)(ka >> 64) <= pa.y, gb = (unsigned long long)(kb >> 64) <= pb.y;
    u128 ca = as_u128(pa), cb = as_u128(pb), oa = 0, ob = 0;
    if (FIRST && ga && ka >= ca) ga = ka < (ca = whole_u128(sa));
    if (FIRST && gb && kb >= cb) gb = kb < (cb = whole_u128(sb));
    if (ga) oa = cas_u128(sa, ca, ka < ca ? ka : ca);
    if (gb) ob = cas_u128(sb, cb, kb < cb ? kb : cb);
    // a swap that took place wrote the smaller of the two; else go on from the value it met
    if (ga && oa != ca)
        for (ca = oa; ka < ca; ca = oa)
            if ((oa = cas_u128(sa, ca, ka)) == ca) break;
    if (gb && ob != cb)
        for (cb = ob; kb < cb; cb = ob)
            if ((ob = cas_u128(sb, cb, kb)) == cb) break;
}

// Limit of a walk in k_m_forest. A path of 3M edges whose gaps fall took 1.3 s
// there; it and k_m_labels take 1.2 ms cut at 256 steps (0.77 at 64, but then
// relays of 30,000 edges stop and start again too, for 0.03 ms more).
constexpr int kMCut = 256;
// The root above label x after the hooks; x's own pointer is moved there when
// the way was longer than one step (by an exchange, not a store: other CTAs
// read these lines meanwhile). A walk is cut after `limit` steps, which *cut
// then says; what is returned is an ancestor short of the root.
__device__ __forceinline__ int new_root(int32_t *par, int x, int limit, unsigned long long *cut) {
    const int p = par[x];
    int r = p;
    for (int it = 0;; it++) {
        const int rr = par[r];
        if (rr == r) break;
        r = rr;
        if ((it & 7) == 7) atomicExch(par + x, r);
        if (it == limit) {
            *(volatile unsigned long long *)cut = 1;
            break;
        }
    }
    if (r != p) atomicExch(par + x, r);
    return r;
}

// Borůvka, all rounds in one cooperative kernel. A root's slot takes the
// smallest bid by 128-bit compare-and-swap: the bid packs (w, u, v) and, in
// its low bits, the label at the edge's other end, so one pass over the live
// edges bids, and the roots then hook from the slots alone. (When the bits do
// not fit -- w bits + 3 id bits > 127 -- the label is left out and a pass over
// the live edges tells each root its winner's other end.) Per round:
//   hook:   each root follows its best edge; a mutual pair keeps the smaller
//           label as root, which is next round's list; every forest edge is
//           appended once;
//   filter: every live edge's labels walk to their new roots (leaving
//           shortcuts), edges inside one component are dropped, the rest is
//           compacted and bids again, in the slots the hooks have cleared.
// If a walk of the filter was cut, the kernel stops there, k_m_labels settles
// the pointers by jumping rounds and does the filter, and the rounds start
// again from its edges (the jumping rounds as a call in here: 0.82 instead of
// 0.65 ms for the last rounds of 20M edges, for the registers).
constexpr int kRes = 1;          // items a thread handles between slot reservations (20,000 edges: 0.15 ms at 1, 0.19 at 2, 0.34 at 4)
__global__ void __launch_bounds__(kBlock, 4) k_m_forest(MsfArgs a) {
    GridBar bar(a.bar);
    if (bar.stopped()) return;
    const int64_t gsize = (int64_t)gridDim.x * blockDim.x, g0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t tile = (int64_t)blockDim.x * kRes;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    const int ib = a.ib, lb = a.lbits;
    const u128 none = ~(u128)0;
    const unsigned lmask = (1u << lb) - 1u, imask = (unsigned)((1ull << ib) - 1ull);
    for (int64_t ix = g0; ix < a.nr0; ix += gsize) {
        const int x = a.roots0 ? a.roots0[ix] : (int)ix;
        a.par[x] = x;
        a.slot[x] = as_pair(none);
    }
    if (!bar.sync()) return;
    auto pack = [&](int64_t x) {
        return ((((u128)(unsigned long long)a.w[x] << ib | (unsigned)a.u[x]) << ib) | (unsigned)a.v[x]) << lb;
    };
    for (int64_t x = g0; x < a.n0; x += gsize) {
        const int cu = a.ru[x], cv = a.rv[x];
        const u128 key = pack(x);
        bid_u128<true>(a.slot + cu, key | (lb ? (unsigned)cv : 0u), a.slot + cv, key | (lb ? (unsigned)cu : 0u));
    }
    if (!bar.sync()) return;
    int64_t n = a.n0, nr = a.nr0, nfe = (int64_t)a.cnt[4];
    ulonglong2 *slot = a.slot, *slot2 = a.slot2;
    const int32_t *roots = a.roots0;
    int32_t *rout = a.roots, *rnext = a.roots2;
    int2 *lin = a.la, *lout = a.lb;
    ulonglong2 *kin = a.ka, *kout = a.kb;
    for (int round = 0;; round++) {
        if (round >= 64) {
            if (lead) a.cnt[5] = 1;
            break;
        }
        if (!lb) {  // the winner of each slot records the label at its other end
            for (int64_t x = g0; x < n; x += gsize) {
                const int2 l = round ? lin[x] : make_int2(a.ru[x], a.rv[x]);
                const u128 key = round ? as_u128(kin[x]) : pack(x);
                if (as_u128(slot[l.x]) == key) a.bp[l.x] = l.y;
                if (as_u128(slot[l.y]) == key) a.bp[l.y] = l.x;
            }
            if (!bar.sync()) return;
        }
        for (int64_t base = (int64_t)blockIdx.x * tile; base < nr; base += gsize * kRes) {  // CTA-uniform
            int xs[kRes], ps[kRes];
            u128 key[kRes];
            unsigned emit = 0, stay = 0;
#pragma unroll
            for (int q = 0; q < kRes; q++) {
                const int64_t ix = base + (int64_t)q * blockDim.x + threadIdx.x;
                xs[q] = ix < nr ? (roots ? roots[ix] : (int)ix) : -1;
            }
#pragma unroll
            for (int q = 0; q < kRes; q++) {
                key[q] = xs[q] >= 0 ? as_u128(slot[xs[q]]) : none;
                ps[q] = -1;
                if (key[q] != none) ps[q] = lb ? (int)((unsigned)key[q] & lmask) : a.bp[xs[q]];
            }
#pragma unroll
            for (int q = 0; q < kRes; q++) {
                if (ps[q] < 0) continue;  // no edge left: par[x] stays x
                const bool mutual = (as_u128(slot[ps[q]]) >> lb) == (key[q] >> lb);
                if (!mutual || xs[q] < ps[q]) emit |= 1u << q;
                if (!mutual || xs[q] > ps[q]) a.par[xs[q]] = ps[q];
                else stay |= 1u << q;
            }
            const unsigned long long at2 = cta_reserve_pair(__popc(emit), __popc(stay), a.cnt + 2 + (round & 1));
            int64_t at = nfe + (int64_t)(unsigned)at2, rat = (int64_t)(at2 >> 32);
#pragma unroll
            for (int q = 0; q < kRes; q++) {
                if ((stay >> q) & 1u) {
                    slot2[xs[q]] = as_pair(none);
                    rout[rat++] = xs[q];
                }
                if (!((emit >> q) & 1u)) continue;
                const u128 k = key[q] >> lb;
                const int u = (int)((unsigned)(k >> ib) & imask), v = (int)((unsigned)k & imask);
                put_fedge(a.fe + at++, u, v, a.rank_of[u], a.rank_of[v], (int64_t)(unsigned long long)(k >> (2 * ib)));
            }
        }
        if (lead) a.cnt[round & 1] = 0;  // the live count written in this round's filter
        if (!bar.sync()) return;
        {
            const unsigned long long c = *(volatile unsigned long long *)(a.cnt + 2 + (round & 1));
            nr = (int64_t)(c >> 32);
            nfe += (int64_t)(unsigned)c;
        }
        for (int64_t base = (int64_t)blockIdx.x * tile; base < n; base += gsize * kRes) {  // CTA-uniform
            int ca[kRes], cb[kRes];
            unsigned keep = 0;
#pragma unroll
            for (int q = 0; q < kRes; q++) {
                const int64_t x = base + (int64_t)q * blockDim.x + threadIdx.x;
                ca[q] = cb[q] = 0;
                if (x < n) {
                    const int2 l = round ? lin[x] : make_int2(a.ru[x], a.rv[x]);
                    ca[q] = new_root(a.par, l.x, a.walk, a.cnt + 6);
                    cb[q] = new_root(a.par, l.y, a.walk, a.cnt + 6);
                    if (ca[q] != cb[q]) keep |= 1u << q;
                }
            }
            long long at = cta_reserve_count(__popc(keep), a.cnt + (round & 1));
#pragma unroll
            for (int q = 0; q < kRes; q++) {
                if (!((keep >> q) & 1u)) continue;
                const int64_t x = base + (int64_t)q * blockDim.x + threadIdx.x;
                const u128 key = round ? as_u128(kin[x]) : pack(x);
                lout[at] = make_int2(ca[q], cb[q]);
                kout[at] = as_pair(key);
                at++;
                bid_u128<false>(slot2 + ca[q], key | (lb ? (unsigned)cb[q] : 0u), slot2 + cb[q], key | (lb ? (unsigned)ca[q] : 0u));
            }
        }
        if (lead) a.cnt[2 + ((round & 1) ^ 1)] = 0;
        if (!bar.sync()) return;
        const int64_t left = (int64_t) * (volatile unsigned long long *)(a.cnt + (round & 1));
        if (left == 0) break;
        if (*(volatile unsigned long long *)(a.cnt + 6)) {  // this round's filter is void: its input is what goes on
            if (lead) {
                a.cnt[7] = (unsigned long long)round + 1;
                a.cnt[8] = (unsigned long long)n;
                a.cnt[9] = (unsigned long long)nr;
            }
            break;
        }
        n = left;
        {
            int32_t *t = rout;
            roots = rout;
            rout = rnext;
            rnext = t;
            int2 *tl = lin;
            lin = lout;
            lout = tl;
            ulonglong2 *tk = kin;
            kin = kout;
            kout = tk;
            tk = slot;
            slot = slot2;
            slot2 = tk;
        }
    }
    if (lead) a.cnt[4] = (unsigned long long)nfe;
    bar.finish();
}

// After k_m_forest stopped at a filter: the pointers of the n live edges'
// labels settle by jumping rounds, and the edges between two components go out
// as columns. cnt: [0] edges out, [1 .. 3] flags of the jumping rounds, zero
// at the start. Labels and keys as k_m_forest keeps them, or (lab null) columns.
struct MLabels {
    int64_t n;
    const int2 *lab;
    const ulonglong2 *key;
    const int32_t *ru, *rv, *u, *v;
    const int64_t *w;
    int32_t *par;
    int32_t *cu2, *cv2, *u2, *v2;
    int64_t *w2;
    unsigned long long *cnt;
    int ib, lbits;
    BarRef bar;
};
struct LabelItem {
    const int2 *lab;
    const int32_t *ru, *rv;
    __device__ __forceinline__ int64_t operator()(int64_t i) const {
        const int64_t x = i >> 1;
        if (lab) return (i & 1) ? lab[x].y : lab[x].x;
        return (i & 1) ? rv[x] : ru[x];
    }
};
__global__ void __launch_bounds__(kBlock) k_m_labels(MLabels a) {
    GridBar bar(a.bar);
    if (bar.stopped()) return;
    const JumpEnd e = jump_rounds(bar, 2 * a.n, LabelItem{a.lab, a.ru, a.rv}, a.par, a.cnt + 1);
    if (e == kJumpBarrier) return;
    if (e == kJumpBound && threadIdx.x == 0) bar.stop(kStopJump);
    const unsigned imask = (unsigned)((1ull << a.ib) - 1ull);
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < a.n; base += (int64_t)gridDim.x * blockDim.x) {  // CTA-uniform
        const int64_t x = base + threadIdx.x;
        int ca = 0, cb = 0;
        if (x < a.n) {
            const int2 l = a.lab ? a.lab[x] : make_int2(a.ru[x], a.rv[x]);
            ca = *(volatile int32_t *)(a.par + l.x);
            cb = *(volatile int32_t *)(a.par + l.y);
        }
        const long long at = cta_reserve(ca != cb, a.cnt);
        if (ca == cb) continue;
        a.cu2[at] = ca;
        a.cv2[at] = cb;
        if (a.lab) {
            const u128 k = as_u128(a.key[x]) >> a.lbits;
            a.u2[at] = (int)((unsigned)(k >> a.ib) & imask);
            a.v2[at] = (int)((unsigned)k & imask);
            a.w2[at] = (int64_t)(unsigned long long)(k >> (2 * a.ib));
        } else {
            a.u2[at] = a.u[x];
            a.v2[at] = a.v[x];
            a.w2[at] = a.w[x];
        }
    }
    bar.finish();
}

__global__ void k_pack_uv_idx(const FEdge *fe, int64_t n, int idbits, unsigned long long *k,
                              unsigned long long *val) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        k[x] = ((unsigned long long)fe[x].u << idbits) | (unsigned long long)fe[x].v;
        val[x] = (unsigned long long)x;
    }
}

__global__ void k_gather_w(const unsigned *stop, const FEdge *fe, const unsigned long long *idx, int64_t n,
                           unsigned long long *k, unsigned long long *val) {
    if (stopped(stop)) return;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long i = idx[x];
        k[x] = (unsigned long long)fe[i].w;
        val[x] = i;
    }
}

// When every w fits 32 bits the w (and graph) passes sort keys only: the
// edge index rides in the low 32 bits, which the passes do not sort on, so
// the order stays that of the previous sort among equal w (LSD stability)
// and each pass moves 8 bytes an edge instead of 16.
__global__ void k_gather_w32(const unsigned *stop, const FEdge *fe, const unsigned long long *idx, int64_t n, unsigned long long *k) {
    if (stopped(stop)) return;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long i = idx[x];
        k[x] = ((unsigned long long)fe[i].w << 32) | i;
    }
}
__global__ void k_gather_graph32(const unsigned *stop, const FEdge *fe, const int32_t *egraph, const unsigned long long *kin, int64_t n,
                                 unsigned long long *k) {
    if (stopped(stop)) return;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long i = kin[x] & 0xffffffffull;
        k[x] = ((unsigned long long)egraph[fe[i].u] << 32) | i;
    }
}

// graph of each sorted forest edge, as a sort key (graph-major output)
__global__ void k_gather_graph(const unsigned *stop, const FEdge *fe, const int32_t *egraph, const unsigned long long *idx,
                               int64_t n, unsigned long long *k, unsigned long long *val) {
    if (stopped(stop)) return;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long i = idx[x];
        k[x] = (unsigned long long)egraph[fe[i].u];
        val[x] = i;
    }
}

// goff[g] = first row of graph g in the graph-major forest (binary search)
__global__ void k_graph_offsets(const unsigned *stop, const int32_t *u, const int32_t *egraph, int64_t n, int G,
                                int64_t *goff) {
    if (stopped(stop)) return;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g <= G;
         g += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = n;  // first row whose graph >= g
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (egraph[u[mid]] < g) lo = mid + 1;
            else hi = mid;
        }
        goff[g] = lo;
    }
}

// one graph: no search (its 20 or more dependent reads take 10 to 18 us)
__global__ void k_one_offset(int64_t *goff, int64_t n) { goff[1] = n; }

__global__ void k_gather_msf(const unsigned *stop, const unsigned long long *idx, unsigned long long imask, int64_t n, const FEdge *fe,
                             int32_t *u, int32_t *v, int32_t *ru, int32_t *rv, int64_t *w) {
    if (stopped(stop)) return;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        FEdge f;
        {
            unsigned long long q0, q1, q2, q3;
            asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                         : "=l"(q0), "=l"(q1), "=l"(q2), "=l"(q3)
                         : "l"(fe + (idx[x] & imask)));
            f.u = (int32_t)q0;
            f.v = (int32_t)(q0 >> 32);
            f.ru = (int32_t)q1;
            f.rv = (int32_t)(q1 >> 32);
            f.w = (int64_t)q2;
        }
        u[x] = f.u;
        v[x] = f.v;
        ru[x] = f.ru;
        rv[x] = f.rv;
        w[x] = f.w;
    }
}

void plan_msf(Arena &ws, const Problem &p, Msf &o) {
    o.goff = ws.take<int64_t>(p.G + 1);
    o.u = ws.take<int32_t>(p.E);
    o.v = ws.take<int32_t>(p.E);
    o.ru = ws.take<int32_t>(p.E);
    o.rv = ws.take<int32_t>(p.E);
    o.w = ws.take<int64_t>(p.E);
}

// Live edges above which the host launches every step of a round by itself:
// the 64-bit bids in three passes at full occupancy beat the one 128-bit pass
// there (100M hub edges, 190M links: the stage takes 40.0 ms, 54.9 with every
// round in the cooperative kernel; 10M edges 5.3 against 6.5), while below, the
// launches and the host's read of every round cost more than they save (3M
// edges 2.07 ms, 2.17 with the line at 2^24).
constexpr int64_t kMLarge = int64_t(1) << 22;
// One side of the live edges: 24 bytes each, as five columns in the large
// rounds, as labels and keys in the cooperative kernel.
struct LiveSide {
    int32_t *cu, *cv, *u, *v;
    int64_t *w;
    ulonglong2 *key;
    int2 *lab;
};
static LiveSide carve_side(Arena &a, int64_t S) {
    const int64_t n = (S + 3) & ~int64_t(3);
    char *p = a.take<char>(24 * n);
    LiveSide s;
    s.cu = (int32_t *)p;
    s.cv = s.cu + n;
    s.u = s.cv + n;
    s.v = s.u + n;
    s.w = (int64_t *)(s.v + n);
    s.key = (ulonglong2 *)p;
    s.lab = (int2 *)(s.key + n);
    return s;
}
struct MsfScratch {
    int32_t *par, *roots, *roots2, *bp, *win;
    LiveSide side[2];
    ulonglong2 *slot, *slot2;
    FEdge *fe;
    unsigned long long *cnt;
    unsigned long long *k1, *k2, *v1, *v2;
    void *radix;
};
static MsfScratch carve_msf(Arena &a, const Problem &p) {
    MsfScratch s;
    int64_t E = p.E, S = link_cap(p);
    s.par = a.take<int32_t>(E);
    s.roots = a.take<int32_t>(E);
    s.roots2 = a.take<int32_t>(E);
    s.bp = a.take<int32_t>(E);
    s.win = a.take<int32_t>(E);
    s.side[0] = carve_side(a, S);
    s.side[1] = carve_side(a, S);
    const int64_t Er = (E + 31) / 32 * 32;
    s.slot = a.take<ulonglong2>(Er);
    s.slot2 = a.take<ulonglong2>(Er);
    s.fe = a.take<FEdge>(E);
    s.cnt = a.take<unsigned long long>(12);
    // the sorts after the rounds, when no bid is read any more
    s.k1 = (unsigned long long *)s.slot;
    s.k2 = s.k1 + Er;
    s.v1 = (unsigned long long *)s.slot2;
    s.v2 = s.v1 + Er;
    s.radix = a.take<char>(radix_scratch_bytes(E));
    return s;
}
size_t msf_scratch_bytes(const Problem &p) {
    Arena a(nullptr, 0);
    carve_msf(a, p);
    return a.off;
}

dgec_status stage_msf(Ctx *c, const Problem &p, const Csr &g, const Skel &sk, Msf &o, void *scratch) {
    cudaStream_t st = c->stream;
    o.n = 0;
    int64_t E = p.E;
    CU_TRY(c, cudaMemsetAsync(o.goff, 0, sizeof(int64_t) * (p.G + 1), st));
    if (E == 0 || sk.n == 0) return DGEC_OK;
    Arena a(scratch, SIZE_MAX);
    MsfScratch s = carve_msf(a, p);
    CU_TRY(c, cudaMemsetAsync(s.cnt, 0, 12 * sizeof(unsigned long long), st));
    // live edges: (cu, cv) component labels, (u, v) original ends, w; the
    // first round reads the skeleton itself (labels = internal ids)
    const int32_t *ccu = sk.ru, *ccv = sk.rv, *cu = sk.u, *cv = sk.v, *roots0 = nullptr;
    const int64_t *cw = sk.w;
    int64_t n = sk.n, nr = E;
    int which = 0;  // the side the next filter writes
    int32_t *roots = s.roots, *roots2 = s.roots2;
    if (n > kMLarge) {
        unsigned long long *bw = (unsigned long long *)s.slot, *buv = bw + E;
        TK(c, "k_m_init", k_m_init<<<grid_for(E, kBlock, kStreamCap), kBlock, 0, st>>>(E, s.par, roots, bw, buv));
        for (int round = 0; n > kMLarge; round++) {
            if (round >= 64) return set_err(c, DGEC_ERR_TIMEOUT, "Boruvka did not finish in 64 rounds");
            const int gn = grid_for(n, kBlock, kStreamCap), gr = grid_for(nr, kBlock, kStreamCap),
                      grk = grid_for(nr, kBlock * kRes8, kStreamCap);
            if (round == 0) TK(c, "k_m_bid", k_m_bid<<<gn, kBlock, 0, st>>>(ccu, ccv, cw, n, bw));
            TK(c, "k_m_bid_uv", k_m_bid_uv<<<gn, kBlock, 0, st>>>(ccu, ccv, cu, cv, cw, n, bw, buv));
            TK(c, "k_m_claim", k_m_claim<<<gn, kBlock, 0, st>>>(ccu, ccv, cu, cv, n, buv, s.bp, s.win));
            TK(c, "k_m_hook", k_m_hook<<<grk, kBlock, 0, st>>>(roots, nr, bw, buv, s.bp, s.win, cu, cv, cw, g.rank_of,
                                                            round == 0 ? g.orig_of : nullptr, s.par, s.fe, s.cnt + 4));
            CU_TRY(c, cudaMemsetAsync(s.cnt, 0, 4 * sizeof(unsigned long long), st));
            if (c->own_walk(kMWalk)) TK(c, "k_m_jump", k_m_jump<true><<<gr, kBlock, 0, st>>>(roots, nr, s.par, kMWalk, s.win, s.cnt));
            else TK(c, "k_m_jump", k_m_jump<false><<<gr, kBlock, 0, st>>>(roots, nr, s.par, c->walk_steps, s.win, s.cnt));
            {
                int grid = 1;
                DG_TRY(coop_grid(c, kCoopMJump, (const void *)k_m_settle, kBlock, 0, &grid));
                unsigned long long *cut = s.cnt;
                BarRef ref = c->next_bar();
                void *args[] = {&s.win, &s.par, &cut, &ref};  // (win: read by the hooks, next written by the claims)
                cudaError_t e;
                TK(c, "k_m_settle", e = cudaLaunchCooperativeKernel((const void *)k_m_settle,
                                                                    dim3((unsigned)std::min({gr, grid, c->num_sms})), dim3(kBlock), args,
                                                                    0, st));
                if (e != cudaSuccess) return set_err(c, DGEC_ERR_CUDA, "k_m_settle launch: %s", cudaGetErrorString(e));
            }
            CU_TRY(c, cudaMemsetAsync(s.cnt, 0, 4 * sizeof(unsigned long long), st));
            TK(c, "k_m_next_roots", k_m_next_roots<<<grk, kBlock, 0, st>>>(roots, nr, s.par, bw, buv, roots2, s.cnt + 1));
            std::swap(roots, roots2);
            const LiveSide &o = s.side[which];
            TK(c, "k_m_filter_bid", k_m_filter_bid<<<grid_for(n, kBlock * kRes8, kStreamCap), kBlock, 0, st>>>(
                                      ccu, ccv, cu, cv, cw, n, s.par, o.cu, o.cv, o.u, o.v, o.w, s.cnt, bw));
            int64_t h[2];
            DG_TRY(read_counters(c, (const int64_t *)s.cnt, 2, h));
            n = h[0];
            nr = h[1];
            ccu = o.cu;
            ccv = o.cv;
            cu = o.u;
            cv = o.v;
            cw = o.w;
            which ^= 1;
        }
        roots0 = roots;
        CU_TRY(c, cudaMemsetAsync(s.cnt, 0, 4 * sizeof(unsigned long long), st));
    }
    int64_t m = 0;
    if (n == 0) DG_TRY(read_counters(c, (const int64_t *)(s.cnt + 4), 1, &m));
    const int lbits = p.tbits + 3 * p.idbits <= 127 ? p.idbits : 0;
    for (int starts = 0; n > 0; starts++) {
        if (starts >= 64) return set_err(c, DGEC_ERR_TIMEOUT, "Boruvka did not finish in 64 starts");
        // the kernel's first filter writes lb/kb: not the side its edges come from
        const LiveSide &in = s.side[which ^ 1], &out = s.side[which];
        MsfArgs f{nr, n, roots0, ccu, ccv, cu, cv, cw, g.rank_of, s.par, roots0 ? roots2 : roots, roots0 ? roots : roots2,
                  s.bp, s.slot, s.slot2, in.lab, out.lab, in.key, out.key, s.fe, s.cnt, p.idbits, lbits, c->walk(kMCut), c->next_bar()};
        int grid = 1;
        DG_TRY(coop_grid(c, kCoopMsf, (const void *)k_m_forest, kBlock, 0, &grid));
        const int64_t want = cdiv(n > nr ? n : nr, kBlock * kRes);
        DG_TRY(coop_launch(c, "k_m_forest", (const void *)k_m_forest, want < grid ? (int)want : grid, kBlock, 0, f));
        int64_t h[6];
        DG_TRY(read_counters(c, (const int64_t *)(s.cnt + 4), 6, h));
        if (h[1]) return set_err(c, DGEC_ERR_TIMEOUT, "Boruvka did not finish in 64 rounds");
        m = h[0];
        if (h[3] == 0) break;
        // a filter's walk was cut: its input's labels settle, and the rounds go on from there
        const int64_t round = h[3] - 1;
        const bool odd = round & 1;  // an odd round reads the side `out`, the others (but the first) `in`
        const LiveSide &from = odd ? out : in, &to = round == 0 ? out : odd ? in : out;
        n = h[4];
        nr = h[5];
        roots = odd ? f.roots2 : f.roots;
        roots2 = odd ? f.roots : f.roots2;
        roots0 = roots;
        CU_TRY(c, cudaMemsetAsync(s.cnt, 0, 4 * sizeof(unsigned long long), st));
        CU_TRY(c, cudaMemsetAsync(s.cnt + 5, 0, 5 * sizeof(unsigned long long), st));
        DG_TRY(coop_grid(c, kCoopMLabels, (const void *)k_m_labels, kBlock, 0, &grid));
        DG_TRY(coop_launch(c, "k_m_labels", (const void *)k_m_labels, (int)std::min<int64_t>(grid, cdiv(n, kBlock)), kBlock, 0,
                           MLabels{n, round ? from.lab : nullptr, from.key, ccu, ccv, cu, cv, cw, s.par, to.cu, to.cv, to.u,
                                   to.v, to.w, s.cnt, p.idbits, lbits, c->next_bar()}));
        DG_TRY(read_counters(c, (const int64_t *)s.cnt, 1, &n));
        CU_TRY(c, cudaMemsetAsync(s.cnt, 0, 4 * sizeof(unsigned long long), st));
        ccu = to.cu;
        ccv = to.cv;
        cu = to.u;
        cv = to.v;
        cw = to.w;
        which = &to == &s.side[0] ? 1 : 0;
    }
    o.n = m;
    if (m == 0) return DGEC_OK;
    // order by (w, u, v): stable radix by the packed original ends, then by w,
    // then (batches) by graph, carrying the edge index; then gather columns
    int gm = grid_for(m, kBlock, kStreamCap);
    unsigned long long *K[2] = {s.k1, s.k2}, *Vb[2] = {s.v1, s.v2};
    int cur = 0;
    bool in_b;
    TK(c, "k_pack_uv_idx", k_pack_uv_idx<<<gm, kBlock, 0, st>>>(s.fe, m, p.idbits, K[0], Vb[0]));
    DG_TRY(radix_sort(c, RadixBuffers{K[cur], K[1 - cur], Vb[cur], Vb[1 - cur]}, m, 0, 2 * p.idbits,
                      s.radix, &in_b));
    if (in_b) cur = 1 - cur;
    if (p.tbits <= 32) {
        TK(c, "k_gather_w", k_gather_w32<<<gm, kBlock, 0, st>>>(c->stop(), s.fe, Vb[cur], m, K[1 - cur]));
        cur = 1 - cur;
        DG_TRY(radix_sort(c, RadixBuffers{K[cur], K[1 - cur], nullptr, nullptr}, m, 32,
                          32 + (p.tbits > 0 ? p.tbits : 1), s.radix, &in_b));
        if (in_b) cur = 1 - cur;
        if (p.G > 1) {
            TK(c, "k_gather_graph", k_gather_graph32<<<gm, kBlock, 0, st>>>(c->stop(), s.fe, p.egraph, K[cur], m, K[1 - cur]));
            cur = 1 - cur;
            DG_TRY(radix_sort(c, RadixBuffers{K[cur], K[1 - cur], nullptr, nullptr}, m, 32,
                              32 + bits_for((uint64_t)(p.G - 1)), s.radix, &in_b));
            if (in_b) cur = 1 - cur;
        }
    } else {
    TK(c, "k_gather_w", k_gather_w<<<gm, kBlock, 0, st>>>(c->stop(), s.fe, Vb[cur], m, K[1 - cur], Vb[1 - cur]));
    cur = 1 - cur;
    DG_TRY(radix_sort(c, RadixBuffers{K[cur], K[1 - cur], Vb[cur], Vb[1 - cur]}, m, 0,
                      p.tbits > 0 ? p.tbits : 1, s.radix, &in_b));
    if (in_b) cur = 1 - cur;
    if (p.G > 1) {
        TK(c, "k_gather_graph", k_gather_graph<<<gm, kBlock, 0, st>>>(c->stop(), s.fe, p.egraph, Vb[cur], m, K[1 - cur],
                                                                     Vb[1 - cur]));
        cur = 1 - cur;
        DG_TRY(radix_sort(c, RadixBuffers{K[cur], K[1 - cur], Vb[cur], Vb[1 - cur]}, m, 0,
                          bits_for((uint64_t)(p.G - 1)), s.radix, &in_b));
        if (in_b) cur = 1 - cur;
    }
    }
    const bool low32 = p.tbits <= 32;  // the index is the sorted key's low word
    const unsigned long long *fin = low32 ? K[cur] : Vb[cur];
    TK(c, "k_gather_msf", k_gather_msf<<<gm, kBlock, 0, st>>>(c->stop(), fin, low32 ? 0xffffffffull : ~0ull, m, s.fe, o.u,
                                                              o.v, o.ru, o.rv, o.w));
    if (p.G == 1) TK(c, "k_graph_offsets", k_one_offset<<<1, 1, 0, st>>>(o.goff, m));
    else TK(c, "k_graph_offsets", k_graph_offsets<<<grid_for(p.G + 1), kBlock, 0, st>>>(c->stop(), o.u, p.egraph, m, p.G, o.goff));
    return DGEC_OK;
}

}  // namespace dgec
