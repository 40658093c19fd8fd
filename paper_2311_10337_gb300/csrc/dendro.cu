// Stage D1: single-linkage dendrogram (Alg. 1, union-find dendrogram) of the sorted
// forest, built in parallel rounds instead of one union-find sweep.
//
// Merge s is the s-th forest edge in (w, u, v) order; its dendrogram node is
// n_edges + s. Every round works on the super-vertices (already merged
// subtrees) and the forest edges not yet placed:
//   1. each super-vertex takes its smallest incident edge (its "pointer");
//      pointers form trees whose root is the one mutual pair, and along a
//      pointer path the edge ranks decrease toward that pair;
//   2. tau(G) = smallest non-pointer edge touching pointer tree G;
//   3. the pointer edges of G below tau(G) are accepted. They form a
//      connected top part of G, and no other edge below them touches it, so
//      in rank order g_1 < g_2 < ... they merge as a chain: g_1 joins the
//      mutual pair's two subtrees, g_k joins g_{k-1} with the subtree of the
//      super-vertex whose pointer g_k is;
//   4. sizes along a chain are a segmented prefix sum; the accepted part of
//      G becomes one super-vertex whose dendrogram root is its last merge.
// Each round accepts at least the mutual edge of every pointer tree, and a
// pointer tree with no interfering edge is placed whole (a star is one
// round), so the round count follows the depth of interference, not the
// dendrogram height.
#include <algorithm>

#include "grids.h"
#include "sort_dev.cuh"
#include "stages.cuh"

namespace dgec {

// Super-vertex labels are internal ids r (a leaf's label is its own r).
// Each super-vertex's dendrogram root (a node id, so a leaf's root is its
// original id) and size share one 16-byte record: a chain step reads both
// with one sector.
struct SvRec {
    int64_t size;
    int32_t root;
    int32_t pad;
};
//
// minr (a super-vertex's smallest live edge) and tau (a pointer tree's
// smallest non-pointer edge) live one round each. A slot holds
// (stamp << 32) | rank with stamp = kStampTop - round: newer rounds have
// smaller stamps, so atomicMin over the whole key keeps this round's
// minimum, and a slot with another stamp holds nothing this round. No pass
// resets them between rounds.
constexpr unsigned kStampTop = 0xFFFFFFF0u;
__device__ __forceinline__ unsigned long long rkey(unsigned stamp, int v) {
    return ((unsigned long long)stamp << 32) | (unsigned)v;
}
__device__ __forceinline__ int rval(unsigned long long k, unsigned stamp) {
    return (unsigned)(k >> 32) == stamp ? (int)(unsigned)k : INT_MAX;
}
__global__ void k_d_init(int64_t E, int64_t n, const int32_t *mu, const int32_t *mv,
                         const int32_t *orig_of, int32_t *svpar, SvRec *sv,
                         unsigned long long *minr, unsigned long long *tau, int32_t *parent, int32_t *act, int32_t *ecu,
                         int32_t *ecv) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < E;
         x += (int64_t)gridDim.x * blockDim.x) {
        parent[x] = -1;
        svpar[x] = (int32_t)x;
        sv[x] = SvRec{1, orig_of[x], 0};
        minr[x] = ~0ull;
        tau[x] = ~0ull;
        if (n == 1 && x == 0) {  // (more rows come ordered, from k_d_order_act)
            act[0] = 0;
            ecu[0] = mu[0];
            ecv[0] = mv[0];
        }
    }
}

// the first active list: forest edges ordered by their internal end, so
// neighbouring threads touch neighbouring labels
// Rows arrive in rank order s, so the key (ru << sbits) | s sorted stably
// over the ru bits alone orders them by ru with ties in s order (no values).
__global__ void k_d_order_keys(const int32_t *ru, int64_t n, int sbits, unsigned long long *k) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x)
        k[x] = ((unsigned long long)(unsigned)ru[x] << sbits) | (unsigned long long)x;
}
__global__ void k_d_order_act(const unsigned *stop, const unsigned long long *k, int64_t n, int sbits, const int32_t *rv,
                              int32_t *act, int32_t *ecu, int32_t *ecv) {
    if (stopped(stop)) return;
    const unsigned long long smask = (1ull << sbits) - 1ull;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long kk = k[j];
        const int s = (int)(kk & smask);
        act[j] = s;
        ecu[j] = (int32_t)(kk >> sbits);  // ru, from the key
        ecv[j] = rv[s];
    }
}

// A dendrogram row as the rounds write it: one whole sector. `parent` is the
// merge above (a node id, -1 at a root).
struct __align__(32) DRow {
    int32_t a, b, parent, pad;
    int64_t size, pad2;
};

__global__ void k_d_split(const DRow *__restrict__ row, int64_t n, int32_t *__restrict__ la,
                          int32_t *__restrict__ lb, int64_t *__restrict__ size, int32_t *__restrict__ mparent) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        const int4 r = *reinterpret_cast<const int4 *>(row + s);
        la[s] = r.x;
        lb[s] = r.y;
        mparent[s] = r.z;
        size[s] = row[s].size;
    }
}

struct DArgs {
    int64_t E, n;
    int lb, sbits;  // bits of a label, of a rank
    int32_t *act, *act2, *ecu, *ecu2, *ecv, *ecv2;  // live edges: rank, labels of the super-vertices at the ends
    unsigned char *st;                              // per live edge: bit 0/1 it is the pointer of ecu/ecv, bit 2 accepted
    unsigned long long *minr, *tau;
    int32_t *gp, *svpar;
    SvRec *sv;
    // accepted edges of small groups, group by group
    int *gcnt;       // [E] by group: its accepted edges (zero between rounds)
    int2 *gseg;      // [E] by group: (first place, edges); first -1: a large group
    int32_t *slot;   // [E] by live edge: place within its group
    int2 *segA;      // (rank, leaves the edge adds)
    int4 *segB;      // (pointer's owner, group, owner's root, the mutual pair's other root or -1)
    int2 *segC;      // its group's (first place, edges)
    unsigned long long *tot;  // [0], [1] places of small groups taken (by round parity), [2], [3] edges of large groups,
                              // [4] cut walks of d_jump, [5 .. 7] flags of the jumping rounds
    // accepted edges of large groups, sorted by (group, rank)
    int2 *kids;          // the nodes the edge merges
    long long *contrib;  // (leaves it adds << 1) | first of its chain
    DRow *row;
    int32_t *parent;     // [E] of the leaves
    SortArgs sort;       // n and bits are set every round
    unsigned *ccnt;      // [CTAs] accepted edges of each CTA's chunk
    SegVal *cagg;        // [CTAs] chain sum over each CTA's chunk
    int *state;          // [0] rounds run, [1] error, [2] live edges (accepted ones after a large round's emit)
    int max_rounds, walk;
    BarRef bar;
};

// The last rounds (k_d_tail) take over at this many live edges; above
// kDLarge the host launches every step by itself: the steps are bound by
// random accesses there and want more threads than the cooperative kernel's
// 1,024 an SM (every round in that kernel: 53.6 ms for the stage at 100M hub
// edges, 34 with the large rounds apart); below, its barriers (about 2 us)
// replace launches and a host read (3M edges: 2.18 ms with the line at 2^19, 2.22
// at 2^20, 2.78 at 2^22).
constexpr int kTailMax = 4096;
constexpr int64_t kDLarge = int64_t(1) << 19;
// Groups of at most this many accepted edges skip the sort: each edge scans
// its group (316,229 edges: 1.08 ms for the stage at 16, 0.92 at 32, 0.87 at 64
// and 128; 10M edges 5.7 at 64, 5.4 at 128).
constexpr int kDSmall = 128;
constexpr int kDItems = 4;
constexpr int kDTile = kSThreads * kDItems;

__device__ __forceinline__ SegVal seg_add(SegVal a, SegVal b) {
    SegVal r;
    r.v = b.f ? b.v : a.v + b.v;
    r.f = a.f | b.f;
    return r;
}
// Ordered exclusive prefix over the CTA's threads; *total: the whole CTA's.
// sm: kSWarps values, free again after the next __syncthreads.
__device__ __forceinline__ SegVal seg_block(SegVal v, SegVal *sm, SegVal *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    SegVal inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        SegVal o;
        o.v = ::__shfl_up_sync(0xffffffffu, inc.v, d);
        o.f = ::__shfl_up_sync(0xffffffffu, inc.f, d);
        if (lane >= d) inc = seg_add(o, inc);
    }
    if (lane == 31) sm[w] = inc;
    SegVal ex;
    ex.v = ::__shfl_up_sync(0xffffffffu, inc.v, 1);
    ex.f = ::__shfl_up_sync(0xffffffffu, inc.f, 1);
    if (lane == 0) ex = SegVal{0, 0};
    __syncthreads();
    SegVal pre{0, 0}, all{0, 0};
#pragma unroll
    for (int i = 0; i < kSWarps; i++) {
        if (i == w) pre = all;
        all = seg_add(all, sm[i]);
    }
    *total = all;
    return seg_add(pre, ex);
}

// A round's state, the same in every CTA.
struct DRound {
    int round, G;  // G: CTAs taking part
    unsigned stamp;
    int64_t na, nacc, nsmall;  // live edges; accepted ones of large and of small groups
    bool odd;  // the live list changes sides every round
};
#define D_LIST                                                       \
    const int32_t *act = w.odd ? a.act2 : a.act;                     \
    int32_t *ecu = w.odd ? a.ecu2 : a.ecu, *ecv = w.odd ? a.ecv2 : a.ecv; \
    const int64_t na = w.na;                                         \
    (void)act, (void)ecu, (void)ecv
#define D_STRIDE \
    const int64_t gsize = (int64_t)w.G * kSThreads, g0 = (int64_t)blockIdx.x * kSThreads + threadIdx.x

// The steps of a round, each a function of its own so that each gets the
// registers it needs.
// Every live edge offers its rank to both super-vertices; the slots are read
// just before (not ahead for several edges): they only fall, and most offers
// to a large super-vertex cannot win once a few have been made.
__device__ __forceinline__ void d_bid(const DArgs &a, const DRound &w) {
    D_STRIDE;
    const int32_t *act = w.odd ? a.act2 : a.act;
    int32_t *ecu = w.odd ? a.ecu2 : a.ecu, *ecv = w.odd ? a.ecv2 : a.ecv;
    const int64_t na = w.na;
    for (int64_t j = g0; j < na; j += gsize) {
        const unsigned long long key = rkey(w.stamp, act[j]);
        int cu = ecu[j], cv = ecv[j];
        if (w.round > 0) {  // labels move one hop after a round's merges
            cu = a.svpar[cu];
            cv = a.svpar[cv];
            ecu[j] = cu;
            ecv[j] = cv;
        }
        if (key < a.minr[cu]) atomicMin(&a.minr[cu], key);
        if (key < a.minr[cv]) atomicMin(&a.minr[cv], key);
    }
}
__device__ __forceinline__ void d_ptr(const DArgs &a, const DRound &w) {
    D_LIST;
    D_STRIDE;
    const unsigned stamp = w.stamp;
    // pointers (a mutual pair points both ends at its smaller label)
    for (int64_t j0 = g0; j0 < na; j0 += gsize * kDItems) {
        int s[kDItems], cu[kDItems], cv[kDItems];
        bool pu[kDItems], pv[kDItems];
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const int64_t j = j0 + q * gsize;
            s[q] = -1;
            if (j >= na) continue;
            s[q] = act[j];
            cu[q] = ecu[j];
            cv[q] = ecv[j];
        }
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            if (s[q] < 0) continue;
            pu[q] = rval(a.minr[cu[q]], stamp) == s[q];
            pv[q] = rval(a.minr[cv[q]], stamp) == s[q];
        }
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            if (s[q] < 0) continue;
            if (pu[q] && pv[q]) {
                const int r = cu[q] < cv[q] ? cu[q] : cv[q];
                a.gp[cu[q]] = r;
                a.gp[cv[q]] = r;
            } else {
                if (pu[q]) a.gp[cu[q]] = cv[q];
                if (pv[q]) a.gp[cv[q]] = cu[q];
            }
            a.st[j0 + q * gsize] = (unsigned char)((pu[q] ? 1 : 0) | (pv[q] ? 2 : 0));
        }
    }
}
// Every pointer to its tree's root, by walks that shorten their own pointer as
// they go. Walks are cut after kDWalk steps, and jump_rounds finishes those:
// on a long chain the threads running meet only pointers as short as their
// own, and the last of them walks all of it. Stage D1 of a path whose gaps fall,
// all walks whole / cut at 256 / 128 / 64 steps: 400,000 edges 166 / 0.88 / 0.61 /
// 0.47 ms, 3M 4.4 s / 3.1 / 2.2 / 1.5 ms; of 200M hub edges 71.0 / 70.6 / 70.6 / 70.6
// (their cut walks settle in 0.08 to 0.11 ms, 14 launches included; 8.3 with rounds
// over all pointers instead of a list of the cut ones).
constexpr int kDWalk = 64;
// OWN: the limit is kDWalk, known when the loop is compiled.
template <bool OWN>
__device__ __forceinline__ void d_jump(const DArgs &a, const DRound &w) {
    const int limit = OWN ? kDWalk : a.walk;
    D_LIST;
    D_STRIDE;
    for (int64_t j = g0; j < na; j += gsize) {
        const int st = a.st[j];
        if (!st) continue;
#pragma unroll
        for (int side = 0; side < 2; side++) {
            if (!((st >> side) & 1)) continue;
            const int c = side ? ecv[j] : ecu[j];
            int r = a.gp[c];
            int it = 0;
            for (; it < limit; it++) {
                const int rr = *(volatile int32_t *)(a.gp + r);
                if (rr == r) break;
                r = rr;
                atomicExch(a.gp + c, r);  // (not a store: see d_alloc)
            }
            if (it == limit) list_cut(a.slot, a.tot + 4, c);
        }
    }
}
// Their number is in tot[4], they lie in `slot`, which d_accept fills later.
__device__ __forceinline__ JumpEnd d_settle(const DArgs &a, GridBar &bar, int64_t n) {
    return jump_rounds(bar, n, ListItem{a.slot}, a.gp, a.tot + 5);
}
__device__ __forceinline__ void d_tau(const DArgs &a, const DRound &w) {
    D_LIST;
    D_STRIDE;
    const unsigned stamp = w.stamp;
    // tau: the smallest non-pointer edge touching each tree
    for (int64_t j = g0; j < na; j += gsize) {
        if (a.st[j]) continue;
        const int gu = a.gp[ecu[j]], gv = a.gp[ecv[j]];
        const unsigned long long key = rkey(stamp, act[j]);
        if (key < a.tau[gu]) atomicMin(&a.tau[gu], key);
        if (key < a.tau[gv]) atomicMin(&a.tau[gv], key);
    }
}
// A place in cnt[g] for every lane with `take`. Two groups of the warp (the
// first lane's, then the first left's) take theirs with one atomic each, so a
// very large group does not serialise on its counter; the others one by one.
__device__ __forceinline__ int group_place(bool take, int g, int *cnt) {
    unsigned left = __ballot_sync(0xffffffffu, take);
    int place = 0;
    const unsigned lt = (1u << lane_id()) - 1u;
#pragma unroll
    for (int i = 0; i < 2; i++) {
        if (!left) return place;
        const int lead = __ffs(left) - 1;
        const int lg = ::__shfl_sync(0xffffffffu, g, lead);
        const unsigned same = left & __ballot_sync(0xffffffffu, g == lg);
        int base = 0;
        if ((int)lane_id() == lead) base = atomicAdd(&cnt[lg], __popc(same));
        base = ::__shfl_sync(0xffffffffu, base, lead);
        if ((same >> lane_id()) & 1u) place = base + __popc(same & lt);
        left &= ~same;
    }
    if ((left >> lane_id()) & 1u) place = atomicAdd(&cnt[g], 1);
    return place;
}

// Accept the pointer edges below their tree's tau; each takes a place in its
// group, and every CTA counts the edges it keeps.
__device__ __forceinline__ void d_accept(const DArgs &a, const DRound &w) {
    __shared__ int s_int[kSWarps];
    D_LIST;
    const int tid = threadIdx.x, me = blockIdx.x, G = w.G;
    const int64_t tiles = (na + kDTile - 1) / kDTile;
    const int64_t t0 = tiles * me / G, t1 = tiles * (me + 1) / G;
    const int64_t j1 = t1 * kDTile < na ? t1 * kDTile : na;
    int cnt = 0;
    for (int64_t b = t0 * kDTile; b < j1; b += kDTile) {  // CTA-uniform
        const int64_t jb = b + tid;
        int s[kDItems], g[kDItems];
        unsigned char st[kDItems];
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const int64_t j = jb + q * kSThreads;
            st[q] = j < j1 ? a.st[j] : 0;
            cnt += j < j1;
            if (st[q]) {
                s[q] = act[j];
                g[q] = ecu[j];
            }
        }
#pragma unroll
        for (int q = 0; q < kDItems; q++)
            if (st[q]) g[q] = a.gp[g[q]];
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const bool acc = st[q] && s[q] < rval(a.tau[g[q]], w.stamp);
            const int place = group_place(acc, acc ? g[q] : -1, a.gcnt);
            if (!acc) continue;
            const int64_t j = jb + q * kSThreads;
            a.st[j] = st[q] | 4;
            a.slot[j] = place;
            cnt--;
        }
    }
    for (int d = 16; d > 0; d >>= 1) cnt += ::__shfl_xor_sync(0xffffffffu, cnt, d);
    if ((tid & 31) == 0) s_int[tid >> 5] = cnt;
    __syncthreads();
    if (tid == 0) {
        int all = 0;
        for (int i = 0; i < kSWarps; i++) all += s_int[i];
        a.ccnt[me] = (unsigned)all;
    }
}

// Every group's stretch of the accepted edges, taken by its mutual edge (the
// one edge that is both ends' pointer, smallest of its group).
__device__ __forceinline__ void d_alloc(const DArgs &a, const DRound &w) {
    D_LIST;
    const int64_t tile = (int64_t)kSThreads * kDItems;
    for (int64_t base = (int64_t)blockIdx.x * tile; base < na; base += (int64_t)w.G * tile) {  // CTA-uniform
        // step by step for all items, so that their loads overlap
        int g[kDItems], gu[kDItems], gv[kDItems], c[kDItems];
        unsigned need = 0;
        unsigned char st[kDItems];
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const int64_t j = base + q * kSThreads + threadIdx.x;
            st[q] = j < na ? a.st[j] : 0;
        }
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const int64_t j = base + q * kSThreads + threadIdx.x;
            gu[q] = gv[q] = -1;
            if (st[q] == 7) {
                gu[q] = ecu[j];
                gv[q] = ecv[j];
            }
        }
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            g[q] = gu[q] < gv[q] ? gu[q] : gv[q];  // the tree's root
            c[q] = 0;
            // read and cleared in one: a load and a store here, among other CTAs'
            // loads of the same lines, takes 8 times as long (0.84 against 0.1 ms
            // for 16M edges)
            if (g[q] >= 0) c[q] = atomicExch(&a.gcnt[g[q]], 0);
        }
#pragma unroll
        for (int q = 0; q < kDItems; q++)
            if (c[q] <= kDSmall) need += (unsigned)c[q];
        long long at = cta_reserve_count(need, a.tot + (w.round & 1));
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            if (g[q] < 0) continue;
            const bool small = c[q] <= kDSmall;
            a.gseg[g[q]] = make_int2(small ? (int)at : -1, c[q]);
            if (small) at += c[q];
        }
    }
}

// The accepted edges to their groups' stretches (those of large groups as
// (group, rank) keys to the sort), the kept ones on to the next round in order.
// Returns how many are kept.
__device__ __forceinline__ int64_t d_emit(const DArgs &a, const DRound &w) {
    __shared__ SegVal s_seg[kSWarps];
    __shared__ int s_int[kSWarps];
    D_LIST;
    const int tid = threadIdx.x, me = blockIdx.x, G = w.G;
    const int64_t tiles = (na + kDTile - 1) / kDTile;
    const int64_t t0 = tiles * me / G, t1 = tiles * (me + 1) / G;
    int64_t kept, pos;
    {
        unsigned before = 0, all = 0;
        for (int i = tid; i < G; i += kSThreads) {
            const unsigned c = a.ccnt[i];
            all += c;
            if (i < me) before += c;
        }
        for (int d = 16; d > 0; d >>= 1) {
            before += ::__shfl_xor_sync(0xffffffffu, before, d);
            all += ::__shfl_xor_sync(0xffffffffu, all, d);
        }
        if ((tid & 31) == 0) s_seg[tid >> 5] = SegVal{(long long)before, (int)all};
        __syncthreads();
        unsigned long long b = 0, t = 0;
        for (int i = 0; i < kSWarps; i++) {
            b += (unsigned long long)s_seg[i].v;
            t += (unsigned)s_seg[i].f;
        }
        kept = (int64_t)t;
        pos = (int64_t)b;
    }
    int32_t *act2 = w.odd ? a.act : a.act2, *ecu2 = w.odd ? a.ecu : a.ecu2, *ecv2 = w.odd ? a.ecv : a.ecv2;
    for (int64_t t = t0; t < t1; t++) {
        const int64_t j = t * kDTile + tid * kDItems;
        int s[kDItems], cu[kDItems], cv[kDItems], sl[kDItems];
        unsigned char st[kDItems];
        if (j + kDItems <= na) {
            const int4 x = *(const int4 *)(act + j), y = *(const int4 *)(ecu + j), z = *(const int4 *)(ecv + j),
                       l = *(const int4 *)(a.slot + j);
            const uchar4 f = *(const uchar4 *)(a.st + j);
            s[0] = x.x, s[1] = x.y, s[2] = x.z, s[3] = x.w;
            cu[0] = y.x, cu[1] = y.y, cu[2] = y.z, cu[3] = y.w;
            cv[0] = z.x, cv[1] = z.y, cv[2] = z.z, cv[3] = z.w;
            sl[0] = l.x, sl[1] = l.y, sl[2] = l.z, sl[3] = l.w;
            st[0] = f.x, st[1] = f.y, st[2] = f.z, st[3] = f.w;
        } else {
#pragma unroll
            for (int q = 0; q < kDItems; q++) {
                const bool in = j + q < na;
                s[q] = in ? act[j + q] : -1;
                cu[q] = in ? ecu[j + q] : 0;
                cv[q] = in ? ecv[j + q] : 0;
                sl[q] = in ? a.slot[j + q] : 0;
                st[q] = in ? a.st[j + q] : 0;
            }
        }
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < kDItems; q++) cnt += s[q] >= 0 && !(st[q] & 4);
        __syncthreads();  // s_int and s_seg are free again
        int64_t at = pos + sort_block_exclusive(cnt, s_int);
        int g[kDItems];
        int2 sg[kDItems];
        unsigned large = 0;
#pragma unroll
        for (int q = 0; q < kDItems; q++) g[q] = s[q] >= 0 && (st[q] & 4) ? a.gp[cu[q]] : -1;
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            sg[q] = g[q] >= 0 ? a.gseg[g[q]] : make_int2(0, 0);
            large += sg[q].x < 0;
        }
        long long lx = 0;
        if (__syncthreads_or(large)) lx = cta_reserve_count(large, a.tot + 2 + (w.round & 1));
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            if (s[q] < 0) continue;
            if (g[q] < 0) {
                act2[at] = s[q];
                ecu2[at] = cu[q];
                ecv2[at] = cv[q];
                at++;
                continue;
            }
            const bool mutual = (st[q] & 3) == 3;
            int Y = (st[q] & 1) ? cu[q] : cv[q], O = (st[q] & 1) ? cv[q] : cu[q];
            if (mutual && Y == g[q]) {  // the pair's other end, so that the root's own label needs no change
                Y = O;
                O = g[q];
            }
            if (sg[q].x >= 0) {
                const SvRec ry = a.sv[Y];
                int add = (int)ry.size, ro = -1;
                if (mutual) {
                    const SvRec o = a.sv[O];
                    add += (int)o.size;
                    ro = o.root;
                }
                const int x = sg[q].x + sl[q];
                a.segA[x] = make_int2(s[q], add);
                a.segB[x] = make_int4(Y, g[q], ry.root, ro);
                a.segC[x] = sg[q];
            } else {
                a.sort.ka[lx] = ((unsigned long long)(unsigned)g[q] << a.sbits) | (unsigned)s[q];
                a.sort.va[lx] = ((unsigned long long)(unsigned)Y << 32) | (unsigned)O;
                lx++;
            }
        }
        int tot = 0;
        for (int i = 0; i < kSWarps; i++) tot += s_int[i];
        pos += tot;
    }
    return kept;
}

// The chains of the small groups: an edge finds the edges before and after it
// among its group's few, and the leaves below.
__device__ __forceinline__ void d_small(const DArgs &a, const DRound &w, int64_t n) {
    D_STRIDE;
    for (int64_t x = g0; x < n; x += gsize) {
        const int2 c = a.segC[x];
        const int4 e = a.segB[x];
        const int2 me = a.segA[x];
        int prev = -1, next = INT_MAX, size = me.y;
        for (int i = 0; i < c.y; i++) {
            const int2 o = a.segA[c.x + i];
            if (o.x < me.x) {
                size += o.y;
                if (o.x > prev) prev = o.x;
            } else if (o.x > me.x && o.x < next) {
                next = o.x;
            }
        }
        const int node = (int)(a.E + me.x);
        const int n1 = prev < 0 ? e.w : (int)(a.E + prev), n2 = e.z;
        DRow *r = a.row + me.x;
        store_sector(r, pack_i32(n1 < n2 ? n1 : n2, n1 < n2 ? n2 : n1),
                     pack_i32(next == INT_MAX ? -1 : (int)(a.E + next), 0), (unsigned long long)size, 0ull);
        if (n2 < a.E) a.parent[n2] = node;
        else a.row[n2 - a.E].parent = node;
        if (prev < 0) {
            if (n1 < a.E) a.parent[n1] = node;
            else a.row[n1 - a.E].parent = node;
        }
        a.svpar[e.x] = e.y;
        if (next == INT_MAX) a.sv[e.y] = SvRec{size, node, 0};
    }
}

__device__ __forceinline__ void d_chain(const DArgs &a, const DRound &w, const unsigned long long *__restrict__ key, const unsigned long long *__restrict__ val) {
    __shared__ SegVal s_seg[kSWarps];
    const int tid = threadIdx.x, me = blockIdx.x, G = w.G;
    const int64_t nacc = w.nacc, ct = (nacc + kDTile - 1) / kDTile;
    const int64_t c0 = ct * me / G, c1 = ct * (me + 1) / G;
    const unsigned long long smask = (1ull << a.sbits) - 1ull;
    // the chains: g_1 joins the mutual pair, g_k joins g_{k-1} with the
    // super-vertex whose pointer it is
    SegVal agg{0, 0};
    for (int64_t t = c0; t < c1; t++) {
        const int64_t x0 = t * kDTile + tid * kDItems;
        unsigned long long k[kDItems], v[kDItems];
        unsigned long long kp = x0 > 0 && x0 < nacc ? key[x0 - 1] : ~0ull;
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const bool in = x0 + q < nacc;
            k[q] = in ? key[x0 + q] : 0;
            v[q] = in ? val[x0 + q] : 0;
        }
        SvRec y[kDItems];
#pragma unroll
        for (int q = 0; q < kDItems; q++)
            if (x0 + q < nacc) y[q] = a.sv[v[q] >> 32];
        SegVal mine{0, 0};
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const int64_t x = x0 + q;
            if (x >= nacc) continue;
            const bool h = x == 0 || (kp >> a.sbits) != (k[q] >> a.sbits);
            int n1;
            long long add = y[q].size;
            if (h) {
                const SvRec o = a.sv[v[q] & 0xffffffffull];
                n1 = o.root;
                add += o.size;
            } else {
                n1 = (int)(a.E + (int64_t)(kp & smask));
            }
            a.kids[x] = make_int2(n1, y[q].root);
            a.contrib[x] = (add << 1) | (h ? 1 : 0);
            mine = seg_add(mine, SegVal{add, h ? 1 : 0});
            kp = k[q];
        }
        SegVal tot;
        __syncthreads();  // s_seg is free again
        seg_block(mine, s_seg, &tot);
        agg = seg_add(agg, tot);
    }
    if (tid == 0) a.cagg[me] = agg;
}
__device__ __forceinline__ void d_rows(const DArgs &a, const DRound &w, const unsigned long long *__restrict__ key, const unsigned long long *__restrict__ val) {
    __shared__ SegVal s_seg[kSWarps];
    const int tid = threadIdx.x, me = blockIdx.x, G = w.G;
    const int64_t nacc = w.nacc, ct = (nacc + kDTile - 1) / kDTile;
    const int64_t c0 = ct * me / G, c1 = ct * (me + 1) / G;
    const unsigned long long smask = (1ull << a.sbits) - 1ull;
    // sizes along the chains, rows, and the merged super-vertices
    SegVal run{0, 0};
    for (int i0 = 0; i0 < me; i0 += kSThreads) {
        SegVal v = i0 + tid < me ? a.cagg[i0 + tid] : SegVal{0, 0};
        SegVal tot;
        __syncthreads();
        seg_block(v, s_seg, &tot);
        run = seg_add(run, tot);
    }
    for (int64_t t = c0; t < c1; t++) {
        const int64_t x0 = t * kDTile + tid * kDItems;
        unsigned long long k[kDItems + 1], v[kDItems];
        long long cb[kDItems];
        int2 kid[kDItems];
        SegVal mine{0, 0};
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const bool in = x0 + q < nacc;
            k[q] = in ? key[x0 + q] : ~0ull;
            v[q] = in ? val[x0 + q] : 0;
            cb[q] = in ? a.contrib[x0 + q] : 0;
            if (in) kid[q] = a.kids[x0 + q];
        }
        k[kDItems] = x0 + kDItems < nacc ? key[x0 + kDItems] : ~0ull;
#pragma unroll
        for (int q = 0; q < kDItems; q++)
            if (x0 + q < nacc) mine = seg_add(mine, SegVal{cb[q] >> 1, (int)(cb[q] & 1)});
        SegVal tot;
        __syncthreads();  // s_seg is free again
        SegVal pre = seg_add(run, seg_block(mine, s_seg, &tot));
        run = seg_add(run, tot);
#pragma unroll
        for (int q = 0; q < kDItems; q++) {
            const int64_t x = x0 + q;
            if (x >= nacc) continue;
            const bool h = cb[q] & 1;
            pre = seg_add(pre, SegVal{cb[q] >> 1, h ? 1 : 0});
            const int grp = (int)(k[q] >> a.sbits), s = (int)(k[q] & smask);
            const bool tail = x == nacc - 1 || (k[q + 1] >> a.sbits) != (k[q] >> a.sbits);
            const int node = (int)(a.E + s), n1 = kid[q].x, n2 = kid[q].y;
            DRow *r = a.row + s;
            store_sector(r, pack_i32(n1 < n2 ? n1 : n2, n1 < n2 ? n2 : n1),
                         pack_i32(tail ? -1 : (int)(a.E + (int64_t)(k[q + 1] & smask)), 0), (unsigned long long)pre.v, 0ull);
            // the children's parent (a chain's merge below knows already)
            if (n2 < a.E) a.parent[n2] = node;
            else a.row[n2 - a.E].parent = node;
            a.svpar[v[q] >> 32] = grp;
            if (h) {
                if (n1 < a.E) a.parent[n1] = node;
                else a.row[n1 - a.E].parent = node;
                a.svpar[v[q] & 0xffffffffull] = grp;
            }
            if (tail) a.sv[grp] = SvRec{pre.v, node, 0};
        }
    }
}
// Large rounds: every step a kernel of its own, at the occupancy its
// registers allow.
#define D_KERNEL(name, call)                                                                          \
    __global__ void __launch_bounds__(kSThreads, 2) k_d_##name(const __grid_constant__ DArgs a,       \
                                                               const __grid_constant__ DRound w) { \
        if (stopped(a.bar.word + 2)) return;                                                              \
        call;                                                                                             \
    }
D_KERNEL(bid, d_bid(a, w))
D_KERNEL(ptr, d_ptr(a, w))
D_KERNEL(jump, d_jump<true>(a, w))
D_KERNEL(jump_n, d_jump<false>(a, w))
D_KERNEL(tau, d_tau(a, w))
D_KERNEL(accept, d_accept(a, w))
D_KERNEL(alloc, d_alloc(a, w))
D_KERNEL(emit, const int64_t n = d_emit(a, w); if (blockIdx.x == 0 && threadIdx.x == 0) a.state[2] = (int)n)
D_KERNEL(small, d_small(a, w, w.nsmall))
#undef D_KERNEL
__global__ void __launch_bounds__(kSThreads, 2) k_d_chain(const __grid_constant__ DArgs a, const __grid_constant__ DRound w,
                                                       const unsigned long long *key, const unsigned long long *val) {
    if (stopped(a.bar.word + 2)) return;
    d_chain(a, w, key, val);
}
__global__ void __launch_bounds__(kSThreads, 2) k_d_rows(const __grid_constant__ DArgs a, const __grid_constant__ DRound w,
                                                       const unsigned long long *key, const unsigned long long *val) {
    if (stopped(a.bar.word + 2)) return;
    d_rows(a, w, key, val);
}

// What d_jump left of a large round's walks: nothing unless some were cut.
__global__ void __launch_bounds__(kSThreads, 2) k_d_settle(const __grid_constant__ DArgs a) {
    const int64_t n = (int64_t)a.tot[4];
    if (n == 0) return;  // the same for every CTA: written before this launch
    GridBar bar(a.bar);
    if (bar.stopped()) return;
    const JumpEnd e = d_settle(a, bar, n);
    if (e == kJumpBarrier) return;
    if (e == kJumpBound && threadIdx.x == 0) bar.stop(kStopJump);
    bar.finish();
}

// The same steps inside the cooperative kernel, as calls so that each keeps
// its own registers.
__device__ __noinline__ void dc_bid(const DArgs &a, const DRound &w) { d_bid(a, w); }
__device__ __noinline__ void dc_ptr(const DArgs &a, const DRound &w) { d_ptr(a, w); }
template <bool OWN>
__device__ __noinline__ void dc_jump(const DArgs &a, const DRound &w) { d_jump<OWN>(a, w); }
__device__ __noinline__ JumpEnd dc_settle(const DArgs &a, GridBar &bar, int64_t n) { return d_settle(a, bar, n); }
__device__ __noinline__ void dc_tau(const DArgs &a, const DRound &w) { d_tau(a, w); }
__device__ __noinline__ void dc_accept(const DArgs &a, const DRound &w) { d_accept(a, w); }
__device__ __noinline__ void dc_alloc(const DArgs &a, const DRound &w) { d_alloc(a, w); }
__device__ __noinline__ void dc_small(const DArgs &a, const DRound &w) { d_small(a, w, w.nsmall); }
__device__ __noinline__ int64_t dc_emit(const DArgs &a, const DRound &w) { return d_emit(a, w); }
__device__ __noinline__ void dc_chain(const DArgs &a, const DRound &w, const unsigned long long *key,
                                      const unsigned long long *val) { d_chain(a, w, key, val); }
__device__ __noinline__ void dc_rows(const DArgs &a, const DRound &w, const unsigned long long *key,
                                     const unsigned long long *val) { d_rows(a, w, key, val); }
__device__ __noinline__ bool dc_sort(const DArgs &a, int64_t n, int bits, int most, unsigned long long *sm, GridBar &bar) {
    return sort_run<SortWide, true>(a.sort, n, 0, bits, most, sort_smem<SortWide, true>(sm), bar);
}
#undef D_LIST
#undef D_STRIDE

// Middle rounds in one cooperative kernel: no launch and no host read between
// the steps, from the round the host stops at until at most kTailMax edges
// are live.
__global__ void __launch_bounds__(kSThreads, 2) k_d_rounds(const __grid_constant__ DArgs a, const __grid_constant__ DRound w0) {
    extern __shared__ __align__(16) unsigned long long d_sm[];
    GridBar bar(a.bar);
    if (bar.stopped()) return;
    DRound w = w0;
    w.G = gridDim.x;
    int error = 0;
    for (; w.na > kTailMax; w.round++) {
        if (w.round >= a.max_rounds) {
            error = 1;
            break;
        }
        w.odd = w.round & 1;
        w.stamp = kStampTop - (unsigned)w.round;
        dc_bid(a, w);
        if (!bar.sync()) return;
        dc_ptr(a, w);
        if (!bar.sync()) return;
        if (a.walk == kDWalk) dc_jump<true>(a, w);
        else dc_jump<false>(a, w);
        if (!bar.sync()) return;
        const int64_t cut = (int64_t) * (volatile unsigned long long *)(a.tot + 4);
        if (cut > 0) {
            const JumpEnd e = dc_settle(a, bar, cut);
            if (e == kJumpBarrier) return;
            if (e == kJumpBound) {
                if (threadIdx.x == 0) bar.stop(kStopJump);
                return;
            }
        }
        dc_tau(a, w);
        if (!bar.sync()) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) a.tot[4] = 0;  // every CTA has read it
        dc_accept(a, w);
        if (!bar.sync()) return;
        dc_alloc(a, w);
        if (!bar.sync()) return;
        const int64_t kept = dc_emit(a, w);
        if (kept == w.na) {  // cannot be: every round accepts each tree's mutual edge
            error = 2;
            break;
        }
        if (!bar.sync()) return;
        volatile unsigned long long *tot = a.tot;
        w.nsmall = (int64_t)tot[w.round & 1];
        w.nacc = (int64_t)tot[2 + (w.round & 1)];
        if (blockIdx.x == 0 && threadIdx.x == 0) tot[(w.round & 1) ^ 1] = tot[2 + ((w.round & 1) ^ 1)] = 0;
        dc_small(a, w);
        if (w.nacc > 0) {
            // each large group's chain in rank order
            const int kbits = a.lb + a.sbits;
            if (!dc_sort(a, w.nacc, kbits, kSBits, d_sm, bar)) return;
            if (!bar.sync()) return;
            const bool in_b = sort_in_b(w.nacc, kbits, kSBits);
            const unsigned long long *key = in_b ? a.sort.kb : a.sort.ka, *val = in_b ? a.sort.vb : a.sort.va;
            dc_chain(a, w, key, val);
            if (!bar.sync()) return;
            dc_rows(a, w, key, val);
        }
        if (!bar.sync()) return;
        w.na = kept;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.state[0] = w.round;
        a.state[1] = error;
        a.state[2] = (int)w.na;
    }
    bar.finish();
}

// ------------------------------------------------ one-CTA tail of the rounds
// Once at most kTailMax forest edges are live, one CTA runs every remaining
// round in shared memory: the live edges, and for the super-vertices at their
// ends -- renamed 0 .. 2 kTailMax - 1 through gcnt, which is zero between
// rounds -- the slots, pointers, sizes and roots. Only the rows and parents go
// out. The same steps as above; the accepted edges are sorted by (group, rank)
// by a bitonic network, the live list's order changes no result. Bound by
// the steps' CTA barriers and the network (with the arrays in global memory a
// round took 41 us, nearly all of it L2 latency).
constexpr int kTailThreads = 1024;
constexpr int kTailPer = kTailMax / kTailThreads;  // edges a thread holds
constexpr int kTailLabels = 2 * kTailMax;
constexpr size_t kTailSmem = (size_t)kTailLabels * (4 + 4 + 4 + 4 + 2) + (size_t)kTailMax * (4 + 2 + 2 + 1);

__global__ void __launch_bounds__(kTailThreads) k_d_tail(const __grid_constant__ DArgs a) {
    extern __shared__ __align__(16) unsigned char tsm[];
    unsigned *minr = (unsigned *)tsm;                         // [labels] smallest live rank; the sort's keys once the
    unsigned long long *skey = (unsigned long long *)tsm;     //   pointers are known: (group << 32) | rank
    unsigned *tau = minr + kTailLabels;                       // [labels]
    unsigned short *sown = (unsigned short *)(tau);           // the sort's values, once tau is used: the pointers' owners
    int *size = (int *)(tau + kTailLabels), *root = size + kTailLabels;  // [labels]
    int *rank = root + kTailLabels;                           // [edges]
    unsigned short *gp = (unsigned short *)(rank + kTailMax); // [labels] pointer, then its tree's root; kMerged: merged into it
    unsigned short *lu = gp + kTailLabels, *lv = lu + kTailMax;  // [edges] labels
    unsigned char *st = (unsigned char *)(lv + kTailMax);     // [edges] bit 0/1: it is the pointer of lu/lv
    constexpr unsigned short kMerged = 0x8000;
    static_assert(kTailLabels <= kMerged, "labels in 15 bits");
    __shared__ int s_nlab, s_nacc, s_nkeep;
    __shared__ SegVal s_warp[kTailThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (stopped(a.bar.word + 2) || a.state[1] || a.state[2] > kTailMax) return;  // the rounds before did not end
    int na = a.state[2];
    int round = a.state[0];
    if (na == 0) return;
    const int E = (int)a.E;
    {  // in: edges, renamed labels, their sizes and roots
        const bool odd = round & 1;
        const int32_t *act = odd ? a.act2 : a.act, *ecu = odd ? a.ecu2 : a.ecu, *ecv = odd ? a.ecv2 : a.ecv;
        if (tid == 0) s_nlab = 0;
        __syncthreads();
        int c[2 * kTailPer], id[2 * kTailPer];
#pragma unroll
        for (int q = 0; q < kTailPer; q++) {
            const int j = tid + q * kTailThreads;
            c[2 * q] = c[2 * q + 1] = -1;
            if (j >= na) continue;
            rank[j] = act[j];
            c[2 * q] = ecu[j];
            c[2 * q + 1] = ecv[j];
        }
        if (round > 0) {  // the hop after the last round's merges
#pragma unroll
            for (int q = 0; q < 2 * kTailPer; q++)
                if (c[q] >= 0) c[q] = a.svpar[c[q]];
        }
#pragma unroll
        for (int q = 0; q < 2 * kTailPer; q++)  // one edge end names each label
            id[q] = c[q] >= 0 && atomicExch(&a.gcnt[c[q]], 1) == 0 ? atomicAdd(&s_nlab, 1) : -1;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2 * kTailPer; q++) {
            if (id[q] < 0) continue;
            atomicExch(&a.gcnt[c[q]], id[q] + 2);
            const SvRec r = a.sv[c[q]];
            size[id[q]] = (int)r.size;
            root[id[q]] = r.root;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kTailPer; q++) {
            const int j = tid + q * kTailThreads;
            if (j >= na) continue;
            lu[j] = (unsigned short)(*(volatile int *)&a.gcnt[c[2 * q]] - 2);
            lv[j] = (unsigned short)(*(volatile int *)&a.gcnt[c[2 * q + 1]] - 2);
        }
    }
    __syncthreads();
    const int nlab = s_nlab;
    while (na > 0) {
        if (round >= a.max_rounds) {
            if (tid == 0) a.state[1] = 1;
            return;
        }
        for (int c = tid; c < nlab; c += kTailThreads) minr[c] = tau[c] = ~0u;
        if (tid == 0) s_nacc = s_nkeep = 0;
        __syncthreads();
        // every live edge offers its rank to both super-vertices
        for (int j = tid; j < na; j += kTailThreads) {
            const unsigned s = (unsigned)rank[j];
            if (s < minr[lu[j]]) atomicMin(&minr[lu[j]], s);
            if (s < minr[lv[j]]) atomicMin(&minr[lv[j]], s);
        }
        __syncthreads();
        // pointers (a mutual pair points both ends at its smaller label)
        for (int j = tid; j < na; j += kTailThreads) {
            const unsigned s = (unsigned)rank[j];
            const unsigned short cu = lu[j], cv = lv[j];
            const bool pu = minr[cu] == s, pv = minr[cv] == s;
            if (pu && pv) {
                const unsigned short r = cu < cv ? cu : cv;
                gp[cu] = r;
                gp[cv] = r;
            } else {
                if (pu) gp[cu] = cv;
                if (pv) gp[cv] = cu;
            }
            st[j] = (unsigned char)((pu ? 1 : 0) | (pv ? 2 : 0));
        }
        __syncthreads();
        // every pointer to its tree's root
        for (int j = tid; j < na; j += kTailThreads) {
            for (int side = 0; side < 2; side++) {
                if (!((st[j] >> side) & 1)) continue;
                const int c = side ? lv[j] : lu[j];
                int r = gp[c];
                for (int it = 0; it < kTailLabels; it++) {  // bounded: pointer trees
                    const int rr = *(volatile unsigned short *)(gp + r);
                    if (rr == r) break;
                    r = rr;
                    *(volatile unsigned short *)(gp + c) = (unsigned short)r;
                }
            }
        }
        __syncthreads();
        // tau: the smallest non-pointer edge touching each tree
        for (int j = tid; j < na; j += kTailThreads) {
            if (st[j]) continue;
            const unsigned s = (unsigned)rank[j];
            const int gu = gp[lu[j]], gv = gp[lv[j]];
            if (s < tau[gu]) atomicMin(&tau[gu], s);
            if (s < tau[gv]) atomicMin(&tau[gv], s);
        }
        __syncthreads();
        // accept the pointer edges below their tree's tau (minr's place takes the
        // keys); what is kept waits in registers
        int ks[kTailPer], at[kTailPer];
        unsigned kl[kTailPer];
        unsigned short own[kTailPer];
#pragma unroll
        for (int q = 0; q < kTailPer; q++) {
            const int j = tid + q * kTailThreads;
            ks[q] = at[q] = -1;
            if (j >= na) continue;
            const int s = rank[j];
            const unsigned short cu = lu[j], cv = lv[j];
            const int G = gp[cu];
            if (st[j] && (unsigned)s < tau[G]) {
                at[q] = atomicAdd(&s_nacc, 1);
                own[q] = (st[j] & 1) ? cu : cv;
                if (st[j] == 3 && own[q] == G) own[q] = cv;  // the pair's end that is not the root
                skey[at[q]] = ((unsigned long long)(unsigned)G << 32) | (unsigned)s;
            } else {
                ks[q] = s;
                kl[q] = (unsigned)cu | ((unsigned)cv << 16);
            }
        }
        __syncthreads();
        const int nacc = s_nacc;
        if (nacc == 0) {  // every round accepts each tree's mutual edge
            if (tid == 0) a.state[1] = 2;
            return;
        }
        int N = 1;
        while (N < nacc) N <<= 1;
        for (int i = nacc + tid; i < N; i += kTailThreads) skey[i] = ~0ull;  // padding sorts last
#pragma unroll
        for (int q = 0; q < kTailPer; q++)
            if (at[q] >= 0) sown[at[q]] = own[q];
        __syncthreads();
        for (int sz = 2; sz <= N; sz <<= 1) {
            for (int stride = sz >> 1; stride > 0; stride >>= 1) {
                for (int i = tid; i < (N >> 1); i += kTailThreads) {
                    const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                    const bool up = (lo & sz) == 0;
                    const unsigned long long ka = skey[lo], kb = skey[hi];
                    if ((ka > kb) == up) {
                        skey[lo] = kb;
                        skey[hi] = ka;
                        const unsigned short t = sown[lo];
                        sown[lo] = sown[hi];
                        sown[hi] = t;
                    }
                }
                __syncthreads();
            }
        }
        // chains: each thread a run of consecutive sorted edges
        const int C = (nacc + kTailThreads - 1) / kTailThreads;  // <= kTailPer
        const int x0 = tid * C;
        int add[kTailPer], n1[kTailPer], n2[kTailPer];
        bool hd[kTailPer];
        SegVal agg{0, 0};
#pragma unroll
        for (int q = 0; q < kTailPer; q++) {
            const int x = x0 + q;
            if (q >= C || x >= nacc) continue;
            const unsigned long long k = skey[x];
            const int G = (int)(k >> 32), Y = sown[x];
            hd[q] = x == 0 || (int)(skey[x - 1] >> 32) != G;
            n2[q] = root[Y];
            add[q] = size[Y];
            if (hd[q]) {  // the mutual pair: its other end is the tree's root
                n1[q] = root[G];
                add[q] += size[G];
            } else {
                n1[q] = E + (int)(unsigned)skey[x - 1];
            }
            agg = seg_add(agg, SegVal{add[q], hd[q] ? 1 : 0});
        }
        // sizes along each chain: a segmented inclusive sum over the runs
        SegVal inc = agg;
        for (int d = 1; d < 32; d <<= 1) {
            SegVal o;
            o.v = ::__shfl_up_sync(0xffffffffu, inc.v, d);
            o.f = ::__shfl_up_sync(0xffffffffu, inc.f, d);
            if (lane >= d) inc = seg_add(o, inc);
        }
        if (lane == 31) s_warp[wid] = inc;
        SegVal ex;
        ex.v = ::__shfl_up_sync(0xffffffffu, inc.v, 1);
        ex.f = ::__shfl_up_sync(0xffffffffu, inc.f, 1);
        if (lane == 0) ex = SegVal{0, 0};
        __syncthreads();  // also orders the chains' reads of size and root before the writes below
        SegVal run{0, 0};
        for (int i = 0; i < wid; i++) run = seg_add(run, s_warp[i]);
        run = seg_add(run, ex);
#pragma unroll
        for (int q = 0; q < kTailPer; q++) {
            const int x = x0 + q;
            if (q >= C || x >= nacc) continue;
            run = seg_add(run, SegVal{add[q], hd[q] ? 1 : 0});
            const unsigned long long k = skey[x];
            const int G = (int)(k >> 32), s = (int)(unsigned)k, node = E + s;
            const bool tail = x == nacc - 1 || (int)(skey[x + 1] >> 32) != G;
            DRow *r = a.row + s;
            store_sector(r, pack_i32(min(n1[q], n2[q]), max(n1[q], n2[q])),
                         pack_i32(tail ? -1 : E + (int)(unsigned)skey[x + 1], 0), (unsigned long long)run.v, 0ull);
            if (n2[q] < E) a.parent[n2[q]] = node;
            else a.row[n2[q] - E].parent = node;
            if (hd[q]) {
                if (n1[q] < E) a.parent[n1[q]] = node;
                else a.row[n1[q] - E].parent = node;
            }
            gp[sown[x]] |= kMerged;
            if (tail) {
                size[G] = (int)run.v;
                root[G] = node;
            }
        }
        __syncthreads();
        // the edges not accepted stay live, their labels moved one hop
#pragma unroll
        for (int q = 0; q < kTailPer; q++) {
            if (ks[q] < 0) continue;
            const int i = atomicAdd(&s_nkeep, 1);
            const unsigned short cu = (unsigned short)kl[q], cv = (unsigned short)(kl[q] >> 16);
            rank[i] = ks[q];
            lu[i] = (gp[cu] & kMerged) ? gp[cu] & (kMerged - 1) : cu;
            lv[i] = (gp[cv] & kMerged) ? gp[cv] & (kMerged - 1) : cv;
        }
        __syncthreads();
        na = s_nkeep;
        round++;
        __syncthreads();
    }
    if (tid == 0) a.state[0] = round;
}

void plan_dendro(Arena &ws, const Problem &p, Dendro &o) {
    o.a = ws.take<int32_t>(p.E);
    o.b = ws.take<int32_t>(p.E);
    o.size = ws.take<int64_t>(p.E);
    o.parent = ws.take<int32_t>(2 * p.E + 1);
}

struct DScratch {
    int32_t *svpar, *gp, *act, *act2, *ecu, *ecv, *ecu2, *ecv2;
    unsigned char *st;
    SvRec *sv;
    int *state;
    DRow *row;
    unsigned long long *minr, *tau;  // round-stamped slots (see rkey)
    int *gcnt;
    int2 *gseg, *segA, *segC, *kids;
    int4 *segB;
    int32_t *slot;
    long long *contrib;
    unsigned *ccnt;
    SegVal *cagg;
    unsigned long long *k1, *k2, *v1, *v2;
    void *radix;
};
// CTAs the per-CTA counts have room for, whatever the device.
static int chunk_room(int64_t E) { return std::max(sort_ranges_of(E, kSRanges), mid_ctas(E, kSRanges, kSRanges)); }
static DScratch carve_dendro(Arena &a, const Problem &p) {
    DScratch s;
    int64_t E = p.E;
    s.svpar = a.take<int32_t>(E);
    s.sv = a.take<SvRec>(E);
    s.state = a.take<int>(20);  // state[4], then tot[8] as 64-bit words
    s.row = a.take<DRow>(E);
    s.minr = a.take<unsigned long long>(E);
    s.tau = a.take<unsigned long long>(E);
    s.gp = a.take<int32_t>(E);
    s.act = a.take<int32_t>(E);
    s.act2 = a.take<int32_t>(E);
    s.ecu = a.take<int32_t>(E);
    s.ecv = a.take<int32_t>(E);
    s.ecu2 = a.take<int32_t>(E);
    s.ecv2 = a.take<int32_t>(E);
    s.st = a.take<unsigned char>(E);
    s.gcnt = a.take<int>(E);
    s.gseg = a.take<int2>(E);
    s.slot = a.take<int32_t>(E);
    s.segA = a.take<int2>(E);
    s.segB = a.take<int4>(E);
    s.segC = a.take<int2>(E);
    s.kids = a.take<int2>(E);
    s.contrib = a.take<long long>(E);
    const int64_t ctas = chunk_room(E);
    s.ccnt = a.take<unsigned>(ctas);
    s.cagg = a.take<SegVal>(ctas);
    s.k1 = a.take<unsigned long long>(E);
    s.k2 = a.take<unsigned long long>(E);
    s.v1 = a.take<unsigned long long>(E);
    s.v2 = a.take<unsigned long long>(E);
    s.radix = a.take<char>(radix_scratch_bytes(E));
    return s;
}
size_t dendro_scratch_bytes(const Problem &p) {
    Arena a(nullptr, 0);
    carve_dendro(a, p);
    return a.off;
}

dgec_status stage_dendro(Ctx *c, const Problem &p, const Csr &g, const Msf &m, Dendro &o, void *scratch) {
    cudaStream_t st = c->stream;
    int64_t E = p.E, n = m.n;
    o.rounds = 0;
    if (E == 0) return DGEC_OK;
    Arena a(scratch, SIZE_MAX);
    DScratch s = carve_dendro(a, p);
    TK(c, "k_d_init", k_d_init<<<grid_for(E, kBlock, kStreamCap), kBlock, 0, st>>>(
                          E, n, m.ru, m.rv, g.orig_of, s.svpar, s.sv, s.minr, s.tau,
                          o.parent, s.act, s.ecu, s.ecv));
    const int lb = p.idbits > 0 ? p.idbits : 1;
    const int sbits = bits_for((uint64_t)(n > 1 ? n - 1 : 1));
    if (n > 1) {
        const int gn = grid_for(n, kBlock, kStreamCap);
        TK(c, "k_d_order_keys", k_d_order_keys<<<gn, kBlock, 0, st>>>(m.ru, n, sbits, s.k1));
        bool in_b;
        DG_TRY(radix_sort(c, RadixBuffers{s.k1, s.k2, nullptr, nullptr}, n, sbits, sbits + lb, s.radix, &in_b));
        TK(c, "k_d_order_act", k_d_order_act<<<gn, kBlock, 0, st>>>(c->stop(), in_b ? s.k2 : s.k1, n, sbits, m.rv, s.act,
                                                               s.ecu, s.ecv));
    }
    if (n > 0) {
        DArgs d{E, n, lb, sbits, s.act, s.act2, s.ecu, s.ecu2, s.ecv, s.ecv2, s.st, s.minr, s.tau, s.gp, s.svpar, s.sv,
                s.gcnt, s.gseg, s.slot, s.segA, s.segB, s.segC, (unsigned long long *)(s.state + 4), s.kids, s.contrib,
                s.row, o.parent,
                sort_args(c, RadixBuffers{s.k1, s.k2, s.v1, s.v2}, n, 0, lb + sbits, s.radix, E), s.ccnt, s.cagg,
                s.state, 1 << 16, c->walk(kDWalk), c->bar};
        DRound w{0, 0, kStampTop, n, 0, 0, false};
        CU_TRY(c, cudaMemsetAsync(s.state, 0, sizeof(int) * 20, st));
        CU_TRY(c, cudaMemsetAsync(s.gcnt, 0, sizeof(int) * E, st));
        const int most = std::max(sort_ranges_of(E, kSRanges), mid_ctas(E, c->num_sms, kSRanges));
        for (; w.na > kDLarge; w.round++) {
            if (w.round >= d.max_rounds)
                return set_err(c, DGEC_ERR_TIMEOUT, "dendrogram rounds exceeded %d", d.max_rounds);
            w.odd = w.round & 1;
            w.stamp = kStampTop - (unsigned)w.round;
            const int wide = (int)std::min<int64_t>(cdiv(w.na, kSThreads), c->stream_ctas);
            const int few = (int)std::min<int64_t>(std::min<int64_t>(cdiv(w.na, kDTile), 4 * (int64_t)c->num_sms), most);
            w.G = wide;
            TK(c, "k_d_bid", k_d_bid<<<wide, kSThreads, 0, st>>>(d, w));
            w.G = (int)std::min<int64_t>(cdiv(w.na, kDTile), c->stream_ctas);
            TK(c, "k_d_ptr", k_d_ptr<<<w.G, kSThreads, 0, st>>>(d, w));
            w.G = wide;
            if (d.walk == kDWalk) TK(c, "k_d_gjump", k_d_jump<<<wide, kSThreads, 0, st>>>(d, w));
            else TK(c, "k_d_gjump", k_d_jump_n<<<wide, kSThreads, 0, st>>>(d, w));
            DG_TRY(coop_grid(c, kCoopDJump, (const void *)k_d_settle, kSThreads, 0, &w.G));
            w.G = std::min(w.G, c->num_sms);  // hardly ever with work to do: no more than it takes
            {
                d.bar = c->next_bar();
                void *args[] = {&d};
                cudaError_t e;
                TK(c, "k_d_settle", e = cudaLaunchCooperativeKernel((const void *)k_d_settle, dim3((unsigned)w.G),
                                                                    dim3(kSThreads), args, 0, st));
                if (e != cudaSuccess) return set_err(c, DGEC_ERR_CUDA, "k_d_settle launch: %s", cudaGetErrorString(e));
            }
            w.G = wide;
            TK(c, "k_d_tau", k_d_tau<<<wide, kSThreads, 0, st>>>(d, w));
            w.G = few;
            TK(c, "k_d_accept", k_d_accept<<<few, kSThreads, 0, st>>>(d, w));
            w.G = (int)std::min<int64_t>(cdiv(w.na, kDTile), c->stream_ctas);
            TK(c, "k_d_alloc", k_d_alloc<<<w.G, kSThreads, 0, st>>>(d, w));
            w.G = few;
            TK(c, "k_d_emit", k_d_emit<<<few, kSThreads, 0, st>>>(d, w));
            int64_t h[6];  // state, then tot
            DG_TRY(read_counters(c, (const int64_t *)s.state, 6, h));
            const int64_t kept = (int)(h[1] & 0xffffffff);
            if (kept == w.na) return set_err(c, DGEC_ERR_INTERNAL, "dendrogram round accepted no edge");
            w.nsmall = h[2 + (w.round & 1)];
            w.nacc = h[4 + (w.round & 1)];
            CU_TRY(c, cudaMemsetAsync(d.tot, 0, 8 * sizeof(unsigned long long), st));
            if (w.nsmall > 0) {
                w.G = (int)std::min<int64_t>(cdiv(w.nsmall, kSThreads), c->stream_ctas);
                TK(c, "k_d_small", k_d_small<<<w.G, kSThreads, 0, st>>>(d, w));
            }
            if (w.nacc > 0) {
                bool in_b;
                DG_TRY(radix_sort(c, RadixBuffers{s.k1, s.k2, s.v1, s.v2}, w.nacc, 0, lb + sbits, s.radix, &in_b));
                const unsigned long long *key = in_b ? s.k2 : s.k1, *val = in_b ? s.v2 : s.v1;
                w.G = (int)std::min<int64_t>(std::min<int64_t>(cdiv(w.nacc, kDTile), 4 * (int64_t)c->num_sms), most);
                TK(c, "k_d_chain", k_d_chain<<<w.G, kSThreads, 0, st>>>(d, w, key, val));
                TK(c, "k_d_rows", k_d_rows<<<w.G, kSThreads, 0, st>>>(d, w, key, val));
            }
            w.na = kept;
        }
        {
            const size_t smem = sort_smem_bytes<SortWide, true>();
            int grid = 1;
            DG_TRY(coop_grid(c, kCoopDendro, (const void *)k_d_rounds, kSThreads, smem, &grid));
            grid = w.na > kTailMax ? std::min(grid, mid_ctas(w.na, c->num_sms, most)) : 1;
            d.bar = c->next_bar();
            void *args[] = {&d, &w};
            cudaError_t e;
            TK(c, "k_d_rounds", e = cudaLaunchCooperativeKernel((const void *)k_d_rounds, dim3((unsigned)grid),
                                                                dim3(kSThreads), args, smem, st));
            if (e != cudaSuccess) return set_err(c, DGEC_ERR_CUDA, "k_d_rounds launch: %s", cudaGetErrorString(e));
        }
        CU_TRY(c, cudaFuncSetAttribute(k_d_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmem));
        TK(c, "k_d_tail", k_d_tail<<<1, kTailThreads, kTailSmem, st>>>(d));
    }
    if (n > 0)
        TK(c, "k_d_split", k_d_split<<<grid_for(n, kBlock, kStreamCap), kBlock, 0, st>>>(s.row, n, o.a, o.b, o.size,
                                                                                    o.parent + E));
    if (n > 0) {
        int64_t ts;
        DG_TRY(read_counters(c, (const int64_t *)s.state, 1, &ts));
        const int err = (int)(ts >> 32);
        if (err == 1) return set_err(c, DGEC_ERR_TIMEOUT, "dendrogram rounds exceeded %d", 1 << 16);
        if (err) return set_err(c, DGEC_ERR_INTERNAL, "dendrogram round accepted no edge");
        o.rounds = (int)(ts & 0xffffffff);
    }
    return DGEC_OK;
}

}  // namespace dgec
