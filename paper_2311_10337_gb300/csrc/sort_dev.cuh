// The stable LSD radix sort as device code of cooperative kernels, called by
// k_radix_sort (prims.cu) and by the dendrogram rounds (dendro.cu).
#pragma once

#include "coop.cuh"
#include "prims.cuh"

namespace dgec {

// All passes of a sort run in one cooperative launch. A pass counts the
// digits of every tile, turns the counts into places, and scatters: each
// warp ranks its keys with ballots (keys in position order), the CTA
// combines warp counts, stages the tile in shared memory in digit order and
// writes it out so that runs of one digit land contiguously, while the next
// tile's loads are already in flight.
struct AddI {
    __device__ __forceinline__ int operator()(int a, int b) const { return a + b; }
};
constexpr int kSItems = 8;  // keys a thread holds
template <int THREADS, int BITS>
struct SortForm {
    static constexpr int kThreads = THREADS;
    static constexpr int kTile = THREADS * kSItems;
    static constexpr int kWarps = THREADS / 32;
    static constexpr int kBits = BITS;  // of the widest digit
    static constexpr int kBins = 1 << BITS;
    static constexpr int kPer = (kBins + THREADS - 1) / THREADS;  // digits a thread owns (consecutive)
    static constexpr int kCtas = 1024 / THREADS;                  // an SM
};
// Wide digits need fewer passes; narrow ones make longer runs, and smaller
// CTAs wait less at their barriers. prims.cu says which sort takes which.
using SortWide = SortForm<512, 9>;
using SortNarrow = SortForm<256, 8>;
constexpr int kSThreads = SortWide::kThreads, kSTile = SortWide::kTile, kSWarps = SortWide::kWarps, kSBits = SortWide::kBits;
constexpr int kSDirect = 64;           // up to this many CTAs each adds up the others' counts itself
constexpr int kSRanges = 1024;         // most CTAs of a sort
constexpr int kSDeal = 8;              // tiles a CTA above which they are dealt out
constexpr int kSNextWord = 32;         // barrier word that deals out the tiles (a line of its own)

struct SortSmem {
    unsigned long long *keys, *vals;  // [kTile] staged tile
    unsigned short *wcnt;             // [kWarps][kBins]
    unsigned *goff;                   // [kBins]
    int *scan;                        // [kWarps], then the next tile
};
template <class F, bool VALS>
constexpr size_t sort_smem_bytes() {
    return (size_t)F::kTile * 8 * (VALS ? 2 : 1) + (size_t)F::kWarps * F::kBins * 2 + (size_t)F::kBins * 4 + (F::kWarps + 1) * 4;
}
template <class F, bool VALS>
__device__ __forceinline__ SortSmem sort_smem(unsigned long long *p) {
    SortSmem s;
    s.keys = p;
    s.vals = p + F::kTile;
    s.goff = (unsigned *)(p + (VALS ? 2 : 1) * F::kTile);
    s.wcnt = (unsigned short *)(s.goff + F::kBins);
    s.scan = (int *)(s.wcnt + F::kWarps * F::kBins);
    return s;
}

// Exclusive prefix over the values of the CTA's threads.
template <int WARPS = kSWarps>
__device__ __forceinline__ int sort_block_exclusive(int v, int *sm) {
    const int w = threadIdx.x >> 5;
    const int inc = warp_inclusive(v, AddI{});
    if (lane_id() == 31) sm[w] = inc;
    __syncthreads();
    int base = 0;
#pragma unroll
    for (int i = 0; i < WARPS; i++) base += i < w ? sm[i] : 0;
    return base + inc - v;
}

// The lanes of the warp whose `d` (nb bits) equals this lane's, among the
// lanes in `valid`. One ballot a bit: __match_any_sync takes time with the
// number of distinct values (about 100 cycles of an SM for 32 of them).
template <int BITS>
__device__ __forceinline__ unsigned same_digit(unsigned d, int nb, unsigned valid) {
    unsigned peers = valid;
#pragma unroll
    for (int b = 0; b < BITS; b++) {
        if (b >= nb) break;
        const unsigned bit = (d >> b) & 1u;
        peers &= __ballot_sync(0xffffffffu, bit) ^ (bit - 1u);
    }
    return peers;
}

// Rank the tile's keys (digit = (k >> shift) & mask, nv valid items in this
// lane): on return lpos[i] is item i's place in digit order within the tile,
// and the calling thread's digit has `start` (its first place) and `total`.
template <class F>
__device__ __forceinline__ void sort_rank(const SortSmem &s, const unsigned long long (&k)[kSItems], int nv, int shift,
                                          int nb, unsigned short (&lpos)[kSItems], int (&start)[F::kPer], int (&total)[F::kPer],
                                          int warps = F::kWarps) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned short *mine = s.wcnt + warp * F::kBins;
    // each warp clears its own counters (8 a lane and step)
    for (int i = lane * 8; i < (1 << nb); i += 256) *(uint4 *)(mine + i) = make_uint4(0, 0, 0, 0);
    __syncwarp();
    const unsigned lt = (1u << lane) - 1u, mask = (1u << nb) - 1u;
#pragma unroll
    for (int i = 0; i < kSItems; i++) {
        const unsigned d = (unsigned)(k[i] >> shift) & mask;
        const unsigned peers = same_digit<F::kBits>(d, nb, __ballot_sync(0xffffffffu, i < nv));
        const int before = i < nv ? mine[d] : 0;
        lpos[i] = (unsigned short)(before + __popc(peers & lt));
        __syncwarp();
        if ((peers & lt) == 0 && i < nv) mine[d] = (unsigned short)(before + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    int run = 0, tot[F::kPer];
#pragma unroll
    for (int q = 0; q < F::kPer; q++) {
        const unsigned d = threadIdx.x * F::kPer + q;
        int sum = 0;
        if (d <= mask) {
#pragma unroll
            for (int w = 0; w < F::kWarps; w++)
                if (w < warps) sum += s.wcnt[w * F::kBins + d];
        }
        tot[q] = sum;
        run += sum;
    }
    int st = sort_block_exclusive<F::kWarps>(run, s.scan);
#pragma unroll
    for (int q = 0; q < F::kPer; q++) {
        const unsigned d = threadIdx.x * F::kPer + q;
        start[q] = st;
        total[q] = tot[q];
        if (d <= mask) {
            int at = st;
#pragma unroll
            for (int w = 0; w < F::kWarps; w++) {
                if (w >= warps) break;
                const int c = s.wcnt[w * F::kBins + d];
                s.wcnt[w * F::kBins + d] = (unsigned short)at;
                at += c;
            }
        }
        st += tot[q];
    }
}
// (the caller synchronises, then adds s.wcnt[warp][digit] to lpos)

template <class F, bool VALS>
__device__ __forceinline__ void sort_load(const unsigned long long *kin, const unsigned long long *vin, int64_t n,
                                          int64_t base, unsigned long long (&k)[kSItems],
                                          unsigned long long (&v)[kSItems], int *nv) {
    const int64_t w0 = base + (threadIdx.x >> 5) * (32 * kSItems) + (threadIdx.x & 31);
    const int64_t left = n - w0;
    *nv = left <= 0 ? 0 : left >= 32 * kSItems ? kSItems : (int)((left + 31) >> 5);
#pragma unroll
    for (int i = 0; i < kSItems; i++) {
        k[i] = i < *nv ? kin[w0 + i * 32] : 0ull;
        if (VALS) v[i] = i < *nv ? vin[w0 + i * 32] : 0ull;
    }
}

// Digit width of a pass with `bits_left` to sort: spread evenly over the
// fewest passes of at most `most` bits.
__device__ __forceinline__ int sort_pass_bits(int bits_left, int most) {
    const int passes = (bits_left + most - 1) / most;
    return (bits_left + passes - 1) / passes;
}

struct SortArgs {
    unsigned long long *ka, *kb, *va, *vb;
    int64_t n;
    int begin_bit, end_bit, most;  // most: bits of the widest digit
    unsigned *rtot, *rpre;  // [CTAs][digits]: digit counts of each CTA's range of tiles, and those of the ranges before
    unsigned *total;        // [digits]
    unsigned *tile;         // [tiles][digits]: keys of the digit in the range's tiles before
    BarRef bar;
};

// First places of the calling thread's digits: the keys of smaller digits
// plus those of the same digit in the ranges before `range` (`pre` adds more).
// With few ranges every CTA adds up the counts itself, else k_radix_sort has
// summed them (rpre, total).
template <class F>
__device__ __forceinline__ void sort_bases(const SortArgs &a, int nb, int ranges, int range, unsigned *sm,
                                           unsigned (&base)[F::kPer]) {
    const int tid = threadIdx.x, warp = tid >> 5, bins = 1 << nb;
    unsigned tot[F::kPer], mine = 0;
#pragma unroll
    for (int q = 0; q < F::kPer; q++) {
        const int d = tid * F::kPer + q;
        unsigned t = 0, pre = 0;
        if (d < bins) {
            if (ranges > kSDirect) {
                t = a.total[d];
                if (range >= 0) pre = a.rpre[range * bins + d];
            } else {
#pragma unroll 8
                for (int x = 0; x < ranges; x++) {
                    const unsigned y = a.rtot[x * bins + d];
                    t += y;
                    if (x < range) pre += y;
                }
            }
        }
        tot[q] = t;
        mine += t;
        base[q] = pre;
    }
    const unsigned inc = warp_inclusive((int)mine, AddI{});
    if ((tid & 31) == 31) sm[warp] = inc;
    __syncthreads();
    unsigned run = inc - mine;
#pragma unroll
    for (int w = 0; w < F::kWarps; w++) run += w < warp ? sm[w] : 0u;
#pragma unroll
    for (int q = 0; q < F::kPer; q++) {
        base[q] += run;
        run += tot[q];
    }
    __syncthreads();
}

// Counts of the ranges to exclusive prefixes over the ranges and totals: a
// CTA takes 32 digits, each of its warps a run of ranges.
template <class F>
__device__ __forceinline__ void sort_ranges(const SortArgs &a, int nb, int ranges, unsigned *part) {
    const int bins = 1 << nb, tid = threadIdx.x, warp = tid >> 5;
    for (int g = blockIdx.x; g * 32 < bins; g += gridDim.x) {
        const int d = g * 32 + (tid & 31);
        const int r0 = ranges * warp / F::kWarps, r1 = ranges * (warp + 1) / F::kWarps;
        unsigned sum = 0;
        if (d < bins) {
#pragma unroll 8
            for (int r = r0; r < r1; r++) sum += a.rtot[r * bins + d];
        }
        part[tid] = sum;
        __syncthreads();
        unsigned run = 0;
        for (int w = 0; w < warp; w++) run += part[w * 32 + (tid & 31)];
        if (d < bins) {
            if (warp == F::kWarps - 1) a.total[d] = run + sum;
#pragma unroll 8
            for (int r = r0; r < r1; r++) {
                const unsigned x = a.rtot[r * bins + d];
                a.rpre[r * bins + d] = run;
                run += x;
            }
        }
        __syncthreads();
    }
}

// The ranked tile into shared memory in digit order.
template <class F, bool VALS>
__device__ __forceinline__ void sort_stage(const SortSmem &s, const unsigned long long (&k)[kSItems],
                                           const unsigned long long (&v)[kSItems], int nv, int shift, unsigned mask,
                                           const unsigned short (&lpos)[kSItems]) {
    const unsigned short *mine = s.wcnt + (threadIdx.x >> 5) * F::kBins;
#pragma unroll
    for (int i = 0; i < kSItems; i++) {
        if (i >= nv) continue;
        const int at = lpos[i] + mine[(unsigned)(k[i] >> shift) & mask];
        s.keys[at] = k[i];
        if (VALS) s.vals[at] = v[i];
    }
}

// m staged keys to their places.
template <class F, bool VALS>
__device__ __forceinline__ void sort_write(const SortSmem &s, int m, int shift, unsigned mask, unsigned long long *kout,
                                           unsigned long long *vout) {
#pragma unroll
    for (int i = 0; i < kSItems; i++) {
        const int j = i * F::kThreads + threadIdx.x;
        if (j >= m) continue;
        const unsigned long long key = s.keys[j];
        const unsigned g = s.goff[(unsigned)(key >> shift) & mask] + (unsigned)j;
        kout[g] = key;
        if (VALS) vout[g] = s.vals[j];
    }
}

// Where the sorted keys end up (no key is moved for one or none).
template <class F = SortWide>
__host__ __device__ __forceinline__ bool sort_in_b(int64_t n, int bits, int most) {
    return n > 1 && bits > 0 && (n <= F::kTile || (((bits + most - 1) / most) & 1));
}

// CTAs a sort of n keys uses, of `ctas` there are.
template <class F = SortWide>
__host__ __device__ __forceinline__ int sort_ranges_of(int64_t n, int ctas) {
    const int64_t tiles = (n + F::kTile - 1) / F::kTile;
    int64_t r = tiles < kSRanges ? tiles : kSRanges;
    if (r > ctas) r = ctas;
    return r > 1 ? (int)r : 1;
}

// The sort, called by every CTA of a cooperative grid of F::kThreads threads
// (the last ones only keep the barriers company when there are more CTAs than
// tiles). False when a barrier gave up. No barrier after the last pass.
template <class F, bool VALS>
__device__ __forceinline__ bool sort_run(const SortArgs &a, int64_t n, int begin_bit, int end_bit, int most,
                                         const SortSmem &s, GridBar &bar) {
    const int tid = threadIdx.x, warp = tid >> 5;
    unsigned long long k[kSItems], v[kSItems];
    unsigned short lpos[kSItems];
    int nv, start[F::kPer], total[F::kPer];
    if (n <= 1 || end_bit <= begin_bit) return true;
    if (n <= F::kTile) {  // one tile: every pass in shared memory, result in the b buffers
        if (blockIdx.x != 0) return true;
        const int at0 = warp * (32 * kSItems) + (tid & 31);
        sort_load<F, VALS>(a.ka, a.va, n, 0, k, v, &nv);
        for (int shift = begin_bit; shift < end_bit;) {
            const int nb = sort_pass_bits(end_bit - shift, most);
            sort_rank<F>(s, k, nv, shift, nb, lpos, start, total, ((int)n + 32 * kSItems - 1) / (32 * kSItems));
            __syncthreads();
            sort_stage<F, VALS>(s, k, v, nv, shift, (1u << nb) - 1u, lpos);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kSItems; i++) {
                if (i >= nv) continue;
                k[i] = s.keys[at0 + i * 32];
                if (VALS) v[i] = s.vals[at0 + i * 32];
            }
            shift += nb;
        }
#pragma unroll
        for (int i = 0; i < kSItems; i++) {
            if (i >= nv) continue;
            a.kb[at0 + i * 32] = k[i];
            if (VALS) a.vb[at0 + i * 32] = v[i];
        }
        return true;
    }
    const int tiles = (int)((n + F::kTile - 1) / F::kTile), ranges = sort_ranges_of<F>(n, (int)gridDim.x), me = blockIdx.x;
    const bool in = me < ranges;
    const unsigned long long *kin = a.ka, *vin = a.va;
    unsigned long long *kout = a.kb, *vout = a.vb;
    for (int shift = begin_bit; shift < end_bit;) {
        const int nb = sort_pass_bits(end_bit - shift, most), bins = 1 << nb;
        const unsigned mask = (unsigned)bins - 1u;
        unsigned next[F::kPer];
        if (tiles <= ranges) {
            // one tile a CTA: it stays in registers across the barrier, and its ranking gives its counts
            if (in) {
                sort_load<F, VALS>(kin, vin, n, (int64_t)me * F::kTile, k, v, &nv);
                sort_rank<F>(s, k, nv, shift, nb, lpos, start, total);
#pragma unroll
                for (int q = 0; q < F::kPer; q++)
                    if (tid * F::kPer + q < bins) a.rtot[me * bins + tid * F::kPer + q] = (unsigned)total[q];
            }
            if (!bar.sync()) return false;
            if (ranges > kSDirect) {
                sort_ranges<F>(a, nb, ranges, (unsigned *)s.keys);
                if (!bar.sync()) return false;
            }
            if (in) {
                sort_bases<F>(a, nb, ranges, me, (unsigned *)s.scan, next);
#pragma unroll
                for (int q = 0; q < F::kPer; q++)
                    if (tid * F::kPer + q < bins) s.goff[tid * F::kPer + q] = next[q] - (unsigned)start[q];
                sort_stage<F, VALS>(s, k, v, nv, shift, mask, lpos);
                __syncthreads();
                const int64_t left = n - (int64_t)me * F::kTile;
                sort_write<F, VALS>(s, left < F::kTile ? (int)left : F::kTile, shift, mask, kout, vout);
            }
        } else {
            // digit counts of the CTA's own range of tiles, with the prefix over
            // the range at every tile
            const int t0 = (int)((int64_t)tiles * me / ranges), t1 = (int)((int64_t)tiles * (me + 1) / ranges);
            unsigned run[F::kPer];
#pragma unroll
            for (int q = 0; q < F::kPer; q++) run[q] = 0;
            unsigned *cnt = (unsigned *)s.wcnt;  // 8 copies of the counters, two warps each
            static_assert((F::kWarps / 2) * F::kBins * 4 <= F::kWarps * F::kBins * 2, "counter copies");
            for (int t = t0; in && t < t1; t++) {
                unsigned long long kk[kSItems];
                const int64_t b0 = (int64_t)t * F::kTile + tid;
#pragma unroll
                for (int i = 0; i < kSItems; i++) kk[i] = b0 + i * F::kThreads < n ? kin[b0 + i * F::kThreads] : 0ull;
                for (int i = tid; i < (F::kWarps / 2) * bins; i += F::kThreads) cnt[i] = 0u;
                __syncthreads();
#pragma unroll
                for (int i = 0; i < kSItems; i++)
                    if (b0 + i * F::kThreads < n) atomicAdd(&cnt[(warp >> 1) * bins + ((unsigned)(kk[i] >> shift) & mask)], 1u);
                __syncthreads();
#pragma unroll
                for (int q = 0; q < F::kPer; q++) {
                    const int d = tid * F::kPer + q;
                    if (d >= bins) continue;
                    a.tile[(size_t)t * bins + d] = run[q];
#pragma unroll
                    for (int i = 0; i < F::kWarps / 2; i++) run[q] += cnt[i * bins + d];
                }
                __syncthreads();
            }
#pragma unroll
            for (int q = 0; q < F::kPer; q++)
                if (in && tid * F::kPer + q < bins) a.rtot[me * bins + tid * F::kPer + q] = run[q];
            if (me == 0 && tid == 0) bar.ref.word[kSNextWord] = 0u;
            if (!bar.sync()) return false;
            sort_ranges<F>(a, nb, ranges, (unsigned *)s.keys);
            if (!bar.sync()) return false;
            // the tiles in order: what is written at one time is one contiguous
            // stretch a digit. Over a long pass the CTAs would drift apart, so there
            // each takes the next tile as it comes free (the sorts of pairs of a call
            // on 100M hub edges: 18.3 ms with every CTA's tiles fixed, 17.2 so; of
            // 1M to 6M edges 1 to 2 % longer so).
            unsigned base[F::kPer], tp[F::kPer];
            sort_bases<F>(a, nb, ranges, -1, (unsigned *)s.scan, base);
            auto load_prefix = [&](int t) {
                int r = (int)((int64_t)t * ranges / tiles);
                if ((int)((int64_t)tiles * (r + 1) / ranges) <= t) r++;
#pragma unroll
                for (int q = 0; q < F::kPer; q++) {
                    const int d = tid * F::kPer + q;
                    tp[q] = d < bins ? a.tile[(size_t)t * bins + d] + a.rpre[r * bins + d] : 0u;
                }
            };
            int t = in ? me : tiles;
            if (in) {
                sort_load<F, VALS>(kin, vin, n, (int64_t)t * F::kTile, k, v, &nv);
                load_prefix(t);
            }
            unsigned *next = bar.ref.word + kSNextWord;
            const bool deal = tiles > kSDeal * ranges;
            int ahead = 0;  // (thread 0) the tile after the next, asked for a tile in advance
            if (deal && in && tid == 0) ahead = ranges + (int)atomicAdd(next, 1u);
            while (t < tiles) {
                if (deal && tid == 0) {
                    s.scan[F::kWarps] = ahead;
                    ahead = ranges + (int)atomicAdd(next, 1u);
                }
                sort_rank<F>(s, k, nv, shift, nb, lpos, start, total);
                const int tn = deal ? s.scan[F::kWarps] : t + ranges;
#pragma unroll
                for (int q = 0; q < F::kPer; q++)
                    if (tid * F::kPer + q < bins) s.goff[tid * F::kPer + q] = base[q] + tp[q] - (unsigned)start[q];
                __syncthreads();
                sort_stage<F, VALS>(s, k, v, nv, shift, mask, lpos);
                __syncthreads();
                if (tn < tiles) {
                    sort_load<F, VALS>(kin, vin, n, (int64_t)tn * F::kTile, k, v, &nv);
                    load_prefix(tn);
                }
                const int64_t left = n - (int64_t)t * F::kTile;
                sort_write<F, VALS>(s, left < F::kTile ? (int)left : F::kTile, shift, mask, kout, vout);
                t = tn;
            }
        }
        shift += nb;
        if (shift < end_bit) {
            if (!bar.sync()) return false;
            const unsigned long long *tk = kin, *tv = vin;
            kin = kout;
            vin = vout;
            kout = const_cast<unsigned long long *>(tk);
            vout = const_cast<unsigned long long *>(tv);
        }
    }
    return true;
}


// The arguments of a sort of n keys whose scratch was sized for `cap` keys.
SortArgs sort_args(Ctx *c, RadixBuffers buf, int64_t n, int begin_bit, int end_bit, void *scratch, int64_t cap);

}  // namespace dgec
