// Device-wide scans and the stable LSD radix sort.
#include "sort_dev.cuh"

namespace dgec {

dgec_status exclusive_scan_i32(Ctx *c, const int *in, long long *out, int64_t n,
                               long long *scratch) {
    return device_scan<long long, SumI64, LoadI32AsI64, StorePtr<long long>>(
        c, LoadI32AsI64{in}, StorePtr<long long>{out}, n, SumI64{}, 0ll, false, scratch);
}

dgec_status exclusive_scan_i64(Ctx *c, const long long *in, long long *out, int64_t n,
                               long long *scratch) {
    return device_scan<long long, SumI64, LoadPtr<long long>, StorePtr<long long>>(
        c, LoadPtr<long long>{in}, StorePtr<long long>{out}, n, SumI64{}, 0ll, false, scratch);
}

// ------------------------------------------------------------ radix sort
// What bounds it: up to some 100,000 keys the launch and the two barriers of a
// pass; in L2's reach the latency of a tile's chain (load, ballots, counter
// updates, four CTA barriers); beyond, DRAM and the short write runs. One
// launch a sort, not five a pass: 20,000 pairs of 54 bits 63 us (171 us as
// separate histogram, three scan launches and scatter a pass), 300,000 pairs 88 us
// (186 us), 3M 290 us (384 us). All sorts of a call without clustering (22 to 24
// bits, mostly pairs) on 50M mid / 100M hub edges: 4.7 and 9.4 ms (4.7 and 9.0 a
// pass of launches; 5.4 and 10.8 in wide digits with every CTA's tiles fixed).
// 1,024 threads an SM in CTAs of 512 or 256, 8 keys a thread; larger tiles leave
// one CTA an SM.
template <class F, bool VALS>
__global__ void __launch_bounds__(F::kThreads, F::kCtas) k_radix_sort(SortArgs a) {
    extern __shared__ __align__(16) unsigned long long sort_sm[];
    const SortSmem s = sort_smem<F, VALS>(sort_sm);
    GridBar bar(a.bar);
    if (bar.stopped()) return;
    if (sort_run<F, VALS>(a, a.n, a.begin_bit, a.end_bit, a.most, s, bar)) bar.finish();
}

// (the narrow form needs no more: half the digits, twice the tiles)
size_t radix_scratch_bytes(int64_t n) {
    if (n <= SortWide::kTile) return 256;
    return ((size_t)cdiv(n, SortWide::kTile) + 2 * sort_ranges_of(n, kSRanges) + 1) * SortWide::kBins * sizeof(unsigned);
}

template <class F>
static SortArgs form_args(Ctx *c, RadixBuffers buf, int64_t n, int begin_bit, int end_bit, void *scratch, int64_t cap) {
    unsigned *w = (unsigned *)scratch;
    const size_t R = (size_t)sort_ranges_of<F>(cap, kSRanges) * F::kBins;
    return SortArgs{buf.ka, buf.kb, buf.va, buf.vb, n, begin_bit, end_bit, F::kBits, w, w + R, w + 2 * R, w + 2 * R + F::kBins,
                    c->next_bar()};
}
SortArgs sort_args(Ctx *c, RadixBuffers buf, int64_t n, int begin_bit, int end_bit, void *scratch, int64_t cap) {
    return form_args<SortWide>(c, buf, n, begin_bit, end_bit, scratch, cap);
}

template <class F, bool VALS>
static dgec_status launch_sort(Ctx *c, CoopKernel which, RadixBuffers buf, int64_t n, int begin_bit, int end_bit,
                               void *scratch, bool *in_b) {
    const SortArgs a = form_args<F>(c, buf, n, begin_bit, end_bit, scratch, n);
    *in_b = sort_in_b<F>(n, end_bit - begin_bit, a.most);
    const size_t smem = sort_smem_bytes<F, VALS>();
    const void *fn = (const void *)k_radix_sort<F, VALS>;
    int grid = 1;
    DG_TRY(coop_grid(c, which, fn, F::kThreads, smem, &grid));
    return coop_launch(c, VALS ? "k_radix_sort_kv" : "k_radix_sort", fn, sort_ranges_of<F>(n, grid), F::kThreads, smem, a);
}

// Narrow digits in CTAs of 256 threads for more than 2^24 keys where they need
// no pass more, and for more than 2^26 pairs in any case: the runs of 16 pairs
// then cost less than the passes that wide digits save. Sorts of pairs / of keys
// of a call on mid graphs, wide and narrow: 3M edges 0.65 and 0.65 / 0.23 and 0.26
// ms, 10M 1.65 and 1.65 / 0.52 and 0.52, 30M 4.8 and 4.6 / 1.40 and 1.38; 100M hub
// edges 17.2 and 16.4 / 4.5 and 4.3 (narrow also where it needs a pass more: 3M
// 0.69, 30M 4.6).
static bool narrow_form(int64_t n, int bits, bool vals) {
    const bool same = cdiv(bits, SortNarrow::kBits) == cdiv(bits, SortWide::kBits);
    return (same && n > (int64_t(1) << 24)) || (vals && n > (int64_t(1) << 26));
}

dgec_status radix_sort(Ctx *c, RadixBuffers buf, int64_t n, int begin_bit, int end_bit,
                       void *scratch, bool *in_b) {
    *in_b = false;
    if (n <= 1 || end_bit <= begin_bit) return DGEC_OK;
    if (n >> 32) return set_err(c, DGEC_ERR_TOO_LARGE, "sort of %lld keys: at most 2^32 - 1", (long long)n);
    const bool vals = buf.va != nullptr, narrow = narrow_form(n, end_bit - begin_bit, vals);
    if (vals)
        return narrow ? launch_sort<SortNarrow, true>(c, kCoopSortNarrowKV, buf, n, begin_bit, end_bit, scratch, in_b)
                      : launch_sort<SortWide, true>(c, kCoopSortKV, buf, n, begin_bit, end_bit, scratch, in_b);
    return narrow ? launch_sort<SortNarrow, false>(c, kCoopSortNarrowK, buf, n, begin_bit, end_bit, scratch, in_b)
                  : launch_sort<SortWide, false>(c, kCoopSortK, buf, n, begin_bit, end_bit, scratch, in_b);
}

}  // namespace dgec
