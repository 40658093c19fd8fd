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
// (186 us), 3M 290 us (384 us), 50M 3.33 ms (3.37 ms), 200M keys of 27 bits 4.87 ms (6.55 ms). 512
// threads of 8 keys at 2 CTAs an SM measured best of 128 to 512 threads and 4
// to 16 keys a thread: smaller tiles write shorter runs, larger ones leave one
// CTA an SM.
template <bool VALS>
__global__ void __launch_bounds__(kSThreads, 2) k_radix_sort(SortArgs a) {
    extern __shared__ __align__(16) unsigned long long sort_sm[];
    const SortSmem s = sort_smem<VALS>(sort_sm);
    GridBar bar(a.bar);
    if (bar.stopped()) return;
    if (sort_run<VALS>(a, a.n, a.begin_bit, a.end_bit, a.most, s, bar)) bar.finish();
}

size_t radix_scratch_bytes(int64_t n) {
    if (n <= kSTile) return 256;
    return ((size_t)cdiv(n, kSTile) + 2 * sort_ranges_of(n, kSRanges) + 1) * kSBins * sizeof(unsigned);
}

SortArgs sort_args(Ctx *c, RadixBuffers buf, int64_t n, int begin_bit, int end_bit, void *scratch, int64_t cap) {
    unsigned *w = (unsigned *)scratch;
    const size_t R = (size_t)sort_ranges_of(cap, kSRanges) * kSBins;
    return SortArgs{buf.ka, buf.kb, buf.va, buf.vb, n, begin_bit, end_bit, buf.va && n > kSNarrow ? kSBits - 1 : kSBits,
                    w, w + R, w + 2 * R, w + 2 * R + kSBins, c->next_bar()};
}

template <bool VALS>
static dgec_status launch_sort(Ctx *c, const SortArgs &a) {
    const size_t smem = sort_smem_bytes<VALS>();
    int grid = 1;
    DG_TRY(coop_grid(c, VALS ? kCoopSortKV : kCoopSortK, (const void *)k_radix_sort<VALS>, kSThreads, smem, &grid));
    grid = sort_ranges_of(a.n, grid);
    return coop_launch(c, VALS ? "k_radix_sort_kv" : "k_radix_sort", (const void *)k_radix_sort<VALS>, grid, kSThreads, smem, a);
}

dgec_status radix_sort(Ctx *c, RadixBuffers buf, int64_t n, int begin_bit, int end_bit,
                       void *scratch, bool *in_b) {
    *in_b = false;
    if (n <= 1 || end_bit <= begin_bit) return DGEC_OK;
    if (n >> 32) return set_err(c, DGEC_ERR_TOO_LARGE, "sort of %lld keys: at most 2^32 - 1", (long long)n);
    const SortArgs a = sort_args(c, buf, n, begin_bit, end_bit, scratch, n);
    *in_b = sort_in_b(n, end_bit - begin_bit, a.most);
    return buf.va ? launch_sort<true>(c, a) : launch_sort<false>(c, a);
}

}  // namespace dgec
