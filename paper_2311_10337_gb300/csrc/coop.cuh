// Cooperative building blocks: a grid barrier for kernels whose CTAs are all
// resident (cooperative launches), and pointer jumping inside such a kernel.
#pragma once

#include "common.cuh"

namespace dgec {

// Barrier over every CTA of a cooperative launch. Arrivals count up without
// a reset between barriers (compared by signed difference). CTAs of a
// cooperative launch are co-resident, so the limit on the polls (about a
// microsecond each) only bounds the wait should that ever not hold. A barrier
// that gives up writes the stop word (see BarRef) and returns false in every
// thread of its CTA; the kernel must then return at once. The other CTAs find
// the stop word or their own limit at the next barrier, which cannot complete,
// so no CTA goes on to read what the missing one has not written.
struct GridBar {
    BarRef ref;
    unsigned target;
    __device__ __forceinline__ explicit GridBar(const BarRef &r) : ref(r), target(0) {}
    // A kernel of the call has given up before: return at once, without finish().
    __device__ __forceinline__ bool stopped() const { return __syncthreads_or(*(volatile unsigned *)(ref.word + 2) != 0); }
    __device__ __forceinline__ void stop(StopCode code) {  // one thread or more
        *(volatile unsigned *)ref.err = code;
        *(volatile unsigned *)(ref.word + 2) = code;
    }
    __device__ __forceinline__ bool sync() {
        __syncthreads();
        if (gridDim.x == 1) return true;
        bool bad = false;
        target += gridDim.x;
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(ref.word, 1u);
            for (unsigned polls = 0;; polls++) {
                if (polls >= ref.polls || ((polls & 1023) == 1023 && *(volatile unsigned *)(ref.word + 2))) {
                    bad = true;
                    stop(kStopBarrier);
                    break;
                }
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ref.word) : "memory");
                if ((int)(v - target) >= 0) break;
            }
            __threadfence();
        }
        return !__syncthreads_or(bad);
    }
    // every CTA calls this after its last barrier
    __device__ __forceinline__ void finish() {
        if (gridDim.x == 1 || threadIdx.x != 0) return;
        if (atomicAdd(ref.word + 1, 1u) == gridDim.x - 1) {
            ref.word[0] = 0u;
            ref.word[1] = 0u;
        }
    }
};

// The cut walks of a pass: their pointers' owners, in any order.
__device__ __forceinline__ void list_cut(int32_t *list, unsigned long long *n, int x) {
    const unsigned m = __activemask();  // whichever lanes are here
    const int leader = __ffs(m) - 1;
    unsigned long long at = 0;
    if ((int)lane_id() == leader) at = atomicAdd(n, (unsigned long long)__popc(m));
    at = __shfl_sync(m, at, leader);
    list[at + __popc(m & ((1u << lane_id()) - 1u))] = x;
}

// The items of such a list. They alone are unsettled: the other walks ended at
// a fixed point.
struct ListItem {
    const int32_t *list;
    __device__ __forceinline__ int64_t operator()(int64_t i) const { return list[i]; }
};

// In-place pointer jumping, ptr[x] = ptr[ptr[x]], over the n pointers x =
// item(i) (negative: none), in rounds until none moves. Pointers only move to
// ancestors and fixed points are never written, so reading a neighbour's new
// or old value is equally valid, and every distance to the fixed point at
// least halves per round. flag[0 .. 2] are the rounds' flags in turn; flag[0]
// is zero at the start and at the end.
constexpr int kJumpRounds = 64;  // halvings of any distance below 2^31, twice over
enum JumpEnd { kJumpDone, kJumpBarrier, kJumpBound };
template <class Item>
__device__ __forceinline__ JumpEnd jump_rounds(GridBar &bar, int64_t n, const Item &item, int32_t *ptr,
                                               unsigned long long *flag) {
    for (int it = 0; it < kJumpRounds; it++) {
        unsigned long long *f = flag + it % 3;
        if (blockIdx.x == 0 && threadIdx.x == 0) flag[(it + 1) % 3] = 0;  // last read before the barrier behind us
        bool any = false;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
            const int64_t x = item(i);
            if (x < 0) continue;
            const int p = *(volatile int32_t *)(ptr + x);
            const int pp = *(volatile int32_t *)(ptr + p);
            if (pp != p) {
                *(volatile int32_t *)(ptr + x) = pp;
                any = true;
            }
        }
        if (__syncthreads_or(any) && threadIdx.x == 0) atomicOr(f, 1ull);
        if (!bar.sync()) return kJumpBarrier;
        if (*(volatile unsigned long long *)f == 0) {
            if (blockIdx.x == 0 && threadIdx.x == 0) flag[0] = 0;  // (already zero where others still read it)
            return kJumpDone;
        }
    }
    return kJumpBound;
}

}  // namespace dgec
