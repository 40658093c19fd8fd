// Cooperative building blocks: a grid barrier for kernels whose CTAs are all
// resident (launched through coop_launch), and the stable LSD radix sort as
// one such kernel.
#pragma once

#include "common.cuh"

namespace dgec {

// The barrier words of a call (kBarWords of them): [0] arrivals, [1] exits.
// Zeroed once per call; the last CTA out of a kernel leaves them zero again.

// Polls before a barrier gives up (about a microsecond each). CTAs of a
// cooperative launch are co-resident, so this only bounds the wait should
// that ever not hold.
constexpr unsigned kBarPolls = 1u << 24;

// Barrier over every CTA of a cooperative launch. Arrivals count up without
// a reset between barriers (compared by signed difference). A barrier that
// gives up writes 1 to *err (host-mapped memory) and returns false in every
// thread of its CTA; the kernel must then return at once (the other CTAs
// give up likewise).
struct GridBar {
    unsigned *word;
    unsigned *err;
    unsigned nblk, target;  // nblk = 1 once one CTA goes on alone
    __device__ __forceinline__ GridBar(unsigned *w, unsigned *e) : word(w), err(e), nblk(gridDim.x), target(0) {}
    __device__ __forceinline__ bool sync() {
        if (nblk == 1) {
            __syncthreads();
            return true;
        }
        __syncthreads();
        bool bad = false;
        target += nblk;
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(word, 1u);
            unsigned polls = 0;
            for (;;) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
                if ((int)(v - target) >= 0) break;
                if (++polls > kBarPolls) {
                    bad = true;
                    *(volatile unsigned *)err = 1u;
                    break;
                }
            }
            __threadfence();
        }
        return !__syncthreads_or(bad);
    }
    // every CTA calls this after its last barrier
    __device__ __forceinline__ void finish() {
        if (gridDim.x == 1 || threadIdx.x != 0) return;
        if (atomicAdd(word + 1, 1u) == gridDim.x - 1) {
            word[0] = 0u;
            word[1] = 0u;
        }
    }
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
