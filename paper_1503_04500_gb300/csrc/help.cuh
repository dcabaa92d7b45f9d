// help.cuh -- CTAs that have run out of columns take over part of the trailing
// updates of the columns still running (global bin).
//
// The largest columns of a power-law matrix take as long as hundreds of average
// ones, and one CTA each: with 152 columns in flight the bin's time was set by
// the last few (n = 1111 in FP64: 264 ms, of which all SMs together needed 54).
// The trailing update of a panel is independent per column of B, so its owner
// publishes it as groups of columns; idle CTAs and the owner claim groups one at
// a time.  Each column of B is computed by one warp with the same arithmetic
// whoever claims it.
//
// No CTA ever waits for work to be claimed: the owner claims whatever is left
// itself and then waits only for groups that a helper has already claimed, i.e.
// for a CTA that is running; the wait is bounded all the same.
#pragma once

#include "common.cuh"

namespace rsai {

// One published update: groups of `group` columns of [c_lo, c_hi] of B (ld q; c == p: rhs)
struct HelpTask {
    const void *src, *heads, *tcol;  // panel in B, heads of its reflectors, its T (column t at t * kPanel)
    void *B, *rhs;
    int32_t q, p, qq, nb, j0, c_lo, c_hi, group;
};

// Device memory of the global bin, zeroed before each of its launches
struct HelpBoard {
    unsigned long long *word;  // per owner: epoch << 32 | groups << 16 | next group
    uint32_t *done;            // per owner: groups finished by helpers in this epoch
    HelpTask *task;            // per owner
    uint32_t *idle;            // CTAs without a column
    uint32_t *cols_done;       // columns finished
    int32_t slots;             // owners (CTAs with a workspace)

    static __host__ __device__ size_t bytes(int slots) {
        return (size_t)slots * (sizeof(unsigned long long) + sizeof(HelpTask) + sizeof(uint32_t)) + 2 * sizeof(uint32_t);
    }
    static __host__ __device__ HelpBoard at(void *base, int slots) {
        HelpBoard b;
        b.word = (unsigned long long *)base;
        b.task = (HelpTask *)(b.word + slots);
        b.done = (uint32_t *)(b.task + slots);
        b.idle = b.done + slots;
        b.cols_done = b.idle + 1;
        b.slots = slots;
        return b;
    }
};

// polls before a wait is given up (some hundred nanoseconds each)
constexpr unsigned kHelpPolls = 1u << 24;

__device__ __forceinline__ unsigned long long help_load(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t help_load(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t help_epoch(unsigned long long w) { return (uint32_t)(w >> 32); }
__device__ __forceinline__ int help_groups(unsigned long long w) { return (int)((w >> 16) & 0xffff); }
__device__ __forceinline__ int help_next(unsigned long long w) { return (int)(w & 0xffff); }

// One group of the task of `epoch` at `word`, or -1 (one thread)
__device__ __forceinline__ int help_claim(unsigned long long *word, uint32_t epoch) {
    unsigned long long w = help_load(word);
    for (;;) {
        if (help_epoch(w) != epoch || help_next(w) >= help_groups(w)) return -1;
        const unsigned long long seen = atomicCAS(word, w, w + 1);
        if (seen == w) {
            __threadfence();
            return help_next(w);
        }
        w = seen;
    }
}

}  // namespace rsai
