// Barrier between the blocks of one cooperative launch, carrying the largest of
// the blocks' values.
//
// One 64-bit word per phase counts the arrivals, so a block arrives with a
// single reduction (no value comes back) and one of its threads polls one
// address.  The word also counts the blocks whose value equals the previous
// phase's result and those above it: the values exchanged here (exponents and
// bit lengths of a field's maximum) hardly ever change from phase to phase, and
// when some block still holds the previous value and none exceeds it, the
// arrival word alone gives the result.  Blocks with another value also fold it
// into a second word, which is read only when the first does not decide.
// Three sets of words are used in turn; block 0 clears the next set before it
// arrives, when every block has left it.  (All blocks reading all blocks' values
// instead of counting measured 3.6 us more per phase at 128 blocks.)
//
// Every wait is bounded: one that runs out sets *err, which ends the others.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace hcg {

// Device memory of a barrier: 6 words on lines of their own, all zero between launches.
constexpr int kGridBarStride = 16;   // 64-bit words per line of 128 bytes
constexpr size_t kGridBarBytes = 6 * kGridBarStride * sizeof(unsigned long long);

constexpr long long kGridWaitCycles = 2000000000ll;   // about one second at GB300 clocks

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_add_u64(unsigned long long* p, unsigned long long v)
{
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Arrival of this block at phase `ph` with value m (one thread calls it, after
// a block barrier that follows the block's last store of the phase); prev is
// the previous phase's result.
__device__ __forceinline__ void grid_arrive(unsigned long long* bar, int ph, unsigned m, unsigned prev)
{
    unsigned long long* ctr = bar + (ph % 3) * kGridBarStride;
    unsigned long long* big = ctr + 3 * kGridBarStride;
    if (m != prev) atomicMax(big, (unsigned long long)m);
    if (blockIdx.x == 0) {   // the set of phase ph + 1, last used at ph - 2
        unsigned long long* nxt = bar + ((ph + 1) % 3) * kGridBarStride;
        nxt[0] = 0ull;
        nxt[3 * kGridBarStride] = 0ull;
    }
    __threadfence();
    red_add_u64(ctr, 1ull + (m == prev ? 1ull << 20 : m > prev ? 1ull << 40 : 0ull));
}

// One thread waits until every block has arrived at phase `ph`; *m receives the
// largest value.  False when the wait ran out or another block gave up.
__device__ __forceinline__ bool grid_wait(unsigned long long* bar, int ph, unsigned prev, unsigned* m, int* err)
{
    const unsigned need = gridDim.x;
    unsigned long long* ctr = bar + (ph % 3) * kGridBarStride;
    unsigned long long v = ld_acquire_u64(ctr);
    if ((v & 0xfffffull) != need) {
        const long long t0 = clock64();
        int spins = 0;
        do {
            if ((++spins & 255) == 0 && *(volatile int*)err) return false;
            if (clock64() - t0 > kGridWaitCycles) {
                atomicMax(err, 1);
                return false;
            }
            v = ld_acquire_u64(ctr);
        } while ((v & 0xfffffull) != need);
    }
    const bool same = (v >> 20 & 0xfffffull) != 0 && (v >> 40) == 0;
    *m = same ? prev : (unsigned)ld_acquire_u64(ctr + 3 * kGridBarStride);
    return true;
}

// Clears the barrier for the next launch: block 0, after the last phase's wait.
__device__ __forceinline__ void grid_reset(unsigned long long* bar)
{
#pragma unroll
    for (int i = 0; i < 6; ++i) bar[i * kGridBarStride] = 0ull;
}

}  // namespace hcg
