// grid.cuh -- bounded grid-wide barrier for cooperative launches (all CTAs co-resident).
//
// Every wait is bounded: a CTA that has polled `spins` times without the barrier opening
// raises b->err and leaves; CTAs waiting at the same or a later barrier see the
// flag and leave too, so a kernel whose grid can never meet ends within about the spin
// limit and reports through its own status word instead of hanging. Data that other CTAs
// wrote before a barrier is read after it with L1-bypassing loads (__ldcg).
#pragma once
#include "internal.cuh"

namespace sparc {

constexpr unsigned long long kBarrierSpins = 1ull << 25;  // polls (each an L2 round trip)

// The count only grows (the host zeroes the barrier before each launch), and every CTA counts
// the barriers it has passed in `epoch` (0 at the launch's start): a CTA arrives with a release
// add that returns nothing, and waits with acquire loads until the count reaches epoch x
// nblocks, so the last CTA to arrive opens the barrier with its own add and no CTA waits for
// its own add's answer. Thread 0 arrives and waits for its CTA, between two CTA barriers, the
// second of which hands its result to the others. The error flag is looked at every 64 polls:
// two dependent L2 round trips a poll and one after it made a barrier 2 us, 1 us so.
__device__ __forceinline__ bool grid_barrier(GridBarrier *b, unsigned nblocks, unsigned &epoch,
                                             unsigned long long spins = kBarrierSpins)
{
    ++epoch;
    __syncthreads();
    int fail = 0;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.add.u32 [%0], 1;" ::"l"(&b->count) : "memory");
        const unsigned target = epoch * nblocks;
        unsigned long long it = 0;
        for (;;) {
            unsigned c;
            asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(c) : "l"(&b->count) : "memory");
            if ((int)(c - target) >= 0) break;
            // leaves when another CTA has given up, or after `spins` polls (then it raises the
            // flag itself)
            if ((++it & 63) == 0) {
                if (*((volatile int *)&b->err) != 0) {
                    fail = 1;
                    break;
                }
                if (it > spins) {
                    atomicExch(&b->err, 1);
                    fail = 1;
                    break;
                }
                __nanosleep(32);
            }
        }
    }
    return !__syncthreads_or(fail);
}

}  // namespace sparc
