// A barrier over all CTAs of a launch that are on the GPU together, one word of global memory, by the scheme of the grid barrier in CUDA's cooperative
// groups, split into arrival and wait: CTA 0 adds 2^31 - (CTAs - 1), every other CTA 1, so the top bit flips when the last one has
// arrived and the word is ready for the next round (and the next launch, of as many CTAs as it likes) as it is.
//
// arrive / wait are called by ONE thread, between barriers of its CTA: what the CTA's other threads wrote before the first of these
// is visible to every thread of every CTA after the second one (release and acquire at GPU scope, which cover them).
// Data that crosses the barrier has to be read past L1 (__ldcg).  Waits are bounded.
#pragma once
#include "common.cuh"
#include "ptx_sm100.cuh"

namespace llma {

struct GridBarrier {
    uint32_t* word;
    uint32_t sense;  // top bit of the word before the round in progress ends

    __device__ __forceinline__ explicit GridBarrier(uint32_t* w) : word(w) {
        // (the bit cannot flip before this CTA has arrived)
        sense = ptx::ld_acquire(w) & 0x80000000u;
    }
    __device__ __forceinline__ void arrive() {
        const uint32_t add = blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1u) : 1u;
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(word), "r"(add) : "memory");
    }
    __device__ __forceinline__ bool wait(uint64_t most_ns) {
        const uint32_t old = sense;
        sense ^= 0x80000000u;
        const uint64_t t0 = ptx::globaltimer_ns();
        do {
            if ((ptx::ld_acquire(word) ^ old) & 0x80000000u) return true;
        } while (ptx::globaltimer_ns() - t0 < most_ns);
        return false;
    }
};

}  // namespace llma
