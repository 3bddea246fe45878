// Chunks of a channel handed from block to block through one record per (sequence, channel): used by the CUDA-core kernels and by the
// kernels with split products.  Device code and the host side that makes the tags.
#pragma once

#include "rglru_internal.h"
#include "sm100_ptx.cuh"

namespace rglru {

// One record {A, tag, B, tag2} per (sequence, channel): what the chunks so far hand to the next one.  Chunk c waits for the
// tags of its predecessor and overwrites the record with its own; nobody else reads it, so one slot serves the whole chain.
// The last chunk writes too: what a finished call leaves behind carries a tag that no chunk waits for, also when a CUDA graph
// replays the call with the same tags.  A chunk whose wait ran out says so to the next one, which gives up without a wait of its own.
struct Chain {
    uint4 *slot;        // [B][D]
    uint32_t tag, tag2, flip;   // flip: see wait_flip
    unsigned long long spin_ns;
    uint32_t *status;
};
// All lanes of the warp call it (a lane without a channel passes need = false); false if the wait ran out.
__device__ __forceinline__ bool chain_wait(const Chain &ch, const uint4 *slot, bool need, int link, float &A, float &B) {
    uint64_t t0 = 0;
    for (uint32_t n = 0;; ++n) {
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (need) asm volatile("ld.volatile.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(slot) : "memory");
        const uint32_t ty = ch.tag + (uint32_t)link, tw = ch.tag2 ^ (uint32_t)link;
        const bool ready = !need || (r.y == (ty ^ ch.flip) && r.w == (tw ^ ch.flip));
        if (__all_sync(0xffffffffu, ready)) {
            A = __uint_as_float(r.x); B = __uint_as_float(r.z);
            return true;
        }
        // a failed link, whichever it is: blocks that gave up at once have overwritten one another's
        if (__any_sync(0xffffffffu, need && r.w == ~(ch.tag2 ^ (r.y - ch.tag)))) return false;
        if ((n & 31u) == 31u) {
            const uint64_t t = ptx::gtimer();
            if (t0 == 0) t0 = t;
            if (__any_sync(0xffffffffu, t - t0 > ch.spin_ns)) {
                if ((threadIdx.x & 31) == 0) atomicExch(ch.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT);
                return false;
            }
        }
    }
}
__device__ __forceinline__ void chain_put(const Chain &ch, uint4 *slot, int link, float A, float B) {
    asm volatile("st.global.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(slot), "r"(__float_as_uint(A)), "r"(ch.tag + (uint32_t)link), "r"(__float_as_uint(B)),
                 "r"(ch.tag2 ^ (uint32_t)link) : "memory");
}

__device__ __forceinline__ void chain_fail(const Chain &ch, uint4 *slot, int link) {
    asm volatile("st.global.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(slot), "r"(0u), "r"(ch.tag + (uint32_t)link), "r"(0u), "r"(~(ch.tag2 ^ (uint32_t)link)) : "memory");
}

inline Chain make_chain(uint4 *slots, const FwdArgs &f) {
    const uint32_t tag = next_call_tag();
    return Chain{slots, tag, tag * 0x85EBCA6Bu + 0x27220A95u, wait_flip(f.flags), g_spin_limit_ns, f.status};
}

}  // namespace rglru
