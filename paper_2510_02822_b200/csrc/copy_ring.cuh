// What a block owes its copies when it gives up on a wait: those in flight land before its shared memory is given back.
#pragma once
#include <stdint.h>

#include "sm100_ptx.cuh"

namespace flexiq {

// A ring of `depth` stages that was filled `fills` times in order, full[] its barriers: waits for the last fill of every stage by
// that fill's own parity (the parity before it is always the completed one and says nothing).  Bounded: about four
// milliseconds a stage, for fills whose copies were never all issued.  True when all have landed.
static __device__ __noinline__ bool drain_ring(uint64_t *full, int depth, long long fills)
{
    bool landed = true;
    for (long long i = fills > depth ? fills - depth : 0; i < fills; ++i) {
        const uint32_t bar = ptx::smem_u32(&full[i % depth]), parity = (uint32_t)(i / depth) & 1u;
        bool here = false;
        for (uint32_t w = 0; w < 4096u && !here; ++w) here = ptx::mbar_try_wait_hint_s(bar, parity, 1000u);
        landed = landed && here;
    }
    return landed;
}

}  // namespace flexiq
