// The end of a ring of slots whose uses complete asynchronously (copies into
// shared memory, MMAs that read it): a role that leaves its loop, early or not,
// first waits for what it still has in flight, since a block that ends, or frees
// its tensor memory, under a copy or an MMA lets it write into what another block
// has by then. Host code too, so that the slots and parities can be checked.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define ANN_RING_FN __host__ __device__ __forceinline__
#else
#define ANN_RING_FN inline
#endif

namespace ann {

// wait(slot, parity) for each use of a slot that no later one has replaced:
// use i took slot i % slots, whose barrier's phase i / slots it completes.
template <typename Wait>
ANN_RING_FN void wait_last_uses(uint32_t uses, uint32_t slots, Wait wait)
{
    for (uint32_t i = uses > slots ? uses - slots : 0; i < uses; ++i) wait(i % slots, (i / slots) & 1);
}

// The same where a use completes only after all before it.
template <typename Wait>
ANN_RING_FN void wait_last_use(uint32_t uses, uint32_t slots, Wait wait)
{
    if (uses) wait((uses - 1) % slots, ((uses - 1) / slots) & 1);
}

}  // namespace ann
