// wait_last_uses / wait_last_use (ring_wait.cuh) on mbarriers in miniature: a
// slot's barrier counts completed phases, and a wait for a parity ends when the
// current phase has the other one. For every ring of up to 5 slots, up to 13
// uses and every set of the last uses that are still in flight: after the waits
// nothing is in flight, and no wait is for a use that was never made.
#include <cstdio>
#include <vector>

#include "ring_wait.cuh"

int main()
{
    unsigned bad = 0, runs = 0;
    for (uint32_t slots = 1; slots <= 5; ++slots)
        for (uint32_t uses = 0; uses <= 13; ++uses) {
            const uint32_t first = uses > slots ? uses - slots : 0;
            for (uint32_t late = 0; late < 1u << (uses - first); ++late)
                for (int ordered = 0; ordered < 2; ++ordered) {
                    uint32_t low = 0;   // in order, those in flight are the last ones
                    while (low < uses - first && !(late >> low & 1)) ++low;
                    if (ordered && late >> low != (1u << (uses - first - low)) - 1) continue;
                    std::vector<uint32_t> done(slots, 0);
                    for (uint32_t i = 0; i < uses; ++i)
                        if (i < first || !(late >> (i - first) & 1)) ++done[i % slots];
                    uint32_t made = 0;
                    auto wait = [&](uint32_t slot, uint32_t parity) {
                        if ((done[slot] & 1) != parity) return;   // the phase has completed
                        // blocked on phase done[slot]: is there such a use?
                        const uint32_t i = done[slot] * slots + slot;
                        if (slot >= slots || i >= uses) ++bad;
                        if (!ordered) ++done[slot];
                        else   // the commits before it complete with it
                            for (uint32_t j = first; j <= i && j < uses; ++j)
                                if (done[j % slots] == j / slots) ++done[j % slots];
                        ++made;
                    };
                    if (ordered) ann::wait_last_use(uses, slots, wait);
                    else ann::wait_last_uses(uses, slots, wait);
                    for (uint32_t i = first; i < uses; ++i) bad += done[i % slots] != i / slots + 1;
                    ++runs;
                }
        }
    printf("%u runs, %u wrong\n", runs, bad);
    return bad || !runs;
}
