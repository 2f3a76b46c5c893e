// How the warps of the running serve kernels take queries from one FIFO: three
// monotonic counts, the queries taken, the queries published (made available)
// and the difference of the two. Host code too, over any implementation of the
// counts, so that the interleavings of several warps can be enumerated.
//
// Taking a query is two additions: one to the difference, given back if there
// was none, and one to the count of those taken. (A compare and swap of the
// latter fails for all but one of the warps that try together: 3,000 queries
// took 2.7 ms, 0.9 of which was searching.)
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define ANN_SERVE_FN __host__ __device__ __forceinline__
#else
#define ANN_SERVE_FN inline
#endif

namespace ann {

enum ServeCount : uint32_t { kServeTaken = 0, kServePublished, kServeFree, kServeCounts };

// The tail that a launch publishes: its own, which covers its request, or what
// the host has published since (`live`, 0 if the launch takes no later queries).
ANN_SERVE_FN unsigned long long serve_tail(unsigned long long own, unsigned long long live)
{
    return live > own ? live : own;
}

// Make the queries up to `tail` available.
template <typename Counts>
ANN_SERVE_FN void serve_publish(Counts &c, unsigned long long tail)
{
    if (tail <= c.load(kServePublished)) return;
    c.fence();   // what `tail` counts, before the counts
    const unsigned long long was = c.max(kServePublished, tail);
    if (was < tail) c.add(kServeFree, tail - was);
}

// Take the next query: true and its number in *h.
//
// A warp leaves only when everything published has been taken, not when the
// difference reads as none: that is also what it sees between a publisher's two
// steps, and while other warps hold what they are about to give back. (Leaving
// then can strand a query: the publisher itself may serve just one.) Until the
// two counts agree it looks again, and adds only once something reads as free, so
// that the waiting warps hide nothing from each other. What it waits for is the
// next instruction of a running warp; the looks are bounded all the same, and
// reported when they run out.
template <typename Counts>
ANN_SERVE_FN bool serve_take(Counts &c, unsigned long long *h)
{
    uint32_t look = 0;
    do {
        if ((long long)c.add(kServeFree, ~0ull) > 0) {
            *h = c.add(kServeTaken, 1);
            c.fence();
            return true;
        }
        c.add(kServeFree, 1);
        do {
            if (c.load(kServePublished) <= c.load(kServeTaken)) return false;
        } while ((long long)c.load(kServeFree) <= 0 && ++look < Counts::kLooks);
    } while (++look < Counts::kLooks);
    c.gave_up();
    return false;
}

}  // namespace ann
