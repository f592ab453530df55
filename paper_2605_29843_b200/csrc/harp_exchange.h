// Waits for the counted exchanges of a cluster, and the end of a CTA whose wait gave up.  Every wait has a limit.  A thread whose wait
// runs out sends and stores nothing more, and it keeps its CTA until every other thread of the cluster has sent its last piece or has
// ended, and then, with the same limit, until the pieces on their way have landed: they must not land in the shared memory of a CTA that
// has ended.  A thread whose waits all succeeded has every piece of its CTA and may leave at once.  Plain C++ beside the annotation, so
// that a host program can replay it.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define HARP_EXCHANGE_FN __device__ __forceinline__
#else
#define HARP_EXCHANGE_FN inline
#endif

// arrived(): all bytes of the exchange are here.  False: it gave up.
template <typename Arrived>
HARP_EXCHANGE_FN bool exchange_wait(uint32_t limit, const Arrived &arrived) {
    for (uint32_t tries = 0; tries < limit; ++tries)
        if (arrived()) return true;
    return false;
}

// mask: a bit per phase that ends in an exchange.  others_sent(): returns when every thread of the cluster is here or has ended.
template <typename OthersSent, typename Arrived>
HARP_EXCHANGE_FN void exchange_leave(uint32_t mask, uint32_t limit, const OthersSent &others_sent, const Arrived &arrived) {
    others_sent();
    for (int p = 0; (mask >> p) != 0; ++p)
        if ((mask >> p) & 1u) exchange_wait(limit, [&] { return arrived(p); });
}
