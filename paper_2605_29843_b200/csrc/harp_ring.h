// Buffers that bulk copies fill in turn: which phase of a buffer's barrier a thread waits for next, and which of the loads that it
// issued it has not seen arrive.  A wait has a limit.  One that gives up leaves the phase as it is, because a parity wait for
// the phase after it succeeds while this one is still incomplete: the load would pass for one that has arrived, and could land in
// the shared memory of the CTA that follows.  Plain C++ beside the annotations, so that a host program can replay it.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define HARP_RING_FN __device__ __forceinline__
#else
#define HARP_RING_FN inline
#endif

struct BulkRing {
    uint32_t state = 0;                       // bit b: parity of the phase of buffer b; bit 16 + b: its load in flight (one register)

    HARP_RING_FN void issued(int b) { state |= 0x10000u << b; }
    HARP_RING_FN bool arrived(int b) const { return !((state >> (16 + b)) & 1u); }

    // try_phase(buffer, parity): that phase of the buffer's barrier is complete; stop(): another thread has given up
    template <typename Try, typename Stop>
    HARP_RING_FN bool wait(int b, uint32_t limit, const Try &try_phase, const Stop &stop) {
        for (uint32_t it = 1; !try_phase(b, (state >> b) & 1u); ++it)
            if (it > limit || ((it & 63) == 63 && stop())) return false;
        state = (state ^ (1u << b)) & ~(0x10000u << b);
        return true;
    }

    // before the CTA ends: the loads still in flight
    template <typename Try>
    HARP_RING_FN void drain(int n_buf, uint32_t limit, const Try &try_phase) {
        for (int b = 0; b < n_buf; ++b)
            if (!arrived(b)) wait(b, limit, try_phase, [] { return false; });
    }
};
