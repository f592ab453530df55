// The end of a kernel in which a wait for a bulk copy gave up.  Every such wait has a limit; after it nothing is copied any more, but
// the loads already issued may still arrive, and must not land in the shared memory of the CTA that follows.  The thread that
// issues them waits for them before it leaves.  It can because a wait that gave up leaves its buffer's parity as it is: a
// parity wait for the phase after that one succeeds while this one is incomplete, and would wait for nothing.  (Which buffers
// have a load in flight is not kept: the bookkeeping cost the slab pass of harp_pipe.cu, at its register limit, 2 % -- 2048 rows
// of d = 28672 90.9 -> 92.7 us -- and a buffer with none only takes its limit.)  Plain C++ beside the annotation, so that a host
// program can replay it.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define HARP_RING_FN __device__ __forceinline__
#else
#define HARP_RING_FN inline
#endif

// parity: a bit per buffer, the phase of its barrier that has not been seen complete.  try_phase(buffer, parity): that phase is complete.
template <typename Try>
HARP_RING_FN void ring_drain(uint32_t parity, int n_buf, uint32_t limit, const Try &try_phase) {
    for (int b = 0; b < n_buf; ++b)
        for (uint32_t it = 0; it < limit && !try_phase(b, (parity >> b) & 1u); ++it) {}
}
