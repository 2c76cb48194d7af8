// gc_steps.h -- the steps of the validation's pass over the entries (host and
// device; includes nothing of CUDA, so that the arithmetic compiles anywhere).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define GC_HOST_DEVICE __host__ __device__
#else
#define GC_HOST_DEVICE
#endif

namespace gc {

// Rows and entries of one warp's step together (8 entries a lane, less what
// the 16-byte boundary before the first one can take).
constexpr int kValSlots = 8 * 32;
constexpr int kValChunk = kValSlots - 4;

// The steps [k0, k1] that begin in a row of deg entries which starts at place
// d of the count of rows plus entries (none: k1 < k0).  d is negative only where the
// offsets are malformed, whose steps nobody reads.
GC_HOST_DEVICE inline void row_steps(int64_t d, int32_t deg, int64_t steps, bool narrow, int64_t& k0,
                                          int64_t& k1) {
    k0 = 0;
    k1 = -1;
    if (d < 0) return;
    if (narrow) {  // d and deg below 2^31 (a 64-bit division takes a third of the pass)
        k0 = (static_cast<uint32_t>(d) + (kValChunk - 1u)) / kValChunk;
        k1 = (static_cast<uint32_t>(d) + static_cast<uint32_t>(deg)) / kValChunk;
    } else {
        k0 = (d + kValChunk - 1) / kValChunk;
        k1 = (d + deg) / kValChunk;
    }
    if (k1 > steps - 1) k1 = steps - 1;
}

}  // namespace gc
