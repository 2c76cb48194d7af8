// C entry to the validation's step arithmetic (gc_steps.h), for the host-side test.
#include "gc_steps.h"

extern "C" void row_steps(int64_t d, int32_t deg, int64_t steps, int narrow, int64_t* k) {
    gc::row_steps(d, deg, steps, narrow != 0, k[0], k[1]);
}

extern "C" int step_places() { return gc::kValChunk; }
