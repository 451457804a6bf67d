// The strip kernel (sosfilt_strip.cuh) for section counts 1, 2 (split across translation units so that
// the build compiles them in parallel).
#include "sosfilt_strip.cuh"

namespace sosk {
SOSK_STRIP_INST(1)
SOSK_STRIP_INST(2)
}  // namespace sosk
