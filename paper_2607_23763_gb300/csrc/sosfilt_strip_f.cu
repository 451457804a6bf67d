// The strip kernel (sosfilt_strip.cuh) for section counts 8 (split across translation units so that
// the build compiles them in parallel).
#include "sosfilt_strip.cuh"

namespace sosk {
SOSK_STRIP_INST(8)
}  // namespace sosk
