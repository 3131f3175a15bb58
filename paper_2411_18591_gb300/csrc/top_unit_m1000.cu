// Mixed-radix engine for half-length 1000 (padded size 2000): 50 threads a line, two warps. Three
// stages of radix 10 (two exchanges a transform) measured faster than four-stage plans.
#include "top_unit.cuh"

namespace top {
using Eng1000 = Engine<1000, 50, 10, 10, 10>;
}  // namespace top

#define LIST(X) X(Eng1000)
TOP_DEFINE_UNIT(m1000, LIST)
