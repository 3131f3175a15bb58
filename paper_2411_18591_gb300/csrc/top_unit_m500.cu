// Mixed-radix engine for half-length 500 (padded size 1000): 50 threads a line, two warps.
#include "top_unit.cuh"

namespace top {
using Eng500 = Engine<500, 50, 5, 10, 10>;
}  // namespace top

#define LIST(X) X(Eng500)
TOP_DEFINE_UNIT(m500, LIST)
