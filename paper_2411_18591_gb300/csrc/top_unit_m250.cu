// Mixed-radix engine for half-length 250 (padded size 500): 25 threads a line, one warp.
#include "top_unit.cuh"

namespace top {
using Eng250 = Engine<250, 25, 5, 5, 10>;
}  // namespace top

#define LIST(X) X(Eng250)
TOP_DEFINE_UNIT(m250, LIST)
