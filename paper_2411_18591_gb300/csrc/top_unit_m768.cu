// Mixed-radix engine for half-length 768 (padded size 1536): one warp a line.
#include "top_unit.cuh"

namespace top {
using Eng768 = Engine<768, 32, 12, 8, 8>;
}  // namespace top

#define LIST(X) X(Eng768)
TOP_DEFINE_UNIT(m768, LIST)
