// Engine for half-length 2048 (padded size 4096).
#include "top_unit.cuh"

namespace top {
using Eng2048 = Engine<2048, 64, 16, 16, 8>;
}  // namespace top

#define LIST(X) X(Eng2048)
TOP_DEFINE_UNIT(m2048, LIST)
TOP_DEFINE_CZT(m2048, LIST)
