// Engine for half-length 128 (padded size 256).
#include "top_unit.cuh"

namespace top {
using Eng128 = Engine<128, 8, 8, 16>;
}  // namespace top

#define LIST(X) X(Eng128)
TOP_DEFINE_UNIT(m128, LIST)
TOP_DEFINE_CZT(m128, LIST)
