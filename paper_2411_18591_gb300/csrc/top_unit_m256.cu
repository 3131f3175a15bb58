// Engine for half-length 256 (padded size 512).
#include "top_unit.cuh"

namespace top {
using Eng256 = Engine<256, 16, 16, 16>;
}  // namespace top

#define LIST(X) X(Eng256)
TOP_DEFINE_UNIT(m256, LIST)
TOP_DEFINE_CZT(m256, LIST)
