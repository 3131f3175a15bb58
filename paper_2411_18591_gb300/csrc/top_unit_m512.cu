// Engine for half-length 512 (padded size 1024).
#include "top_unit.cuh"

namespace top {
using Eng512 = Engine<512, 16, 16, 32>;
}  // namespace top

#define LIST(X) X(Eng512)
TOP_DEFINE_UNIT(m512, LIST)
TOP_DEFINE_CZT(m512, LIST)
