// Engine for half-length 4096 (padded size 8192).
#include "top_unit.cuh"

namespace top {
using Eng4096 = Engine<4096, 128, 16, 16, 16>;
}  // namespace top

#define LIST(X) X(Eng4096)
TOP_DEFINE_UNIT(m4096, LIST)
TOP_DEFINE_CZT(m4096, LIST)
TOP_DEFINE_CZT_SPLIT(m4096, LIST)
