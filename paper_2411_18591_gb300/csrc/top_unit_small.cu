// Engines for half-lengths 16, 32 and 64 (padded sizes 32 .. 128).
#include "top_unit.cuh"

namespace top {
using Eng16 = Engine<16, 4, 4, 4>;
using Eng32 = Engine<32, 4, 4, 8>;
using Eng64 = Engine<64, 8, 8, 8>;
}  // namespace top

#define LIST(X) X(Eng16) X(Eng32) X(Eng64)
TOP_DEFINE_UNIT(small, LIST)
TOP_DEFINE_CZT(small, LIST)
