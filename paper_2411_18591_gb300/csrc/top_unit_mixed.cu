// Mixed-radix engines (factors 2, 3, 5) for half-lengths 250, 500, 768 and 1000 (padded sizes 500,
// 1000, 1536 and 2000).
#include "top_unit.cuh"

namespace top {
#ifndef TOP_G500
#define TOP_G500 50
#endif
#ifndef TOP_G1000
#define TOP_G1000 50
#endif
using Eng250 = Engine<250, 25, 5, 5, 10>;
using Eng500 = Engine<500, TOP_G500, 5, 10, 10>;
using Eng768 = Engine<768, 32, 12, 8, 8>;
using Eng1000 = Engine<1000, TOP_G1000, 10, 10, 10>;
}  // namespace top

#define LIST(X) X(Eng250) X(Eng500) X(Eng768) X(Eng1000)
TOP_DEFINE_UNIT(mixed, LIST)
