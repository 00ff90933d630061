// Mixed-radix x passes (mixed_x.cuh), float.
#include "mixed_x.cuh"

namespace boris {
MIXED_X_INST(float)
}  // namespace boris
