// Mixed-radix x passes (mixed_x.cuh), double.
#include "mixed_x.cuh"

namespace boris {
MIXED_X_INST(double)
}  // namespace boris
