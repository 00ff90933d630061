// Plane kernel (plane_conv.cuh), float, class 1 (coarse radices, HZ <= 8).
#include "plane_conv.cuh"

namespace boris {
PLANE_INST(float, 1)
}  // namespace boris
