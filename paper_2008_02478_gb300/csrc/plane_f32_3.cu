// Plane kernel (plane_conv.cuh), float, class 3 (HZ 32).
#include "plane_conv.cuh"

namespace boris {
PLANE_INST(float, 3)
}  // namespace boris
