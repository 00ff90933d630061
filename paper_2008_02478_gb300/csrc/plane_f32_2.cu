// Plane kernel (plane_conv.cuh), float, class 2 (HZ 12..24).
#include "plane_conv.cuh"

namespace boris {
PLANE_INST(float, 2)
}  // namespace boris
