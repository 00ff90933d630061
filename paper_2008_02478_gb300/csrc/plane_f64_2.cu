// Plane kernel (plane_conv.cuh), double, class 2 (HZ 12..24).
#include "plane_conv.cuh"

namespace boris {
PLANE_INST(double, 2)
}  // namespace boris
