// Plane kernel (plane_conv.cuh), double, class 3 (HZ 32).
#include "plane_conv.cuh"

namespace boris {
PLANE_INST(double, 3)
}  // namespace boris
