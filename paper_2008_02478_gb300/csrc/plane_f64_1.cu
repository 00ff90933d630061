// Plane kernel (plane_conv.cuh), double, class 1 (coarse radices, HZ <= 8).
#include "plane_conv.cuh"

namespace boris {
PLANE_INST(double, 1)
}  // namespace boris
