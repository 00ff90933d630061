// Plane kernel (plane_conv.cuh), double, class 0 (fine radices).
#include "plane_conv.cuh"

namespace boris {
PLANE_INST(double, 0)
}  // namespace boris
