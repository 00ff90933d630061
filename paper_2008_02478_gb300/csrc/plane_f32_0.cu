// Plane kernel (plane_conv.cuh), float, class 0 (fine radices).
#include "plane_conv.cuh"

namespace boris {
PLANE_INST(float, 0)
}  // namespace boris
