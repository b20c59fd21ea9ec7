// Fused plane kernel, mode XM_INV.
#include "plane.cuh"

namespace cubic {
CUBIC_PLANE_UNIT(XM_INV)
}  // namespace cubic
