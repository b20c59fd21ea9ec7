// Fused plane kernel, mode XM_RATIO.
#include "plane.cuh"

namespace cubic {
CUBIC_PLANE_UNIT(XM_RATIO)
}  // namespace cubic
