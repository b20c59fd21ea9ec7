// Fused plane kernel, mode XM_ADJ_U.
#include "plane.cuh"

namespace cubic {
CUBIC_PLANE_UNIT(XM_ADJ_U)
}  // namespace cubic
