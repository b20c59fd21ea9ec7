// Fused plane kernel, mode XM_UPDATE.
#include "plane.cuh"

namespace cubic {
CUBIC_PLANE_UNIT(XM_UPDATE)
}  // namespace cubic
