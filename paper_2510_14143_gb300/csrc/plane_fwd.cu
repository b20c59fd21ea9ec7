// Fused plane kernel, mode XM_FWD.
#include "plane.cuh"

namespace cubic {
CUBIC_PLANE_UNIT(XM_FWD)
}  // namespace cubic
