// Fused plane kernel, mode XM_ADJ_R.
#include "plane.cuh"

namespace cubic {
CUBIC_PLANE_UNIT(XM_ADJ_R)
}  // namespace cubic
