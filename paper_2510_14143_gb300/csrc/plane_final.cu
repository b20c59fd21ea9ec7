// Fused plane kernel, mode XM_FINAL.
#include "plane.cuh"

namespace cubic {
CUBIC_PLANE_UNIT(XM_FINAL)
}  // namespace cubic
