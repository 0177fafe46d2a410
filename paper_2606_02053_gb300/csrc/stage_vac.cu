// Stage / RHS / constraint kernels for the "vac" matter variant.
#include "stage_split.cuh"

namespace cosmos {
COSMOS_DEFINE_VARIANT(vac, false, false)
}  // namespace cosmos
