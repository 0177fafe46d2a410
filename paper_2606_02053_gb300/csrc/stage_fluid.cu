// Stage / RHS / constraint kernels for the "fluid" matter variant.
#include "stage_split.cuh"

namespace cosmos {
COSMOS_DEFINE_VARIANT(fluid, true, false)
}  // namespace cosmos
