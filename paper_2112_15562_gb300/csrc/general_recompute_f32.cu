// General column kernels of the recompute mode, float.
#include "general_impl.cuh"

namespace gj {
GJ_RECOMPUTE(float)
}  // namespace gj
