// General column kernels of the recompute mode, double.
#include "general_impl.cuh"

namespace gj {
GJ_RECOMPUTE(double)
}  // namespace gj
