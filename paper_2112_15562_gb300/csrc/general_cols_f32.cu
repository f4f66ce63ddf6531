// General column kernels, float.
#include "general_impl.cuh"

namespace gj {
GJ_COLS(float)
}  // namespace gj
