// General column kernels, double.
#include "general_impl.cuh"

namespace gj {
GJ_COLS(double)
}  // namespace gj
