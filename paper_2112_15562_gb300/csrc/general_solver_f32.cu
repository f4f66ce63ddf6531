// General row kernels of the joint solver, float.
#include "general_impl.cuh"
#include "rrcg_functors.cuh"

namespace gj {
using Model = ProModel<float>;
using Direction = ProDirection<float>;
GJ_ROW_FWD(float, Model)
GJ_ROW_FWD(float, Direction)
GJ_ROW_INV(float, EpiGradient<float>)
GJ_ROW_INV(float, EpiQNorm<float>)
GJ_ROW_RESID(float, EpiResidual<float>)
}  // namespace gj
