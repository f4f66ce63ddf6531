// General row kernels of the joint solver, double.
#include "general_impl.cuh"
#include "rrcg_functors.cuh"

namespace gj {
using Model = ProModel<double>;
using Direction = ProDirection<double>;
GJ_ROW_FWD(double, Model)
GJ_ROW_FWD(double, Direction)
GJ_ROW_INV(double, EpiGradient<double>)
GJ_ROW_INV(double, EpiQNorm<double>)
GJ_ROW_RESID(double, EpiResidual<double>)
}  // namespace gj
