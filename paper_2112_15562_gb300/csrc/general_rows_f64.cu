// General row kernels of the products, double.
#include "general_impl.cuh"

namespace gj {
GJ_ROW_FWD(double, LoadPlain2<double>)
GJ_ROW_INV(double, StorePlain2<double>)
}  // namespace gj
