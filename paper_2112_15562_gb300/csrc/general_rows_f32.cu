// General row kernels of the products, float.
#include "general_impl.cuh"

namespace gj {
GJ_ROW_FWD(float, LoadPlain2<float>)
GJ_ROW_INV(float, StorePlain2<float>)
}  // namespace gj
