// FP64 apply on the tensor pipe: n = 5, 6.
#include "apply_f64x_launch.cuh"

namespace dg {
namespace apply_detail {
DG_X64_INSTANCE(5)
DG_X64_INSTANCE(6)
}  // namespace apply_detail
}  // namespace dg
