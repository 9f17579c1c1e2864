// FP64 apply on the tensor pipe: n = 2, 3, 4.
#include "apply_f64x_launch.cuh"

namespace dg {
namespace apply_detail {
DG_X64_INSTANCE(2)
DG_X64_INSTANCE(3)
DG_X64_INSTANCE(4)
}  // namespace apply_detail
}  // namespace dg
