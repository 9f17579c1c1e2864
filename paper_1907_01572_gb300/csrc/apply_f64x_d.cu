// FP64 apply on the tensor pipe: n = 9.
#include "apply_f64x_launch.cuh"

namespace dg {
namespace apply_detail {
DG_X64_INSTANCE(9)
}  // namespace apply_detail
}  // namespace dg
