// FP64 apply on the tensor pipe: n = 7, 8.
#include "apply_f64x_launch.cuh"

namespace dg {
namespace apply_detail {
DG_X64_INSTANCE(7)
DG_X64_INSTANCE(8)
}  // namespace apply_detail
}  // namespace dg
