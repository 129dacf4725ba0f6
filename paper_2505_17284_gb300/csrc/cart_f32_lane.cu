// Instantiation unit of the general Cartesian stage kernel: FP32 storage. Units are
// compiled in parallel; the dispatcher is cart_dispatch.cu.
#include "cart_kernel.cuh"

namespace rtk {
RTK_CART_DEFINE_UNIT(f32_lane, float)
}  // namespace rtk
