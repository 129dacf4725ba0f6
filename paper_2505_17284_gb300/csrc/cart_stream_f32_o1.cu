// Instantiation unit of the streaming Cartesian stage kernel: FP32 storage, first order.
#include "cart_stream.cuh"

namespace rtk {
RTK_STR_UNIT(f32_o1, 1, float)
}  // namespace rtk
