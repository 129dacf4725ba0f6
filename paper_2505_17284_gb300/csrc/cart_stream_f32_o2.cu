// Instantiation unit of the streaming Cartesian stage kernel: FP32 storage, MUSCL.
#include "cart_stream.cuh"

namespace rtk {
RTK_STR_UNIT(f32_o2, 2, float)
}  // namespace rtk
