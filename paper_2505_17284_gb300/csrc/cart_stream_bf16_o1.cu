// Instantiation unit of the streaming Cartesian stage kernel: BF16 storage, first order.
#include "cart_stream.cuh"

namespace rtk {
RTK_STR_UNIT(bf16_o1, 1, __nv_bfloat16)
}  // namespace rtk
