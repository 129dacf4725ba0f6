// Instantiation unit of the streaming Cartesian stage kernel: BF16 storage, MUSCL.
#include "cart_stream.cuh"

namespace rtk {
RTK_STR_UNIT(bf16_o2, 2, __nv_bfloat16)
}  // namespace rtk
