// Instantiation unit of the general Cartesian stage kernel: BF16 storage. Units are
// compiled in parallel; the dispatcher is cart_dispatch.cu.
#include "cart_kernel.cuh"

namespace rtk {
RTK_CART_DEFINE_UNIT(bf16_lane, __nv_bfloat16)
}  // namespace rtk
