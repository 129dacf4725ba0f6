// Dispatch over the Cartesian kernels' instantiation units and the static facts the
// host needs about the variants (tile width, shared memory per CTA).
#include "cart_kernel.cuh"
#include "cart_stream.cuh"

namespace rtk {

#define RTK_UNIT_DECL(NAME)                                                                     \
  cudaError_t cart_prepare_##NAME(int, int, int, int);                                          \
  cudaError_t cart_launch_##NAME(const InstDesc*, const WorkItem*, int, int, int, int, int, cudaStream_t);
RTK_UNIT_DECL(f32_lane)
RTK_UNIT_DECL(bf16_lane)
#undef RTK_UNIT_DECL
#define RTK_STR_DECL(NAME)                                                                                  \
  cudaError_t str_prepare_##NAME(int stage, int tx, int ly, int form);                                      \
  cudaError_t str_launch_##NAME(const InstDesc*, const WorkItem*, int n_items, int stage, int tx, int ly,    \
                                int form, cudaStream_t, bool chained);                                      \
  size_t str_smem_##NAME(int stage, int tx, int ly, int form);
RTK_STR_DECL(f32_o1)
RTK_STR_DECL(f32_o2)
RTK_STR_DECL(bf16_o1)
RTK_STR_DECL(bf16_o2)
#undef RTK_STR_DECL
#define RTK_STR_PICK(FN) \
  (storage == 0 ? (order == 1 ? FN##_f32_o1 : FN##_f32_o2) : (order == 1 ? FN##_bf16_o1 : FN##_bf16_o2))

int cart_tile_width(int run) { return kCartWarps * run; }
int cart_stream_chunk_groups(int tx) { return kStrWarps * kStrCells / tx; }

// Streaming kernel (uni != 0): tiles of 16 or 32 cells; general kernel: tiles of 16
// cells, 1, 2 or 4 ordinates per lane.
static bool variant_exists(int order, int run, int vec, int uni) {
  if (order != 1 && order != 2) return false;
  if (uni) return (run == 2 || run == 4) && (order == 2 || uni == STREAM_PLAIN);
  return run == 2 && (vec == 1 || vec == 2 || vec == 4);
}

cudaError_t prepare_cart_stage(int stage, int order, int storage, int run, int vec, int ly_max, int uni) {
  if (!variant_exists(order, run, vec, uni)) return cudaErrorInvalidValue;
  if (uni) return RTK_STR_PICK(str_prepare)(stage, cart_tile_width(run), ly_max, uni);
  return (storage == 0 ? cart_prepare_f32_lane : cart_prepare_bf16_lane)(stage, order, vec, ly_max);
}

cudaError_t launch_cart_stage(const InstDesc* d_desc, const WorkItem* d_items, int n_items, int stage, int order,
                              int storage, int run, int vec, int ly_max, cudaStream_t stream, int uni,
                              bool chained) {
  if (n_items <= 0) return cudaSuccess;
  if (!variant_exists(order, run, vec, uni)) return cudaErrorInvalidValue;
  if (uni) return RTK_STR_PICK(str_launch)(d_desc, d_items, n_items, stage, cart_tile_width(run), ly_max, uni, stream,
                                         chained);
  return (storage == 0 ? cart_launch_f32_lane : cart_launch_bf16_lane)(d_desc, d_items, n_items, stage, order, vec,
                                                                       ly_max, stream);
}

template <typename T>
static size_t smem_of(int order, int vec, int ly, int stage) {
#define RTK_SMC(O, VV, ST, TT) \
  if (order == O && vec == VV && stage == ST) return cart_smem_for<O, 2, VV, ST, TT>(ly);
  RTK_CART_ALL(RTK_SMC, T)
#undef RTK_SMC
  return 0;
}

size_t cart_smem_bytes(int order, int storage, int run, int vec, int ly, int stage, int uni) {
  if (!variant_exists(order, run, vec, uni)) return 0;
  if (uni) return RTK_STR_PICK(str_smem)(stage, cart_tile_width(run), ly, uni);
  return storage == 0 ? smem_of<float>(order, vec, ly, stage) : smem_of<__nv_bfloat16>(order, vec, ly, stage);
}

}  // namespace rtk
