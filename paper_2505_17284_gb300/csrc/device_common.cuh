// Device helpers for the S_N kernels: mbarrier and TMA wrappers (inline PTX for
// sm_103a), bounded waits, storage conversions, warp/block reductions and the
// deterministic QoI finalize that closes every stage launch.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "rt_internal.h"

namespace rtk {

// ------------------------------------------------------------------ storage
template <typename T> struct Store;
template <> struct Store<float> {
  static __device__ __forceinline__ float load(const float* p) { return *p; }
  static __device__ __forceinline__ float from_smem(const float v) { return v; }
  static __device__ __forceinline__ float round(float v) { return v; }
  static __device__ __forceinline__ float round_sr(float v, uint32_t) { return v; }
  static __device__ __forceinline__ float2 round_sr2(float2 v, uint32_t) { return v; }
  static __device__ __forceinline__ void store(float* p, float v) { *p = v; }
};
template <> struct Store<__nv_bfloat16> {
  static __device__ __forceinline__ float load(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  static __device__ __forceinline__ float from_smem(const __nv_bfloat16 v) { return __bfloat162float(v); }
  // round-to-nearest-even to bf16 and back
  static __device__ __forceinline__ float round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
  // stochastic rounding to bf16 and back, with 16 random bits r: the magnitude
  // is rounded up with probability (dropped low 16 bits) / 2^16, so the stored
  // value is unbiased; exactly representable values are kept
  static __device__ __forceinline__ float round_sr(float v, uint32_t r) {
    return __uint_as_float((__float_as_uint(v) + (r & 0xffffu)) & 0xffff0000u);
  }
  // the pair (a, b) with the 32 random bits r: low half for a, high half for b
  static __device__ __forceinline__ float2 round_sr2(float2 v, uint32_t r) {
    return make_float2(__uint_as_float((__float_as_uint(v.x) + (r & 0xffffu)) & 0xffff0000u),
                       __uint_as_float((__float_as_uint(v.y) + (r >> 16)) & 0xffff0000u));
  }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
};

// ------------------------------------------------------------------ random bits for BF16 stores
// BF16 keeps 8 significant bits. Rounding every stored state to nearest drops
// any per-step change smaller than half a unit in the last place; with small
// time steps (a triangle mesh takes dt from its smallest cells, so most cells
// change by a small fraction per step) the state then stops moving where it
// varies slowly and particles are lost. The stage kernels therefore round BF16
// stores stochastically (Store::round_sr) with 16 random bits per element.
// The bits are a counter-based hash of (cell, ordinate, step, stage), so a run
// is reproducible, independent of the launch configuration (tiles, ordinates
// per lane, batching), and different from step to step:
//   salt  = mix(4 step + stage + c)                  once per launch
//   gkey  = g * K1 ^ salt                             per group g = k / 4 of
//                                                     four ordinates
//   h     = mix(cell * K2 + gkey)                     per cell and group
//   h2    = xorshift-multiply of h
// ordinate 4g + e takes the low (e even) or high (e odd) half of h (e < 2) or
// h2 (e >= 2). mix is Wellons' "lowbias32" 32-bit integer mixer; K1, K2 odd
// constants (cell * K2 is a bijection of the 32-bit cell index, so no index
// wraps: cells are below 2^31). One mixer call serves four elements.
__device__ __forceinline__ uint32_t sr_mix(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}
// salt of one stage launch: step counter and stage (Euler, Heun 1, Heun 2)
__device__ __forceinline__ uint32_t sr_salt(int64_t step, int stage) {
  return sr_mix((uint32_t)step * 4u + (uint32_t)stage + 0x2545f491u);
}
// key of the ordinate group g (ordinates 4g .. 4g+3) in one launch
__device__ __forceinline__ uint32_t sr_gkey(int g, uint32_t salt) { return ((uint32_t)g * 0x85ebca77u) ^ salt; }
// 64 random bits of the group's four elements in one cell: .x for ordinates
// 4g, 4g+1 (low, high half), .y for 4g+2, 4g+3
__device__ __forceinline__ uint2 sr_bits4(uint32_t cell, uint32_t gkey) {
  const uint32_t h = sr_mix(cell * 0x9e3779b1u + gkey);
  uint32_t h2 = (h ^ (h >> 15)) * 0x2c1b3c6du;
  h2 ^= h2 >> 13;
  return make_uint2(h, h2);
}
// the 16 random bits (low half) of ordinate 4g + e
__device__ __forceinline__ uint32_t sr_elem(uint2 b, int e) {
  const uint32_t w = (e & 2) ? b.y : b.x;
  return (e & 1) ? (w >> 16) : w;
}

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Make the initialised barriers visible to the async (TMA) proxy.
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Order this thread's earlier generic-proxy shared-memory accesses (and those
// made visible to it by a barrier) before later async-proxy (TMA) writes.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

constexpr int64_t kDrainCycles = 4000000000LL;   // bound of a wait for copies in flight (about two seconds)

// Wait for phase `parity` of `bar` to complete, for at most `limit` SM clock
// cycles. Returns false if the limit ran out.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, int64_t limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (clock64() - t0 > limit) return false;
  }
}

// Stage kernels of a run of steps are launched with programmatic serialisation: a grid's
// blocks become resident when those of the stage before have left, before its writes are
// flushed and its end is reported, and run what depends on set-up data alone (descriptors,
// work items, mesh data) until grid_wait() returns: the stage before has then completed and
// its writes are visible (at once in a launch without the attribute). Every thread calls it,
// in every block and before any return: a grid that completed without waiting would let the
// one after it start too early. No grid lets the next one in before its own blocks leave
// (griddepcontrol.launch_dependents): that cost 2 us a launch, and the next stage's blocks
// then filled whichever SMs emptied first, two to an SM on grids below one wave (140^2 x 128
// Heun 52 -> 59 us). Without it 60^2 x 64 triangles 14.6 -> 12.3 us a first-order step and
// 55.7 -> 45.8 a second-order one, 130^2 x 64 20.7 -> 18.4 and 100.8 -> 97.7.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The instance's position in time, read past L1.
struct StepHead {
  int64_t step;
  int32_t parity, status;
};
__device__ __forceinline__ StepHead step_head(const InstState* st) {
  return {__ldcg(&st->step), __ldcg(&st->parity), __ldcg(&st->status)};
}

// 3-D tiled TMA load of one box into shared memory, completing on `bar`.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}

// The tensor maps live in global memory (written before the launch); make
// them visible to the tensormap proxy before the first TMA use.
__device__ __forceinline__ void fence_tensormap_acquire(const CUtensorMap* map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(map))
               : "memory");
}

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// ------------------------------------------------------------------ math
// Three-operand minimum and maximum (one instruction each).
__device__ __forceinline__ float fmin3f(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float fmax3f(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum V per-lane values over the 32 lanes of a warp with log2(V) + 5 - log2(V)
// butterfly steps; afterwards lane l holds the total of value index
// (l >> (5 - log2 V)). Fixed order: deterministic.
template <int V>
__device__ __forceinline__ float multi_warp_sum(float (&v)[V], int lane) {
  static_assert(V == 1 || V == 2 || V == 4 || V == 8, "V must be 1, 2, 4 or 8");
  if constexpr (V == 1) {
    return warp_sum(v[0]);
  } else {
    // step with offset 16: keep half of the values, send the other half
    constexpr int H = V / 2;
    float a[H];
    const bool hi = (lane & 16) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const float keep = hi ? v[H + i] : v[i];
      const float send = hi ? v[i] : v[H + i];
      a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
    if constexpr (H == 1) {
      float s = a[0];
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      return s;
    } else {
      constexpr int Q = H / 2;
      float b[Q];
      const bool hi8 = (lane & 8) != 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const float keep = hi8 ? a[Q + i] : a[i];
        const float send = hi8 ? a[i] : a[Q + i];
        b[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
      }
      if constexpr (Q == 1) {
        float s = b[0];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
      } else {
        const bool hi4 = (lane & 4) != 0;
        float s = (hi4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, hi4 ? b[0] : b[1], 4);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        return s;
      }
    }
  }
}

// ------------------------------------------------------------------ QoI finalize
// Block-wide FP64 reduction of `acc` (nq values per thread, nq <= NQ) into
// red[0..nq) in shared memory, in a fixed order. Must be called by all threads.
template <int NT>
__device__ __forceinline__ void block_reduce_q(const double (&acc)[NQ], int nq, double* red /*[NT/32][NQ]*/) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    if (q < nq) {
      const double s = warp_sum_d(acc[q]);
      if (lane == 0) red[warp * NQ + q] = s;
    }
  }
  __syncthreads();
  if (threadIdx.x < nq) {
    double s = 0.0;
    for (int w = 0; w < NT / 32; ++w) s += red[w * NQ + threadIdx.x];
    red[threadIdx.x] = s;    // row 0 reused for the result (read above by this thread only)
  }
  __syncthreads();
}

// Sum over a block of one FP32 value per thread (v[0 .. NT) in shared memory), in
// FP64, by one warp; every lane returns it. A lane first adds its NT / 32 values
// with Knuth's two-sum, twice: the rounding errors of the FP32 sum are kept beside
// it, and those of their sum beside them, which together hold more bits than an
// FP64 sum (s + e alone holds about 48). So three conversions and 7 additions run
// on the FP64 pipe instead of 5 additions in each of the block's warps: that pipe
// adds about 2 lanes per cycle and SM here, and the block sums were most of a small
// launch's tail.
template <int NT>
__device__ __forceinline__ double warp_block_sum(const float* v) {
  const int lane = threadIdx.x & 31;
  float s = 0.f, e = 0.f, f = 0.f;
#pragma unroll
  for (int j = 0; j < NT / 32; ++j) {
    const float x = v[lane + 32 * j];
    const float t = s + x, z = t - s;
    const float y = (s - (t - z)) + (x - z);   // t + y = s + x
    const float u = e + y, w = u - e;
    f += (e - (u - w)) + (y - w);
    s = t;
    e = u;
  }
  double r = (double)s + ((double)e + (double)f);
  if (!isfinite(r)) {   // a value, or the FP32 sum of finite ones, is not finite
    r = 0.0;
    for (int j = 0; j < NT / 32; ++j) r += (double)v[lane + 32 * j];
  }
  return warp_sum_d(r);
}

// Sum over rows [0, n) of one quantity by one warp, FP64, fixed order.
__device__ __forceinline__ double warp_rows_sum(const double* row, int n) {
  const int lane = threadIdx.x & 31;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  for (int i = lane; i < n; i += 128) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i + 32 * j < n) a[j] += __ldcg(row + i + 32 * j);
  }
  return warp_sum_d((a[0] + a[1]) + (a[2] + a[3]));
}

// Write this work item's QoI partial (red[0..nq)), and if it is the last item of
// its instance in this launch, reduce all partials in item order and apply the
// time-integration update of `stage`. Must be called by all threads. Partials are
// kept quantity by quantity ([nq][count]): the last item's warps read a quantity
// each, 32 items at a time, and one thread per quantity then updates the state.
// Bound by latency: it is the tail of every launch. With the block sums taken by
// all warps on the FP64 pipe, a fence by every thread and a serial update of 18
// quantities by one thread, a 70^2 x 64 first-order step took 72 us with its QoIs
// read, 140^2 x 128 Heun 111 us; now 58 and 89 us.
template <int NT>
__device__ void finalize_item(const InstDesc& d, const WorkItem& it, const double* red, int stage,
                              double* scratch /*[NQ]*/) {
  __shared__ uint32_t s_last;
  const int nreg = d.n_regions, nq = nreg + 2;
  InstState* st = d.st;
  if (threadIdx.x < nq) d.partials[(size_t)threadIdx.x * it.count + it.item] = red[threadIdx.x];
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();   // the block's partials (ordered before by the barrier) before its ticket
    const uint32_t t = atomicAdd(&st->ticket, 1u);
    s_last = (t == static_cast<uint32_t>(it.count - 1)) ? 1u : 0u;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  for (int q = threadIdx.x >> 5; q < nq; q += NT / 32) {
    const double v = warp_rows_sum(d.partials + (size_t)q * it.count, it.count);
    if ((threadIdx.x & 31) == 0) scratch[q] = v;
  }
  __syncthreads();
  // compact order (regions..., mass, outflow) to the NQ layout, one thread each
  const int q = threadIdx.x;
  if (q < NQ) {
    double S = 0.0;
    if (q < nreg) S = scratch[q];
    if (q == kQMass) S = scratch[nreg];
    if (q == kQOut) S = scratch[nreg + 1];
    const double dt = d.dt_d;
    if (stage == STAGE_EULER) {
      st->I[q] += dt * st->S_cur[q];
      st->S_cur[q] = S;
    } else if (stage == STAGE_HEUN1) {
      st->I[q] += 0.5 * dt * st->S_cur[q];
      st->S_mid[q] = S;
    } else if (stage == STAGE_HEUN2) {
      st->I[q] += 0.5 * dt * st->S_mid[q];
      st->S_cur[q] = S;
    } else {  // STAGE_INIT
      st->S_cur[q] = S;
    }
    if (!isfinite(S)) atomicCAS(&st->status, DEV_OK, DEV_NONFINITE);
  }
  if (q == 0) {
    if (stage == STAGE_EULER) {
      st->step += 1;
      st->parity ^= 1;
    } else if (stage == STAGE_HEUN2) {
      st->step += 1;
    }
    st->ticket = 0u;
  }
}

// Launch of a stage kernel; `chained`: it follows another kernel of the same run of steps.
template <typename... P, typename... A>
inline cudaError_t launch_stage_kernel(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t stream,
                                       bool chained, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace rtk
