// Helpers shared by the Cartesian stage kernels: vector loads and stores of psi
// rows, paired FP32 arithmetic, minmod, and the epilogue that closes a work item.
#pragma once
#include <cuda_bf16.h>

#include "device_common.cuh"

namespace rtk {

// Index of cell or row g on a periodic axis of n cells (g may lie a few cells
// outside 0..n-1).
__device__ __forceinline__ int wrap_index(int g, int n) { return ((g % n) + n) % n; }

// minmod(a, b) = median(a, b, 0): 0 unless a and b share a sign, else the one of
// smaller magnitude.
__device__ __forceinline__ float minmod_med(float a, float b) {
  const float lo = fminf(a, b), hi = fmaxf(a, b);
  return fmaxf(lo, fminf(hi, 0.f));
}

template <typename T, int V>
__device__ __forceinline__ void lds_vec(const T* p, float (&out)[V]) {
  if constexpr (sizeof(T) == 4) {
    if constexpr (V == 4) {
      const float4 x = *reinterpret_cast<const float4*>(p);
      out[0] = x.x; out[1] = x.y; out[2] = x.z; out[3] = x.w;
    } else if constexpr (V == 2) {
      const float2 x = *reinterpret_cast<const float2*>(p);
      out[0] = x.x; out[1] = x.y;
    } else {
      out[0] = *reinterpret_cast<const float*>(p);
    }
  } else {
    if constexpr (V == 4) {
      const uint2 x = *reinterpret_cast<const uint2*>(p);
      const float2 fa = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x.x));
      const float2 fb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x.y));
      out[0] = fa.x; out[1] = fa.y; out[2] = fb.x; out[3] = fb.y;
    } else if constexpr (V == 2) {
      const float2 fa = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
      out[0] = fa.x; out[1] = fa.y;
    } else {
      out[0] = __bfloat162float(*p);
    }
  }
}

template <typename T, int V>
__device__ __forceinline__ void stg_vec(T* p, const float (&in)[V]) {
  if constexpr (sizeof(T) == 4) {
    if constexpr (V == 4) {
      *reinterpret_cast<float4*>(p) = make_float4(in[0], in[1], in[2], in[3]);
    } else if constexpr (V == 2) {
      *reinterpret_cast<float2*>(p) = make_float2(in[0], in[1]);
    } else {
      *reinterpret_cast<float*>(p) = in[0];
    }
  } else {
    if constexpr (V == 4) {
      __nv_bfloat162 a = __floats2bfloat162_rn(in[0], in[1]);
      __nv_bfloat162 b = __floats2bfloat162_rn(in[2], in[3]);
      uint2 x;
      x.x = *reinterpret_cast<uint32_t*>(&a);
      x.y = *reinterpret_cast<uint32_t*>(&b);
      *reinterpret_cast<uint2*>(p) = x;
    } else if constexpr (V == 2) {
      *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(in[0], in[1]);
    } else {
      *p = __float2bfloat16_rn(in[0]);
    }
  }
}

// ---- paired FP32 helpers (two values per instruction on sm_100 and later)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);   // a - b, rounded once
}
__device__ __forceinline__ float2 relu2(float2 a) { return make_float2(fmaxf(a.x, 0.f), fmaxf(a.y, 0.f)); }
// minmod(a, b) = min(max(a, b), max(a, 0), max(b, 0)), the last two given: for
// a <= b this is a when 0 <= a, 0 when a < 0 <= b and b when b < 0, i.e. the
// median of (a, b, 0). A difference feeds two faces, so its max(., 0) is shared.
__device__ __forceinline__ float2 minmod2r(float2 a, float2 b, float2 ra, float2 rb) {
  return make_float2(fmin3f(fmaxf(a.x, b.x), ra.x, rb.x), fmin3f(fmaxf(a.y, b.y), ra.y, rb.y));
}

template <typename T, int V>
__device__ __forceinline__ void lds_vec2(const T* p, float2 (&out)[V / 2]) {
  static_assert(V == 2 || V == 4, "pairs need V = 2 or 4");
  if constexpr (sizeof(T) == 4) {
    if constexpr (V == 4) {
      const float4 x = *reinterpret_cast<const float4*>(p);
      out[0] = make_float2(x.x, x.y);
      out[1] = make_float2(x.z, x.w);
    } else {
      out[0] = *reinterpret_cast<const float2*>(p);
    }
  } else {
    if constexpr (V == 4) {
      const uint2 x = *reinterpret_cast<const uint2*>(p);
      out[0] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x.x));
      out[1] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x.y));
    } else {
      out[0] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
    }
  }
}

template <typename T, int V>
__device__ __forceinline__ void stg_vec2(T* p, const float2 (&in)[V / 2]) {
  if constexpr (sizeof(T) == 4) {
    if constexpr (V == 4) {
      *reinterpret_cast<float4*>(p) = make_float4(in[0].x, in[0].y, in[1].x, in[1].y);
    } else {
      *reinterpret_cast<float2*>(p) = in[0];
    }
  } else {
    if constexpr (V == 4) {
      __nv_bfloat162 a = __floats2bfloat162_rn(in[0].x, in[0].y);
      __nv_bfloat162 b = __floats2bfloat162_rn(in[1].x, in[1].y);
      uint2 x;
      x.x = *reinterpret_cast<uint32_t*>(&a);
      x.y = *reinterpret_cast<uint32_t*>(&b);
      *reinterpret_cast<uint2*>(p) = x;
    } else {
      *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(in[0].x, in[0].y);
    }
  }
}

// Epilogue of a work item: write phi_out of the tile and reduce the FP64 QoI
// partials of the output state (absorption per region, mass, boundary outflow),
// then close the launch for this work item. scr: scr_n >= NT floats of shared
// memory that nothing else uses any more (the ring).
template <int STAGE, int NT>
__device__ __forceinline__ void cart_epilogue(const InstDesc& d, const WorkItem& it, float* __restrict__ phi_out,
                                              const float* tile_acc, double* red, float* scr, int scr_n, int x0,
                                              int ya, int nrows, int TX, float bacc) {
  const int tid = threadIdx.x;
  const int nx = d.nx;
  const int nreg = d.n_regions, nq = nreg + 2;
  float fa[kMaxReg];
#pragma unroll
  for (int g = 0; g < kMaxReg; ++g) fa[g] = 0.f;
  float fm = 0.f;
  const int tx_shift = 31 - __clz(TX);   // tile widths are powers of two
  for (int i = tid; i < nrows * TX; i += NT) {
    const int r = i >> tx_shift, xl = i & (TX - 1);
    const int gx = x0 + xl;
    if (gx >= nx) continue;
    const size_t cell = (size_t)(ya + r) * nx + gx;
    const float ph = tile_acc[i];
    phi_out[cell] = ph;
    const int reg = d.region[cell];
    const float va = d.sig_a_f[d.mat[cell]] * ph;
#pragma unroll
    for (int g = 0; g < kMaxReg; ++g)
      if (g == reg) fa[g] += va;
    fm += ph;
  }
  // per-thread FP32 terms to shared memory, as many quantities at a time as fit;
  // a warp per quantity adds them in FP64
  const int batch = min(nq, scr_n / NT);
  for (int q0 = 0; q0 < nq; q0 += batch) {
    const int q1 = min(nq, q0 + batch);
    __syncthreads();
#pragma unroll
    for (int g = 0; g < kMaxReg; ++g)
      if (g < nreg && g >= q0 && g < q1) scr[(g - q0) * NT + tid] = fa[g];
    if (nreg >= q0 && nreg < q1) scr[(nreg - q0) * NT + tid] = fm;
    if (nreg + 1 >= q0 && nreg + 1 < q1) scr[(nreg + 1 - q0) * NT + tid] = bacc;
    __syncthreads();
    for (int q = q0 + (tid >> 5); q < q1; q += NT / 32) {
      const double v = warp_block_sum<NT>(scr + (q - q0) * NT);
      if ((tid & 31) == 0) red[q] = q <= nreg ? v * d.area_d : v;
    }
  }
  __syncthreads();
  finalize_item<NT>(d, it, red, STAGE, red + NQ);
}

}  // namespace rtk
