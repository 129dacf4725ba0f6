// Second-order finite volumes on triangle meshes (Sec. 4.2, the paper's own
// scheme): the trace on edge e of cell i is R_i = psi_i + L_i g_i . r_ie at the
// edge midpoint (r_ie = x_e - x_i, x_i the centroid), with the Green-Gauss
// gradient g_i = (1/A_i) sum_e l_e n_e (psi_i + psi_e)/2 and the Venkatakrishnan
// limiter L_i = min_e L_ie (Eq. V_limiter: Delta = (1/2) g_i . r_ie, beta from
// the max / min of psi over the cell and its neighbours, epsilon = A_i^3).
// Boundary edges see the ghost value psi^- (the side's inflow value for
// entering ordinates, 0 otherwise) in the gradient and the max / min, and carry
// first-order fluxes.
//
// Two kernels per stage, both persistent over 64-cell chunks like the
// first-order stage kernel (chunk metadata staged in shared memory by bulk
// copies, one warp per cell, lanes over ordinates, FP32 pairs; the grid has
// as many CTAs as are resident at once; a warp fetches the rows of its next
// cell to L2 while it works on one, since only neighbours' rows are there
// already):
//   tri_grad_kernel    reads psi of a cell and its three neighbours and writes
//                      the limited gradient L g (two FP32 rows per cell);
//   tri_stage2_kernel  reads psi and L g of a cell and its neighbours, takes
//                      the upwind reconstructed trace on each edge (the
//                      neighbour's R at the shared midpoint) and writes the
//                      stage output, phi
//                      and the FP64 QoI partials as the first-order kernel does.
//
// Bound by the latency of the gathers (24 warps per SM in the gradient pass, 16 in
// the stage pass; DRAM at 58 - 66 % of the copy rate, issue slots at 56 and 46 %). Differences
// to the cell's value, not values, are summed over the edges: the sums of the normals
// vanish, and the rounding error is smaller (650^2 x 256, one step against FP64: 4.22e-8
// of psi, 4.33e-8 with values). At 400^2 x 256 (FP32), with IEEE divisions in divergent
// branches and 2 ordinates per lane in the stage pass: gradient 0.82 ms, stage 0.45 ms;
// now 0.25 and 0.37 ms. A Heun step at 650^2 x 256: 6.65 -> 3.27 ms.
#include <cuda_bf16.h>

#include <type_traits>

#include "device_common.cuh"

namespace rtk {

namespace {

constexpr int kT2Threads = 256;
constexpr int kT2Warps = kT2Threads / 32;
// With 4 ordinates per lane the stage pass needs 128 registers (two CTAs per SM); the
// gradient pass needs 80, and takes 12 warps per CTA then, so that its two hold 24.
constexpr int t2_ctas(int vec) { return vec == 4 ? 2 : 3; }
constexpr int t2_grad_threads(int vec) { return vec == 4 ? 384 : 256; }
constexpr int kT2Chunk = 64;
constexpr uint32_t kT2MetaBytes = 16u + 32u + 48u;   // per cell: neighbours, geometry, second-order geometry

template <typename T, int VEC>
struct alignas(sizeof(T) * VEC) Vec2T {
  T v[VEC];
};

template <typename T, int VEC>
__device__ __forceinline__ void ld_vec(const T* p, float (&out)[VEC]) {
  const Vec2T<T, VEC> x = *reinterpret_cast<const Vec2T<T, VEC>*>(p);
#pragma unroll
  for (int l = 0; l < VEC; ++l) out[l] = Store<T>::from_smem(x.v[l]);
}

template <typename T, int VEC>
__device__ __forceinline__ void st_vec(T* p, const float (&in)[VEC]) {
  Vec2T<T, VEC> x;
#pragma unroll
  for (int l = 0; l < VEC; ++l) {
    if constexpr (sizeof(T) == 4) {
      x.v[l] = in[l];
    } else {
      x.v[l] = __float2bfloat16_rn(in[l]);
    }
  }
  *reinterpret_cast<Vec2T<T, VEC>*>(p) = x;
}

__device__ __forceinline__ void t2_bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Arithmetic on a pair of ordinates (FP32 pairs: two values per instruction), or on the one
// ordinate of a lane (a pair of itself would take twice the scalar operations: 260^2 x 32
// Heun 241 us against 222).
__device__ __forceinline__ float t2_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 t2_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float t2_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 t2_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float t2_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 t2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float t2_neg(float a) { return -a; }
__device__ __forceinline__ float2 t2_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float t2_abs(float a) { return fabsf(a); }
__device__ __forceinline__ float2 t2_abs(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ float t2_min3(float a, float b, float c) { return fmin3f(a, b, c); }
__device__ __forceinline__ float2 t2_min3(float2 a, float2 b, float2 c) {
  return make_float2(fmin3f(a.x, b.x, c.x), fmin3f(a.y, b.y, c.y));
}
__device__ __forceinline__ float t2_max3(float a, float b, float c) { return fmax3f(a, b, c); }
__device__ __forceinline__ float2 t2_max3(float2 a, float2 b, float2 c) {
  return make_float2(fmax3f(a.x, b.x, c.x), fmax3f(a.y, b.y, c.y));
}
__device__ __forceinline__ float t2_pos(float a) { return fmaxf(a, 0.f); }
__device__ __forceinline__ float2 t2_pos(float2 a) { return make_float2(fmaxf(a.x, 0.f), fmaxf(a.y, 0.f)); }
__device__ __forceinline__ float t2_pick(float s, float a, float b) { return s > 0.f ? a : b; }   // a where s > 0
__device__ __forceinline__ float2 t2_pick(float2 s, float2 a, float2 b) {
  return make_float2(s.x > 0.f ? a.x : b.x, s.y > 0.f ? a.y : b.y);
}
__device__ __forceinline__ float t2_least(float a) { return a; }
__device__ __forceinline__ float t2_least(float2 a) { return fminf(a.x, a.y); }
__device__ __forceinline__ float t2_most(float a) { return a; }
__device__ __forceinline__ float t2_most(float2 a) { return fmaxf(a.x, a.y); }
template <typename P>
__device__ __forceinline__ P t2_dup(float a) {
  if constexpr (sizeof(P) == 4) return a;
  else return make_float2(a, a);
}
__device__ __forceinline__ float t2_rcp(float a) {   // approximate reciprocal of a float in the normal range
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ float2 t2_rcp(float2 a) { return make_float2(t2_rcp(a.x), t2_rcp(a.y)); }

// psi^- of boundary side s for an ordinate: the side's inflow value if the
// ordinate enters through it (outward normals x- (-1,0), x+ (1,0), y- (0,-1),
// y+ (0,1)), else 0
__device__ __forceinline__ float ghost_value(const InstDesc& d, int s, float xi, float eta) {
  const float on = (s == 0) ? -xi : (s == 1) ? xi : (s == 2) ? -eta : eta;
  return on < 0.f ? d.ghost[s] : 0.f;
}

// Venkatakrishnan value of one edge (Eq. V_limiter with the 1/Delta factor
// cancelled), from x = |Delta| and y = |beta| on Delta's side: with p = x y and
// c = y^2 + eps^2 + p it is (c + p) / (c + 2 x^2), and 1 where that is 0 / 0.
__device__ __forceinline__ float venkat_exact(float x, float y, float eps2) {
  const float p = x * y, c = fmaf(y, y, eps2) + p;
  const float den = fmaf(x + x, x, c);
  return den > 0.f ? (c + p) / den : 1.f;
}

// Quotients a / b of positive floats, b and 1 / b in the normal range: the product with the
// approximate reciprocal, corrected once by its residual a - q b, which a fused operation
// gives exactly (P. Markstein, Computation of elementary functions on the IBM RISC System/6000
// processor, 1990). Off from the rounded quotient only where a / b lies within 2^-21 ulp of the
// middle of two floats (or, for a below 2^-102, whose residuals are subnormal, 2^-126 / a ulp).
template <typename P>
__device__ __forceinline__ P quotient(P a, P b) {
  const P r = t2_rcp(b), q = t2_mul(a, r);
  return t2_fma(t2_fma(t2_neg(q), b, a), r, q);
}

// Smallest of the three edges' limiter values outside the range of quotient for the values as
// they are. Denominators below 2^-118 are formed again, with their numerators, from x and y
// times 2^63, the quotient being homogeneous: a front's foot has them where epsilon^2 = A^6 is
// small (10^-36 at 2 * 650^2 cells). (Numerators of epsilon^2 over larger denominators, at every
// extremum of the state, are near enough as they are: testing for them too took 4 % of a step at
// 650^2 x 256, scaling every cell's terms 3 %.) Only states above 10^18 divide by IEEE.
__device__ __forceinline__ float limiter_rescaled(float gx, float gy, float up, float dn, const float (&rxh)[3],
                                                  const float (&ryh)[3], float eps2) {
  float x[3], y[3], den[3], L[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const float D = fmaf(ryh[e], gy, rxh[e] * gx);
    x[e] = fabsf(D);
    y[e] = D > 0.f ? up : dn;
    den[e] = fmaf(x[e] + x[e], x[e], fmaf(y[e], y[e], eps2) + x[e] * y[e]);
  }
  const bool ieee = !(fmax3f(den[0], den[1], den[2]) <= 1e36f);
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    if (ieee) {
      L[e] = venkat_exact(x[e], y[e], eps2);
    } else {
      const float s = den[e] < 0x1p-100f ? 0x1p63f : 1.f;
      const float xs = x[e] * s, ys = y[e] * s, p = xs * ys, c = fmaf(ys, ys, eps2 * s * s) + p;
      const float d = fmaf(xs + xs, xs, c);
      L[e] = d > 0.f ? quotient(c + p, d) : 1.f;   // 0 / 0 without a spread
    }
  }
  return fminf(fminf(L[0], L[1]), L[2]);
}

// Limited gradient L g of a pair of ordinates (or one) from the cell's values c and its
// neighbours' n0, n1, n2. The normals of a triangle sum to zero, so the Green-Gauss sum of
// l n (c + n_e)/2 is that of l n (n_e - c)/2, whose rounding error scales with the differences,
// not the values.
template <typename P>
__device__ __forceinline__ void limited_gradient(P c, P n0, P n1, P n2, const float (&axh)[3], const float (&ayh)[3],
                                                 const float (&rxh)[3], const float (&ryh)[3], float eps2, P& lx, P& ly) {
  auto dup = [](float a) { return t2_dup<P>(a); };
  const P mc = t2_neg(c), s0 = t2_add(n0, mc), s1 = t2_add(n1, mc), s2 = t2_add(n2, mc);
  const P gx = t2_fma(dup(axh[2]), s2, t2_fma(dup(axh[1]), s1, t2_mul(dup(axh[0]), s0)));
  const P gy = t2_fma(dup(ayh[2]), s2, t2_fma(dup(ayh[1]), s1, t2_mul(dup(ayh[0]), s0)));
  // beta_max and -beta_min
  const P up = t2_pos(t2_max3(s0, s1, s2)), dn = t2_pos(t2_neg(t2_min3(s0, s1, s2)));
  P num[3], den[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const P D = t2_fma(dup(ryh[e]), gy, t2_mul(dup(rxh[e]), gx));
    const P x = t2_abs(D), y = t2_pick(D, up, dn), p = t2_mul(x, y);
    const P q = t2_add(t2_fma(y, y, dup(eps2)), p);
    num[e] = t2_add(q, p);
    den[e] = t2_fma(t2_add(x, x), x, q);
  }
  // The smallest of the edges' values. Three IEEE divisions in divergent branches were 200 of
  // 269 instructions per cell and ordinate.
  P L;
  const float lo = t2_least(t2_min3(den[0], den[1], den[2])), hi = t2_most(t2_max3(den[0], den[1], den[2]));
  if (lo >= 0x1p-118f && hi <= 1e36f) {
    L = t2_min3(quotient(num[0], den[0]), quotient(num[1], den[1]), quotient(num[2], den[2]));
  } else if (t2_most(t2_max3(t2_abs(gx), t2_abs(gy), dup(0.f))) == 0.f) {
    L = dup(1.f);   // no gradient: a state of zeros
  } else if constexpr (sizeof(P) == 4) {
    L = limiter_rescaled(gx, gy, up, dn, rxh, ryh, eps2);
  } else {
    L = make_float2(limiter_rescaled(gx.x, gy.x, up.x, dn.x, rxh, ryh, eps2), limiter_rescaled(gx.y, gy.y, up.y, dn.y, rxh, ryh, eps2));
  }
  lx = t2_mul(L, gx);
  ly = t2_mul(L, gy);
}

// Fetch the rows of a cell to L2, a 128-byte line per lane at a time: na lines at a,
// nb at b, and the rest at c.
__device__ __forceinline__ void prefetch_lines(const void* a, int na, const void* b, int nb, const void* c, int nc) {
  for (int o = threadIdx.x & 31; o < na + nb + nc; o += 32) {
    const char* p = reinterpret_cast<const char*>(o < na ? a : (o < na + nb ? b : c));
    const int q = o < na ? o : (o < na + nb ? o - na : o - na - nb);
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 128 * q));
  }
}

// Chunk metadata in shared memory, double-buffered.
struct T2Meta {
  int4 nbr[2][kT2Chunk];
  float4 geo[2][2 * kT2Chunk];
  float4 geo2[2][3 * kT2Chunk];
  uint64_t bar[2];
};

__device__ __forceinline__ void t2_stage_meta(const InstDesc& d, T2Meta& m, int k, int b, int n_cells) {
  const int c0 = k * kT2Chunk;
  const int cells = min(kT2Chunk, n_cells - c0);
  mbar_arrive_expect_tx(&m.bar[b], (uint32_t)cells * kT2MetaBytes);
  t2_bulk_load(m.nbr[b], d.tri_nbr + c0, (uint32_t)cells * 16u, &m.bar[b]);
  t2_bulk_load(m.geo[b], d.tri_geo + 2 * (size_t)c0, (uint32_t)cells * 32u, &m.bar[b]);
  t2_bulk_load(m.geo2[b], d.tri_geo2 + 3 * (size_t)c0, (uint32_t)cells * 48u, &m.bar[b]);
}

// -------------------------------------------------------------------- gradient
template <int VEC, typename T>
__global__ void __launch_bounds__(t2_grad_threads(VEC), t2_ctas(VEC))
    tri_grad_kernel(const InstDesc* __restrict__ descs, const WorkItem* __restrict__ items, int stage) {
  constexpr int kGradWarps = t2_grad_threads(VEC) / 32;
  __shared__ __align__(16) T2Meta meta;
  const WorkItem it = items[blockIdx.x];
  const InstDesc& d = descs[it.inst];
  InstState* st = d.st;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int Mpad = d.Mpad;
  const int nv = Mpad / (32 * VEC);
  const int psi_lines = (Mpad * (int)sizeof(T) + 127) / 128;
  const int n_cells = (int)d.n_cells;
  const int n_chunks = (n_cells + kT2Chunk - 1) / kT2Chunk;
  const int G = it.b;
  const int64_t limit = d.wait_limit;
  if (threadIdx.x == 0) {
    mbar_init(&meta.bar[0], 1);
    mbar_init(&meta.bar[1], 1);
    fence_barrier_init();
    if (it.a < n_chunks) t2_stage_meta(d, meta, it.a, 0, n_cells);
    if (it.a + G < n_chunks) t2_stage_meta(d, meta, it.a + G, 1, n_cells);
  }
  grid_wait();
  const StepHead head = step_head(st);
  if (head.step >= d.n_steps || head.status != DEV_OK) {
    // finished or failed instances are masked; no copy may be in flight when the block leaves
    if (threadIdx.x == 0)
      for (int j = 0; j < 2; ++j)
        if (it.a + j * G < n_chunks) mbar_wait_bounded(&meta.bar[j], 0u, kDrainCycles);
    return;
  }
  const int in_buf = (stage == STAGE_EULER) ? head.parity : (stage == STAGE_HEUN1 ? 0 : 1);
  const T* __restrict__ psi = reinterpret_cast<const T*>(d.psi[in_buf]);
  float* __restrict__ lg = d.tri_lg;
  __syncthreads();
  bool ok = true;
  int i = 0;
  for (int k = it.a; k < n_chunks; k += G, ++i) {
    const int b = i & 1;
    const bool mok = mbar_wait_bounded(&meta.bar[b], (uint32_t)((i >> 1) & 1), limit);
    if (__syncthreads_or(!mok)) {
      ok = false;
      break;
    }
    const int c0 = k * kT2Chunk;
    const int c_end = min(n_cells, c0 + kT2Chunk);
    for (int cell = c0 + warp; cell < c_end; cell += kGradWarps) {
      const int li = cell - c0;
      const int4 nb = meta.nbr[b][li];
      const float4 g0 = meta.geo[b][2 * li], g1 = meta.geo[b][2 * li + 1];
      const float4 h0 = meta.geo2[b][3 * li], h1 = meta.geo2[b][3 * li + 1];
      // halves: of the face average in the gradient, and of Delta = (1/2) g . r
      const float axh[3] = {0.5f * g0.x, 0.5f * g0.z, 0.5f * g1.x}, ayh[3] = {0.5f * g0.y, 0.5f * g0.w, 0.5f * g1.y};
      const float rxh[3] = {0.5f * h0.x, 0.5f * h0.z, 0.5f * h1.x}, ryh[3] = {0.5f * h0.y, 0.5f * h0.w, 0.5f * h1.y};
      const float eps2 = g1.w;
      const int nbr[3] = {nb.x, nb.y, nb.z};
      const bool has_bnd = (nbr[0] < 0) | (nbr[1] < 0) | (nbr[2] < 0);
      {
        const int64_t nc = cell + kGradWarps < c_end ? cell + kGradWarps : (int64_t)(k + G) * kT2Chunk + warp;
        if (nc < n_cells) prefetch_lines(psi + (size_t)nc * Mpad, psi_lines, nullptr, 0, nullptr, 0);
      }
      const T* row_c = psi + (size_t)cell * Mpad + lane * VEC;
      const T* row_n[3];
#pragma unroll
      for (int e = 0; e < 3; ++e) row_n[e] = psi + (size_t)(nbr[e] >= 0 ? nbr[e] : cell) * Mpad + lane * VEC;
      float* row_g = lg + (size_t)cell * 2 * Mpad + lane * VEC;
      for (int v = 0; v < nv; ++v) {
        float c[VEC], nb3[3][VEC], ox[VEC], oy[VEC];
        ld_vec<T, VEC>(row_c, c);
#pragma unroll
        for (int e = 0; e < 3; ++e) ld_vec<T, VEC>(row_n[e], nb3[e]);
        if (has_bnd) {
          const int kk = (v * 32 + lane) * VEC;
#pragma unroll
          for (int e = 0; e < 3; ++e)
            if (nbr[e] < 0) {
#pragma unroll
              for (int l = 0; l < VEC; ++l) nb3[e][l] = ghost_value(d, -1 - nbr[e], d.xi[kk + l], d.eta[kk + l]);
            }
        }
        if constexpr (VEC >= 2) {
#pragma unroll
          for (int l = 0; l < VEC; l += 2) {
            float2 gx, gy;
            limited_gradient<float2>(make_float2(c[l], c[l + 1]), make_float2(nb3[0][l], nb3[0][l + 1]),
                              make_float2(nb3[1][l], nb3[1][l + 1]), make_float2(nb3[2][l], nb3[2][l + 1]), axh, ayh, rxh,
                              ryh, eps2, gx, gy);
            ox[l] = gx.x;
            ox[l + 1] = gx.y;
            oy[l] = gy.x;
            oy[l + 1] = gy.y;
          }
        } else {
          limited_gradient<float>(c[0], nb3[0][0], nb3[1][0], nb3[2][0], axh, ayh, rxh, ryh, eps2, ox[0], oy[0]);
        }
        st_vec<float, VEC>(row_g, ox);
        st_vec<float, VEC>(row_g + Mpad, oy);
        row_c += 32 * VEC;
        row_g += 32 * VEC;
#pragma unroll
        for (int e = 0; e < 3; ++e) row_n[e] += 32 * VEC;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0 && k + 2 * G < n_chunks) t2_stage_meta(d, meta, k + 2 * G, b, n_cells);
  }
  if (!ok && threadIdx.x == 0) {
    for (int j = i; j < i + 2; ++j) {
      const int kj = it.a + j * G;
      if (kj < n_chunks) mbar_wait_bounded(&meta.bar[j & 1], (uint32_t)((j >> 1) & 1), limit);
    }
    atomicCAS(&st->status, DEV_OK, DEV_TIMEOUT);
    st->timeout_where = ((int64_t)blockIdx.x << 32) | (int64_t)i;
  }
}

// -------------------------------------------------------------------- stage
template <int VEC, int STAGE, typename T>
__global__ void __launch_bounds__(kT2Threads, t2_ctas(VEC))
    tri_stage2_kernel(const InstDesc* __restrict__ descs, const WorkItem* __restrict__ items) {
  __shared__ __align__(16) T2Meta meta;
  __shared__ double red[(kT2Warps + 1) * NQ];
  __shared__ float wacc[kT2Warps][NQ];
  __shared__ double wdacc[kT2Warps][NQ];
  const WorkItem it = items[blockIdx.x];
  const InstDesc& d = descs[it.inst];
  InstState* st = d.st;

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float* __restrict__ d_xi = d.xi;
  const float* __restrict__ d_eta = d.eta;
  const float* __restrict__ d_w = d.w;
  const int Mpad = d.Mpad;
  const int nv = Mpad / (32 * VEC);
  const int psi_lines = (Mpad * (int)sizeof(T) + 127) / 128;
  const float dt = d.dt;
  const int nreg = d.n_regions, nq = nreg + 2;
  const int n_cells = (int)d.n_cells;
  const int n_chunks = (n_cells + kT2Chunk - 1) / kT2Chunk;
  const int G = it.b;
  const int64_t limit = d.wait_limit;

  if (lane < NQ) {
    wacc[warp][lane] = 0.f;
    wdacc[warp][lane] = 0.0;
  }
  if (threadIdx.x == 0) {
    mbar_init(&meta.bar[0], 1);
    mbar_init(&meta.bar[1], 1);
    fence_barrier_init();
    if (it.a < n_chunks) t2_stage_meta(d, meta, it.a, 0, n_cells);
    if (it.a + G < n_chunks) t2_stage_meta(d, meta, it.a + G, 1, n_cells);
  }
  grid_wait();
  const StepHead head = step_head(st);
  if (head.step >= d.n_steps || head.status != DEV_OK) {
    // finished or failed instances are masked; no copy may be in flight when the block leaves
    if (threadIdx.x == 0)
      for (int j = 0; j < 2; ++j)
        if (it.a + j * G < n_chunks) mbar_wait_bounded(&meta.bar[j], 0u, kDrainCycles);
    return;
  }
  const int parity = (STAGE == STAGE_EULER) ? head.parity : 0;
  [[maybe_unused]] const uint32_t salt = sr_salt(head.step, STAGE);   // BF16 stochastic rounding
  const int in_buf = (STAGE == STAGE_EULER) ? parity : (STAGE == STAGE_HEUN1 ? 0 : 1);
  const int out_buf = (STAGE == STAGE_EULER) ? (1 - parity) : (STAGE == STAGE_HEUN1 ? 1 : 0);
  const T* __restrict__ psi_in = reinterpret_cast<const T*>(d.psi[in_buf]);
  const T* __restrict__ psi_base = reinterpret_cast<const T*>(d.psi[0]);
  T* __restrict__ psi_out = reinterpret_cast<T*>(d.psi[out_buf]);
  const float* __restrict__ lg = d.tri_lg;
  const float* __restrict__ phi_in = d.phi[in_buf];
  float* __restrict__ phi_out = d.phi[out_buf];
  __syncthreads();
  bool ok = true;
  int ncell = 0;
  int i = 0;
  for (int k = it.a; k < n_chunks; k += G, ++i) {
    const int b = i & 1;
    const bool mok = mbar_wait_bounded(&meta.bar[b], (uint32_t)((i >> 1) & 1), limit);
    if (__syncthreads_or(!mok)) {
      ok = false;
      break;
    }
    const int c0 = k * kT2Chunk;
    const int c_end = min(n_cells, c0 + kT2Chunk);
    for (int cell = c0 + warp; cell < c_end; cell += kT2Warps) {
      const int li = cell - c0;
      const int4 nb = meta.nbr[b][li];
      const float4 g0 = meta.geo[b][2 * li], g1 = meta.geo[b][2 * li + 1];
      const float4 h0 = meta.geo2[b][3 * li], h1 = meta.geo2[b][3 * li + 1], h2 = meta.geo2[b][3 * li + 2];
      const float ax[3] = {g0.x, g0.z, g1.x}, ay[3] = {g0.y, g0.w, g1.y};
      float rx[3] = {h0.x, h0.z, h1.x}, ry[3] = {h0.y, h0.w, h1.y};
      // the neighbour's centroid-to-midpoint vector of the shared edge
      float sx[3] = {h1.z, h2.x, h2.z}, sy[3] = {h1.w, h2.y, h2.w};
      const int nbr[3] = {nb.x, nb.y, nb.z};
      const int m = nb.w & 255, reg = (nb.w >> 8) & 255;
      const float area = g1.z;
      const float sig_t = d.sig_t[m];
      const float src = d.sig_s2pi[m] * phi_in[cell] + d.q_src[m];
      const bool has_bnd = (nbr[0] < 0) | (nbr[1] < 0) | (nbr[2] < 0);
      {
        // the rows of the warp's next cell: their first use goes to DRAM, the neighbours' mostly to L2
        const int64_t nc = cell + kT2Warps < c_end ? cell + kT2Warps : (int64_t)(k + G) * kT2Chunk + warp;
        if (nc < n_cells)
          prefetch_lines(psi_in + (size_t)nc * Mpad, psi_lines, lg + (size_t)nc * 2 * Mpad, Mpad / 16,
                         psi_base + (size_t)nc * Mpad, STAGE == STAGE_HEUN2 ? psi_lines : 0);
      }
      // the lane's pieces of the rows: its own, and per edge the neighbour's (psi, then L g in x and y)
      const T* row_c = psi_in + (size_t)cell * Mpad + lane * VEC;
      const float* row_g = lg + (size_t)cell * 2 * Mpad + lane * VEC;
      const T* nrow[3];
      const float* ngrow[3];
      float gh[3];
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const size_t j = nbr[e] >= 0 ? nbr[e] : cell;   // (a boundary edge reads its own cell's, unused)
        nrow[e] = psi_in + j * Mpad + lane * VEC;
        ngrow[e] = lg + j * 2 * Mpad + lane * VEC;
        gh[e] = 0.f;
        if (nbr[e] < 0) {   // first order on the boundary: the traces are the cell value and psi^-
          gh[e] = d.ghost[-1 - nbr[e]];
          rx[e] = ry[e] = sx[e] = sy[e] = 0.f;
        }
      }

      float phi_part = 0.f, bpart = 0.f;
      for (int v = 0; v < nv; ++v) {
        const int kk = (v * 32 + lane) * VEC;
        float c[VEC], cx[VEC], cy[VEC], nbv[3][VEC], nx[3][VEC], ny[3][VEC];
        [[maybe_unused]] float base[VEC];
        ld_vec<T, VEC>(row_c, c);
        ld_vec<float, VEC>(row_g, cx);
        ld_vec<float, VEC>(row_g + Mpad, cy);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          ld_vec<T, VEC>(nrow[e], nbv[e]);
          ld_vec<float, VEC>(ngrow[e], nx[e]);
          ld_vec<float, VEC>(ngrow[e] + Mpad, ny[e]);
          nrow[e] += 32 * VEC;
          ngrow[e] += 32 * VEC;
        }
        if constexpr (STAGE == STAGE_HEUN2) ld_vec<T, VEC>(psi_base + (row_c - psi_in), base);
        row_c += 32 * VEC;
        row_g += 32 * VEC;
        if (has_bnd) {
#pragma unroll
          for (int e = 0; e < 3; ++e)
            if (nbr[e] < 0) {
#pragma unroll
              for (int l = 0; l < VEC; ++l) nbv[e][l] = gh[e];
            }
        }
        float xi[VEC], eta[VEC], w[VEC], out[VEC];
        ld_vec<float, VEC>(d_xi + kk, xi);
        ld_vec<float, VEC>(d_eta + kk, eta);
        ld_vec<float, VEC>(d_w + kk, w);
        // BF16 rounding bits of the lane's ordinates kk .. kk+VEC-1 (one group of four)
        [[maybe_unused]] uint2 rb4;
        if constexpr (sizeof(T) == 2) rb4 = sr_bits4((uint32_t)cell, sr_gkey(kk >> 2, salt));
        // ordinate pairs (two FP32 values per instruction), or the lane's one ordinate
        using P = std::conditional_t<(VEC > 1), float2, float>;
#pragma unroll
        for (int l = 0; l < VEC; l += 2) {
          auto pair = [&](const float (&a)[VEC]) {
            if constexpr (VEC > 1) return make_float2(a[l], a[l + 1]);
            else return a[l];
          };
          auto dup = [](float a) { return t2_dup<P>(a); };
          const P c2 = pair(c), xi2 = pair(xi), eta2 = pair(eta), cx2 = pair(cx), cy2 = pair(cy);
          // traces less the cell's value: omega . n l / A sums to zero over the edges
          const P mc2 = t2_neg(c2);
          P div = dup(0.f);
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const P on = t2_fma(eta2, dup(ay[e]), t2_mul(xi2, dup(ax[e])));
            const P mine = t2_fma(cx2, dup(rx[e]), t2_mul(cy2, dup(ry[e])));
            const P other = t2_fma(pair(nx[e]), dup(sx[e]), t2_fma(pair(ny[e]), dup(sy[e]), t2_add(pair(nbv[e]), mc2)));
            div = t2_fma(on, t2_pick(on, mine, other), div);
          }
          const P F = t2_add(t2_fma(dup(-sig_t), c2, t2_neg(div)), dup(src));
          P o;
          if constexpr (STAGE == STAGE_HEUN2) {
            o = t2_mul(dup(0.5f), t2_fma(dup(dt), F, t2_add(pair(base), c2)));
          } else {
            o = t2_fma(dup(dt), F, c2);
          }
          if constexpr (VEC > 1) {
            if constexpr (sizeof(T) == 2) {
              o.x = Store<T>::round_sr(o.x, sr_elem(rb4, (kk + l) & 3));
              o.y = Store<T>::round_sr(o.y, sr_elem(rb4, (kk + l + 1) & 3));
            }
            out[l] = o.x;
            out[l + 1] = o.y;
          } else {
            if constexpr (sizeof(T) == 2) o = Store<T>::round_sr(o, sr_elem(rb4, kk & 3));
            out[l] = o;
          }
        }
        st_vec<T, VEC>(psi_out + (size_t)cell * Mpad + kk, out);
#pragma unroll
        for (int l = 0; l < VEC; ++l) {
          phi_part = fmaf(w[l], out[l], phi_part);
          if (has_bnd) {
#pragma unroll
            for (int e = 0; e < 3; ++e)
              if (nbr[e] < 0) {
                const float on = xi[l] * ax[e] + eta[l] * ay[e];
                bpart += w[l] * on * ((on > 0.f) ? out[l] : gh[e]);
              }
          }
        }
      }
      const float ph = warp_sum(phi_part);
      float bsum = 0.f;
      if (has_bnd) bsum = warp_sum(bpart);
      if (lane == 0) {
        phi_out[cell] = ph;
        wacc[warp][reg] += d.sig_a_f[m] * area * ph;
        wacc[warp][nreg] += area * ph;
        wacc[warp][nreg + 1] += bsum * area;
      }
      if ((++ncell & 31) == 0) {
        __syncwarp();
        if (lane < nq) {
          wdacc[warp][lane] += (double)wacc[warp][lane];
          wacc[warp][lane] = 0.f;
        }
        __syncwarp();
      }
    }
    __syncthreads();
    if (threadIdx.x == 0 && k + 2 * G < n_chunks) t2_stage_meta(d, meta, k + 2 * G, b, n_cells);
  }
  if (!ok && threadIdx.x == 0) {
    for (int j = i; j < i + 2; ++j) {
      const int kj = it.a + j * G;
      if (kj < n_chunks) mbar_wait_bounded(&meta.bar[j & 1], (uint32_t)((j >> 1) & 1), limit);
    }
    atomicCAS(&st->status, DEV_OK, DEV_TIMEOUT);
    st->timeout_where = ((int64_t)blockIdx.x << 32) | (int64_t)i;
  }
  __syncwarp();
  if (lane < nq) wdacc[warp][lane] += (double)wacc[warp][lane];
  __syncthreads();
  if (threadIdx.x < nq) {
    double s = 0.0;
    for (int w2 = 0; w2 < kT2Warps; ++w2) s += wdacc[w2][threadIdx.x];
    red[threadIdx.x] = s;
  }
  __syncthreads();
  finalize_item<kT2Threads>(d, it, red, STAGE, red + NQ);
}

}  // namespace

int tri2_ctas_per_sm(int vec) { return t2_ctas(vec); }

cudaError_t launch_tri2_stage(const InstDesc* d_desc, const WorkItem* d_items, int n_items, int stage, int storage,
                              int vec, cudaStream_t s, bool chained) {
  if (n_items <= 0) return cudaSuccess;
#define RTK_T2(V, ST, TT)                                                                       \
  if (vec == V && stage == ST) {                                                                \
    cudaError_t e = launch_stage_kernel(tri_grad_kernel<V, TT>, n_items, t2_grad_threads(V), 0, s, chained, \
                                        d_desc, d_items, ST);                                   \
    if (e != cudaSuccess) return e;                                                             \
    return launch_stage_kernel(tri_stage2_kernel<V, ST, TT>, n_items, kT2Threads, 0, s, true, d_desc, d_items); \
  }
#define RTK_T2_ALL(TT)                                                                          \
  RTK_T2(1, STAGE_EULER, TT) RTK_T2(1, STAGE_HEUN1, TT) RTK_T2(1, STAGE_HEUN2, TT)              \
  RTK_T2(2, STAGE_EULER, TT) RTK_T2(2, STAGE_HEUN1, TT) RTK_T2(2, STAGE_HEUN2, TT)              \
  RTK_T2(4, STAGE_EULER, TT) RTK_T2(4, STAGE_HEUN1, TT) RTK_T2(4, STAGE_HEUN2, TT)
  if (storage == 0) { RTK_T2_ALL(float) } else { RTK_T2_ALL(__nv_bfloat16) }
#undef RTK_T2_ALL
#undef RTK_T2
  return cudaErrorInvalidValue;
}

}  // namespace rtk
