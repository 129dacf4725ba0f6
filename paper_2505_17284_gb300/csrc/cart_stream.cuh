// Cartesian stage kernel of the explicit S_N step (Sec. 4.2-4.3), streaming form:
// every warp walks its own strip of cells along the flow, fed by its own ring of
// shared-memory rows, and never waits for another warp until the tile is done.
//
// Work split. A CTA of 8 warps owns a tile of TX = 8 WX cells in x by a segment
// of `ly` rows; warp w takes the 8 columns w mod WX of the tile and the chunks
// w / WX, w / WX + WC, ... of ordinates (WC = 8 / WX). A chunk is a window of 32
// consecutive ordinates that share the sign of eta; lane l holds the ordinates
// 4 (l mod 8) .. + 3 of the window for the pair of cells 2 (l / 8), + 1 of the
// strip, so that 8 lanes read one cell's 32 ordinates as one 128-byte row of shared
// memory, without bank conflicts whichever cell a lane is at: lanes may walk x in
// opposite directions. A window may begin or end inside the 32 (the quadrature's
// sign changes need not fall on multiples of 32): ordinates outside [lo, hi) carry
// no weight and are not stored, and a neighbouring window covers them.
//
// Row walk. For each chunk the warp takes its rows along the flow in y, two at a
// time. The rows of a pair, (8 + 2H) cells x 32 ordinates each (Heun stage 2: and 8
// cells of psi^n), arrive by 16-byte asynchronous copies, one or two pairs ahead, into
// a slot that the warp frees with a __syncwarp. (Loads by one lane through tensor maps
// cost 60 issue slots per row, more than half of the arithmetic, and a tensor-map
// fence per warp took 9 us at a tile's start.) When a row is read,
//   z = - dt |xi|/dx (F_right - F_left)    and the part of  - dt |eta|/dy (G_up - G_low)
// known by then are kept, with
//   F_right - F_left = (u_0 - u_-1) + (m_0 - m_-1)/2,  m_f = minmod of the two
// differences beside face f's upwind cell, cells numbered along the flow. The face
// above the previous row is known once this row is, so the previous row is completed
// with out = (a c + b) + (z + ...). Domain faces are first order: m = 0 there. The
// window carried from row to row is (c, its difference to the row before, z): no row
// is read twice and there is no barrier between rows, so the 16 warps of an SM drift
// apart and cover each other's waits.
//
// Update. With a = 1 - dt sigma_t and b = dt (sigma_s/(2 pi) phi + Q) per cell:
//   Euler / Heun stage 1: out = a psi + b - dt (div_x + div_y)
//   Heun stage 2:         out = psi^n / 2 + (a psi1 + b - dt (div_x + div_y)) / 2
// (Eq. sn_2d_eqn_fv and Sec. 4.3; the halves are exact, the last sum rounds once). phi_out = sum_k w_k out_k: two rows are summed over
// 8 lanes by shuffles, chunks in the warp's own accumulators, the WC warps of a column
// in fixed order at the end. The boundary outflow is taken from the stored rows after
// the walk; the epilogue writes phi_out and the FP64 QoI partials.
//
// Ordered form (second order, grids of at most 1e5 cells; kOrderedMaxCells has the reason).
// The sums above add differences, and phi in another order than the kernels that read whole
// chunks of 32 V ordinates do (V ordinates per lane). Where runs are long enough for the
// scheme to amplify that, the operations of those kernels are kept, value for value: face
// values F = u + m/2 and G, then div = ax (F_1 - F_0) + ay (G_1 - G_0) with the last product
// fused (y for per-lane directions, x for chunk-uniform ones), out = (a c + b) - div; and the
// lanes leave their terms of phi in shared memory (128 bytes per cell, or all ordinates where
// V = 1; no shuffles in the walk), which are then added in the order of a warp's butterfly
// over the chunk. The face values take 8 more registers (spilled, mostly at sides), the terms
// limit a segment to 13 rows with two CTAs per SM (fewer for V = 1, which takes one CTA per SM
// then), and rules of more than 128 ordinates meet at a barrier of the column's warps per
// 128. Per Heun step, sums of differences, ordered, and the general kernel: 140^2 x 128 52, 56
// and 111 us, 280^2 x 256 163, 179 and 320, 140^2 x 100 56, 66 and 135, 272^2 x 64 52, 65 and
// 143 (300^2).
//
// Bound by: HBM on large grids (1400^2 x 512 FP32 Heun: 20 bytes per cell and ordinate
// at 5.6 TB/s; a pair of rows is about 500 instructions for 16 values a lane, issue
// slots half used), by instruction latency and the fixed cost of a launch on small ones.
// Per Heun step, against the kernels that it replaced (one CTA barrier per row with
// chunk-uniform directions; for mixed directions the general kernel of
// cart_kernel.cuh): 1400^2 x 512 4.12 -> 3.57 ms (BF16 4.42 -> 3.69, first-order Euler
// 1.51 -> 1.36), 700^2 x 484 1.36 -> 1.13, 531^2 x 100 0.57 -> 0.25. Measured and not
// kept: 4 cells per lane (12 warps per SM: spills, and a loop too long for the instruction
// cache), scalar instead of paired FP32 (24 % slower), prefetching the pair after next to L2.
#pragma once
#include <cuda_bf16.h>

#include <atomic>

#include "cart_common.cuh"

namespace rtk {

constexpr int kStrThreads = 256;
constexpr int kStrWarps = kStrThreads / 32;
constexpr int kStrRun = 2;                   // consecutive cells of a lane
constexpr int kStrCells = 4 * kStrRun;       // cells of a warp's strip
constexpr int kStrOrds = 32;                 // ordinates of a chunk
enum StrForm { STR_DIFF = 0, STR_LANE = 1, STR_UNI = 2 };   // order of the operations (str_chunk)

template <int ORDER, int STAGE, typename T>
struct StrCfg {
  static constexpr int H = ORDER;
  // rows loaded per chunk beyond the segment: H before it, and at second order one after it
  static constexpr int EXTRA = ORDER == 2 ? 3 : 1;
  // ring slots, of two rows each: two CTAs per SM leave about 80 KB of an SM's shared memory to each ring
  static constexpr int NS = (STAGE == STAGE_HEUN2 ? 2 : 3) + (sizeof(T) == 2 ? 1 : 0);
  static constexpr int cell_bytes = kStrOrds * (int)sizeof(T);
  static constexpr int row_cells = kStrCells + 2 * H;
  static constexpr int halo_bytes = row_cells * cell_bytes;
  static constexpr int base_bytes = STAGE == STAGE_HEUN2 ? kStrCells * cell_bytes : 0;
  static constexpr int row_bytes = halo_bytes + base_bytes;
  static constexpr int ring_bytes = kStrWarps * NS * 2 * row_bytes;
  // 16-byte copies: a lane takes piece lane % pieces of cells lane / pieces + j * per_copy
  static constexpr int pieces = cell_bytes / 16;
  static constexpr int per_copy = 32 / pieces;
  static constexpr int copies = (row_cells + per_copy - 1) / per_copy;
  static constexpr int last_lanes = (row_cells - (copies - 1) * per_copy) * pieces;   // lanes of the last copy
};

// Floats per cell that hold the lanes' terms of phi in the ordered form (form: CartForm).
__host__ __device__ inline int str_parts(int form) { return form >> 1; }
// (a, b) of every cell, and one phi accumulator per cell and chunk group; in the ordered
// form one per cell, and the lanes' terms
__host__ __device__ inline size_t str_tile_bytes(int tx, int ly, int parts) {
  return (size_t)ly * tx * 8 + (parts ? (size_t)ly * tx * 4 * (1 + parts) : (size_t)ly * kStrWarps * kStrCells * 4);
}
constexpr size_t kStrRedBytes = (kStrWarps + 1) * NQ * 8;

template <int ORDER, int STAGE, typename T>
size_t str_smem_for(int tx, int ly, int form) {
  return StrCfg<ORDER, STAGE, T>::ring_bytes + str_tile_bytes(tx, ly, str_parts(form)) + kStrRedBytes + 128;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// copies 16 bytes, or fills with zeros (bytes = 0; src is not read)
__device__ __forceinline__ void cp_async16z(uint32_t dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// What only strips at the domain's edge need, in shared memory (one per CTA).
struct StrEdge {
  int nx, ny, periodic_x, periodic_y;
  float ghost[4];   // psi^- of the sides
};

// One warp's strip: what the row walk needs from the descriptor and the tile.
struct StrWarp {
  uint32_t ring;       // this warp's slots (shared address)
  uint8_t* ring_p;
  const float2* ab;    // [ly][TX] of the tile
  float* acc;          // [ly][TX] of the warp's chunk group
  float* part;         // ordered form: the lanes' terms of phi, [ly][TX][parts]
  int parts, slots;    // ordered form: floats per cell, and windows that they hold
  const StrEdge* ed;
  const uint8_t* src;  // the lane's piece of the strip's row 0, ordinate 0: copy 0 of the halo row
  int64_t to_base;     // from there to its piece of the row of psi^n beside it, in bytes (Heun stage 2)
  int64_t row_bytes;   // one grid row of psi
  int col_bytes;       // cells between the copies of a lane
  int xw, xl;          // first cell of the strip: global, in the tile
  int ya, yb, TX;
  int ahead;           // slots in flight: NS - 1, or the row pairs of a chunk if they are fewer
};

// Start the copies of rows 2q, 2q + 1 of a chunk (first ordinate kb, flow dy) into a
// slot. Cells and rows outside the domain are filled with zeros (vacuum); inflow values
// and, on a periodic x axis, the wrapped cells are set when the row is used.
template <int ORDER, int STAGE, typename T, bool EDGE>
__device__ __forceinline__ void str_load(const StrWarp& w, uint32_t dst, int kb, int dy, int q) {
  using L = StrCfg<ORDER, STAGE, T>;
  const int lane = threadIdx.x & 31;
  int p = (dy > 0 ? w.ya : w.yb - 1) + dy * (2 * q - L::H);
  const uint8_t* src0 = w.src + kb * (int)sizeof(T);
  dst += 16 * lane;
  if constexpr (!EDGE) {
    const uint8_t* src = src0 + p * w.row_bytes;
    const int64_t rb = dy > 0 ? w.row_bytes : -w.row_bytes;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const uint8_t* s = src;
#pragma unroll
      for (int j = 0; j < L::copies; ++j) {
        if (j + 1 < L::copies || lane < L::last_lanes) cp_async16(dst + r * L::row_bytes + j * 512, s);
        s += w.col_bytes;
      }
      if (STAGE == STAGE_HEUN2 && (ORDER == 1 || q > 0)) {   // psi^n of the row that row 2q + r completes
        const uint8_t* sb = src + w.to_base - (ORDER == 2 ? rb : 0);
#pragma unroll
        for (int j = 0; j * L::per_copy < kStrCells; ++j) {
          cp_async16(dst + r * L::row_bytes + L::halo_bytes + j * 512, sb);
          sb += w.col_bytes;
        }
      }
      src += rb;
    }
    return;
  }
  const int nx = w.ed->nx, ny = w.ed->ny;
  const int g0 = w.xw - L::H + lane / L::pieces;
#pragma unroll 1
  for (int r = 0; r < 2; ++r) {
    int pl = p;
    bool in = p >= 0 && p < ny;
    if (!in && w.ed->periodic_y) { pl = wrap_index(p, ny); in = true; }
    const uint8_t* s = src0 + (in ? pl : 0) * w.row_bytes;
#pragma unroll
    for (int j = 0; j < L::copies; ++j) {
      const int g = g0 + j * L::per_copy;
      if (j + 1 < L::copies || lane < L::last_lanes)
        cp_async16z(dst + j * 512, s, in && g >= 0 && g < nx ? 16u : 0u);
      s += w.col_bytes;
    }
    if constexpr (STAGE == STAGE_HEUN2) {
      const int pb = ORDER == 2 ? p - dy : p;
      const bool inb = pb >= 0 && pb < ny;
      const uint8_t* sb = src0 + w.to_base + (inb ? pb : 0) * w.row_bytes;
#pragma unroll
      for (int j = 0; j * L::per_copy < kStrCells; ++j) {
        cp_async16z(dst + L::halo_bytes + j * 512, sb, inb && g0 + L::H + j * L::per_copy < nx ? 16u : 0u);
        sb += w.col_bytes;
      }
    }
    dst += L::row_bytes;
    p += dy;
  }
}

// Window of one row: values, difference to the row before along the flow, and the flux
// terms known when the row arrives (all of x, and of y the face below it); in the ordered
// form the differences of the face values in x.
struct StrRow {
  float2 c[kStrRun][2], d[kStrRun][2], z[kStrRun][2];
};

// One chunk of one warp; c_next is the warp's next chunk (or past the last), whose first
// rows are loaded while this one ends. EDGE: the strip with its halo touches a side of
// the domain. Strips away from the sides have a body of their own: testing for the sides
// in the row cost 48 of 291 instructions and 17 % of the time at 560^2 x 512.
// FORM: STR_DIFF, or the ordered form with the operations of per-lane (STR_LANE) or of
// chunk-uniform directions (STR_UNI) and with V ordinates per term of phi.
template <int ORDER, int STAGE, typename T, bool EDGE, int FORM, int V>
__device__ __forceinline__ void str_chunk(const InstDesc& d, const StrWarp& w, const int4 ch, const int c, const int c_next,
                                          int& slot, const int in_buf, T* __restrict__ psi_out,
                                          [[maybe_unused]] const uint32_t salt) {
  constexpr bool ORD = FORM != STR_DIFF;
  using L = StrCfg<ORDER, STAGE, T>;
  constexpr int H = L::H, R = kStrRun, NS = L::NS;
  constexpr int NU = R + H + ORDER - 1;   // cells read per row: -H .. R + ORDER - 2 along the flow
  const int lane = threadIdx.x & 31, l8 = lane & 7, grp = lane >> 3;
  const bool more = c_next < d.n_chunks;
  int nkb = 0, ndy = 1;
  if (more) {
    const int4 cn = d.str_chunks[c_next];
    nkb = cn.x;
    ndy = cn.z;
  }
  const int k0 = ch.x + 4 * l8;
  const int dys = ch.z;
  const int n = w.yb - w.ya + L::EXTRA;                // rows of the chunk
  const int npair = (n + 1) / 2;
  constexpr bool PARTIAL = !ORD || V == 1;             // windows may be partial
  const bool part = PARTIAL && ch.y != (32 << 8);

  float2 w2[2], ax2[2], ay2[2];
  float xsum = 0.f;
  {
    const float dt = d.dt;
    // stage 2 averages psi^n and the update: the halves (of a and b, too) are exact
    const float half = (ORD ? 1.f : -1.f) * (STAGE == STAGE_HEUN2 ? 0.5f : 1.f);
    const int lo = ch.x + (ch.y & 255), hi = ch.x + (ch.y >> 8);
    float wv[4], ax[4], ay[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const bool own = k0 + v >= lo && k0 + v < hi;
      const float x = own ? d.xi[k0 + v] : 0.f, y = own ? d.eta[k0 + v] : 0.f;
      wv[v] = own ? d.w[k0 + v] : 0.f;
      xsum += x;
      ax[v] = half * (dt * fabsf(x) * d.inv_dx);
      ay[v] = half * (dt * fabsf(y) * d.inv_dy);
    }
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      w2[v] = make_float2(wv[2 * v], wv[2 * v + 1]);
      ax2[v] = make_float2(ax[2 * v], ax[2 * v + 1]);
      ay2[v] = make_float2(ay[2 * v], ay[2 * v + 1]);
    }
  }
  const int dxs = xsum >= 0.f ? 1 : -1;               // the lane's flow direction in x
  const int s0 = R * grp + (dxs > 0 ? 0 : R - 1);      // the lane's first cell along the flow, within the strip
  const int step_b = dxs * L::cell_bytes;              // next cell along the flow, in a slot
  const int start = dys > 0 ? w.ya : w.yb - 1;
  const int gx0 = w.xw + s0;
  const uint8_t* ring_l = w.ring_p + (s0 + H) * L::cell_bytes + 4 * l8 * (int)sizeof(T);
  const int astep = dys * w.TX;
  // row completed by row 0 of the chunk: EXTRA rows before the first (never touched)
  T* op = psi_out + ((int64_t)(start - dys * L::EXTRA) * d.nx + gx0) * d.Mpad + k0;
  const int64_t ostep = (int64_t)dys * d.nx * d.Mpad;
  const int mstep = dxs * d.Mpad;
  const float2* tab = w.ab + (start - w.ya) * w.TX - L::EXTRA * astep + w.xl + s0;
  float* tacc = w.acc + (start - w.ya) * w.TX - L::EXTRA * astep + w.xl + R * grp + (l8 >> 2) + ((l8 >> 1) & 1) * astep;
  // ordered form: the lane's terms of the row's cells (a pair of cells has 2 parts floats in
  // blocks of 32 / V, rotated by the pair so that the four of a row lie in different banks)
  [[maybe_unused]] float* tpart = nullptr;
  [[maybe_unused]] int poff[R], pstep = 0;
  [[maybe_unused]] bool second = false;   // the term is added to that of the window 64 ordinates before
  if constexpr (ORD && V == 1) {   // one ordinate per term: all ordinates of a cell in order
    tpart = w.part + ((start - w.ya) * w.TX - L::EXTRA * astep + w.xl + R * grp) * w.parts + k0;
    pstep = astep * w.parts;
#pragma unroll
    for (int r = 0; r < R; ++r) poff[r] = (dxs > 0 ? r : 1 - r) * w.parts;
  } else if constexpr (ORD) {
    static_assert(R == 2, "pairs of cells");
    const int wslot = c & (w.slots - 1);
    tpart = w.part + ((start - w.ya) * w.TX - L::EXTRA * astep + w.xl + R * grp) * w.parts + l8 * (4 / V);
    pstep = astep * w.parts;
#pragma unroll
    for (int r = 0; r < R; ++r)
      poff[r] = (((dxs > 0 ? r : 1 - r) * w.slots + wslot + grp) & (2 * w.slots - 1)) * (32 / V);
    second = V == 4 && w.slots == 2 && (c & 2);
  }
  const bool odd = part || w.xw + kStrCells > d.nx;    // a partial window, or the domain ends inside the strip

  // strips at an x side: which cells of a row lie outside (bits m), which of them upstream
  // (bits 8 + m: they hold psi^-), and which of the run's faces are on the domain boundary
  // (bits 16 + f: first order)
  [[maybe_unused]] uint32_t xbits = 0;
  if constexpr (EDGE) {
#pragma unroll
    for (int m = 0; m < NU; ++m) {
      const int g = gx0 + dxs * (m - H);
      if (g < 0 || g >= d.nx) xbits |= (1u << m) | ((g < 0) == (dxs > 0) ? 1u << (8 + m) : 0u);
    }
    if (!d.periodic_x) xbits |= (((xbits & 255u) | (xbits & 255u) >> 1) >> (H - 1)) << 16;   // face f: cells f + H - 1, f + H
  }

  // Row i of the chunk arrives in X; Y holds the row before it, which is completed
  // here (second order; first order completes the row itself). c: w-weighted sums of
  // the completed cells.
  [[maybe_unused]] float2 G[R][2];   // ordered form: y face values before the row that is completed next
  auto row = [&](const int i, const int in_slot, const bool done, StrRow& X, const StrRow& Y, float (&c)[R]) {
    const uint8_t* cur = ring_l + in_slot;
    float2 u[NU][2];
#pragma unroll
    for (int m = 0; m < NU; ++m) lds_vec2<T, 4>(reinterpret_cast<const T*>(cur + (m - H) * step_b), u[m]);
    [[maybe_unused]] bool face2 = true;   // the face between the row before and this one is second order
    if constexpr (EDGE) {
      const StrEdge& ed = *w.ed;
      const int p = start + dys * (i - H), ny = ed.ny;
      if (!ed.periodic_y) {
        const bool gy = p < 0 || p >= ny;
        face2 = gy == (p - dys < 0 || p - dys >= ny);
        if (gy) {
          // psi^- of the side for the rows before the domain; the row after it only meets a first-order face
          const float gv = (dys > 0 ? p < 0 : p >= ny) ? ed.ghost[dys > 0 ? 2 : 3] : 0.f;
#pragma unroll
          for (int m = 0; m < NU; ++m)
#pragma unroll
            for (int v = 0; v < 2; ++v) u[m][v] = make_float2(gv, gv);
        }
      }
      if (!ed.periodic_x) {
        // entering ordinates see psi^- of the side; leaving ones meet first-order faces only
        const float gup = ed.ghost[dxs > 0 ? 0 : 1];
#pragma unroll
        for (int m = 0; m < NU; ++m)
          if (xbits >> m & 1) {
            const float gv = (xbits >> (8 + m) & 1) ? gup : 0.f;
            u[m][0] = u[m][1] = make_float2(gv, gv);
          }
      } else if (p >= 0 && p < ny) {
        // periodic: the wrapped cell of the same row, from the input state
#pragma unroll
        for (int m = 0; m < NU; ++m)
          if (xbits >> m & 1)
            lds_vec2<T, 4>(reinterpret_cast<const T*>(d.psi[in_buf]) +
                               ((size_t)p * ed.nx + wrap_index(gx0 + dxs * (m - H), ed.nx)) * d.Mpad + k0, u[m]);
      }
    }
    float2 out[R][2];
    const StrRow& C = ORDER == 2 ? Y : X;   // the row completed
    if constexpr (ORD) {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        float2 D[NU], RD[NU], F[R + 1];   // F: face before cell f
#pragma unroll
        for (int m = 1; m < NU; ++m) {
          D[m] = sub2(u[m][v], u[m - 1][v]);
          RD[m] = relu2(D[m]);
        }
#pragma unroll
        for (int f = 0; f <= R; ++f) {
          float2 M = minmod2r(D[f + 2], D[f + 1], RD[f + 2], RD[f + 1]);
          if (EDGE && (xbits >> (16 + f) & 1)) M = make_float2(0.f, 0.f);   // domain faces are first order
          F[f] = __ffma2_rn(make_float2(0.5f, 0.5f), M, u[f + 1][v]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          X.z[r][v] = sub2(F[r + 1], F[r]);
          X.c[r][v] = u[r + H][v];
          X.d[r][v] = sub2(X.c[r][v], Y.c[r][v]);
          float2 M = minmod2r(X.d[r][v], Y.d[r][v], relu2(X.d[r][v]), relu2(Y.d[r][v]));
          if (EDGE && !face2) M = make_float2(0.f, 0.f);
          float2 up = Y.c[r][v];   // the face's upwind value; the general kernel walks +y whatever the flow
          if (FORM == STR_LANE && dys < 0) up = sub2(X.c[r][v], X.d[r][v]);
          const float2 g = __ffma2_rn(make_float2(0.5f, 0.5f), M, up);
          const float2 dg = sub2(g, G[r][v]);
          G[r][v] = g;
          out[r][v] = FORM == STR_UNI ? __ffma2_rn(ax2[v], Y.z[r][v], __fmul2_rn(ay2[v], dg))
                                      : __ffma2_rn(ay2[v], dg, __fmul2_rn(ax2[v], Y.z[r][v]));
        }
      }
    } else {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        // x: the flux terms of the row
        float2 D[NU];   // D[m] = u[m] - u[m-1]
        [[maybe_unused]] float2 M[R + 1];
#pragma unroll
        for (int m = 1; m < NU; ++m) D[m] = sub2(u[m][v], u[m - 1][v]);
        if constexpr (ORDER == 2) {
          float2 RD[NU];
#pragma unroll
          for (int m = 1; m < NU; ++m) RD[m] = relu2(D[m]);
#pragma unroll
          for (int f = 0; f <= R; ++f) M[f] = minmod2r(D[f + 2], D[f + 1], RD[f + 2], RD[f + 1]);   // face before cell f
          if constexpr (EDGE) {   // domain faces are first order
#pragma unroll
            for (int f = 0; f <= R; ++f)
              if (xbits >> (16 + f) & 1) M[f] = make_float2(0.f, 0.f);
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          float2 g = D[r + H];
          if constexpr (ORDER == 2) g = __ffma2_rn(make_float2(0.5f, 0.5f), sub2(M[r + 1], M[r]), g);
          float2 z = __fmul2_rn(ax2[v], g);
          // y: difference to the row before, half the limited difference at the face between them
          X.c[r][v] = u[r + H][v];
          X.d[r][v] = sub2(X.c[r][v], Y.c[r][v]);
          if constexpr (ORDER == 2) {
            float2 h = __fmul2_rn(make_float2(0.5f, 0.5f),
                                  minmod2r(X.d[r][v], Y.d[r][v], relu2(X.d[r][v]), relu2(Y.d[r][v])));
            if (EDGE && !face2) h = make_float2(0.f, 0.f);
            out[r][v] = __ffma2_rn(ay2[v], h, Y.z[r][v]);
            X.z[r][v] = __ffma2_rn(ay2[v], sub2(X.d[r][v], h), z);
          } else {
            out[r][v] = __ffma2_rn(ay2[v], X.d[r][v], z);
          }
        }
      }
    }
    if (done) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float2 ab = tab[dxs * r];
        [[maybe_unused]] float2 base[2];
        if constexpr (STAGE == STAGE_HEUN2)
          lds_vec2<T, 4>(reinterpret_cast<const T*>(cur + (r * step_b + L::halo_bytes - H * L::cell_bytes)), base);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          float2 t = __ffma2_rn(make_float2(ab.x, ab.x), C.c[r][v], make_float2(ab.y, ab.y));
          t = ORD ? sub2(t, out[r][v]) : __fadd2_rn(t, out[r][v]);
          // (the sum of the update first: psi^n and it are of one size, and their sum rounds at twice that)
          out[r][v] = STAGE == STAGE_HEUN2 ? __ffma2_rn(make_float2(0.5f, 0.5f), base[v], t) : t;
        }
      }
      if constexpr (sizeof(T) == 2) {
        const uint32_t gkey = sr_gkey(k0 >> 2, salt);   // the lane's group of 4 ordinates
        const int cell = (start + dys * (i - L::EXTRA)) * d.nx + gx0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const uint2 rb = sr_bits4((uint32_t)(cell + dxs * r), gkey);
          out[r][0] = Store<T>::round_sr2(out[r][0], rb.x);
          out[r][1] = Store<T>::round_sr2(out[r][1], rb.y);
        }
      }
      if (!odd) {
#pragma unroll
        for (int r = 0; r < R; ++r) stg_vec2<T, 4>(op + r * mstep, out[r]);
      } else {
        const int lo = ch.x + (ch.y & 255), hi = ch.x + (ch.y >> 8);
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (gx0 + dxs * r < d.nx) {
#pragma unroll
            for (int v = 0; v < 4; ++v)
              if (k0 + v >= lo && k0 + v < hi)
                Store<T>::store(op + r * mstep + v, (v & 1) ? out[r][v / 2].y : out[r][v / 2].x);
          }
      }
    }
    op += ostep;
    tab += astep;
    if constexpr (ORD) {
      if (done) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          float* p = tpart + poff[r];
          const float2 p0 = __fmul2_rn(w2[0], out[r][0]);
          if constexpr (V == 1) {
            const float2 p1 = __fmul2_rn(w2[1], out[r][1]);
            if (!part) {
              *reinterpret_cast<float4*>(p) = make_float4(p0.x, p0.y, p1.x, p1.y);
            } else {
              const int lo = ch.x + (ch.y & 255), hi = ch.x + (ch.y >> 8);
#pragma unroll
              for (int v = 0; v < 4; ++v)
                if (k0 + v >= lo && k0 + v < hi) p[v] = v == 0 ? p0.x : v == 1 ? p0.y : v == 2 ? p1.x : p1.y;
            }
          } else if constexpr (V == 4) {
            float t;
            if constexpr (FORM == STR_UNI) {
              const float2 pw = __ffma2_rn(w2[1], out[r][1], p0);
              t = pw.x + pw.y;
            } else {
              t = fmaf(w2[1].y, out[r][1].y, fmaf(w2[1].x, out[r][1].x, fmaf(w2[0].y, out[r][0].y, p0.x)));
            }
            *p = second ? *p + t : t;
          } else {
            const float2 p1 = __fmul2_rn(w2[1], out[r][1]);
            *reinterpret_cast<float2*>(p) =
                FORM == STR_UNI ? make_float2(p0.x + p0.y, p1.x + p1.y)
                                : make_float2(fmaf(w2[0].y, out[r][0].y, p0.x), fmaf(w2[1].y, out[r][1].y, p1.x));
          }
        }
      }
      tpart += pstep;
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float2 pw = __ffma2_rn(w2[1], out[r][1], __fmul2_rn(w2[0], out[r][0]));
        c[r] = pw.x + pw.y;
      }
    }
  };

  StrRow A, B;
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int v = 0; v < 2; ++v) B.c[r][v] = B.d[r][v] = B.z[r][v] = G[r][v] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int q = 0; q < npair; ++q) {
    if (NS > 2 && w.ahead == NS - 1) cp_async_wait<NS - 2>();
    else cp_async_wait<0>();
    __syncwarp();   // the rows have arrived for every lane, and every lane has read the pair before
    {
      // that pair's slot takes the load `ahead` pairs on (this chunk's, or the warp's next one's)
      const int tq = q + w.ahead;
      const int free_slot = slot == 0 ? w.ahead : slot - 1;
      const bool here = tq < npair;
      if (here || more)
        str_load<ORDER, STAGE, T, EDGE>(w, w.ring + free_slot * (2 * L::row_bytes), here ? ch.x : nkb, here ? dys : ndy,
                                  here ? tq : tq - npair);
      cp_async_commit();
    }
    const int in_slot = slot * (2 * L::row_bytes);
    if (++slot > w.ahead) slot = 0;
    const int i = 2 * q;
    const bool done0 = i >= L::EXTRA && i < n, done1 = i + 1 >= L::EXTRA && i + 1 < n;   // a row is completed
    float c0[R], c1[R];
    row(i, in_slot, done0, A, B, c0);
    row(i + 1, in_slot + L::row_bytes, done1, B, A, c1);
    if constexpr (ORD) continue;
    // phi of both completed rows, summed over the pair's 8 lanes: lanes 0, 1 end with the left cell of
    // the first row, 2, 3 with that of the second, 4 .. 7 with the right ones (a cell beyond a ragged
    // edge has an accumulator that nothing reads)
    const bool h4 = (lane & 4) != 0, h2 = (lane & 2) != 0, fwd = dxs > 0;
    const bool k4 = h4 == fwd;   // keeps cell 1 along the flow
    const float e0 = (k4 ? c0[1] : c0[0]) + __shfl_xor_sync(0xffffffffu, (fwd ? !h4 : h4) ? c0[1] : c0[0], 4);
    const float e1 = (k4 ? c1[1] : c1[0]) + __shfl_xor_sync(0xffffffffu, (fwd ? !h4 : h4) ? c1[1] : c1[0], 4);
    float s = (h2 ? e1 : e0) + __shfl_xor_sync(0xffffffffu, h2 ? e0 : e1, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if ((lane & 1) == 0 && (h2 ? done1 : done0)) *tacc += s;
    tacc += 2 * astep;
  }
}

// Barrier of the WC warps of strip wx (at most four strips; the ids are constants, so that
// a CTA reserves no more barriers than these).
__device__ __forceinline__ void str_strip_barrier(int wx, int WC) {
  const int threads = 32 * WC;
  if (wx == 0) asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
  else if (wx == 1) asm volatile("bar.sync 2, %0;" ::"r"(threads) : "memory");
  else if (wx == 2) asm volatile("bar.sync 3, %0;" ::"r"(threads) : "memory");
  else asm volatile("bar.sync 4, %0;" ::"r"(threads) : "memory");
}

// Ordered form: phi of the strip's cells from the lanes' terms of `n` windows, added to acc.
// A lane of the kernel whose order is kept holds V consecutive ordinates of a chunk of 32 V,
// and a warp's butterfly adds lanes 16 apart, then 8, 4, 2 and 1: the same tree here, windows
// first. The WC warps of the strip (this one is wc) share the cells.
template <int V>
__device__ __forceinline__ void str_phi_ordered(const StrWarp& w, int wc, int WC, int n) {
  const int lane = threadIdx.x & 31, l8 = lane & 7, grp = lane >> 3;
  const int mask = 2 * w.slots - 1;
#pragma unroll 2
  for (int i = wc; i < kStrRun * (w.yb - w.ya); i += WC) {
    const int phys = i & 1, pair = (i >> 1) * w.TX + w.xl + kStrRun * grp;
    const float* p = w.part + pair * w.parts + l8 * (4 / V);
    auto at = [&](int slot) { return p + ((phys * w.slots + slot + grp) & mask) * (32 / V); };
    float a = w.acc[pair + phys];
    if constexpr (V == 4) {
      float s = w.slots == 4 ? (*at(0) + *at(2)) + (*at(1) + *at(3)) : *at(0) + *at(1);
      s += __shfl_xor_sync(0xffffffffu, s, 4);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      a += s;
    } else {
      for (int k = 0; k < n; k += 2) {
        float2 s = __fadd2_rn(*reinterpret_cast<const float2*>(at(k)), *reinterpret_cast<const float2*>(at(k + 1)));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
          s = __fadd2_rn(s, make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o)));
        a += s.x + s.y;
      }
    }
    if (l8 == 0) w.acc[pair + phys] = a;
  }
}

// The same for one ordinate per lane: n ordinates, of which a lane here takes four in a row.
__device__ __forceinline__ void str_phi_ordered1(const StrWarp& w, int wc, int WC, int n) {
  const int lane = threadIdx.x & 31, l8 = lane & 7, grp = lane >> 3;
  for (int i = wc; i < kStrRun * (w.yb - w.ya); i += WC) {
    const int cell = (i >> 1) * w.TX + w.xl + kStrRun * grp + (i & 1);
    const float* p = w.part + cell * w.parts;
    float a = 0.f;
    for (int k = 4 * l8; k - 4 * l8 < n; k += 32) {
      float4 x = *reinterpret_cast<const float4*>(p + k);
      float2 s = make_float2(k < n ? x.x : 0.f, k + 1 < n ? x.y : 0.f), t = make_float2(k + 2 < n ? x.z : 0.f, k + 3 < n ? x.w : 0.f);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        s = __fadd2_rn(s, make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o)));
        t = __fadd2_rn(t, make_float2(__shfl_xor_sync(0xffffffffu, t.x, o), __shfl_xor_sync(0xffffffffu, t.y, o)));
      }
      s = __fadd2_rn(s, t);
      a += s.x + s.y;
    }
    if (l8 == 0) w.acc[cell] = a;
  }
}

// Ordered form: the chunks of a warp. The warps of a strip meet where their windows complete
// chunks of 32 V ordinates.
template <int STAGE, typename T, int FORM, int V>
__device__ __forceinline__ void str_chunks_ordered(const InstDesc& d, const StrWarp& w, int wx, int wc, int WC, bool active,
                                                   bool edge, int in_buf, T* __restrict__ psi_out, uint32_t salt) {
  const int n_chunks = d.n_chunks;
  [[maybe_unused]] const int per = max(V, WC);
  if (active) {
    int slot = 0;
#pragma unroll 1
    for (int c = wc; c < n_chunks; c += WC) {
      const int4 ch = d.str_chunks[c];
      if (edge) str_chunk<2, STAGE, T, true, FORM, V>(d, w, ch, c, c + WC, slot, in_buf, psi_out, salt);
      else str_chunk<2, STAGE, T, false, FORM, V>(d, w, ch, c, c + WC, slot, in_buf, psi_out, salt);
      [[maybe_unused]] const int next = c - wc + WC;   // first window of the strip's next round
      if constexpr (V > 1) {
        if (next % per == 0 && next < n_chunks) {
          str_strip_barrier(wx, WC);
          str_phi_ordered<V>(w, wc, WC, per);
          str_strip_barrier(wx, WC);
        }
      }
    }
    cp_async_wait<0>();
  }
  __syncthreads();
  if constexpr (V > 1) str_phi_ordered<V>(w, wc, WC, n_chunks - (n_chunks - 1) / per * per);
  else str_phi_ordered1(w, wc, WC, d.M);
  __syncthreads();
}

// Boundary outflow of a tile's output state (first-order traces: what leaves through a
// side of the domain less what enters with psi^-), from the stored state: a warp takes a
// cell, its lanes the ordinates.
template <typename T>
__device__ __noinline__ float str_boundary(const InstDesc& d, const T* psi, int x0, int x1, int ya, int yb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float bacc = 0.f;
#pragma unroll 1
  for (int side = 0; side < 4; ++side) {
    const bool xs = side < 2, low = (side & 1) == 0;
    if (xs ? d.periodic_x : d.periodic_y) continue;
    if (xs ? (low ? x0 > 0 : x1 < d.nx) : (low ? ya > 0 : yb < d.ny)) continue;
    const int cnt = xs ? yb - ya : x1 - x0;
    const float len = (float)(xs ? d.dy_d : d.dx_d), gh = d.ghost[side];
    const float* dir = xs ? d.xi : d.eta;
#pragma unroll 1
    for (int i = warp; i < cnt; i += kStrWarps) {
      const int gx = xs ? (low ? 0 : d.nx - 1) : x0 + i, gy = xs ? ya + i : (low ? 0 : d.ny - 1);
      const T* cell = psi + ((size_t)gy * d.nx + gx) * d.Mpad;
      for (int k = lane; k < d.Mpad; k += 32) {
        const float on = low ? -dir[k] : dir[k];
        float o;
        if constexpr (sizeof(T) == 2) o = __bfloat162float(__ldcg(cell + k));
        else o = __ldcg(cell + k);
        bacc += len * (d.w[k] * on * (on > 0.f ? o : (on < 0.f ? gh : 0.f)));
      }
    }
  }
  return bacc;
}

template <int ORDER, int STAGE, typename T, int FORM>
__global__ void __launch_bounds__(kStrThreads, 2)
    cart_stream_kernel(const InstDesc* __restrict__ descs, const WorkItem* __restrict__ items) {
  using L = StrCfg<ORDER, STAGE, T>;
  constexpr bool ORD = FORM != STR_DIFF;
  const WorkItem it = items[blockIdx.x];
  const InstDesc& d = descs[it.inst];
  InstState* st = d.st;
  grid_wait();
  const StepHead head = step_head(st);
  // finished or failed instances are masked
  if (head.step >= d.n_steps || head.status != DEV_OK) return;
  if (d.drop_load >= 0) {
    // test hook: a load that never arrives. Nothing here waits on a barrier that a load
    // completes, so the launch gives up at once instead of after the wait limit.
    if (threadIdx.x == 0) atomicCAS(&st->status, DEV_OK, DEV_TIMEOUT);
    return;
  }
  extern __shared__ __align__(128) uint8_t smem_raw[];
  __shared__ StrEdge s_edge;
  uint8_t* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int TX = d.tx, tx_shift = 31 - __clz(TX), WX = TX / kStrCells, WC = kStrWarps / WX;
  const int wx = warp & (WX - 1), wc = warp / WX;
  const int parity = (STAGE == STAGE_EULER) ? head.parity : 0;
  const uint32_t salt = sr_salt(head.step, STAGE);   // BF16 stochastic rounding
  const int in_buf = (STAGE == STAGE_EULER) ? parity : (STAGE == STAGE_HEUN1 ? 0 : 1);
  const int out_buf = (STAGE == STAGE_EULER) ? (1 - parity) : (STAGE == STAGE_HEUN1 ? 1 : 0);
  const float* __restrict__ phi_in = d.phi[in_buf];
  T* __restrict__ psi_out = reinterpret_cast<T*>(d.psi[out_buf]);
  const int nx = d.nx, ny = d.ny;
  const int x0 = it.a * TX, ya = it.b * d.ly, yb = min(ny, ya + d.ly), nrows = yb - ya;

  float2* tile_ab = reinterpret_cast<float2*>(smem + L::ring_bytes);
  float* tile_acc = reinterpret_cast<float*>(tile_ab + d.ly * TX);   // [WC][ly][TX]; ordered form [ly][TX]
  const int parts = ORD ? d.ord_parts : 0;
  double* red = reinterpret_cast<double*>(smem + L::ring_bytes + str_tile_bytes(TX, d.ly, parts));

  StrWarp w;
  w.ring_p = smem + warp * (L::NS * 2 * L::row_bytes);
  w.ring = smem_u32(w.ring_p);
  w.ab = tile_ab;
  w.acc = tile_acc + (ORD ? 0 : wc * d.ly * TX);
  w.part = tile_acc + d.ly * TX;
  w.parts = parts;
  w.slots = ORD ? parts * d.ord_vec / 32 : 0;
  w.ed = &s_edge;
  w.xl = wx * kStrCells;
  w.xw = x0 + w.xl;
  w.ya = ya;
  w.yb = yb;
  w.TX = TX;
  // rows 2q, 2q + 1 reach from H rows before the segment to at most two after it
  const bool edge = (w.xw - L::H < 0) || (w.xw + kStrCells + L::H > nx) || (ya - 2 < 0) || (yb + 2 > ny);
  w.ahead = min(L::NS - 1, (nrows + L::EXTRA + 1) / 2);
  const int64_t cell_b = (int64_t)d.Mpad * (int)sizeof(T);
  w.row_bytes = nx * cell_b;
  w.col_bytes = (int)(L::per_copy * cell_b);
  w.src = reinterpret_cast<const uint8_t*>(d.psi[in_buf]) + (w.xw - L::H + lane / L::pieces) * cell_b + 16 * (lane % L::pieces);
  w.to_base = reinterpret_cast<const uint8_t*>(d.psi[0]) - reinterpret_cast<const uint8_t*>(d.psi[in_buf]) + L::H * cell_b;
  const bool active = w.xw < nx && wc < d.n_chunks;
  if (tid == 0) {
    s_edge.nx = nx;
    s_edge.ny = ny;
    s_edge.periodic_x = d.periodic_x;
    s_edge.periodic_y = d.periodic_y;
    for (int s = 0; s < 4; ++s) s_edge.ghost[s] = d.ghost[s];
  }
  __syncthreads();

  if (active) {
    const int4 ch = d.str_chunks[wc];
#pragma unroll 1
    for (int s = 0; s < w.ahead; ++s) {
      if (edge) str_load<ORDER, STAGE, T, true>(w, w.ring + s * (2 * L::row_bytes), ch.x, ch.z, s);
      else str_load<ORDER, STAGE, T, false>(w, w.ring + s * (2 * L::row_bytes), ch.x, ch.z, s);
      cp_async_commit();
    }
  }
  // per-cell constants of the tile: a = 1 - dt sigma_t, b = dt (sigma_s/(2 pi) phi + Q)
  const float dt = d.dt, half = STAGE == STAGE_HEUN2 ? 0.5f : 1.f;
  for (int i = tid; i < nrows * TX; i += kStrThreads) {
    const int gx = x0 + (i & (TX - 1));
    float a = 1.f, b = 0.f;
    if (gx < nx) {
      const size_t cell = (size_t)(ya + (i >> tx_shift)) * nx + gx;
      const int m = d.mat[cell];
      a = 1.f - dt * d.sig_t[m];
      b = dt * (d.sig_s2pi[m] * phi_in[cell] + d.q_src[m]);
    }
    tile_ab[i] = make_float2(half * a, half * b);
  }
  for (int i = tid; i < (ORD ? 1 : WC) * d.ly * TX; i += kStrThreads) tile_acc[i] = 0.f;
  __syncthreads();

  const int n_chunks = d.n_chunks;
  if constexpr (ORD) {
    if (d.ord_vec == 4) str_chunks_ordered<STAGE, T, FORM, 4>(d, w, wx, wc, WC, active, edge, in_buf, psi_out, salt);
    else if (d.ord_vec == 2) str_chunks_ordered<STAGE, T, FORM, 2>(d, w, wx, wc, WC, active, edge, in_buf, psi_out, salt);
    else if constexpr (FORM == STR_LANE) str_chunks_ordered<STAGE, T, FORM, 1>(d, w, wx, wc, WC, active, edge, in_buf, psi_out, salt);
  } else {
    if (active) {
      int slot = 0;
#pragma unroll 1
      for (int c = wc; c < n_chunks; c += WC) {
        const int4 ch = d.str_chunks[c];
        if (edge) str_chunk<ORDER, STAGE, T, true, STR_DIFF, 4>(d, w, ch, c, c + WC, slot, in_buf, psi_out, salt);
        else str_chunk<ORDER, STAGE, T, false, STR_DIFF, 4>(d, w, ch, c, c + WC, slot, in_buf, psi_out, salt);
      }
      cp_async_wait<0>();
    }
    __syncthreads();
    // phi of a cell: its chunk groups in order
    for (int i = tid; i < nrows * TX; i += kStrThreads) {
      float s = tile_acc[i];
      for (int g = 1; g < WC; ++g) s += tile_acc[g * d.ly * TX + i];
      tile_acc[i] = s;   // read back by the same thread only
    }
  }
  const int x1 = min(nx, x0 + TX);
  float bacc = 0.f;
  if (x0 == 0 || x1 == nx || ya == 0 || yb == ny) bacc = str_boundary<T>(d, psi_out, x0, x1, ya, yb);
  cart_epilogue<STAGE, kStrThreads>(d, it, d.phi[out_buf], tile_acc, red, reinterpret_cast<float*>(smem),
                                    L::ring_bytes / 4, x0, ya, nrows, TX, bacc);
}

template <int ORDER, int STAGE, typename T, int FORM>
static cudaError_t str_prepare_one(int tx, int ly, int form) {
  // The dynamic shared-memory limit belongs to the current device and the kernel;
  // it is only ever raised (atomics: host threads may race here, harmlessly).
  constexpr int kDev = 64;
  static std::atomic<size_t> s_limit[kDev];
  const size_t smem = str_smem_for<ORDER, STAGE, T>(tx, ly, form);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool tracked = dev >= 0 && dev < kDev;
  if (tracked && smem <= s_limit[dev].load(std::memory_order_acquire)) return cudaSuccess;
  e = cudaFuncSetAttribute(cart_stream_kernel<ORDER, STAGE, T, FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (tracked) {
    size_t cur = s_limit[dev].load(std::memory_order_relaxed);
    while (cur < smem && !s_limit[dev].compare_exchange_weak(cur, smem, std::memory_order_release)) {
    }
  }
  return cudaSuccess;
}

template <int ORDER, int STAGE, typename T, int FORM>
static cudaError_t str_launch_one(const InstDesc* d, const WorkItem* items, int n, int tx, int ly, int form, cudaStream_t s,
                                  bool chained) {
  cudaError_t e = str_prepare_one<ORDER, STAGE, T, FORM>(tx, ly, form);
  if (e != cudaSuccess) return e;
  return launch_stage_kernel(cart_stream_kernel<ORDER, STAGE, T, FORM>, n, kStrThreads,
                             str_smem_for<ORDER, STAGE, T>(tx, ly, form), s, chained, d, items);
}

// Calls FN<..., FORM>(args) for the kernel of `form` (the ordered form: second order only).
#define RTK_STR_FORM(FN, ...)                                                     \
  if (form == STREAM_PLAIN) return FN<ORDER, STAGE, T, STR_DIFF>(__VA_ARGS__);    \
  if constexpr (ORDER == 2) {                                                     \
    if (form & STREAM_UNI) return FN<ORDER, STAGE, T, STR_UNI>(__VA_ARGS__);      \
    return FN<ORDER, STAGE, T, STR_LANE>(__VA_ARGS__);                            \
  }                                                                               \
  return cudaErrorInvalidValue;
template <int ORDER, int STAGE, typename T>
static cudaError_t str_prepare(int tx, int ly, int form) {
  RTK_STR_FORM(str_prepare_one, tx, ly, form)
}
template <int ORDER, int STAGE, typename T>
static cudaError_t str_launch(const InstDesc* d, const WorkItem* items, int n, int tx, int ly, int form, cudaStream_t s,
                              bool chained) {
  RTK_STR_FORM(str_launch_one, d, items, n, tx, ly, form, s, chained)
}
#undef RTK_STR_FORM

// One translation unit per (order, storage type): the three stages.
#define RTK_STR_UNIT(NAME, ORDER, TT)                                                                         \
  cudaError_t str_prepare_##NAME(int stage, int tx, int ly, int form) {                                       \
    if (stage == STAGE_EULER) return str_prepare<ORDER, STAGE_EULER, TT>(tx, ly, form);                       \
    if (stage == STAGE_HEUN1) return str_prepare<ORDER, STAGE_HEUN1, TT>(tx, ly, form);                       \
    return str_prepare<ORDER, STAGE_HEUN2, TT>(tx, ly, form);                                                 \
  }                                                                                                           \
  size_t str_smem_##NAME(int stage, int tx, int ly, int form) {                                               \
    return stage == STAGE_HEUN2 ? str_smem_for<ORDER, STAGE_HEUN2, TT>(tx, ly, form)                          \
                                : str_smem_for<ORDER, STAGE_EULER, TT>(tx, ly, form);                         \
  }                                                                                                           \
  cudaError_t str_launch_##NAME(const InstDesc* d, const WorkItem* items, int n, int stage, int tx, int ly,   \
                                int form, cudaStream_t s, bool chained) {                                     \
    if (stage == STAGE_EULER) return str_launch<ORDER, STAGE_EULER, TT>(d, items, n, tx, ly, form, s, chained); \
    if (stage == STAGE_HEUN1) return str_launch<ORDER, STAGE_HEUN1, TT>(d, items, n, tx, ly, form, s, chained); \
    return str_launch<ORDER, STAGE_HEUN2, TT>(d, items, n, tx, ly, form, s, chained);                         \
  }

}  // namespace rtk
