// Staged first-order stage kernel on triangle meshes (Sec. 4.2 on triangles,
// Eq. upwind1stOrder and Eq. sn_2d_eqn_fv; Euler or either Heun stage).
//
// The arithmetic per cell and ordinate is that of tri_stage_kernel: with the edge
// normals of a cell summing to zero, the upwind flux sum over the edges is
// sum_e min((omega_k . n_e) l_e / A_i, 0) (psi_e - psi_i) (psi_e the neighbour's
// value or the side's psi^-; edges that the ordinate leaves through contribute
// nothing); then the Euler or Heun update, phi_out = sum_k w_k out_k and the FP64 QoI
// partials.
//
// What differs is how the rows arrive. Cells are stored in the Morton order of
// their centroids, so a chunk of 32 consecutive cells is a compact patch whose
// edges lead to about 23 other cells (at most 32 on the jittered split
// meshes): its halo, listed per chunk on the host. For each block of W = 32 VEC
// ordinates the CTA copies the block's segment of every row the chunk needs, its own
// rows, its halo rows and, in Heun stage 2, the rows of psi^n, into shared memory
// (16-byte asynchronous copies, one row per warp instruction at 4 ordinates per lane)
// while it computes the block before from the other buffer. Each row is read
// from L2/DRAM about 1.7 times per chunk instead of 4 (a cell's own row plus
// three gathers by its neighbours). The chunk metadata (neighbour ids, edge
// geometry, neighbour slots in the staged rows, the halo list) arrives by bulk
// copies three chunks ahead, and the last warp turns it into a table of the cells'
// constants during the chunk before.
//
// Persistent: CTA g of G takes chunks g, g + G, ... (two CTAs of 8 warps per
// SM); warp w owns cells w, w + 8, .. of a chunk and keeps their phi
// and outflow partial sums in registers across the blocks. One barrier per block.
// Chunks without boundary edges, nearly all, run a body without their tests. Every
// wait on a barrier is bounded; one that runs out stops the whole CTA at the next
// block's end, drains the copies in flight and reports RT_ETIMEOUT.
//
// Bound by issue slots and fixed latencies at 16 warps per SM (256 instructions per
// cell of 256 ordinates, 44 % of the slots; DRAM 8.1 bytes per cell and ordinate at
// half of its peak). 1300^2 x 256 first-order Euler, FP32: with selects between the
// traces, two barriers per block, one thread's QoI sums per cell and per-row bulk copies
// (which a warp issues lane by lane) 2.28 ms; now 1.70. 650^2 x 256 BF16 0.61 -> 0.42.
#include <cuda_bf16.h>

#include <type_traits>

#include "device_common.cuh"

namespace rtk {

namespace {

constexpr int kStgThreads = 256;
constexpr int kStgWarps = kStgThreads / 32;
constexpr int kStgChunk = kTriStgChunk;   // cells per chunk (32)
constexpr int kStgCellsPerWarp = kStgChunk / kStgWarps;
constexpr int kStgMeta = 4;   // metadata buffers: chunks i .. i+3
constexpr int kStgTab = 16;   // cell table entries: n.l/A x and y per edge, -sigma_t, source, offsets
                              // of the neighbours' staged rows, boundary flags, area, area sigma_a, QoI region

__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void stg_copy16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void stg_copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename T, int VEC>
__device__ __forceinline__ void ld_row(const T* p, float (&out)[VEC]) {
  if constexpr (sizeof(T) == 4) {
    if constexpr (VEC == 4) {
      const float4 x = *reinterpret_cast<const float4*>(p);
      out[0] = x.x; out[1] = x.y; out[2] = x.z; out[3] = x.w;
    } else if constexpr (VEC == 2) {
      const float2 x = *reinterpret_cast<const float2*>(p);
      out[0] = x.x; out[1] = x.y;
    } else {
      out[0] = *reinterpret_cast<const float*>(p);
    }
  } else {
    if constexpr (VEC == 4) {
      const uint2 x = *reinterpret_cast<const uint2*>(p);
      out[0] = __uint_as_float(x.x << 16); out[1] = __uint_as_float(x.x & 0xffff0000u);
      out[2] = __uint_as_float(x.y << 16); out[3] = __uint_as_float(x.y & 0xffff0000u);
    } else if constexpr (VEC == 2) {
      const uint32_t x = *reinterpret_cast<const uint32_t*>(p);
      out[0] = __uint_as_float(x << 16); out[1] = __uint_as_float(x & 0xffff0000u);
    } else {
      out[0] = __bfloat162float(*p);
    }
  }
}

template <typename T, int VEC>
__device__ __forceinline__ void st_row(T* p, const float (&in)[VEC]) {
  if constexpr (sizeof(T) == 4) {
    if constexpr (VEC == 4) {
      *reinterpret_cast<float4*>(p) = make_float4(in[0], in[1], in[2], in[3]);
    } else if constexpr (VEC == 2) {
      *reinterpret_cast<float2*>(p) = make_float2(in[0], in[1]);
    } else {
      *reinterpret_cast<float*>(p) = in[0];
    }
  } else {
    if constexpr (VEC == 4) {
      __nv_bfloat162 a = __floats2bfloat162_rn(in[0], in[1]);
      __nv_bfloat162 b = __floats2bfloat162_rn(in[2], in[3]);
      uint2 x;
      x.x = *reinterpret_cast<uint32_t*>(&a);
      x.y = *reinterpret_cast<uint32_t*>(&b);
      *reinterpret_cast<uint2*>(p) = x;
    } else if constexpr (VEC == 2) {
      *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(in[0], in[1]);
    } else {
      *p = __float2bfloat16_rn(in[0]);
    }
  }
}

}  // namespace

// Shared-memory layout of the staged kernel: two row buffers of `rows` rows of
// W values (the chunk's own rows, hmax halo rows, and in Heun stage 2 the rows of
// psi^n), then kStgMeta metadata buffers (neighbour records, edge geometry, neighbour
// slots, halo ids), two cell tables, the mbarriers and counters.
struct StgLayout {
  size_t row_bytes, rows, buf_bytes, meta_bytes, total;
  int hmax;
};

__host__ __device__ inline StgLayout stg_layout(int vec, int es, int hmax, bool base) {
  StgLayout L;
  L.hmax = hmax;
  L.row_bytes = (size_t)32 * vec * es;
  L.rows = (size_t)kStgChunk + hmax + (base ? kStgChunk : 0);
  L.buf_bytes = (L.rows * L.row_bytes + 127) / 128 * 128;
  L.meta_bytes = ((size_t)kStgChunk * 16 + 2 * kStgChunk * 16 + kStgChunk * 4 + (size_t)hmax * 4 + 127) / 128 * 128;
  // + two cell tables, control, slack
  L.total = 2 * L.buf_bytes + kStgMeta * L.meta_bytes + 2 * kStgChunk * kStgTab * 4 + 128 + 128;
  return L;
}

template <int VEC, int STAGE, typename T>
__global__ void __launch_bounds__(kStgThreads, 2)
    tri_staged_kernel(const InstDesc* __restrict__ descs, const WorkItem* __restrict__ items) {
  __shared__ double red[2 * NQ];
  __shared__ float facc[NQ][kStgChunk];
  __shared__ double dacc[kStgWarps][NQ];
  __shared__ int plain_chunk[2];
  extern __shared__ __align__(128) uint8_t stg_raw[];
  const WorkItem it = items[blockIdx.x];
  const InstDesc& d = descs[it.inst];
  InstState* st = d.st;

  constexpr int W = 32 * VEC;
  constexpr bool kBase = STAGE == STAGE_HEUN2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float* __restrict__ d_xi = d.xi;
  const float* __restrict__ d_eta = d.eta;
  const float* __restrict__ d_w = d.w;
  const int Mpad = d.Mpad;
  const int nb = Mpad / W;
  const float dt = d.dt;
  const int nreg = d.n_regions, nq = nreg + 2;
  const int n_cells = (int)d.n_cells;
  const int n_chunks = (n_cells + kStgChunk - 1) / kStgChunk;
  const int G = it.b;
  const int64_t limit = d.wait_limit;
  const StgLayout L = stg_layout(VEC, (int)sizeof(T), d.tri_hmax, kBase);
  const int base_row = kStgChunk + L.hmax;

  uint8_t* smem = stg_raw + ((128u - (smem_u32(stg_raw) & 127u)) & 127u);
  uint8_t* rowbuf[2] = {smem, smem + L.buf_bytes};
  uint8_t* meta0 = smem + 2 * L.buf_bytes;
  float* tabs = reinterpret_cast<float*>(meta0 + kStgMeta * L.meta_bytes);   // [2][kStgChunk][kStgTab]
  uint64_t* meta_bar = reinterpret_cast<uint64_t*>(tabs + 2 * kStgChunk * kStgTab);   // [kStgMeta]
  int* ctl = reinterpret_cast<int*>(meta_bar + kStgMeta);
  int* s_hcount = ctl;                  // [kStgMeta] halo rows of the chunk in each metadata buffer
  int* s_meta_last = ctl + kStgMeta;    // [kStgMeta] last chunk ordinal issued into each, -1 none

  auto metabuf = [&](int mb) { return meta0 + (size_t)mb * L.meta_bytes; };
  auto meta_nbr = [&](int mb) { return reinterpret_cast<const int4*>(metabuf(mb)); };
  auto meta_geo = [&](int mb) { return reinterpret_cast<const float4*>(metabuf(mb) + kStgChunk * 16); };
  auto meta_lidx = [&](int mb) { return reinterpret_cast<const uint32_t*>(metabuf(mb) + 3 * kStgChunk * 16); };
  auto meta_halo = [&](int mb) {
    return reinterpret_cast<const int32_t*>(metabuf(mb) + 3 * kStgChunk * 16 + kStgChunk * 4);
  };
  const int n_my = (it.a < n_chunks) ? (n_chunks - 1 - it.a) / G + 1 : 0;
  const int J = n_my * nb;

  // metadata of chunk ordinal i into buffer i % kStgMeta (thread 0)
  auto issue_meta = [&](int i) {
    const int mb = i % kStgMeta;
    const int k = it.a + i * G;
    const int c0 = k * kStgChunk;
    const int cells = min(kStgChunk, n_cells - c0);
    const int2 oc = d.tri_halo_oc[k];
    const int hpad = (oc.y + 3) & ~3;
    s_hcount[mb] = oc.y;
    s_meta_last[mb] = i;
    uint8_t* m = metabuf(mb);
    mbar_arrive_expect_tx(&meta_bar[mb], (uint32_t)(cells * 48 + kStgChunk * 4 + hpad * 4));
    bulk_copy(m, d.tri_nbr + c0, (uint32_t)cells * 16u, &meta_bar[mb]);
    bulk_copy(m + kStgChunk * 16, d.tri_geo + 2 * (size_t)c0, (uint32_t)cells * 32u, &meta_bar[mb]);
    bulk_copy(m + 3 * kStgChunk * 16, d.tri_lidx + (size_t)k * kStgChunk, kStgChunk * 4u, &meta_bar[mb]);
    if (hpad > 0) bulk_copy(m + 3 * kStgChunk * 16 + kStgChunk * 4, d.tri_halo + oc.x, (uint32_t)hpad * 4u, &meta_bar[mb]);
  };

  if (threadIdx.x < kStgChunk)
    for (int q = 0; q < nq; ++q) facc[q][threadIdx.x] = 0.f;
  if (lane < NQ) dacc[warp][lane] = 0.0;
  if (threadIdx.x == 0) {
    for (int q = 0; q < kStgMeta; ++q) {
      mbar_init(&meta_bar[q], 1);
      s_meta_last[q] = -1;
    }
    fence_barrier_init();
    for (int i = 0; i < min(n_my, kStgMeta - 1); ++i) issue_meta(i);
  }
  grid_wait();
  const StepHead head = step_head(st);
  if (head.step >= d.n_steps || head.status != DEV_OK) {
    // finished or failed instances are masked; no copy may be in flight when the block leaves
    if (threadIdx.x == 0)
      for (int i = 0; i < min(n_my, kStgMeta - 1); ++i) mbar_wait_bounded(&meta_bar[i], 0u, kDrainCycles);
    return;
  }
  const int parity = (STAGE == STAGE_EULER) ? head.parity : 0;
  [[maybe_unused]] const uint32_t salt = sr_salt(head.step, STAGE);   // BF16 stochastic rounding
  const int in_buf = (STAGE == STAGE_EULER) ? parity : (STAGE == STAGE_HEUN1 ? 0 : 1);
  const int out_buf = (STAGE == STAGE_EULER) ? (1 - parity) : (STAGE == STAGE_HEUN1 ? 1 : 0);
  const T* __restrict__ psi_in = reinterpret_cast<const T*>(d.psi[in_buf]);
  const T* __restrict__ psi_base = reinterpret_cast<const T*>(d.psi[0]);
  T* __restrict__ psi_out = reinterpret_cast<T*>(d.psi[out_buf]);
  const float* __restrict__ phi_in = d.phi[in_buf];
  float* __restrict__ phi_out = d.phi[out_buf];
  const int64_t to_base = psi_base - psi_in;
  __syncthreads();

  // Start the copies of block bb of chunk ordinal ii (whose metadata must have arrived: false
  // if waiting for it ran out) into row buffer rb, 16 bytes per lane: a warp takes rows
  // warp * RPI .. + RPI - 1 and every kStgWarps * RPI-th group after them.
  constexpr int kPieces = W * (int)sizeof(T) / 16;   // 16-byte pieces of a row
  constexpr int RPI = 32 / kPieces;                  // rows per copy instruction of a warp
  const int r_lane = warp * RPI + lane / kPieces, p_lane = lane % kPieces;
  auto issue_rows = [&](int ii, int bb, int rb) -> bool {
    const int mb = ii % kStgMeta;
    const bool mok = mbar_wait_bounded(&meta_bar[mb], (uint32_t)((ii / kStgMeta) & 1), limit);
    if (!__all_sync(0xffffffffu, mok)) return false;
    const int c0 = (it.a + ii * G) * kStgChunk;
    const int cells = min(kStgChunk, n_cells - c0);
    const int H = s_hcount[mb];
    const int32_t* halo = meta_halo(mb);
    const T* col = psi_in + bb * W + p_lane * (16 / (int)sizeof(T));
    const uint32_t dst = smem_u32(rowbuf[rb]) + 16 * p_lane;
    const uint32_t rbytes = (uint32_t)L.row_bytes;
    for (int r = r_lane; r < cells; r += kStgWarps * RPI) {
      const T* s = col + (size_t)(c0 + r) * Mpad;
      stg_copy16(dst + r * rbytes, s);
      if constexpr (kBase) stg_copy16(dst + (base_row + r) * rbytes, s + to_base);
    }
    for (int r = r_lane; r < H; r += kStgWarps * RPI)
      stg_copy16(dst + (kStgChunk + r) * rbytes, col + (size_t)halo[r] * Mpad);
    return true;
  };

  // add a warp's FP32 QoI sums (its cells of a chunk) to its FP64 ones
  auto flush = [&]() {
    __syncwarp();
    for (int q = 0; q < nq; ++q) {
      const int li = warp + (lane & 3) * kStgWarps;
      double s = (double)facc[q][li];
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      if (lane < 4) facc[q][li] = 0.f;
      if (lane == 0) dacc[warp][q] += s;
    }
    __syncwarp();
  };
  // Cell table of chunk ordinal i, lane l of the last warp for cell l: what a cell needs
  // besides its rows. Built while the chunk before it is computed, in two halves, so that
  // the load of phi has that long.
  float src_next = 0.f;
  auto table_load = [&](int i) {
    const int c0 = (it.a + i * G) * kStgChunk;
    if (c0 + lane < n_cells) {
      const int m = meta_nbr(i % kStgMeta)[lane].w & 255;
      src_next = d.sig_s2pi[m] * phi_in[c0 + lane] + d.q_src[m];
    }
  };
  auto table_store = [&](int i) {
    const int mb = i % kStgMeta, c0 = (it.a + i * G) * kStgChunk;
    uint32_t flags = 1u;   // (a missing cell makes the chunk not plain)
    if (c0 + lane < n_cells) {
      const int4 nb4 = meta_nbr(mb)[lane];
      const float4 g0 = meta_geo(mb)[2 * lane], g1 = meta_geo(mb)[2 * lane + 1];
      const uint32_t lx = meta_lidx(mb)[lane];
      float* t = tabs + ((i & 1) * kStgChunk + lane) * kStgTab;
      t[0] = g0.x; t[1] = g0.z; t[2] = g1.x;   // x components of (n.l)/A for edges 0, 1, 2
      t[3] = g0.y; t[4] = g0.w; t[5] = g1.y;   // y components
      t[6] = -d.sig_t[nb4.w & 255];
      t[7] = src_next;
      flags = 0;
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const uint32_t slot = (lx >> (8 * e)) & 255u;   // 255: a boundary edge (reads the cell's own row, unused)
        if (slot == 255u) flags |= 1u << e;
        t[8 + e] = __uint_as_float((slot == 255u ? (uint32_t)lane : slot) * (uint32_t)L.row_bytes);
      }
      t[11] = __uint_as_float(flags);
      t[12] = g1.z;
      t[13] = g1.z * d.sig_a_f[nb4.w & 255];
      t[14] = __uint_as_float((uint32_t)(nb4.w >> 8) & 255u);
    }
    const bool any = __any_sync(0xffffffffu, flags != 0);
    if (lane == 0) plain_chunk[i & 1] = any ? 0 : 1;
  };
  // the first block; afterwards block j + 1 is loaded while block j is computed
  bool iok = J > 0 ? issue_rows(0, 0, 0) : true;
  if (J > 0 && warp == kStgWarps - 1 && iok) {
    table_load(0);
    table_store(0);
  }
  stg_copy_wait();
  bool stop = __syncthreads_or(!iok);

  bool ok = true;
  float phi_part[kStgCellsPerWarp], bpart[kStgCellsPerWarp];
  int j = 0;
  for (int i = 0, b = 0; j < J; ++j) {
    if (stop) {
      ok = false;
      break;
    }
    const int mb = i % kStgMeta, rb = j & 1;
    const bool chunk_end = b == nb - 1;
    // the next block's rows, and the next chunk's table, while this block is computed; a wait
    // that runs out stops all warps after the block
    const bool go = j + 1 < J ? issue_rows(chunk_end ? i + 1 : i, chunk_end ? 0 : b + 1, rb ^ 1) : true;
    const bool next_tab = warp == kStgWarps - 1 && chunk_end && i + 1 < n_my;
    if (next_tab && go) table_load(i + 1);
    const int k = it.a + i * G;
    const int c0 = k * kStgChunk;
    const int cells = min(kStgChunk, n_cells - c0);
    const float* tab = tabs + (i & 1) * kStgChunk * kStgTab;
    if (b == 0) {
#pragma unroll
      for (int q = 0; q < kStgCellsPerWarp; ++q) {
        phi_part[q] = 0.f;
        bpart[q] = 0.f;
      }
    }
    const uint8_t* rows = rowbuf[rb] + lane * (VEC * (int)sizeof(T));
    const int kk = b * W + lane * VEC;
    float xi[VEC], eta[VEC], w[VEC];
    ld_row<float, VEC>(d_xi + kk, xi);
    ld_row<float, VEC>(d_eta + kk, eta);
    ld_row<float, VEC>(d_w + kk, w);
    T* out_row = psi_out + (size_t)(c0 + warp) * Mpad + kk;
    // PLAIN: a whole chunk without boundary edges (all but a few)
    auto cells_of_warp = [&](auto plain) {
      constexpr bool PLAIN = decltype(plain)::value;
#pragma unroll
      for (int q = 0; q < kStgCellsPerWarp; ++q, out_row += (size_t)kStgWarps * Mpad) {
        const int li = warp + q * kStgWarps;
        if (!PLAIN && li >= cells) break;
        const float4 t0 = *reinterpret_cast<const float4*>(tab + li * kStgTab);
        const float4 t1 = *reinterpret_cast<const float4*>(tab + li * kStgTab + 4);
        const uint4 t2 = *reinterpret_cast<const uint4*>(tab + li * kStgTab + 8);
        const float ax[3] = {t0.x, t0.y, t0.z};
        const float ay[3] = {t0.w, t1.x, t1.y};
        float c[VEC], nbv[3][VEC];
        [[maybe_unused]] float base[VEC];
        ld_row<T, VEC>(reinterpret_cast<const T*>(rows + (uint32_t)li * (uint32_t)L.row_bytes), c);
        ld_row<T, VEC>(reinterpret_cast<const T*>(rows + t2.x), nbv[0]);
        ld_row<T, VEC>(reinterpret_cast<const T*>(rows + t2.y), nbv[1]);
        ld_row<T, VEC>(reinterpret_cast<const T*>(rows + t2.z), nbv[2]);
        if constexpr (kBase) ld_row<T, VEC>(reinterpret_cast<const T*>(rows + (uint32_t)(base_row + li) * (uint32_t)L.row_bytes), base);
        if (!PLAIN && t2.w) {
          // boundary edges: psi^- of the side
          const int4 nb4 = meta_nbr(mb)[li];
          const int nbr[3] = {nb4.x, nb4.y, nb4.z};
#pragma unroll
          for (int e = 0; e < 3; ++e)
            if (t2.w >> e & 1) {
              const float gh = d.ghost[-1 - nbr[e]];
#pragma unroll
              for (int l = 0; l < VEC; ++l) nbv[e][l] = gh;
            }
        }
        // BF16 rounding bits of the lane's ordinates kk .. kk+VEC-1 (one group of four)
        [[maybe_unused]] uint2 rb4;
        if constexpr (sizeof(T) == 2) rb4 = sr_bits4((uint32_t)(c0 + li), sr_gkey(kk >> 2, salt));
        float out[VEC];
        // ordinate pairs (two FP32 values per instruction); a single ordinate is a pair of itself
        float2 pw = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < VEC; l += 2) {
          const int l1 = VEC > 1 ? l + 1 : l;
          auto pair = [&](const float (&a)[VEC]) { return make_float2(a[l], a[l1]); };
          auto dup = [](float a) { return make_float2(a, a); };
          const float2 c2 = pair(c), xi2 = pair(xi), eta2 = pair(eta);
          float2 F = __ffma2_rn(dup(t1.z), c2, dup(t1.w));
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const float2 on = __ffma2_rn(eta2, dup(ay[e]), __fmul2_rn(xi2, dup(ax[e])));
            const float2 n2 = pair(nbv[e]);
            F = __ffma2_rn(make_float2(fminf(on.x, 0.f), fminf(on.y, 0.f)), __fadd2_rn(c2, make_float2(-n2.x, -n2.y)), F);
          }
          // dt enters last: rounded into the cell's constants, it would be off by the same amount in every step
          float2 o = __ffma2_rn(dup(dt), F, c2);
          if constexpr (kBase) o = __fmul2_rn(dup(0.5f), __fadd2_rn(pair(base), o));
          if constexpr (sizeof(T) == 2) {
            o.x = Store<T>::round_sr(o.x, sr_elem(rb4, (kk + l) & 3));
            o.y = Store<T>::round_sr(o.y, sr_elem(rb4, (kk + l1) & 3));
          }
          out[l] = o.x;
          if constexpr (VEC > 1) out[l1] = o.y;
          pw = __ffma2_rn(pair(w), o, pw);
        }
        phi_part[q] += VEC > 1 ? pw.x + pw.y : pw.x;
        if (!PLAIN && t2.w) {
          const float4 g0 = meta_geo(mb)[2 * li], g1 = meta_geo(mb)[2 * li + 1];
          const float bx[3] = {g0.x, g0.z, g1.x}, by[3] = {g0.y, g0.w, g1.y};
#pragma unroll
          for (int e = 0; e < 3; ++e)
            if (t2.w >> e & 1) {
#pragma unroll
              for (int l = 0; l < VEC; ++l) {
                const float on = xi[l] * bx[e] + eta[l] * by[e];
                bpart[q] += w[l] * on * ((on > 0.f) ? out[l] : nbv[e][l]);
              }
            }
        }
        st_row<T, VEC>(out_row, out);
      }
    };
    if (plain_chunk[i & 1]) cells_of_warp(std::true_type{});
    else cells_of_warp(std::false_type{});
    if (chunk_end) {
      // phi and the QoI terms of the warp's cells: lane 8 q holds cell q (FP32 over 32 chunks, then FP64)
      static_assert(kStgCellsPerWarp == 4, "four cells, eight lanes each in the sums");
      const float ph = multi_warp_sum<kStgCellsPerWarp>(phi_part, lane);
      const float bsum = plain_chunk[i & 1] ? 0.f : multi_warp_sum<kStgCellsPerWarp>(bpart, lane);
      const int li = warp + (lane >> 3) * kStgWarps;
      if ((lane & 7) == 0 && li < cells) {
        const float4 q4 = *reinterpret_cast<const float4*>(tab + li * kStgTab + 12);
        phi_out[c0 + li] = ph;
        facc[__float_as_uint(q4.z)][li] += q4.y * ph;
        facc[nreg][li] += q4.x * ph;
        facc[nreg + 1][li] += bsum * q4.x;
      }
      if ((i & 31) == 31) flush();
    }
    if (next_tab && go) table_store(i + 1);
    // every warp is done with row buffer rb, the next block's rows have arrived, and at the
    // chunk's end the next chunk's table is there
    stg_copy_wait();
    stop = __syncthreads_or(!go);
    if (chunk_end) {
      if (threadIdx.x == 0 && i + kStgMeta - 1 < n_my) {
        fence_proxy_async_smem();
        issue_meta(i + kStgMeta - 1);   // into buffer (i - 1) % kStgMeta, free since chunk i - 1 ended
      }
    }
    if (chunk_end) { b = 0; ++i; } else { ++b; }
  }
  if (!ok) {
    if (threadIdx.x == 0) {
      // drain: the last copies issued into each metadata buffer may still be in flight
      for (int q = 0; q < kStgMeta; ++q)
        if (s_meta_last[q] >= 0) mbar_wait_bounded(&meta_bar[q], (uint32_t)((s_meta_last[q] / kStgMeta) & 1), limit);
      atomicCAS(&st->status, DEV_OK, DEV_TIMEOUT);
      st->timeout_where = ((int64_t)blockIdx.x << 32) | (int64_t)j;
    }
  }
  flush();
  __syncthreads();
  if (threadIdx.x < nq) {
    double s = 0.0;
    for (int w2 = 0; w2 < kStgWarps; ++w2) s += dacc[w2][threadIdx.x];
    red[threadIdx.x] = s;
  }
  __syncthreads();
  finalize_item<kStgThreads>(d, it, red, STAGE, red + NQ);
}

size_t tri_staged_smem_bytes(int vec, int storage, int hmax, int stage) {
  return stg_layout(vec, storage == 1 ? 2 : 4, hmax, stage == STAGE_HEUN2).total;
}

template <int VEC, int STAGE, typename T>
static cudaError_t stg_prepare_one(size_t smem) {
  return cudaFuncSetAttribute(tri_staged_kernel<VEC, STAGE, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

template <int VEC, int STAGE, typename T>
static cudaError_t stg_launch_one(const InstDesc* d_desc, const WorkItem* d_items, int n_items, size_t smem,
                                  cudaStream_t s, bool chained) {
  return launch_stage_kernel(tri_staged_kernel<VEC, STAGE, T>, n_items, kStgThreads, smem, s, chained, d_desc, d_items);
}

#define RTK_STG_ALL(X, TT)                                                                          \
  X(1, STAGE_EULER, TT) X(1, STAGE_HEUN1, TT) X(1, STAGE_HEUN2, TT) X(2, STAGE_EULER, TT)           \
  X(2, STAGE_HEUN1, TT) X(2, STAGE_HEUN2, TT) X(4, STAGE_EULER, TT) X(4, STAGE_HEUN1, TT)           \
  X(4, STAGE_HEUN2, TT)

// The dynamic shared memory of any instance (the host keeps it below
// kStgSmemCap, else it takes the gathering kernel): every variant's limit is
// raised to that cap once, the same for all instances, so that preparing one
// instance never lowers the limit another one launches with.
constexpr size_t kStgSmemCap = 108 * 1024;   // two CTAs per SM

cudaError_t prepare_tri_staged(int stage, int storage, int vec, int hmax) {
  if (tri_staged_smem_bytes(vec, storage, hmax, stage) > kStgSmemCap) return cudaErrorInvalidValue;
  const size_t smem = kStgSmemCap;
#define RTK_P(V, ST, TT) \
  if (vec == V && stage == ST) return stg_prepare_one<V, ST, TT>(smem);
  if (storage == 0) { RTK_STG_ALL(RTK_P, float) } else { RTK_STG_ALL(RTK_P, __nv_bfloat16) }
#undef RTK_P
  return cudaErrorInvalidValue;
}

cudaError_t launch_tri_staged(const InstDesc* d_desc, const WorkItem* d_items, int n_items, int stage, int storage,
                              int vec, int hmax, cudaStream_t s, bool chained) {
  if (n_items <= 0) return cudaSuccess;
  const size_t smem = tri_staged_smem_bytes(vec, storage, hmax, stage);
#define RTK_L(V, ST, TT) \
  if (vec == V && stage == ST) return stg_launch_one<V, ST, TT>(d_desc, d_items, n_items, smem, s, chained);
  if (storage == 0) { RTK_STG_ALL(RTK_L, float) } else { RTK_STG_ALL(RTK_L, __nv_bfloat16) }
#undef RTK_L
  return cudaErrorInvalidValue;
}

}  // namespace rtk
