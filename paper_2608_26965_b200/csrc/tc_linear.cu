// Tensor-core (tcgen05 + TMEM + TMA) kernels for the tall-skinny linear algebra
// of the clustering stage (Section 3.2.2 metric matrices, Section 3.2.1
// covariance and projection on the principal components):
//   gram_tc       G = X^T X and column sums of X   (X [N, d] bf16)
//   transform_tc  Y = g(X W) + b, g = identity or row normalisation
//                 (W [d, d] fp32 used as bf16 hi + lo parts; Y fp32)
//   rep_gram_tc   G = R^T R and column sums of R = g(X W), R never written to memory
// A value v kept as hi + lo (hi = bf16(v), lo = bf16(v - hi)) keeps 16 bits of
// mantissa; products use hi*hi + hi*lo + lo*hi with fp32 accumulation.
#include "kernels.h"
#include "tc_ptx.cuh"

namespace ca {

using namespace ptx;

constexpr int kLinThreads = 192;     // warp 0: TMA, warp 1: MMA, warps 2-5: epilogue
constexpr int kRows = 128;           // rows per tile

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, int x, int y, int z, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
               ::"l"(map), "r"(x), "r"(y), "r"(z), "r"(src)
               : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ===========================================================================
// Gram matrix + column sums
// ===========================================================================
template <int D>
struct GramCfg {
  static constexpr int PANELS = D / 64;
  static constexpr int PANEL_BYTES = kRows * 128;
  static constexpr int TILE_BYTES = PANELS * PANEL_BYTES;       // one part (hi or lo)
  static constexpr int M = D;                                   // 64 or 128 accumulator rows
};

struct GramParams {
  float* partial;        // [(p * n_chunks + chunk) * (D*D + D)]
  int* status;
  int n_rows, chunk_rows, n_chunks, stages, normalize;    // normalize: of the representation
};

// One of the four epilogue warps writes its rows of the accumulated Gram matrix.
template <int D>
__device__ __forceinline__ void write_gram(uint32_t tmem_acc, int quarter, int lane, bool any, float* __restrict__ out) {
  // accumulator row m sits in lane m (D = 128) or in lane (m % 16) + 32 (m / 16) (D = 64)
  const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
  const int m = D == 128 ? quarter * 32 + lane : quarter * 16 + lane;
  const bool live = any && (D == 128 || lane < 16);
#pragma unroll
  for (int c4 = 0; c4 < D / 32; ++c4) {
    uint32_t v[32];
    tmem_ld32(tmem_acc + lane_addr + c4 * 32, v);
    tmem_wait_ld();
    if (live) {
      float4* dst = reinterpret_cast<float4*>(out + m * D + c4 * 32);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        dst[j] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                             __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
    }
  }
}

template <int D>
__global__ void __launch_bounds__(kLinThreads, 1)
gram_tc_kernel(const __grid_constant__ CUtensorMap tm_x, const GramParams prm) {
  wait_for_previous();
  using C = GramCfg<D>;
  extern __shared__ unsigned char smem_unaligned[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_unaligned) + 1023) & ~uintptr_t(1023));
  constexpr int stage_bytes = C::TILE_BYTES;
  const uint32_t s_base = smem_u32(smem);
  const uint32_t s_ones = s_base + prm.stages * stage_bytes;                // 2 KB of bf16 1.0
  const uint32_t bar0 = s_ones + 2048;
  auto b_full = [&](int s) { return bar0 + 8 * s; };
  auto b_empty = [&](int s) { return bar0 + 8 * (prm.stages + s); };
  const uint32_t b_done = bar0 + 8 * (2 * prm.stages);
  unsigned char* misc = smem + prm.stages * stage_bytes + 2048 + 8 * (2 * prm.stages + 1);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p = blockIdx.y, chunk = blockIdx.x;
  const int r_begin = chunk * prm.chunk_rows;
  const int r_end = min(prm.n_rows, r_begin + prm.chunk_rows);
  const int n_tiles = (r_end - r_begin + kRows - 1) / kRows;
  constexpr uint32_t kCols = (D + 16 <= 128) ? 128 : 256;

  if (tid == 0) {
    for (int s = 0; s < prm.stages; ++s) { mbar_init(b_full(s), 1); mbar_init(b_empty(s), 1); }
    mbar_init(b_done, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  for (int e = tid; e < 1024; e += kLinThreads)
    reinterpret_cast<__nv_bfloat16*>(smem + prm.stages * stage_bytes)[e] = __float2bfloat16_rn(1.0f);
  fence_proxy_async();                 // the ones are read by the tensor core (async proxy)
  if (warp == 1) { tmem_alloc(smem_u32(tmem_slot), kCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_acc = *tmem_slot, tmem_sum = tmem_acc + D;

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int s = t % prm.stages;
        if (t >= prm.stages) ok = mbar_wait(b_empty(s), ((t / prm.stages) - 1) & 1, abort_flag, prm.status);
        if (!ok) break;
        mbar_expect_tx(b_full(s), stage_bytes);
        const uint32_t dst = s_base + s * stage_bytes;
        for (int pn = 0; pn < C::PANELS; ++pn)
          tma_load_3d(dst + pn * C::PANEL_BYTES, &tm_x, pn * 64, r_begin + t * kRows, p, b_full(s));
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(C::M, D, 1, 1);        // X^T X: both operands MN-major
      constexpr uint32_t idesc_sum = idesc_bf16_f32(C::M, 16, 1, 1);
      bool ok = true;
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int s = t % prm.stages;
        ok = mbar_wait(b_full(s), (t / prm.stages) & 1, abort_flag, prm.status);
        if (!ok) break;
        tc_fence_after();
        const uint32_t x = s_base + s * stage_bytes;
#pragma unroll
        for (int ks = 0; ks < kRows / 16; ++ks) {
          // 16 rows (the contraction index) per step = 2048 bytes; 64-column panels along M and N
          const uint64_t dh = smem_desc_sw128(x + ks * 2048, C::PANEL_BYTES, 1024);
          const uint64_t ones = smem_desc_sw128(s_ones, C::PANEL_BYTES, 1024);
          const uint32_t acc = (t > 0 || ks > 0) ? 1u : 0u;
          mma_ss(tmem_acc, dh, dh, idesc, acc);
          mma_ss(tmem_sum, dh, ones, idesc_sum, acc);
        }
        mma_commit(b_empty(s));
      }
      mma_commit(b_done);
    }
  } else {
    const int quarter = warp & 3;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(b_done, 0, abort_flag, prm.status));
    if (warp == 2) let_next_start();
    tc_fence_after();
    if (ok) {
      float* out = prm.partial + ((size_t)p * prm.n_chunks + chunk) * (D * D + D);
      write_gram<D>(tmem_acc, quarter, lane, n_tiles > 0, out);
      const uint32_t sum = tmem_ld1(tmem_sum + ((uint32_t)(quarter * 32) << 16));     // one of 16 identical sums
      tmem_wait_ld();
      if (n_tiles > 0 && (D == 128 || lane < 16))
        out[D * D + (D == 128 ? quarter * 32 + lane : quarter * 16 + lane)] = __uint_as_float(sum);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_acc, kCols);
}

// ===========================================================================
// Row transform
// ===========================================================================
template <int D>
struct LinCfg {
  static constexpr int PANELS = D / 64;
  static constexpr int PANEL_BYTES = kRows * 128;               // X panels: 128 rows x 128 bytes
  static constexpr int TILE_BYTES = PANELS * PANEL_BYTES;       // one part of an X tile
  static constexpr int W_PANEL_BYTES = D * 128;                 // W^T panels: D rows x 128 bytes
  static constexpr int W_BYTES = PANELS * W_PANEL_BYTES;        // one part of W^T
  static constexpr int OUT_BYTES = kRows * D * 4;               // fp32 tile
};

struct LinParams {
  const float* bias;      // [P][D] or null
  float* out_t;           // [P][kSplitCols][n_rows] or null: the first coordinates once more, coordinate-major
  int* status;
  int n_rows, tiles_per_cta, stages, normalize;       // normalize: rows are divided by their norm before the bias
};

template <int D>
__global__ void __launch_bounds__(kLinThreads, 1)
transform_tc_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_whi,
                    const __grid_constant__ CUtensorMap tm_wlo, const __grid_constant__ CUtensorMap tm_out,
                    const LinParams prm) {
  wait_for_previous();
  using C = LinCfg<D>;
  extern __shared__ unsigned char smem_unaligned[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_unaligned) + 1023) & ~uintptr_t(1023));
  constexpr int stage_bytes = C::TILE_BYTES;
  const uint32_t s_base = smem_u32(smem);
  const uint32_t s_w = s_base;                                   // W^T hi, W^T lo
  const uint32_t s_x = s_w + 2 * C::W_BYTES;
  const uint32_t s_out = s_x + prm.stages * stage_bytes;
  unsigned char* out_ptr = smem + 2 * C::W_BYTES + prm.stages * stage_bytes;
  const uint32_t bar0 = s_out + C::OUT_BYTES;
  const uint32_t b_w = bar0;
  auto b_full = [&](int s) { return bar0 + 8 + 8 * s; };
  auto b_empty = [&](int s) { return bar0 + 8 + 8 * (prm.stages + s); };
  auto b_acc_full = [&](int a) { return bar0 + 8 + 8 * (2 * prm.stages + a); };
  auto b_acc_empty = [&](int a) { return bar0 + 8 + 8 * (2 * prm.stages + 2 + a); };
  unsigned char* misc = out_ptr + C::OUT_BYTES + 8 * (2 * prm.stages + 5);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);
  float* s_bias = reinterpret_cast<float*>(misc + 16);            // [D]

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p = blockIdx.y;
  const int total_tiles = (prm.n_rows + kRows - 1) / kRows;
  const int t_begin = blockIdx.x * prm.tiles_per_cta;
  const int n_tiles = max(0, min(total_tiles, t_begin + prm.tiles_per_cta) - t_begin);
  constexpr uint32_t kCols = 2 * D;                              // two accumulators

  if (tid == 0) {
    mbar_init(b_w, 1);
    for (int s = 0; s < prm.stages; ++s) { mbar_init(b_full(s), 1); mbar_init(b_empty(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(b_acc_full(a), 1); mbar_init(b_acc_empty(a), 128); }
    *abort_flag = 0;
    fence_mbar_init();
  }
  for (int j = tid; j < D; j += kLinThreads) s_bias[j] = prm.bias ? prm.bias[(size_t)p * D + j] : 0.f;
  if (warp == 1) { tmem_alloc(smem_u32(tmem_slot), kCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(b_w, 2 * C::W_BYTES);
      for (int pn = 0; pn < C::PANELS; ++pn) {
        tma_load_2d(s_w + pn * C::W_PANEL_BYTES, &tm_whi, pn * 64, p * D, b_w);
        tma_load_2d(s_w + C::W_BYTES + pn * C::W_PANEL_BYTES, &tm_wlo, pn * 64, p * D, b_w);
      }
      bool ok = true;
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int s = t % prm.stages;
        if (t >= prm.stages) ok = mbar_wait(b_empty(s), ((t / prm.stages) - 1) & 1, abort_flag, prm.status);
        if (!ok) break;
        mbar_expect_tx(b_full(s), stage_bytes);
        const uint32_t dst = s_x + s * stage_bytes;
        const int row = (t_begin + t) * kRows;
        for (int pn = 0; pn < C::PANELS; ++pn) {
          tma_load_3d(dst + pn * C::PANEL_BYTES, &tm_x, pn * 64, row, p, b_full(s));
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(kRows, D, 0, 0);    // X (K-major) times W^T (K-major)
      bool ok = mbar_wait(b_w, 0, abort_flag, prm.status);
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int s = t % prm.stages, a = t & 1;
        if (t >= 2) ok = mbar_wait(b_acc_empty(a), ((t >> 1) - 1) & 1, abort_flag, prm.status);
        if (ok) ok = mbar_wait(b_full(s), (t / prm.stages) & 1, abort_flag, prm.status);
        if (!ok) break;
        tc_fence_after();
        const uint32_t xh = s_x + s * stage_bytes;
        const uint32_t acc = tmem_base + a * D;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint32_t xo = (ks / 4) * C::PANEL_BYTES + (ks % 4) * 32;
          const uint32_t wo = (ks / 4) * C::W_PANEL_BYTES + (ks % 4) * 32;
          const uint64_t dxh = smem_desc_sw128(xh + xo, 16, 1024);
          const uint64_t dwh = smem_desc_sw128(s_w + wo, 16, 1024);
          const uint64_t dwl = smem_desc_sw128(s_w + C::W_BYTES + wo, 16, 1024);
          mma_ss(acc, dxh, dwh, idesc, ks > 0 ? 1u : 0u);
          mma_ss(acc, dxh, dwl, idesc, 1u);
        }
        mma_commit(b_empty(s));
        mma_commit(b_acc_full(a));
      }
    }
  } else {
    const int st = tid - 64;
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    bool ok = true;
    for (int t = 0; t < n_tiles && ok; ++t) {
      const int a = t & 1;
      ok = __all_sync(0xffffffffu, mbar_wait(b_acc_full(a), (t >> 1) & 1, abort_flag, prm.status));
      if (!ok) break;
      tc_fence_after();
      float v[D];
#pragma unroll
      for (int c4 = 0; c4 < D / 32; ++c4) {
        uint32_t r[32];
        tmem_ld32(tmem_base + a * D + lane_addr + c4 * 32, r);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; ++j) v[c4 * 32 + j] = __uint_as_float(r[j]);
      }
      tc_fence_before();
      mbar_arrive(b_acc_empty(a));                    // the accumulator may be overwritten
      if (prm.normalize) {
        float ss = 0.f;
#pragma unroll
        for (int j = 0; j < D; ++j) ss = fmaf(v[j], v[j], ss);
        const float nrm = sqrtf(ss);
        const float inv = nrm >= 1e-30f ? 1.f / nrm : 0.f;
#pragma unroll
        for (int j = 0; j < D; ++j) v[j] = fmaf(v[j], inv, s_bias[j]);
      } else {
#pragma unroll
        for (int j = 0; j < D; ++j) v[j] += s_bias[j];
      }
      if (prm.out_t) {
        // coordinate-major copy of the coordinates that the splitter reads one at a time: for one
        // coordinate the 128 threads of the tile write 512 consecutive bytes
        const int grow = (t_begin + t) * kRows + row;
        if (grow < prm.n_rows) {
          float* dst = prm.out_t + (size_t)p * kSplitCols * prm.n_rows + grow;
#pragma unroll
          for (int j = 0; j < kSplitCols; ++j) dst[(size_t)j * prm.n_rows] = v[j];
        }
      }
      // the previous tile's stores must have finished reading the staging buffer
      if (st == 0) tma_store_wait_read();
      asm volatile("bar.sync 1, 128;" ::: "memory");
      // fp32 tile as 32-column panels with the 128-byte swizzle the store expects
#pragma unroll
      for (int pn = 0; pn < D / 32; ++pn)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          float4 w = make_float4(v[pn * 32 + 4 * c], v[pn * 32 + 4 * c + 1], v[pn * 32 + 4 * c + 2], v[pn * 32 + 4 * c + 3]);
          *reinterpret_cast<float4*>(out_ptr + pn * 16384 + row * 128 + ((c ^ (row & 7)) * 16)) = w;
        }
      fence_proxy_async();
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (st == 0) {
        const int grow = (t_begin + t) * kRows;
        for (int pn = 0; pn < D / 32; ++pn) tma_store_3d(&tm_out, pn * 32, grow, p, s_out + pn * 16384);
        tma_store_commit();
      }
    }
    let_next_start();
    if (st == 0) tma_store_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, kCols);
}

// ===========================================================================
// Gram matrix and column sums of the row representation R = g(X W), g = identity or division by the row's norm
// ===========================================================================
// Two chained products per tile of 128 rows: T = X W into tensor memory, from where the epilogue
// warps normalise a row per thread and write it to shared memory as H + L, bf16 hi + lo parts in the
// layout of a loaded tile, then the Gram matrix.  H^T H + H^T 2L is what is accumulated: its
// symmetric part is H^T H + H^T L + L^T H, and the decomposition takes the symmetric part of what it is given.
// T of the next tile is issued before R of this one is waited for.
// r(q) used to be written by the row transform and read back by its Gram matrix and by the projection
// (12 d bytes per row): the query side of 40 heads of 32,760 rows, d = 128, took 0.63 ms in these
// kernels and takes 0.35, 0.16 of them here (0.20 with column sums from 16-column products).  What bounds it is
// the epilogue's chain per tile: 3,400 cycles at d = 128, 1,400 of which the 32 KB of X take from HBM.
template <int D>
struct RepCfg {
  static constexpr int PANELS = D / 64;
  static constexpr int PANEL_BYTES = kRows * 128;
  static constexpr int TILE_BYTES = PANELS * PANEL_BYTES;
  static constexpr int W_PANEL_BYTES = D * 128;
  static constexpr int W_BYTES = PANELS * W_PANEL_BYTES;
  static constexpr int STAGES = D == 64 ? 3 : 2;
  static constexpr int OFF_X = 2 * W_BYTES;
  static constexpr int OFF_R = OFF_X + STAGES * TILE_BYTES;             // hi tile, 2 lo tile
  static constexpr int GROUPS = D / 64;                                 // epilogue warps per 32 rows: 64 columns each
  static constexpr int THREADS = 64 + 128 * GROUPS;
  static constexpr int OFF_NORM = OFF_R + 2 * TILE_BYTES;               // [2][GROUPS][128 rows] partial squared norms
  static constexpr int OFF_BAR = OFF_NORM + 2 * GROUPS * kRows * 4;
  static constexpr int NUM_BARS = 2 + 2 * STAGES + 4 + 3;               // weights, done; x full/empty; acc full/empty x 2; r full/empty; norms
  static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;
  static constexpr int SMEM = 1024 + OFF_MISC + 16;
  static constexpr uint32_t TMEM_COLS = D == 64 ? 256 : 512;            // two T accumulators, G
  static constexpr int CTAS_PER_SM = D == 64 ? 2 : 1;
};

template <int D>
__global__ void __launch_bounds__(RepCfg<D>::THREADS, RepCfg<D>::CTAS_PER_SM)
rep_gram_tc_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_whi,
                   const __grid_constant__ CUtensorMap tm_wlo, const GramParams prm) {
  wait_for_previous();
  using C = RepCfg<D>;
  extern __shared__ unsigned char smem_unaligned[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_unaligned) + 1023) & ~uintptr_t(1023));
  const uint32_t s_base = smem_u32(smem);
  const uint32_t s_w = s_base, s_x = s_base + C::OFF_X, s_r = s_base + C::OFF_R;
  unsigned char* r_ptr = smem + C::OFF_R;
  const uint32_t bar0 = s_base + C::OFF_BAR;
  const uint32_t b_w = bar0, b_done = bar0 + 8;
  auto b_full = [&](int s) { return bar0 + 16 + 8 * s; };
  auto b_empty = [&](int s) { return bar0 + 16 + 8 * (C::STAGES + s); };
  auto b_acc_full = [&](int a) { return bar0 + 16 + 8 * (2 * C::STAGES + a); };
  auto b_acc_empty = [&](int a) { return bar0 + 16 + 8 * (2 * C::STAGES + 2 + a); };
  const uint32_t b_r_full = bar0 + 16 + 8 * (2 * C::STAGES + 4), b_r_empty = b_r_full + 8, b_norm = b_r_full + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p = blockIdx.y, chunk = blockIdx.x;
  const int r_begin = chunk * prm.chunk_rows;
  const int r_end = min(prm.n_rows, r_begin + prm.chunk_rows);
  const int n_tiles = (r_end - r_begin + kRows - 1) / kRows;

  if (tid == 0) {
    mbar_init(b_w, 1);
    mbar_init(b_done, 1);
    for (int s = 0; s < C::STAGES; ++s) { mbar_init(b_full(s), 1); mbar_init(b_empty(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(b_acc_full(a), 1); mbar_init(b_acc_empty(a), 4 * C::GROUPS); }
    mbar_init(b_r_full, 4 * C::GROUPS);
    mbar_init(b_r_empty, 1);
    mbar_init(b_norm, 4 * C::GROUPS);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_t = *tmem_slot, tmem_g = tmem_t + 2 * D;

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(b_w, 2 * C::W_BYTES);
      for (int pn = 0; pn < C::PANELS; ++pn) {
        tma_load_2d(s_w + pn * C::W_PANEL_BYTES, &tm_whi, pn * 64, p * D, b_w);
        tma_load_2d(s_w + C::W_BYTES + pn * C::W_PANEL_BYTES, &tm_wlo, pn * 64, p * D, b_w);
      }
      bool ok = true;
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int s = t % C::STAGES;
        if (t >= C::STAGES) ok = mbar_wait(b_empty(s), ((t / C::STAGES) - 1) & 1, abort_flag, prm.status);
        if (!ok) break;
        mbar_expect_tx(b_full(s), C::TILE_BYTES);
        for (int pn = 0; pn < C::PANELS; ++pn)
          tma_load_3d(s_x + s * C::TILE_BYTES + pn * C::PANEL_BYTES, &tm_x, pn * 64, r_begin + t * kRows, p, b_full(s));
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc_t = idesc_bf16_f32(kRows, D, 0, 0);     // X (K-major) times W^T (K-major)
      constexpr uint32_t idesc_g = idesc_bf16_f32(D, D, 1, 1);         // R^T R: both operands MN-major
      bool ok = mbar_wait(b_w, 0, abort_flag, prm.status);
      auto product_t = [&](int t) {
        const int s = t % C::STAGES, a = t & 1;
        if (t >= 2 && !mbar_wait(b_acc_empty(a), ((t >> 1) - 1) & 1, abort_flag, prm.status)) return false;
        if (!mbar_wait(b_full(s), (t / C::STAGES) & 1, abort_flag, prm.status)) return false;
        tc_fence_after();
        const uint32_t x = s_x + s * C::TILE_BYTES, acc = tmem_t + a * D;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint64_t dx = smem_desc_sw128(x + (ks / 4) * C::PANEL_BYTES + (ks % 4) * 32, 16, 1024);
          const uint32_t wo = (ks / 4) * C::W_PANEL_BYTES + (ks % 4) * 32;
          mma_ss(acc, dx, smem_desc_sw128(s_w + wo, 16, 1024), idesc_t, ks > 0 ? 1u : 0u);
          mma_ss(acc, dx, smem_desc_sw128(s_w + C::W_BYTES + wo, 16, 1024), idesc_t, 1u);
        }
        mma_commit(b_empty(s));
        mma_commit(b_acc_full(a));
        return true;
      };
      if (ok && n_tiles > 0) ok = product_t(0);
      for (int t = 0; t < n_tiles && ok; ++t) {
        if (t + 1 < n_tiles) ok = product_t(t + 1);
        if (ok) ok = mbar_wait(b_r_full, t & 1, abort_flag, prm.status);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int ks = 0; ks < kRows / 16; ++ks) {
          // 16 rows (the contraction index) per step = 2048 bytes; 64-column panels along M and N
          const uint64_t dh = smem_desc_sw128(s_r + ks * 2048, C::PANEL_BYTES, 1024);
          const uint64_t dl = smem_desc_sw128(s_r + C::TILE_BYTES + ks * 2048, C::PANEL_BYTES, 1024);
          const uint32_t acc = (t > 0 || ks > 0) ? 1u : 0u;
          mma_ss(tmem_g, dh, dh, idesc_g, acc);
          mma_ss(tmem_g, dh, dl, idesc_g, 1u);
        }
        mma_commit(b_r_empty);
      }
      mma_commit(b_done);
    }
  } else {
    const int quarter = warp & 3, group = (warp - 2) >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    float* s_norm = reinterpret_cast<float*>(smem + C::OFF_NORM);
    auto wait = [&](uint32_t bar, uint32_t parity) {
      return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, prm.status));
    };
    float sum[64];                                     // of this thread's row of every tile
#pragma unroll
    for (int j = 0; j < 64; ++j) sum[j] = 0.f;
    bool ok = true;
#pragma unroll 1
    for (int t = 0; t < n_tiles && ok; ++t) {
      const int a = t & 1;
      ok = wait(b_acc_full(a), (t >> 1) & 1);
      if (!ok) break;
      tc_fence_after();
      float v[64];
      {
        uint32_t r0[32], r1[32];
        tmem_ld32(tmem_t + a * D + group * 64 + lane_addr, r0);
        tmem_ld32(tmem_t + a * D + group * 64 + 32 + lane_addr, r1);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; ++j) { v[j] = __uint_as_float(r0[j]); v[32 + j] = __uint_as_float(r1[j]); }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_acc_empty(a));
      if (prm.normalize) {
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
        for (int j = 0; j < 64; j += 4) {
          s0 = fmaf(v[j], v[j], s0); s1 = fmaf(v[j + 1], v[j + 1], s1);
          s2 = fmaf(v[j + 2], v[j + 2], s2); s3 = fmaf(v[j + 3], v[j + 3], s3);
        }
        float ss = (s0 + s1) + (s2 + s3);
        if constexpr (C::GROUPS > 1) {                 // the other half of the row is another warp's
          float* norms = s_norm + a * C::GROUPS * kRows + row;
          norms[group * kRows] = ss;
          __syncwarp();
          if (lane == 0) mbar_arrive(b_norm);
          ok = wait(b_norm, t & 1);
          if (!ok) break;
          ss = norms[0] + norms[kRows];
        }
        const float nrm = sqrtf(ss);
        const float inv = nrm >= 1e-30f ? 1.f / nrm : 0.f;
#pragma unroll
        for (int j = 0; j < 64; ++j) v[j] *= inv;
      }
      uint32_t hi[32], lo[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const float x0 = v[2 * j], x1 = v[2 * j + 1];
        sum[2 * j] += x0;
        sum[2 * j + 1] += x1;
        hi[j] = pack_bf16x2(x0, x1);
        lo[j] = pack_bf16x2(2.f * (x0 - __uint_as_float(hi[j] << 16)), 2.f * (x1 - __uint_as_float(hi[j] & 0xffff0000u)));
      }
      if (t > 0) ok = wait(b_r_empty, (t - 1) & 1);
      if (!ok) break;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int off = group * C::PANEL_BYTES + row * 128 + ((c ^ (row & 7)) * 16);
        *reinterpret_cast<uint4*>(r_ptr + off) = make_uint4(hi[4 * c], hi[4 * c + 1], hi[4 * c + 2], hi[4 * c + 3]);
        *reinterpret_cast<uint4*>(r_ptr + C::TILE_BYTES + off) = make_uint4(lo[4 * c], lo[4 * c + 1], lo[4 * c + 2], lo[4 * c + 3]);
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_r_full);
    }
    if (warp == 2) let_next_start();
    if (ok) ok = wait(b_done, 0);
    tc_fence_after();
    float* out = prm.partial + ((size_t)p * prm.n_chunks + chunk) * (D * D + D);
    if (ok && group == 0) write_gram<D>(tmem_g, quarter, lane, n_tiles > 0, out);
    // the tensor core is done with R: its space takes the sums per row, [D / 64][128 rows][64 columns]
    if (ok) {
      float* mine = reinterpret_cast<float*>(r_ptr) + (group * kRows + row) * 64;
#pragma unroll
      for (int j = 0; j < 64; j += 4)
        *reinterpret_cast<float4*>(mine + (j ^ (4 * (lane & 7)))) = make_float4(sum[j], sum[j + 1], sum[j + 2], sum[j + 3]);
    }
  }
  __syncthreads();
  if (tid < D && !*abort_flag) {
    const float* rows = reinterpret_cast<const float*>(r_ptr) + (tid >> 6) * kRows * 64;
    float total = 0.f;
#pragma unroll 8
    for (int r = 0; r < kRows; ++r) total += rows[r * 64 + ((tid & 63) ^ (4 * (r & 7)))];
    prm.partial[((size_t)p * prm.n_chunks + chunk) * (D * D + D) + D * D + tid] = total;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_t, C::TMEM_COLS);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static EncodeTiledFn lin_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// [P][n][D] tensor; box = box_cols x box_rows x 1, 128-byte swizzle
static bool map_3d(CUtensorMap* map, const void* base, int P, int n, int D, int elem_bytes, int box_cols,
                   int box_rows) {
  EncodeTiledFn fn = lin_encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)n, (cuuint64_t)P};
  cuuint64_t strides[2] = {(cuuint64_t)D * elem_bytes, (cuuint64_t)n * D * elem_bytes};
  cuuint32_t box[3] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
            const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
static bool map_2d(CUtensorMap* map, const void* base, size_t rows, int D, int box_rows) {
  EncodeTiledFn fn = lin_encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)D, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)D * 2};
  cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Chunks of rows per problem, one CTA each, `ctas_per_sm` of them resident per SM: the count that
// minimises rounds x (tiles per chunk + 3), the time of the launch in tiles when every CTA pays
// about three tiles' worth of start-up and epilogue and a last round that is nearly empty costs a
// full round (320 CTAs on 148 slots run as long as 444); chunks of at least four tiles.
int gram_tc_chunking(int n_rows, int problems, int ctas_per_sm, int* chunk_rows, int* n_chunks) {
  int sms = 148, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
    (void)cudaGetLastError();
    sms = 148;
  }
  const long long slots = (long long)sms * (ctas_per_sm > 0 ? ctas_per_sm : 1);
  const int tiles = ceil_div(n_rows, kRows);
  int best_c = 1, best_cr = tiles * kRows;
  long long best_cost = -1;
  for (int c = 1; c <= tiles; ++c) {
    const int ct = ceil_div(tiles, c);                     // tiles per chunk
    if (c > 1 && ct < 4) break;
    const int cr = ct * kRows;
    const int chunks = ceil_div(n_rows, cr);
    const long long total = (long long)chunks * problems;
    const long long rounds = (total + slots - 1) / slots;
    const long long cost = rounds * (ct + 3);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best_c = chunks; best_cr = cr; }
    if (rounds > 8) break;
  }
  // the buffer of partial sums is sized for the chunk count of the CUDA-core moments kernel
  int m_cr, m_chunks;
  moments_chunking(n_rows, problems, &m_cr, &m_chunks);
  if (best_c > m_chunks) {
    best_cr = ceil_div(ceil_div(n_rows, m_chunks), kRows) * kRows;
    best_c = ceil_div(n_rows, best_cr);
  }
  *chunk_rows = best_cr;
  *n_chunks = best_c;
  return 0;
}

int launch_gram_tc(const void* X, int problems, int n_rows, int D, float* partial, double* gram, double* colsum,
                   int* status, LaunchStream st) {
  GramParams prm{};
  prm.partial = partial; prm.status = status; prm.n_rows = n_rows;
  const int tile = kRows * D * 2;
  // three stages, so that two CTAs share an SM and one's start-up and epilogue overlap the other's
  // streaming (video480: 0.36 -> 0.34 ms for the step's three launches)
  prm.stages = 3;
  const size_t smem = 1024 + (size_t)prm.stages * tile + 2048 + 8 * (2 * prm.stages + 1) + 64;
  {
    int per_sm = (int)((227 * 1024) / (smem + 1024));
    const int by_tmem = 512 / ((D + 16 <= 128) ? 128 : 256);
    if (per_sm > by_tmem) per_sm = by_tmem;
    gram_tc_chunking(n_rows, problems, per_sm, &prm.chunk_rows, &prm.n_chunks);
  }
  CUtensorMap mx;
  if (!map_3d(&mx, X, problems, n_rows, D, 2, 64, kRows)) return CA_ERR_CUDA;
  auto k = D == 64 ? gram_tc_kernel<64> : gram_tc_kernel<128>;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  launch_chained(k, dim3(prm.n_chunks, problems), kLinThreads, smem, st, mx, prm);
  CA_LAUNCH_CHECK();
  return launch_gram_finalize(partial, problems, prm.n_chunks, D, gram, colsum, st);
}

template <int D>
static int launch_rep_gram(const void* X, int problems, int n_rows, int normalize, float* partial, double* gram,
                           double* colsum, const void* wt_hi, const void* wt_lo, int* status, LaunchStream st) {
  using C = RepCfg<D>;
  GramParams prm{};
  prm.partial = partial; prm.status = status; prm.n_rows = n_rows; prm.normalize = normalize;
  gram_tc_chunking(n_rows, problems, C::CTAS_PER_SM, &prm.chunk_rows, &prm.n_chunks);
  CUtensorMap mx, mwh, mwl;
  if (!map_3d(&mx, X, problems, n_rows, D, 2, 64, kRows) || !map_2d(&mwh, wt_hi, (size_t)problems * D, D, D) ||
      !map_2d(&mwl, wt_lo, (size_t)problems * D, D, D))
    return CA_ERR_CUDA;
  auto k = rep_gram_tc_kernel<D>;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
  launch_chained(k, dim3(prm.n_chunks, problems), C::THREADS, C::SMEM, st, mx, mwh, mwl, prm);
  CA_LAUNCH_CHECK();
  return launch_gram_finalize(partial, problems, prm.n_chunks, D, gram, colsum, st);
}

int launch_rep_gram_tc(const void* X, int problems, int n_rows, int D, int normalize, float* partial, double* gram,
                       double* colsum, const void* wt_hi, const void* wt_lo, int* status, LaunchStream st) {
  return D == 64 ? launch_rep_gram<64>(X, problems, n_rows, normalize, partial, gram, colsum, wt_hi, wt_lo, status, st)
                 : launch_rep_gram<128>(X, problems, n_rows, normalize, partial, gram, colsum, wt_hi, wt_lo, status, st);
}

int launch_transform_tc(const void* X, int problems, int n_rows, int D, const float* bias, int normalize, float* out,
                        const void* wt_hi, const void* wt_lo, int* status, LaunchStream st, float* out_t) {
  LinParams prm{};
  prm.bias = bias; prm.out_t = out_t; prm.status = status; prm.n_rows = n_rows; prm.normalize = normalize;
  const int tile = kRows * D * 2;
  const int fixed = 2 * D * D * 2 + kRows * D * 4 + 4096;
  prm.stages = (200 * 1024 - fixed) / tile;
  if (prm.stages > 4) prm.stages = 4;
  if (prm.stages < 1) return CA_ERR_UNSUPPORTED;
  const int total_tiles = ceil_div(n_rows, kRows);
  int ctas = 296 / problems;
  if (ctas < 1) ctas = 1;
  prm.tiles_per_cta = ceil_div(total_tiles, ctas);
  if (prm.tiles_per_cta < 2) prm.tiles_per_cta = 2;
  CUtensorMap mx, mwh, mwl, mo;
  if (!map_3d(&mx, X, problems, n_rows, D, 2, 64, kRows) || !map_2d(&mwh, wt_hi, (size_t)problems * D, D, D) ||
      !map_2d(&mwl, wt_lo, (size_t)problems * D, D, D) || !map_3d(&mo, out, problems, n_rows, D, 4, 32, kRows))
    return CA_ERR_CUDA;
  const size_t smem = 1024 + (size_t)fixed + (size_t)prm.stages * tile + D * 4;
  auto k = D == 64 ? transform_tc_kernel<64> : transform_tc_kernel<128>;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  launch_chained(k, dim3(ceil_div(total_tiles, prm.tiles_per_cta), problems), kLinThreads, smem, st, mx, mwh, mwl, mo, prm);
  CA_LAUNCH_CHECK();
  return CA_OK;
}

}  // namespace ca
