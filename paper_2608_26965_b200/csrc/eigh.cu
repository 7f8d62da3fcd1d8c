// Cholesky factors of the metric matrices (Section 3.2.2); the metric matrices themselves
// for the basic splitting variant.  (Covariances and principal components: eigh_tql.cu.)
#include "kernels.h"

namespace ca {

// ---------------------------------------------------------------------------
// Factor of a positive semi-definite matrix: lower-triangular F with F F^T = A
// (right-looking Cholesky in double, one CTA per matrix).  A pivot
// that is not above 1e-12 of the largest diagonal entry marks a direction in
// which the (pseudo-)metric is zero: its column of F is set to zero, which is the
// counterpart of clamping small or negative eigenvalues (Section 3.2.2).
// Any factor of the metric matrix gives the same principal-component
// coordinates as its symmetric root, because the two differ by a rotation.
//
// The matrix is formed on load from a Gram matrix and column sums: gram * scale (the query metric
// M = Q^T Q / n_q, `sum` null) or (gram - s s^T / n) * scale (the centred scatter of the keys).
// Besides F in double and float, F^T can be written as bf16 hi + lo parts, the layout in which the
// tensor-core projection takes its weights (the query representation multiplies by F).
//
// The elimination goes by panels of eight columns, a row per lane in registers; every lane factors the panel's 8 x 8 head for itself
// as well, so that the chain of a column (pivot, reciprocal, update: some 80 cycles) waits for no other lane.  Then all
// threads take the eight columns off the trailing block at once: two barriers per eight columns.  (With the panel's rows in one
// warp and pivots and heads by shuffles a factor took 15 us at d = 64 and 50 us at d = 128; now 12.5 and 33.)  The trailing block is kept
// in registers as the accumulators of double-precision matrix instructions, tiles of 8 x 8 of the lower triangle dealt out so
// that the shrinking block stays spread over all warps; finished columns stay in shared memory, unscaled, and are scaled by 1 / sqrt(pivot)
// on the way out.  The trailing block takes A[r][k] -= A[r][j] A[k][j] / pivot_j with the unscaled columns;
// a dropped pivot (reciprocal 0) leaves it alone and gives a zero column.
// ---------------------------------------------------------------------------
constexpr int kPanel = 8;

// reciprocal: the hardware's estimate (a relative error e of 2^-20) and one step of third order, 1 + e + e^2
__device__ __forceinline__ double reciprocal(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// C (8 x 8) += A (8 x 4) B (4 x 8) in double: lane l holds A[l / 4][l % 4], B[l % 4][l / 4], C[l / 4][2 (l % 4) + 0, 1]
__device__ __forceinline__ void mma_f64(double (&c)[2], double a, double b) {
  asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

template <int D>
__global__ void __launch_bounds__(4 * D) cholesky_factor_kernel(const double* __restrict__ gram,
                                                                const double* __restrict__ sum, double n,
                                                                double scale, double* __restrict__ out64,
                                                                float* __restrict__ out32,
                                                                __nv_bfloat16* __restrict__ wt_hi,
                                                                __nv_bfloat16* __restrict__ wt_lo) {
  constexpr int NT = 4 * D, NW = NT / 32;
  constexpr int NB = D / kPanel;              // blocks of eight rows, of eight columns
  constexpr int TILES = NB * (NB + 1) / 2, SLOTS = (TILES + NW - 1) / NW;
  constexpr int LD = D + 1;                   // pitch of a column
  constexpr int LP = D + 8;                   // of a panel column: the four columns of a fragment in two runs of banks
  extern __shared__ __align__(16) double chol_smem[];
  double* F = chol_smem;                      // [D][LD]  finished columns, column-major, unscaled; a panel before it is factored
  double* P = F + D * LD;                     // [kPanel][LP]  panel columns
  double* G = P + kPanel * LP;                // [kPanel][LP]  ... over their pivots
  double* pivots = G + kPanel * LP;           // [D]
  __shared__ double s_tol;
  constexpr double kDrop = 1e-12;             // share of the largest diagonal entry below which a pivot drops out
  const int tid = threadIdx.x, w = tid >> 5, q = tid & 31, fr = q >> 2, fk = q & 3;
  const double* A = gram + (size_t)blockIdx.x * D * D;
  const double* sm = sum ? sum + (size_t)blockIdx.x * D : nullptr;
  // Tiles (I, J), I >= J, of eight rows by eight columns, the last column of blocks first: those that a step still
  // has to do are the first ones of the list, dealt out to the warps in turn.
  int row0[SLOTS], col0[SLOTS];
  double a[SLOTS][2];
  const double per_n = sm ? scale / n : 0.0;
#pragma unroll
  for (int i = 0; i < SLOTS; ++i) {
    const int t = w + NW * i;
    const int m = (int)((sqrtf((float)(8 * t + 1)) - 1.f) * 0.5f) + 1;   // blocks in the tile's column of blocks
    col0[i] = t < TILES ? kPanel * (NB - m) : -1;
    row0[i] = t < TILES ? kPanel * (NB - m + t - m * (m - 1) / 2) : 0;
  }
  wait_for_previous();                        // (what stands above needs nothing of the kernel before)
  {
    double2 g[SLOTS];
    double sr[SLOTS], s0[SLOTS], s1[SLOTS];
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) {
      const int r = row0[i] + fr, k = max(col0[i], 0) + 2 * fk;
      g[i] = *reinterpret_cast<const double2*>(&A[r * D + k]);
      // the centring needs double precision: the Gram matrix is n mean^2 + scatter
      sr[i] = sm ? sm[r] : 0.0;
      s0[i] = sm ? sm[k] : 0.0;
      s1[i] = sm ? sm[k + 1] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) {
      const int r = row0[i] + fr, k = col0[i] + 2 * fk;
      const double row_term = sr[i] * per_n;
      a[i][0] = fma(-row_term, s0[i], g[i].x * scale);
      a[i][1] = fma(-row_term, s1[i], g[i].y * scale);
      if (col0[i] >= 0) {                       // (a slot without a tile holds entries of another one's)
        if (k == r) pivots[r] = a[i][0];
        if (k + 1 == r) pivots[r] = a[i][1];
      }
    }
  }
  __syncthreads();
  if (tid < 32) {
    double mx = 0.0;
    for (int t = tid; t < D; t += 32) mx = max(mx, pivots[t]);
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (tid == 0) s_tol = kDrop * mx;
  }
#pragma unroll 1
  for (int p0 = 0; p0 < D; p0 += kPanel) {
    // the panel's columns, from their owners to shared memory
#pragma unroll
    for (int i = 0; i < SLOTS; ++i)
      if (col0[i] == p0) {
        F[(p0 + 2 * fk) * LD + row0[i] + fr] = a[i][0];
        F[(p0 + 2 * fk + 1) * LD + row0[i] + fr] = a[i][1];
      }
    __syncthreads();
    if (tid < D && (w + 1) * 32 > p0) {
      // row `tid` of the panel, and its 8 x 8 head, which every lane factors for itself
      const double tol = s_tol;
      double head[kPanel][kPanel], x[kPanel];
#pragma unroll
      for (int c = 0; c < kPanel; ++c) {
        x[c] = F[(p0 + c) * LD + tid];
#pragma unroll
        for (int k = c; k < kPanel; ++k) head[c][k] = F[(p0 + c) * LD + p0 + k];
      }
      __syncwarp();
#pragma unroll
      for (int c = 0; c < kPanel; ++c) {
        const double pivot = head[c][c];
        const double ip = pivot > tol ? reciprocal(pivot) : 0.0;
        const double f = x[c] * ip;
#pragma unroll
        for (int j = c + 1; j < kPanel; ++j) {
          const double fj = head[c][j] * ip;
#pragma unroll
          for (int k = c + 1; k <= j; ++k) head[k][j] = fma(-fj, head[c][k], head[k][j]);
          x[j] = fma(-f, head[c][j], x[j]);
        }
        P[c * LP + tid] = x[c];
        G[c * LP + tid] = -f;
        if (tid >= p0 + kPanel) F[(p0 + c) * LD + tid] = x[c];
        if (tid == p0 + c) pivots[tid] = pivot > tol ? pivot : 0.0;
      }
    }
    __syncthreads();
    if (tid < kPanel * kPanel) F[(p0 + tid / kPanel) * LD + p0 + tid % kPanel] = P[(tid / kPanel) * LP + p0 + tid % kPanel];
    // trailing block, by groups of a warp's tiles without a branch in between (tiles that are done take anything)
    constexpr int GROUP = D == 64 ? SLOTS : 3;
#pragma unroll
    for (int i0 = 0; i0 < SLOTS; i0 += GROUP) {
      if (col0[i0] <= p0) break;
#pragma unroll
      for (int i = i0; i < i0 + GROUP && i < SLOTS; ++i) {
        mma_f64(a[i], G[fk * LP + row0[i] + fr], P[fk * LP + max(col0[i], 0) + fr]);
        mma_f64(a[i], G[(4 + fk) * LP + row0[i] + fr], P[(4 + fk) * LP + max(col0[i], 0) + fr]);
      }
    }
  }
  let_next_start();
  __syncthreads();
  if (tid < D) pivots[tid] = pivots[tid] > 0.0 ? rsqrt(pivots[tid]) : 0.0;
  __syncthreads();
  const size_t mat = (size_t)blockIdx.x * D * D;
#pragma unroll 8
  for (int e = tid; e < D * D; e += NT) {
    const int r = e / D, k = e % D;
    const double v = k <= r ? F[k * LD + r] * pivots[k] : 0.0;
    out64[mat + e] = v;
    if (out32) out32[mat + e] = (float)v;
  }
  if (wt_hi) {                                // F^T [out k][in r] = F[r][k] as bf16 hi + lo
#pragma unroll 8
    for (int e = tid; e < D * D; e += NT) {
      const int k = e / D, r = e % D;
      const float vf = k <= r ? (float)(F[k * LD + r] * pivots[k]) : 0.f;
      const __nv_bfloat16 h = __float2bfloat16_rn(vf);
      wt_hi[mat + e] = h;
      wt_lo[mat + e] = __float2bfloat16_rn(vf - __bfloat162float(h));
    }
  }
}

int launch_cholesky_factor(const double* gram, const double* sum, double n, double scale, int count, int D,
                           double* out64, float* out32, void* wt_hi, void* wt_lo, LaunchStream st) {
  __nv_bfloat16* hi = static_cast<__nv_bfloat16*>(wt_hi);
  __nv_bfloat16* lo = static_cast<__nv_bfloat16*>(wt_lo);
  const size_t smem = sizeof(double) * ((size_t)D * (D + 1) + 2 * kPanel * (D + 8) + D);
  auto k = D == 64 ? cholesky_factor_kernel<64> : cholesky_factor_kernel<128>;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  launch_chained(k, count, 4 * D, smem, st, gram, sum, n, scale, out64, out32, hi, lo);
  CA_LAUNCH_CHECK();
  return CA_OK;
}

// ---------------------------------------------------------------------------
// d x d algebra in double (one CTA per problem unless noted).
// ---------------------------------------------------------------------------
// M = gramQ / n_q ;  C_K = (gramK - sumK sumK^T / n_k) ck_scale   (centred scatter), rounded to float
__global__ void metric_kernel(const double* __restrict__ gramQ, const double* __restrict__ gramK,
                              const double* __restrict__ sumK, int D, double n_q, double n_k,
                              double ck_scale, float* __restrict__ M, float* __restrict__ CK) {
  wait_for_previous();
  let_next_start();
  const int p = blockIdx.y;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= D * D) return;
  const int i = e / D, j = e % D;
  const size_t o = (size_t)p * D * D + e;
  M[o] = (float)(gramQ[o] / n_q);
  CK[o] = (float)((gramK[o] - sumK[(size_t)p * D + i] * sumK[(size_t)p * D + j] / n_k) * ck_scale);
}

int launch_metric(const double* gramQ, const double* gramK, const double* sumK, int P, int D, int n_q,
                  int n_k, double ck_scale, float* M, float* CK, LaunchStream st) {
  launch_chained(metric_kernel, dim3(ceil_div(D * D, 256), P), 256, 0, st, gramQ, gramK, sumK, D, (double)n_q,
                 (double)n_k, ck_scale, M, CK);
  CA_LAUNCH_CHECK();
  return CA_OK;
}
}  // namespace ca
