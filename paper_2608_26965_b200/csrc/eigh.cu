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
// The elimination goes by panels of eight columns.  One warp factors a panel with its rows in
// registers and shuffles instead of barriers (the chain of a column: pivot, reciprocal, update), then all
// threads take the eight columns off the trailing block at once: two barriers per eight columns.  With a
// column and a barrier of 1,024 threads per step, and the one division of the step in its chain, a factor
// took 26 us at d = 64 and 59 us at d = 128 (per launch); now 17.5 and 50.  Warp w keeps the entries (w + NW a, q + 32 b) of the trailing block in
// registers, rows dealt out cyclically, so that the shrinking block stays spread over all warps and tests on
// rows are uniform; finished columns stay in shared memory, unscaled, and are scaled by 1 / sqrt(pivot)
// on the way out.  The trailing block takes A[r][k] -= A[r][j] A[k][j] / pivot_j with the unscaled columns;
// a dropped pivot (reciprocal 0) leaves it alone and gives a zero column.
// ---------------------------------------------------------------------------
constexpr int kPanel = 8;

// reciprocal by Newton's iteration on the hardware's estimate (relative error of a few 1e-16)
__device__ __forceinline__ double reciprocal(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

template <int D>
__global__ void __launch_bounds__(4 * D) cholesky_factor_kernel(const double* __restrict__ gram,
                                                                const double* __restrict__ sum, double n,
                                                                double scale, double* __restrict__ out64,
                                                                float* __restrict__ out32,
                                                                __nv_bfloat16* __restrict__ wt_hi,
                                                                __nv_bfloat16* __restrict__ wt_lo) {
  constexpr int NT = 4 * D, NW = NT / 32;
  constexpr int RT = D / NW, CT = D / 32;     // rows and columns of a thread's tile
  constexpr int LD = D + 1;                   // pitch of a column
  extern __shared__ __align__(16) double chol_smem[];
  double* F = chol_smem;                      // [D][LD]  finished columns and the panel, column-major, unscaled
  double* G = F + D * LD;                     // [kPanel][D]  panel columns over their pivots
  double* pivots = G + kPanel * D;            // [D]
  __shared__ double s_tol;
  constexpr double kDrop = 1e-12;             // share of the largest diagonal entry below which a pivot drops out
  wait_for_previous();
  const int tid = threadIdx.x, w = tid >> 5, q = tid & 31;
  const double* A = gram + (size_t)blockIdx.x * D * D;
  const double* sm = sum ? sum + (size_t)blockIdx.x * D : nullptr;
  double a[RT][CT];
  const double per_n = sm ? scale / n : 0.0;
#pragma unroll
  for (int ta = 0; ta < RT; ++ta) {
    const int r = w + NW * ta;
    // the centring needs double precision: the Gram matrix is n mean^2 + scatter
    const double row_term = sm ? sm[r] * per_n : 0.0;
#pragma unroll
    for (int tb = 0; tb < CT; ++tb) {
      const int k = q + 32 * tb;
      a[ta][tb] = 0.0;
      if (k <= r) a[ta][tb] = sm ? fma(-row_term, sm[k], A[r * D + k] * scale) : A[r * D + k] * scale;
      if (k == r) pivots[r] = a[ta][tb];
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
    const int b0 = p0 >> 5, at = q - (p0 & 31);
    if (at >= 0 && at < kPanel) {
#pragma unroll
      for (int ta = 0; ta < RT; ++ta) {
        double v = a[ta][0];
#pragma unroll
        for (int tb = 1; tb < CT; ++tb) v = tb == b0 ? a[ta][tb] : v;
        F[(p0 + at) * LD + w + NW * ta] = v;
      }
    }
    __syncthreads();
    if (w == 0) {
      const double tol = s_tol;
      double x[CT][kPanel];                   // rows q + 32 s
#pragma unroll
      for (int s = 0; s < CT; ++s)
#pragma unroll
        for (int c = 0; c < kPanel; ++c) x[s][c] = F[(p0 + c) * LD + q + 32 * s];
#pragma unroll
      for (int c = 0; c < kPanel; ++c) {
        // rows p0 .. p0 + 7 of the panel lie in slot b0 of eight neighbouring lanes
        double own = x[0][c];
#pragma unroll
        for (int s = 1; s < CT; ++s) own = s == b0 ? x[s][c] : own;
        const double pivot = __shfl_sync(0xffffffffu, own, (p0 + c) & 31);
        double head[kPanel];
#pragma unroll
        for (int k = c + 1; k < kPanel; ++k) head[k] = __shfl_sync(0xffffffffu, own, (p0 + k) & 31);
        const double ip = pivot > tol ? reciprocal(pivot) : 0.0;
#pragma unroll
        for (int s = 0; s < CT; ++s) {
          const double f = x[s][c] * ip;
#pragma unroll
          for (int k = c + 1; k < kPanel; ++k) x[s][k] = fma(-f, head[k], x[s][k]);
          F[(p0 + c) * LD + q + 32 * s] = x[s][c];
          G[c * D + q + 32 * s] = f;
        }
        if (q == 0) pivots[p0 + c] = pivot > tol ? pivot : 0.0;
      }
    }
    __syncthreads();
    // trailing block: columns from p0 + 8 on
#pragma unroll
    for (int half = 0; half < kPanel; half += 4) {
      double cv[CT][4];
#pragma unroll
      for (int tb = 0; tb < CT; ++tb)
#pragma unroll
        for (int c = 0; c < 4; ++c) cv[tb][c] = q + 32 * tb >= p0 + kPanel ? F[(p0 + half + c) * LD + q + 32 * tb] : 0.0;
#pragma unroll
      for (int ta = 0; ta < RT; ++ta) {
        const int r = w + NW * ta;
        if (r < p0 + kPanel) continue;        // uniform over the warp
        double f[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) f[c] = G[(half + c) * D + r];
#pragma unroll
        for (int tb = 0; tb < CT; ++tb) {
          if (32 * tb > r || 32 * tb + 31 < p0 + kPanel) continue;   // uniform: above the diagonal, or finished
#pragma unroll
          for (int c = 0; c < 4; ++c) a[ta][tb] = fma(-f[c], cv[tb][c], a[ta][tb]);
        }
      }
    }
  }
  let_next_start();
  __syncthreads();
  if (tid < D) pivots[tid] = pivots[tid] > 0.0 ? rsqrt(pivots[tid]) : 0.0;
  __syncthreads();
  const size_t mat = (size_t)blockIdx.x * D * D;
#pragma unroll 4
  for (int e = tid; e < D * D; e += NT) {
    const int r = e / D, k = e % D;
    const double v = k <= r ? F[k * LD + r] * pivots[k] : 0.0;
    out64[mat + e] = v;
    if (out32) out32[mat + e] = (float)v;
  }
  if (wt_hi) {                                // F^T [out k][in r] = F[r][k] as bf16 hi + lo
#pragma unroll 4
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
  const size_t smem = sizeof(double) * ((size_t)D * (D + 1) + kPanel * D + D);
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
