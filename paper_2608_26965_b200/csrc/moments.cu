// Second moments of row sets and row transforms (Section 3.2.2: metric matrices
// Q^T Q and K_c^T K_c; Section 3.2.1: covariance for the global principal
// components; projection of the rows).
#include "kernels.h"

namespace ca {

// ---------------------------------------------------------------------------
// Gram matrix and column sums of a chunk of rows.  One CTA per (chunk, problem),
// 256 threads; thread (ti, tj) owns a TM x TM tile of the D x D result.
// partial[(p * n_chunks + chunk) * (D*D + D)] : D*D Gram (row-major) then D sums.
// ---------------------------------------------------------------------------
template <typename T, int D>
__global__ void __launch_bounds__(256) gram_chunk_kernel(const T* __restrict__ X, int n_rows,
                                                         int chunk_rows, int n_chunks,
                                                         float* __restrict__ partial) {
  wait_for_previous();
  constexpr int TR = 32;            // rows staged per step
  constexpr int TM = D / 16;        // 4 (D=64) or 8 (D=128)
  __shared__ __align__(16) float xs[TR][D + 4];
  const int p = blockIdx.y, chunk = blockIdx.x;
  const T* Xp = X + (size_t)p * n_rows * D;
  const int r_begin = chunk * chunk_rows;
  const int r_end = min(n_rows, r_begin + chunk_rows);
  const int ti = threadIdx.x / 16, tj = threadIdx.x % 16;
  float acc[TM][TM];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) acc[i][j] = 0.f;
  float colsum = 0.f;
  for (int r0 = r_begin; r0 < r_end; r0 += TR) {
    const int nr = min(TR, r_end - r0);
#pragma unroll
    for (int i = 0; i < TR * D / 1024; ++i) {
      const int e = threadIdx.x + 256 * i, r = e / (D / 4), col = 4 * (e % (D / 4));
      *reinterpret_cast<float4*>(&xs[r][col]) =
          (r < nr) ? load4(Xp + (size_t)(r0 + r) * D + col) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
#pragma unroll 4
    for (int r = 0; r < TR; ++r) {
      float a[TM], b[TM];
#pragma unroll
      for (int i = 0; i < TM; i += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&xs[r][ti * TM + i]);
        a[i] = v.x; a[i + 1] = v.y; a[i + 2] = v.z; a[i + 3] = v.w;
      }
      // columns 4 tj + 64 g of a thread: its neighbours' loads are next to its own
#pragma unroll
      for (int j = 0; j < TM; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&xs[r][4 * tj + 16 * j]);
        b[j] = v.x; b[j + 1] = v.y; b[j + 2] = v.z; b[j + 3] = v.w;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (threadIdx.x < D) {
#pragma unroll 8
      for (int r = 0; r < TR; ++r) colsum += xs[r][threadIdx.x];
    }
    __syncthreads();
  }
  let_next_start();
  float* out = partial + ((size_t)p * n_chunks + chunk) * (D * D + D);
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) out[(ti * TM + i) * D + 4 * tj + 16 * (j & ~3) + (j & 3)] = acc[i][j];
  if (threadIdx.x < D) out[D * D + threadIdx.x] = colsum;
}

// Sums the chunk partials in a fixed order, in double.
__global__ void gram_finalize_kernel(const float* __restrict__ partial, int n_chunks, int elems,
                                     double* __restrict__ gram, double* __restrict__ colsum,
                                     int dd) {
  wait_for_previous();
  let_next_start();
  const int p = blockIdx.y;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= elems) return;
  const float* src = partial + (size_t)p * n_chunks * elems + e;
  double s = 0.0;
  for (int c = 0; c < n_chunks; ++c) s += (double)src[(size_t)c * elems];
  if (e < dd) gram[(size_t)p * dd + e] = s;
  else colsum[(size_t)p * (elems - dd) + (e - dd)] = s;
}

int moments_chunking(int n_rows, int problems, int* chunk_rows, int* n_chunks) {
  long long target = ((long long)n_rows * problems + 1183) / 1184;   // ~8 CTAs per SM
  int cr = (int)((target + 63) / 64 * 64);
  // chunks of 64 rows where there are few rows: 4 heads of 5,003 rows at d = 128 took 75 us in 80 CTAs
  // of 256 rows and take 46 in 316
  if (cr < 64) cr = 64;
  if (cr > 8192) cr = 8192;
  *chunk_rows = cr;
  *n_chunks = ceil_div(n_rows, cr);
  return 0;
}

int launch_gram_finalize(const float* partial, int problems, int n_chunks, int D, double* gram,
                         double* colsum, LaunchStream st) {
  const int elems = D * D + D;
  launch_chained(gram_finalize_kernel, dim3(ceil_div(elems, 256), problems), 256, 0, st, partial, n_chunks, elems, gram,
                 colsum, D * D);
  CA_LAUNCH_CHECK();
  return CA_OK;
}

template <typename T>
static int launch_moments_t(const T* X, int problems, int n_rows, int D, float* partial,
                            double* gram, double* colsum, LaunchStream st) {
  int chunk_rows, n_chunks;
  moments_chunking(n_rows, problems, &chunk_rows, &n_chunks);
  dim3 grid(n_chunks, problems);
  auto k = D == 64 ? gram_chunk_kernel<T, 64> : gram_chunk_kernel<T, 128>;
  launch_chained(k, grid, 256, 0, st, X, n_rows, chunk_rows, n_chunks, partial);
  CA_LAUNCH_CHECK();
  return launch_gram_finalize(partial, problems, n_chunks, D, gram, colsum, st);
}

int launch_moments(const void* X, int dtype, int problems, int n_rows, int D, float* partial,
                   double* gram, double* colsum, LaunchStream st) {
  if (dtype == CA_DTYPE_BF16)
    return launch_moments_t(static_cast<const __nv_bfloat16*>(X), problems, n_rows, D, partial, gram, colsum, st);
  return launch_moments_t(static_cast<const float*>(X), problems, n_rows, D, partial, gram, colsum, st);
}

// ---------------------------------------------------------------------------
// Row transform: out[r,:] = g(X[r,:] W + b), W [D,D] row-major fp32, b [D] (may
// be null).  g = identity, or division by the row's Euclidean norm (rows whose
// norm is below 1e-30 map to zero).  Output fp32.  One CTA per 64 rows.
// ---------------------------------------------------------------------------
// Bound by the fp32 pipe and the shared-memory loads in front of it: a thread computes 4 rows by 4 (d = 64) or
// 8 (d = 128) columns from 16-byte loads, 12 of them per 128 multiply-adds; the results are staged over
// the rows they came from, so that two CTAs share an SM at d = 128 (4 heads of 5,003 rows: 54 -> 33 us).
template <typename T, int D>
__global__ void __launch_bounds__(256) transform_rows_kernel(const T* __restrict__ X, int n_rows,
                                                             const float* __restrict__ W,
                                                             const float* __restrict__ bias,
                                                             int normalize, float* __restrict__ out) {
  constexpr int TR = 64;
  constexpr int LD = D + 4;
  constexpr int CG = D / 64;              // groups of four columns per thread (4 tc + 64 g), rows per thread = 4
  extern __shared__ __align__(16) float smem[];
  float* Ws = smem;                       // [D][D]
  float* xs = Ws + D * D;                 // [TR][LD]  rows, then results
  __shared__ float inv_norm[TR];
  wait_for_previous();
  const int p = blockIdx.y;
  const int r0 = blockIdx.x * TR;
  const int nr = min(TR, n_rows - r0);
  const T* Xp = X + (size_t)p * n_rows * D;
  const float* Wp = W + (size_t)p * D * D;
#pragma unroll 4
  for (int e = threadIdx.x; e < D * D / 4; e += 256)
    *reinterpret_cast<float4*>(&Ws[4 * e]) = *reinterpret_cast<const float4*>(&Wp[4 * e]);
#pragma unroll 4
  for (int e = threadIdx.x; e < TR * D / 4; e += 256) {
    const int r = e / (D / 4), col = 4 * (e % (D / 4));
    *reinterpret_cast<float4*>(&xs[r * LD + col]) =
        (r < nr) ? load4(Xp + (size_t)(r0 + r) * D + col) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  const int tr = threadIdx.x / 16;        // 16 row groups of 4 rows
  const int tc = threadIdx.x % 16;
  float acc[4][CG][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int g = 0; g < CG; ++g)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][g][c] = 0.f;
#pragma unroll 2
  for (int k = 0; k < D; k += 4) {
    float4 a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(&xs[(tr * 4 + i) * LD + k]);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
      for (int g = 0; g < CG; ++g) {
        const float4 b = *reinterpret_cast<const float4*>(&Ws[(k + kk) * D + 64 * g + 4 * tc]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float x = kk == 0 ? a[i].x : kk == 1 ? a[i].y : kk == 2 ? a[i].z : a[i].w;
          acc[i][g][0] = fmaf(x, b.x, acc[i][g][0]); acc[i][g][1] = fmaf(x, b.y, acc[i][g][1]);
          acc[i][g][2] = fmaf(x, b.z, acc[i][g][2]); acc[i][g][3] = fmaf(x, b.w, acc[i][g][3]);
        }
      }
  }
  __syncthreads();                        // the rows have been read
  const float* bp = bias ? bias + (size_t)p * D : nullptr;
#pragma unroll
  for (int g = 0; g < CG; ++g) {
    const float4 b = bp ? *reinterpret_cast<const float4*>(&bp[64 * g + 4 * tc]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<float4*>(&xs[(tr * 4 + i) * LD + 64 * g + 4 * tc]) =
          make_float4(acc[i][g][0] + b.x, acc[i][g][1] + b.y, acc[i][g][2] + b.z, acc[i][g][3] + b.w);
  }
  __syncthreads();
  if (normalize) {
    // 4 threads per row, fixed summation order
    const int r = threadIdx.x / 4, q = threadIdx.x % 4;
    float s = 0.f;
    for (int col = q; col < D; col += 4) { float v = xs[r * LD + col]; s = fmaf(v, v, s); }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (q == 0) { float n = sqrtf(s); inv_norm[r] = (n >= 1e-30f) ? 1.f / n : 0.f; }
    __syncthreads();
  }
  float* op = out + ((size_t)p * n_rows + r0) * D;
#pragma unroll 4
  for (int e = threadIdx.x; e < nr * D / 4; e += 256) {
    const int r = e / (D / 4), col = 4 * (e % (D / 4));
    float4 v = *reinterpret_cast<const float4*>(&xs[r * LD + col]);
    if (normalize) { const float s = inv_norm[r]; v.x *= s; v.y *= s; v.z *= s; v.w *= s; }
    *reinterpret_cast<float4*>(&op[(size_t)r * D + col]) = v;
  }
}

template <typename T>
static int launch_transform_t(const T* X, int problems, int n_rows, int D, const float* W,
                              const float* bias, int normalize, float* out, LaunchStream st) {
  dim3 grid(ceil_div(n_rows, 64), problems);
  size_t smem = (size_t)(D * D + 64 * (D + 4)) * sizeof(float);
  if (D == 64) {
    auto k = transform_rows_kernel<T, 64>;
    CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    launch_chained(k, grid, 256, smem, st, X, n_rows, W, bias, normalize, out);
  } else {
    auto k = transform_rows_kernel<T, 128>;
    CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    launch_chained(k, grid, 256, smem, st, X, n_rows, W, bias, normalize, out);
  }
  CA_LAUNCH_CHECK();
  return CA_OK;
}

int launch_transform_rows(const void* X, int dtype, int problems, int n_rows, int D, const float* W,
                          const float* bias, int normalize, float* out, LaunchStream st) {
  if (dtype == CA_DTYPE_BF16)
    return launch_transform_t(static_cast<const __nv_bfloat16*>(X), problems, n_rows, D, W, bias, normalize, out, st);
  return launch_transform_t(static_cast<const float*>(X), problems, n_rows, D, W, bias, normalize, out, st);
}

}  // namespace ca
