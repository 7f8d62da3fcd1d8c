// 8-bit storage of queries, keys and key centroids for the attention variant
// with a quantised Q K^T (Section 3.1: the paper's block-sparse kernel is a
// quantised one).  Scheme: E4M3 codes (4 exponent bits, 3 mantissa bits, largest
// finite value 448), one scale per query row, per key cluster and per run of 64
// key centroids.  A scale maps the largest magnitude of its group to 448; all of
// it in float32 with IEEE operations, so that any implementation gets the same
// codes:  amax = max |x|;  inv = 448 / amax;  s = amax / 448  (both 0 when amax
// is 0);  code = E4M3(x * inv), round to nearest even, saturating.  The logits
// are formed from the codes and multiplied by the two scales afterwards.
#include <cuda_fp8.h>

#include "kernels.h"

namespace ca {

namespace {

// two codes, the first in the low byte (one conversion instruction for both)
__device__ __forceinline__ uint32_t to_e4m3x2(float y0, float y1) {
  return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(y0, y1), __NV_SATFINITE, __NV_E4M3);
}

__device__ __forceinline__ float warp_max(float v) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// A run of 64 key centroids (fp32) per CTA: `live` of them exist, the rest is written as zero codes.
template <int D>
__global__ void __launch_bounds__(256) quantize_centroids_kernel(const float* __restrict__ X, int n_kc, int cen_tiles,
                                                                 unsigned char* __restrict__ codes,
                                                                 float* __restrict__ scales) {
  __shared__ float part[8];
  __shared__ float s_inv;
  const int g = blockIdx.x, p = blockIdx.y;
  const int first = g * 64;
  const int live = min(64, max(0, n_kc - first));
  const float4* src = reinterpret_cast<const float4*>(X + ((size_t)p * n_kc + first) * D);
  uint32_t* dst = reinterpret_cast<uint32_t*>(codes + ((size_t)p * cen_tiles * 64 + first) * D);
  constexpr int VPT = 64 * D / 4 / 256;
  const int n_live = live * D / 4;
  float4 x[VPT];
  float mx = 0.f;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int e = threadIdx.x + v * 256;
    x[v] = e < n_live ? src[e] : make_float4(0.f, 0.f, 0.f, 0.f);
    mx = fmaxf(mx, fmaxf(fmaxf(fabsf(x[v].x), fabsf(x[v].y)), fmaxf(fabsf(x[v].z), fabsf(x[v].w))));
  }
  mx = warp_max(mx);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    float amax = 0.f;
    for (int w = 0; w < 8; ++w) amax = fmaxf(amax, part[w]);
    s_inv = amax > 0.f ? __fdiv_rn(448.f, amax) : 0.f;
    scales[(size_t)p * cen_tiles + g] = amax > 0.f ? __fdiv_rn(amax, 448.f) : 0.f;
  }
  __syncthreads();
  const float inv = s_inv;
#pragma unroll
  for (int v = 0; v < VPT; ++v)
    dst[threadIdx.x + v * 256] = to_e4m3x2(__fmul_rn(x[v].x, inv), __fmul_rn(x[v].y, inv)) |
                                 (to_e4m3x2(__fmul_rn(x[v].z, inv), __fmul_rn(x[v].w, inv)) << 16);
}

// largest magnitude of eight bf16 values (16 bytes), exact
__device__ __forceinline__ __nv_bfloat162 absmax8(const uint4& raw, __nv_bfloat162 m) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&raw);
  return __hmax2(__hmax2(__hmax2(m, __habs2(h[0])), __habs2(h[1])), __hmax2(__habs2(h[2]), __habs2(h[3])));
}
__device__ __forceinline__ float larger(__nv_bfloat162 m) { return fmaxf(__low2float(m), __high2float(m)); }
__device__ __forceinline__ uint2 codes8(const uint4& raw, float inv) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
  uint32_t c[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    c[i] = to_e4m3x2(__fmul_rn(__uint_as_float(w[i] << 16), inv), __fmul_rn(__uint_as_float(w[i] & 0xffff0000u), inv));
  return make_uint2(c[0] | (c[1] << 16), c[2] | (c[3] << 16));
}

// One key cluster (c_k rows of D bf16) per CTA of 256 threads: the rows are read once with 16-byte
// loads and stay in registers between the maximum and the codes (c_k * D / 2048 vectors per thread).
template <int D, int VPT>
__global__ void __launch_bounds__(256) quantize_clusters_kernel(const __nv_bfloat16* __restrict__ X, int c_k,
                                                                unsigned char* __restrict__ codes,
                                                                float* __restrict__ scales) {
  __shared__ float part[8];
  __shared__ float s_inv;
  const size_t group = blockIdx.x;                                   // cluster index over all problems
  const uint4* src = reinterpret_cast<const uint4*>(X + group * (size_t)c_k * D);
  uint2* dst = reinterpret_cast<uint2*>(codes + group * (size_t)c_k * D);
  const int n_vec = c_k * D / 8;
  uint4 x[VPT];
  __nv_bfloat162 m = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int e = threadIdx.x + v * 256;
    x[v] = e < n_vec ? src[e] : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int v = 0; v < VPT; ++v) m = absmax8(x[v], m);
  const float mx = warp_max(larger(m));
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    float amax = 0.f;
    for (int w = 0; w < 8; ++w) amax = fmaxf(amax, part[w]);
    s_inv = amax > 0.f ? __fdiv_rn(448.f, amax) : 0.f;
    scales[group] = amax > 0.f ? __fdiv_rn(amax, 448.f) : 0.f;
  }
  __syncthreads();
  const float inv = s_inv;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int e = threadIdx.x + v * 256;
    if (e < n_vec) dst[e] = codes8(x[v], inv);
  }
}

// Query rows, 16 threads per row (8 values each), four rows per thread and 64 per CTA, so that four loads are in
// flight (with one row per thread and one conversion per value the whole preparation of 40 heads of 32,760 rows
// took 295 us and takes 177, 1.0 GB read and written).
template <int D>
__global__ void __launch_bounds__(256) quantize_rows_kernel(const __nv_bfloat16* __restrict__ X, size_t n_rows,
                                                            unsigned char* __restrict__ codes,
                                                            float* __restrict__ scales) {
  static_assert(D == 128, "one 16-byte vector per thread, 16 threads per row");
  const size_t row0 = (size_t)blockIdx.x * 64 + (threadIdx.x >> 4);
  const int sub = threadIdx.x & 15;
  uint4 x[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const size_t row = row0 + 16 * u;
    x[u] = row < n_rows ? reinterpret_cast<const uint4*>(X + row * D)[sub] : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const size_t row = row0 + 16 * u;
    float mx = larger(absmax8(x[u], __floats2bfloat162_rn(0.f, 0.f)));
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (row >= n_rows) continue;
    const float inv = mx > 0.f ? __fdiv_rn(448.f, mx) : 0.f;
    if (sub == 0) scales[row] = mx > 0.f ? __fdiv_rn(mx, 448.f) : 0.f;
    reinterpret_cast<uint2*>(codes + row * D)[sub] = codes8(x[u], inv);
  }
}

}  // namespace

// Qp [P * n_qc * c_q, D] -> codes + one scale per row; Kp [P, n_kc * c_k, D] -> codes + one scale per
// cluster; ck [P, n_kc, D] fp32 -> codes [P, cen_tiles * 64, D] (zero rows behind the last centroid)
// + one scale per run of 64.
int launch_quantize_qk(const void* Qp, const void* Kp, const float* ck, int P, int n_qc, int c_q, int n_kc, int c_k,
                       int cen_tiles, int D, unsigned char* q8, float* sq, unsigned char* k8, float* sk,
                       unsigned char* c8, float* sc, LaunchStream st) {
  if (D != 128) return CA_ERR_UNSUPPORTED;
  const size_t q_rows = (size_t)P * n_qc * c_q;
  quantize_rows_kernel<128><<<(unsigned)((q_rows + 63) / 64), 256, 0, st>>>(static_cast<const __nv_bfloat16*>(Qp), q_rows, q8, sq);
  CA_LAUNCH_CHECK();
  const __nv_bfloat16* kp = static_cast<const __nv_bfloat16*>(Kp);
  const unsigned clusters = (unsigned)((size_t)P * n_kc);
  if (c_k == 64) quantize_clusters_kernel<128, 4><<<clusters, 256, 0, st>>>(kp, c_k, k8, sk);
  else if (c_k == 128) quantize_clusters_kernel<128, 8><<<clusters, 256, 0, st>>>(kp, c_k, k8, sk);
  else if (c_k == 256) quantize_clusters_kernel<128, 16><<<clusters, 256, 0, st>>>(kp, c_k, k8, sk);
  else return CA_ERR_UNSUPPORTED;
  CA_LAUNCH_CHECK();
  if (ck) {
    quantize_centroids_kernel<128><<<dim3(cen_tiles, P), 256, 0, st>>>(ck, n_kc, cen_tiles, c8, sc);
    CA_LAUNCH_CHECK();
  }
  return CA_OK;
}

}  // namespace ca
