// FP32 CUDA-core kernel for block-sparse attention with striped
// mean-compensation (eq. 2 over the selected clusters; Appendix A: an excluded
// cluster enters through its centroid key and value with weight
// |c| exp(q . kbar / sqrt(d)), in numerator and denominator).
// Serves fp32 storage, unusual cluster sizes, and as an on-device cross-check of
// the tensor-core kernel.  Flash-style online softmax, fp32 throughout.
//
// Bound by the fp32 pipe and by what feeds it from shared memory: 16 threads share RY = 4 query
// rows, a thread computes 4 x 2 scores and 4 x D / 16 outputs, so that six 16-byte loads feed 32 (scores)
// and 12 feed 128 (outputs) multiply-adds; the rows of the next tile of keys are fetched from global memory
// while a tile is computed.  4 heads of 5,003 rows, d = 128, 5 of 40 clusters of 128 kept: 0.80 ->
// 0.36 ms; 2 heads of 1,024 rows, d = 64: 49 -> 26 us (before: 16 query rows per CTA, scalar loads).
// A CTA takes 64 query rows where that still gives every SM one, otherwise 32; of a query cluster of 16
// rows it takes those, with RY = 2: in a tile of 32 half of the threads computed nothing, and calls with such
// clusters took up to 1.4 times as long as with the scalar kernel (60 shapes: 1.00 of its speed in the mean, 0.71 at worst; with the narrow
// tile 1.37 and 0.99, with RY = 4 in it 1.35 and 0.94).
#include "kernels.h"

namespace ca {

constexpr int kRefKT = 32;       // keys per staged tile
// Key clusters that the bitmap of the selected ones covers at a time (128 KB, beside the widest tile), so that their number
// has no bound in shared memory.  With more of them (`many`, an instance of its own: moving the window costs the others
// registers) the bitmap is set anew per window; a second pass never has as many (the tensor-core kernel takes an eighth).
constexpr int kRefWindow = 1 << 20;

template <typename T, int D, int QR, int RY, bool many>
__global__ void __launch_bounds__(16 * QR / RY)
attn_ref_kernel(const T* __restrict__ Qp, const T* __restrict__ Kp, const T* __restrict__ Vp,
                const float* __restrict__ ck, const float* __restrict__ cv,
                const int32_t* __restrict__ count_k, const int32_t* __restrict__ block_idx,
                const int32_t* __restrict__ keep_count, int list_stride,
                const int32_t* __restrict__ perm_q, int n_q, int n_k, int c_q, int c_k, int keep_all,
                int compensate, float scale, T* __restrict__ O, float* __restrict__ lse,
                int* __restrict__ status, const int32_t* __restrict__ redo, int redo_tiles,
                int* __restrict__ redo_count, int per_cta, int n_clusters) {
  wait_for_previous();
  constexpr int NT = 16 * QR / RY;       // threads: 16 per RY query rows
  constexpr int LD = D + 4;              // row pitch: rows of eight threads in distinct banks
  constexpr int LP = kRefKT + 4;
  constexpr int CG = D / 64;             // groups of four output columns per thread
  constexpr int KI = kRefKT / 16;        // keys per thread
  constexpr int PF = kRefKT * D / 4 / NT;   // float4 of keys (of values) per thread and tile
  extern __shared__ __align__(16) float smem[];
  float* qs = smem;                      // [QR][LD]
  float* ks = qs + QR * LD;              // [KT][LD]
  float* vs = ks + kRefKT * LD;          // [KT][LD]
  float* ps = vs + kRefKT * LD;          // [QR][LP]
  float* bias = ps + QR * LP;            // [KT] per-key additive term (ln|c| or -inf)
  unsigned* selected = reinterpret_cast<unsigned*>(bias + kRefKT);   // bitmap over a window of key clusters

  const int n_qc = (n_q + c_q - 1) / c_q, n_kc = (n_k + c_k - 1) / c_k;
  const int tiles_per_cluster = (c_q + QR - 1) / QR;
  const int tid = threadIdx.x;
  const int tr = tid >> 4, tc = tid & 15;
  // first pass of a problem: one CTA per tile of QR query rows.  Second pass behind the
  // tensor-core kernel (`redo` given): a CTA looks at `per_cta` query clusters, returns at once unless one
  // of them is marked ([B*H, n_qc, 2]) and otherwise walks over the tiles of the marked ones.
  if (redo) {
    const int g = blockIdx.x * per_cta + tid;
    bool marked = false;
    if (tid < per_cta && g < n_clusters)
      for (int t = 0; t < redo_tiles; ++t) marked |= redo[(size_t)g * 2 + t] != 0;
    if (!__syncthreads_or(marked)) return;
  }
#pragma unroll 1
  for (int turn = 0; turn < per_cta; ++turn) {
  const int g = redo ? blockIdx.x * per_cta + turn : 0;
  if (redo) {
    if (g >= n_clusters) break;
    bool marked = false;
    for (int t = 0; t < redo_tiles; ++t) marked |= redo[(size_t)g * 2 + t] != 0;
    if (!marked) continue;                                  // uniform over the CTA
    if (tid == 0 && redo_count) atomicAdd(redo_count, 1);   // statistics: clusters recomputed
    __syncthreads();                                        // the cluster before is done with the shared arrays
  }
  const int p = redo ? g / n_qc : blockIdx.y;
  const int qc = redo ? g % n_qc : blockIdx.x / tiles_per_cluster;
  const int r0_first = redo ? 0 : (blockIdx.x % tiles_per_cluster) * QR;
  const int r0_end = redo ? c_q : r0_first + QR;
  const size_t q_base = ((size_t)p * n_qc + qc) * (size_t)c_q;
  const T* Kh = Kp + (size_t)p * n_kc * (size_t)c_k * D;
  const T* Vh = Vp + (size_t)p * n_kc * (size_t)c_k * D;
  const float* ckh = ck + (size_t)p * n_kc * D;
  const float* cvh = cv + (size_t)p * n_kc * D;
  const int32_t* sel = block_idx + ((size_t)p * n_qc + qc) * list_stride;
  int keep = keep_count ? keep_count[(size_t)p * n_qc + qc] : keep_all;   // ragged lists carry their length
  // indices from the caller are range-checked before use: a bad one sets CA_ERR_BAD_INDEX (6) in the
  // status word and is skipped (a list length is clamped to its row, a cluster that does not exist
  // is left out, a row of O that does not exist is not written)
  if (keep < 0 || keep > list_stride) {
    if (tid == 0) atomicCAS(status, 0, 6);
    keep = keep < 0 ? 0 : list_stride;
  }
  const int32_t* cnt = count_k + (size_t)p * n_kc;

  auto mark = [&](int first) {             // the selected ones among the clusters [first, first + kRefWindow)
    const int words = many ? kRefWindow / 32 : (n_kc + 31) / 32;
    for (int w = tid; w < words; w += NT) selected[w] = 0u;
    __syncthreads();
    for (int t = tid; t < keep; t += NT) {
      const int j = sel[t];
      if (j < 0 || j >= n_kc) atomicCAS(status, 0, 6);
      else if (!many || (j >= first && j - first < kRefWindow)) atomicOr(&selected[(j - first) >> 5], 1u << (j & 31));
    }
  };
  mark(0);

  for (int r0 = r0_first; r0 < r0_end; r0 += QR) {
    __syncthreads();                       // the previous tile's readers are done with the staged rows
    for (int e = tid; e < QR * D / 4; e += NT) {
      const int r = e / (D / 4), col = 4 * (e % (D / 4));
      const int pos = qc * c_q + r0 + r;
      const float4 v = (r0 + r < c_q && pos < n_q) ? load4(Qp + (q_base + r0 + r) * D + col) : make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(&qs[r * LD + col]) = v;
    }

    float m_run[RY], l_run[RY], acc[RY][CG][4];
#pragma unroll
    for (int y = 0; y < RY; ++y) {
      m_run[y] = -INFINITY;
      l_run[y] = 0.f;
#pragma unroll
      for (int g = 0; g < CG; ++g)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[y][g][c] = 0.f;
    }

    // Tiles of keys: the members of the selected clusters in list order (t, row t0), then, 32 at a time, the
    // centroids (t = keep, first centroid t0).  `rows` = 0: no tile left.
    int t = 0, t0 = 0, rows = 0, members = 0;
    auto settle = [&]() {                  // the first tile at or behind (t, t0)
      while (t < keep) {
        const int j = sel[t];
        members = (j < 0 || j >= n_kc) ? 0 : min(max(cnt[j], 0), c_k);       // out of range: flagged above
        if (t0 < members) { rows = min(kRefKT, members - t0); return; }
        ++t;
        t0 = 0;
      }
      rows = compensate ? min(kRefKT, n_kc - t0) : 0;
    };
    float4 kf[PF], vf[PF];
    float next_bias = 0.f;
    auto fetch = [&]() {
      const bool cen = t >= keep;
      const size_t base = cen ? (size_t)t0 * D : ((size_t)sel[t] * c_k + t0) * D;
#pragma unroll
      for (int i = 0; i < PF; ++i) {
        const int e = tid + i * NT, r = e / (D / 4), col = 4 * (e % (D / 4));
        kf[i] = vf[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rows) {
          const size_t at = base + (size_t)r * D + col;
          kf[i] = cen ? load4(ckh + at) : load4(Kh + at);
          vf[i] = cen ? load4(cvh + at) : load4(Vh + at);
        }
      }
      if (tid < kRefKT) {
        bool use = tid < rows;
        if (cen && use) {
          const int j = t0 + tid;
          use = !((selected[(many ? j % kRefWindow : j) >> 5] >> (j & 31)) & 1u);
          next_bias = use ? logf((float)cnt[j]) : -INFINITY;
        } else {
          next_bias = use ? 0.f : -INFINITY;
        }
      }
    };
    settle();
    if (rows > 0) fetch();
    while (rows > 0) {
      __syncthreads();                     // the tile before has been read
#pragma unroll
      for (int i = 0; i < PF; ++i) {
        const int e = tid + i * NT, r = e / (D / 4), col = 4 * (e % (D / 4));
        *reinterpret_cast<float4*>(&ks[r * LD + col]) = kf[i];
        *reinterpret_cast<float4*>(&vs[r * LD + col]) = vf[i];
      }
      if (tid < kRefKT) bias[tid] = next_bias;
      __syncthreads();
      t0 += kRefKT;
      rows = 0;
      if (t < keep) settle();
      else rows = max(0, min(kRefKT, n_kc - t0));
      if constexpr (many) {
        if (rows > 0 && t >= keep && t0 > 0 && t0 % kRefWindow == 0) {
          __syncthreads();                 // the window before has been read
          mark(t0);
          __syncthreads();
        }
      }
      if (rows > 0) fetch();

      // scores of rows RY tr + y, keys tc + 16 i
      float s[RY][KI];
#pragma unroll
      for (int y = 0; y < RY; ++y)
#pragma unroll
        for (int i = 0; i < KI; ++i) s[y][i] = 0.f;
#pragma unroll 4
      for (int k = 0; k < D; k += 4) {
        float4 q4[RY], k4[KI];
#pragma unroll
        for (int y = 0; y < RY; ++y) q4[y] = *reinterpret_cast<const float4*>(&qs[(RY * tr + y) * LD + k]);
#pragma unroll
        for (int i = 0; i < KI; ++i) k4[i] = *reinterpret_cast<const float4*>(&ks[(tc + 16 * i) * LD + k]);
#pragma unroll
        for (int y = 0; y < RY; ++y)
#pragma unroll
          for (int i = 0; i < KI; ++i) {
            s[y][i] = fmaf(q4[y].x, k4[i].x, s[y][i]); s[y][i] = fmaf(q4[y].y, k4[i].y, s[y][i]);
            s[y][i] = fmaf(q4[y].z, k4[i].z, s[y][i]); s[y][i] = fmaf(q4[y].w, k4[i].w, s[y][i]);
          }
      }
      // online softmax: the 16 threads of a row are half a warp
      float tmax[RY];
#pragma unroll
      for (int y = 0; y < RY; ++y) {
        tmax[y] = -INFINITY;
#pragma unroll
        for (int i = 0; i < KI; ++i) {
          s[y][i] = s[y][i] * scale + bias[tc + 16 * i];
          tmax[y] = fmaxf(tmax[y], s[y][i]);
        }
      }
#pragma unroll
      for (int o = 1; o < 16; o <<= 1)
#pragma unroll
        for (int y = 0; y < RY; ++y) tmax[y] = fmaxf(tmax[y], __shfl_xor_sync(0xffffffffu, tmax[y], o));
      float psum[RY], alpha[RY];
#pragma unroll
      for (int y = 0; y < RY; ++y) {
        const float m_new = fmaxf(m_run[y], tmax[y]);
        const bool any = m_new > -INFINITY;
        alpha[y] = any ? expf(m_run[y] - m_new) : 1.f;
        psum[y] = 0.f;
#pragma unroll
        for (int i = 0; i < KI; ++i) {
          const float pv = any ? expf(s[y][i] - m_new) : 0.f;
          ps[(RY * tr + y) * LP + tc + 16 * i] = pv;
          psum[y] += pv;
        }
        m_run[y] = m_new;
      }
#pragma unroll
      for (int o = 1; o < 16; o <<= 1)
#pragma unroll
        for (int y = 0; y < RY; ++y) psum[y] += __shfl_xor_sync(0xffffffffu, psum[y], o);
#pragma unroll
      for (int y = 0; y < RY; ++y) {
        l_run[y] = l_run[y] * alpha[y] + psum[y];
#pragma unroll
        for (int g = 0; g < CG; ++g)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[y][g][c] *= alpha[y];
      }
      __syncwarp();
#pragma unroll 2
      for (int key = 0; key < kRefKT; key += 4) {
        float4 p4[RY];
#pragma unroll
        for (int y = 0; y < RY; ++y) p4[y] = *reinterpret_cast<const float4*>(&ps[(RY * tr + y) * LP + key]);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int g = 0; g < CG; ++g) {
            const float4 v4 = *reinterpret_cast<const float4*>(&vs[(key + kk) * LD + 64 * g + 4 * tc]);
#pragma unroll
            for (int y = 0; y < RY; ++y) {
              const float pv = kk == 0 ? p4[y].x : kk == 1 ? p4[y].y : kk == 2 ? p4[y].z : p4[y].w;
              acc[y][g][0] = fmaf(pv, v4.x, acc[y][g][0]); acc[y][g][1] = fmaf(pv, v4.y, acc[y][g][1]);
              acc[y][g][2] = fmaf(pv, v4.z, acc[y][g][2]); acc[y][g][3] = fmaf(pv, v4.w, acc[y][g][3]);
            }
          }
      }
    }

#pragma unroll
    for (int y = 0; y < RY; ++y) {
      const int row = r0 + RY * tr + y, pos = qc * c_q + row;
      if (row >= c_q || pos >= n_q) continue;
      const int orig = perm_q[(size_t)p * n_q + pos];
      if (orig < 0 || orig >= n_q) {
        atomicCAS(status, 0, 6);
        continue;
      }
      // a row without a single live entry (an empty list without compensation): zeros, lse = -inf
      const bool empty = !(l_run[y] > 0.f);
      const float inv = empty ? 0.f : 1.f / l_run[y];
      T* out = O + ((size_t)p * n_q + orig) * D;
#pragma unroll
      for (int g = 0; g < CG; ++g)
        store4(out + 64 * g + 4 * tc, make_float4(acc[y][g][0] * inv, acc[y][g][1] * inv, acc[y][g][2] * inv, acc[y][g][3] * inv));
      if (lse && tc == 0) lse[(size_t)p * n_q + orig] = empty ? -INFINITY : m_run[y] + logf(l_run[y]);
    }
  }   // tiles of the cluster
  }   // clusters of the CTA
}

template <typename T, int D, int QR, int RY = 4, bool many = false>
static int launch_rows(const ca_problem_t& pr, const T* Qp, const T* Kp, const T* Vp, const float* ck,
                       const float* cv, const int32_t* count_k, const int32_t* block_idx,
                       const int32_t* keep_count, int list_stride, const int32_t* perm_q, float scale, T* O,
                       float* lse, int* status, LaunchStream st, const int32_t* redo, int redo_tiles,
                       int* redo_count) {
  const int n_qc = ceil_div(pr.n_q, pr.cluster_q), n_kc = ceil_div(pr.n_k, pr.cluster_k);
  const size_t smem = sizeof(float) * ((size_t)(QR + 2 * kRefKT) * (D + 4) + QR * (kRefKT + 4) + kRefKT) +
                      sizeof(unsigned) * (((n_kc < kRefWindow ? n_kc : kRefWindow) + 31) / 32);
  // second pass: some 600 CTAs that look at their share of the marks (10,240 CTAs that each looked at one took 18 us)
  const int n_clusters = pr.batch * pr.heads * n_qc;
  constexpr int NT = 16 * QR / RY;
  const int per_cta = redo ? (ceil_div(n_clusters, 592) < NT ? ceil_div(n_clusters, 592) : NT) : 1;
  const dim3 grid = redo ? dim3(ceil_div(n_clusters, per_cta))
                         : dim3(n_qc * ceil_div(pr.cluster_q, QR), pr.batch * pr.heads);
  auto k = attn_ref_kernel<T, D, QR, RY, many>;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  launch_chained(k, grid, NT, smem, st, Qp, Kp, Vp, ck, cv, count_k, block_idx, keep_count, list_stride, perm_q, pr.n_q, pr.n_k,
                                pr.cluster_q, pr.cluster_k, pr.keep, pr.compensate, scale, O, lse, status, redo,
                                redo_tiles, redo_count, per_cta, n_clusters);
  CA_LAUNCH_CHECK();
  return CA_OK;
}

template <typename T>
static int launch_t(const ca_problem_t& pr, const T* Qp, const T* Kp, const T* Vp, const float* ck,
                    const float* cv, const int32_t* count_k, const int32_t* block_idx,
                    const int32_t* keep_count, int list_stride, const int32_t* perm_q, float scale, T* O,
                    float* lse, int* status, LaunchStream st, const int32_t* redo, int redo_tiles,
                    int* redo_count) {
  // 64 query rows per CTA read every key half as often as 32; 32 where 64 would leave SMs without a CTA
  const int n_kc = ceil_div(pr.n_k, pr.cluster_k);
  const long long ctas = (long long)pr.batch * pr.heads * ceil_div(pr.n_q, 64);
  const bool wide = !redo && pr.cluster_q >= 64 && ctas >= 148;
  auto go = [&](auto launch) {
    return launch(pr, Qp, Kp, Vp, ck, cv, count_k, block_idx, keep_count, list_stride, perm_q, scale, O, lse, status, st,
                  redo, redo_tiles, redo_count);
  };
  const bool narrow = pr.cluster_q < 32;       // (never a second pass: the tensor-core kernel takes 64 rows and more)
  if (n_kc > kRefWindow) return pr.head_dim == 64 ? go(launch_rows<T, 64, 32, 4, true>) : go(launch_rows<T, 128, 32, 4, true>);
  if (pr.head_dim == 64) return narrow ? go(launch_rows<T, 64, 16, 2>) : wide ? go(launch_rows<T, 64, 64>) : go(launch_rows<T, 64, 32>);
  return narrow ? go(launch_rows<T, 128, 16, 2>) : wide ? go(launch_rows<T, 128, 64>) : go(launch_rows<T, 128, 32>);
}

int launch_attn_ref(const ca_problem_t& pr, const void* Qp, const void* Kp, const void* Vp,
                    const float* ck, const float* cv, const int32_t* count_k, const int32_t* block_idx,
                    const int32_t* keep_count, int list_stride, const int32_t* perm_q, float scale, void* O,
                    float* lse, int* status, LaunchStream st, const int32_t* redo, int redo_tiles,
                    int* redo_count) {
  if (pr.dtype == CA_DTYPE_BF16)
    return launch_t(pr, static_cast<const __nv_bfloat16*>(Qp), static_cast<const __nv_bfloat16*>(Kp),
                    static_cast<const __nv_bfloat16*>(Vp), ck, cv, count_k, block_idx, keep_count, list_stride,
                    perm_q, scale,
                    static_cast<__nv_bfloat16*>(O), lse, status, st, redo, redo_tiles, redo_count);
  return launch_t(pr, static_cast<const float*>(Qp), static_cast<const float*>(Kp),
                  static_cast<const float*>(Vp), ck, cv, count_k, block_idx, keep_count, list_stride, perm_q, scale,
                  static_cast<float*>(O), lse, status, st, redo, redo_tiles, redo_count);
}

}  // namespace ca
