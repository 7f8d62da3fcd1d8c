// FP32 CUDA-core kernel for block-sparse attention with striped
// mean-compensation (eq. 2 over the selected clusters; Appendix A: an excluded
// cluster enters through its centroid key and value with weight
// |c| exp(q . kbar / sqrt(d)), in numerator and denominator).
// Serves fp32 storage, unusual cluster sizes, and as an on-device cross-check of
// the tensor-core kernel.  Flash-style online softmax, fp32 throughout.
//
// Bound by the fp32 pipe and by what feeds it from shared memory: 16 threads share RY query
// rows, a thread computes RY x KT / 16 scores and RY x D / 16 outputs, so that (RY = 4, KT = 64) eight 16-byte loads feed 64
// (scores) and 12 feed 128 (outputs) multiply-adds.  fp32 storage: the keys of the next tile are copied to shared memory
// asynchronously while the softmax and the outputs of a tile are computed, its values during the scores of the next, without
// passing registers, which leaves room for 16 warps per SM; with registers in between (8 to 16 warps, 64 rows per CTA) 4
// heads of 5,003 rows, d = 128, 5 of 40 clusters of 128 kept took 357 us, now 310, 4 heads of 8,192 rows 805 -> 599, 2 heads of 1,024
// rows, d = 64 29 -> 23.  (5,003 rows are 628 CTAs, four to an SM: 36 too many for one wave.)  bf16 storage (the cross-check and
// the second pass behind the tensor-core kernel) converts, so its rows pass through registers.
// Of a query cluster of 16 rows a CTA takes those, with RY = 2: in a tile of 32 half of the threads would compute nothing.
#include "kernels.h"

namespace ca {

// 16 bytes global -> shared memory, zeros where `use` is false
__device__ __forceinline__ void copy_async16(float* dst, const float* src, bool use) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(use ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void copies_close() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int left>                // all groups of copies but the last `left` have arrived
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(left) : "memory"); }

// Key clusters that the bitmap of the selected ones covers at a time (128 KB, beside the widest tile), so that their number
// has no bound in shared memory.  With more of them (`many`, an instance of its own: moving the window costs the others
// registers) the bitmap is set anew per window; a second pass never has as many (the tensor-core kernel takes an eighth).
constexpr int kRefWindow = 1 << 20;

template <typename T, int D, int QR, int RY, int KT, bool direct, bool many>
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
  constexpr int LP = KT + 4;
  constexpr int CG = D / 64;             // groups of four output columns per thread
  constexpr int KI = KT / 16;            // keys per thread
  constexpr int PF = KT * D / 4 / NT;    // float4 of keys (of values) per thread and tile
  extern __shared__ __align__(16) float smem[];
  float* qs = smem;                      // [QR][LD]
  float* ks = qs + QR * LD;              // [KT][LD]
  float* vs = ks + KT * LD;              // [KT][LD]
  float* ps = vs + KT * LD;              // [QR][LP]
  float* bias = ps + QR * LP;            // [2][KT] per-key additive term (ln|c| or -inf), of two tiles in turn
  unsigned* selected = reinterpret_cast<unsigned*>(bias + 2 * KT);   // bitmap over a window of key clusters

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

    // Tiles of keys: the members of the selected clusters in list order (t, row t0), then, KT at a time, the
    // centroids (t = keep, first centroid t0).  `rows` = 0: no tile left.
    int t = 0, t0 = 0, rows = 0, members = 0;
    auto settle = [&]() {                  // the first tile at or behind (t, t0)
      while (t < keep) {
        const int j = sel[t];
        members = (j < 0 || j >= n_kc) ? 0 : min(max(cnt[j], 0), c_k);       // out of range: flagged above
        if (t0 < members) { rows = min(KT, members - t0); return; }
        ++t;
        t0 = 0;
      }
      rows = compensate ? min(KT, n_kc - t0) : 0;
    };
    float4 kf[direct ? 1 : PF], vf[direct ? 1 : PF];
    int parity = 0;                        // of the tile that is computed
    const T *k_src = nullptr, *v_src = nullptr;   // (direct) rows of the next tile
    int src_rows = 0;
    auto copy_tile = [&](float* dst, const T* src) {
      if constexpr (direct) {
#pragma unroll 4
        for (int i = 0; i < PF; ++i) {
          const int e = tid + i * NT, r = e / (D / 4), col = 4 * (e % (D / 4));
          copy_async16(&dst[r * LD + col], src + (r < src_rows ? (size_t)r * D + col : 0), r < src_rows);
        }
      }
      copies_close();
    };
    // Of this thread's key of the next tile: how many rows it stands for (1, or a centroid's; 0: not in use), waited for at the tile's
    // turn; or its additive term, formed where the rows are fetched.  bf16, us, at the tile's turn / at the fetch: 5 heads of 318 x
    // 38,642 rows, clusters of 16, d = 128 (16 rows) 390 / 314, d = 64 193 / 199; 4 heads of 8,000 rows, d = 128, clusters of
    // 64 (64 rows) 687 / 828; fp32, 2 heads of 2,500 rows, d = 64, clusters of 64 x 32 (32 rows) 51.2 / 49.7.
    constexpr bool late = direct || QR == 64 || (QR == 16 && D == 64);
    int next_count = 0;
    float next_bias = 0.f;
    auto fetch = [&]() {
      const bool cen = t >= keep;
      const size_t base = cen ? (size_t)t0 * D : ((size_t)sel[t] * c_k + t0) * D;
      if constexpr (direct) {
        k_src = (cen ? ckh : Kh) + base;
        v_src = (cen ? cvh : Vh) + base;
        src_rows = rows;
      } else {
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
      }
      if (tid < KT) {
        const int j = t0 + tid;
        const bool centroid = cen && tid < rows;
        const bool use = centroid ? !((selected[(many ? j % kRefWindow : j) >> 5] >> (j & 31)) & 1u) : tid < rows;
        if constexpr (late) {
          next_count = use ? 1 : 0;
          if (centroid && use) next_count = cnt[j];
        } else {
          next_bias = use ? 0.f : -INFINITY;
          if (centroid && use) next_bias = logf((float)cnt[j]);
        }
      }
    };
    settle();
    if (rows > 0) {
      fetch();
      if constexpr (direct) { copy_tile(ks, k_src); copy_tile(vs, v_src); }
    }
    while (rows > 0) {
      if (late && tid < KT) bias[parity * KT + tid] = next_count == 1 ? 0.f : logf((float)next_count);   // (of 0: -inf)
      if constexpr (direct) {
        copies_wait<1>();
        __syncthreads();                   // the keys have arrived
      } else {
        __syncthreads();                   // the tile before has been read
#pragma unroll
        for (int i = 0; i < PF; ++i) {
          const int e = tid + i * NT, r = e / (D / 4), col = 4 * (e % (D / 4));
          *reinterpret_cast<float4*>(&ks[r * LD + col]) = kf[i];
          *reinterpret_cast<float4*>(&vs[r * LD + col]) = vf[i];
        }
        if (!late && tid < KT) bias[tid] = next_bias;
        __syncthreads();
      }
      t0 += KT;
      rows = 0;
      if (t < keep) settle();
      else rows = max(0, min(KT, n_kc - t0));
      if constexpr (many) {
        if (rows > 0 && t >= keep && t0 > 0 && t0 % kRefWindow == 0) {
          __syncthreads();                 // the window before has been read
          mark(t0);
          __syncthreads();
        }
      }
      const float* b_tile = bias + parity * KT;
      if constexpr (late) parity ^= 1;
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
      if constexpr (direct) {
        copies_wait<0>();
        __syncthreads();                   // the keys have been read, the values have arrived
        if (rows > 0) copy_tile(ks, k_src);
      }
      // online softmax: the 16 threads of a row are half a warp
      float tmax[RY];
#pragma unroll
      for (int y = 0; y < RY; ++y) {
        tmax[y] = -INFINITY;
#pragma unroll
        for (int i = 0; i < KI; ++i) {
          s[y][i] = s[y][i] * scale + b_tile[tc + 16 * i];
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
      for (int key = 0; key < KT; key += 4) {
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
      if constexpr (direct) {
        __syncthreads();                   // the values have been read
        if (rows > 0) copy_tile(vs, v_src);
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

// direct: tiles are copied to shared memory asynchronously, not by way of registers
template <typename T, int D, int QR, int RY, int KT, bool direct = sizeof(T) == 4, bool many = false>
static int launch_rows(const ca_problem_t& pr, const T* Qp, const T* Kp, const T* Vp, const float* ck,
                       const float* cv, const int32_t* count_k, const int32_t* block_idx,
                       const int32_t* keep_count, int list_stride, const int32_t* perm_q, float scale, T* O,
                       float* lse, int* status, LaunchStream st, const int32_t* redo, int redo_tiles,
                       int* redo_count) {
  const int n_qc = ceil_div(pr.n_q, pr.cluster_q), n_kc = ceil_div(pr.n_k, pr.cluster_k);
  const size_t smem = sizeof(float) * ((size_t)(QR + 2 * KT) * (D + 4) + QR * (KT + 4) + 2 * KT) +
                      sizeof(unsigned) * (((n_kc < kRefWindow ? n_kc : kRefWindow) + 31) / 32);
  // second pass: some 600 CTAs that look at their share of the marks (10,240 CTAs that each looked at one took 18 us)
  const int n_clusters = pr.batch * pr.heads * n_qc;
  constexpr int NT = 16 * QR / RY;
  const int per_cta = redo ? (ceil_div(n_clusters, 592) < NT ? ceil_div(n_clusters, 592) : NT) : 1;
  const dim3 grid = redo ? dim3(ceil_div(n_clusters, per_cta))
                         : dim3(n_qc * ceil_div(pr.cluster_q, QR), pr.batch * pr.heads);
  auto k = attn_ref_kernel<T, D, QR, RY, KT, direct, many>;
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
  const int n_qc = ceil_div(pr.n_q, pr.cluster_q), n_kc = ceil_div(pr.n_k, pr.cluster_k);
  auto go = [&](auto launch) {
    return launch(pr, Qp, Kp, Vp, ck, cv, count_k, block_idx, keep_count, list_stride, perm_q, scale, O, lse, status, st,
                  redo, redo_tiles, redo_count);
  };
  if (n_kc > kRefWindow) return pr.head_dim == 64 ? go(launch_rows<T, 64, 32, 4, 32, false, true>) : go(launch_rows<T, 128, 32, 4, 32, false, true>);
  const bool narrow = pr.cluster_q < 32;       // (never a second pass: the tensor-core kernel takes 64 rows and more)
  if constexpr (sizeof(T) == 4) {
    // Query rows per CTA: 8 or 16 where every CTA still has an SM for itself (a CTA is a chain of latencies then, which shared
    // work shortens) and of clusters of 16, otherwise 32.  Keys per tile: 64 (fewer rounds of the softmax), but 32 where
    // clusters are smaller (a tile holds one cluster), at d = 128 with more than two CTAs per SM, of which four fit with 32 and two
    // with 64, and where lists and centroids fill tiles of 64 so badly that an eighth of the columns is added (12 heads of
    // 1,370 rows, 2 of 22 clusters of 64, d = 64 35.2 us with 32, 37.2 with 64), unless every CTA has an SM for itself.
    // us, tiles of 32 rows and 32 keys / 64 keys / 16 rows and 64 keys / 8 rows:
    //   1 head of 1,024 rows, d = 64     20.7 / 19.5 / 16.6 / 14.9      2 heads of 1,024     31 / 27 / 22.8 / 26.8
    //   4 heads of 1,024                 30 / 26.8 / 28.9 / 37          4 heads of 8,192     619 / 537 / 733
    //   1 head of 1,500, d = 128         59 / 51 / 41 / 54              2 heads of 2,500     134 / 115 / 146
    //   2 heads of 5,003, 10 clusters    321 / 395                      4 heads of 8,192     599 / 709
    //   4 heads of 5,000 in clusters of 32    331 / 671             1 head of 1,000, key clusters of 16     93 / - / 77
    // Query clusters of 16, d = 128, 16 rows and 32 keys / 64 keys: 2 heads of 1,400 rows, key clusters of 128 (176 CTAs) 80 / 74,
    // 2 of 2,500 (314 CTAs, 18 more than two to an SM) 60 / 76, 4 of 8,000 688 / 720.
    // By way of registers where small clusters leave at most two CTAs to an SM: two barriers per tile instead of three (2 heads of
    // 2,500 rows, clusters of 64 x 32, d = 64 49.6 us, and 51 with asynchronous copies, d = 128 76.2 and 78; at
    // d = 128 16 rows take the same time either way).
    auto columns = [&](int keys) {       // of a list in tiles of `keys`
      return (long long)pr.keep * ceil_div(pr.cluster_k, keys) * keys + (pr.compensate ? (long long)ceil_div(n_kc, keys) * keys : 0);
    };
    const bool full = keep_count || 7 * columns(64) <= 8 * columns(32);     // (lists of lengths not known here: taken as long)
    auto ctas = [&](int rows) { return (long long)pr.batch * pr.heads * n_qc * ceil_div(pr.cluster_q, rows); };
    const bool few = ctas(32) <= 296, short_rows = narrow || ctas(16) <= 148, wide_keys = pr.cluster_k >= 64;
    if (wide_keys && ctas(8) <= 148) return pr.head_dim == 64 ? go(launch_rows<T, 64, 8, 1, 64>) : go(launch_rows<T, 128, 8, 1, 64>);
    if (pr.head_dim == 64) {
      if (short_rows && wide_keys && (full || ctas(16) <= 148)) return go(launch_rows<T, 64, 16, 2, 64>);
      if (short_rows) return few ? go(launch_rows<T, 64, 16, 2, 32, false>) : go(launch_rows<T, 64, 16, 2, 32>);
      if (wide_keys && full) return go(launch_rows<T, 64, 32, 4, 64>);
      return few ? go(launch_rows<T, 64, 32, 4, 32, false>) : go(launch_rows<T, 64, 32, 4, 32>);
    }
    if (short_rows) return wide_keys && (ctas(16) <= 148 || (full && ctas(16) <= 296)) ? go(launch_rows<T, 128, 16, 2, 64>) : go(launch_rows<T, 128, 16, 2, 32>);
    if (!few) return go(launch_rows<T, 128, 32, 4, 32>);
    return wide_keys && full ? go(launch_rows<T, 128, 32, 4, 64>) : go(launch_rows<T, 128, 32, 4, 32, false>);
  } else {
    // 64 query rows per CTA read every key half as often as 32; 32 where 64 would leave SMs without a CTA
    const bool wide = !redo && pr.cluster_q >= 64 && (long long)pr.batch * pr.heads * ceil_div(pr.n_q, 64) >= 148;
    if (pr.head_dim == 64) return narrow ? go(launch_rows<T, 64, 16, 2, 32>) : wide ? go(launch_rows<T, 64, 64, 4, 32>) : go(launch_rows<T, 64, 32, 4, 32>);
    return narrow ? go(launch_rows<T, 128, 16, 2, 32>) : wide ? go(launch_rows<T, 128, 64, 4, 32>) : go(launch_rows<T, 128, 32, 4, 32>);
  }
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
