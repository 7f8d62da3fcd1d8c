// Diagonalized recursive splitting (Section 3.2.1) on fp32 principal-component
// coordinates.
//
// A set [lo, lo+s) keeps its rows in ascending original order.  A split
//   1. takes m = min(d, s) rows at positions floor(j*s/m), estimates the variance
//      of each coordinate over them in float32 with a fixed operation order and
//      picks the coordinate of largest variance, lowest index on exact ties;
//   2. finds, by counting into bins and ranking one bin, the L-th smallest
//      (value, row) along it, L = c * floor((s + c) / (2c));
//   3. moves the L smallest rows to [lo, lo+L) and the others to [lo+L, lo+s),
//      both sides keeping their order (stable partition by prefix sums).
// Nothing depends on floating-point rounding except step 1, whose operation
// order is fixed, so the permutation is reproducible bit for bit.
//
// Two kernels.  Large sets: one launch per tree level, a thread-block cluster of
// up to 8 CTAs per set; each CTA keeps its slice of keys and rows in shared
// memory, histograms and partition offsets are combined through distributed
// shared memory (hardware cluster barriers, no spin waits).  Sets of at most
// kTailRows rows: one CTA finishes the whole subtree in shared memory, all
// subsets of a level side by side, and writes the permutation once.
//
// The basic variant of the splitting (a power iteration per set instead of a
// coordinate choice, at the end of this file) computes its keys in kernels of
// its own and reuses the per-level kernel for selection and partition.
#include <climits>
#include <cooperative_groups.h>

#include "kernels.h"
#include "sample_position.h"

namespace ca {

namespace cg = cooperative_groups;

constexpr int kSplitThreads = 1024;      // subtree kernel of the basic variant
constexpr int kSmemRowsMax = 24576;      // rows a CTA stages (8 bytes each)
constexpr int kMaxCluster = 8;
constexpr int kLevelBins = 1024;
constexpr int kLevelList = 512;          // candidates that the level kernel ranks from a list
constexpr int kTailRowsMax = 1024;       // rows of a subtree
constexpr int kTailSegs = 16;            // subsets a tail CTA splits side by side
constexpr int kBasicRowsMax = 4096;      // the same of the basic variant
constexpr int kBasicSegs = 32;

struct SegmentRef { int lo, size, active; };

// Walks from the root to slot `slot` of `level` (most significant bit first).
// A set of at most c rows is final; its slot at deeper levels is the all-zero
// continuation (it only has to be copied to the output buffer).
__device__ __forceinline__ SegmentRef locate_segment(int n, int c, int level, int slot) {
  SegmentRef r{0, n, 1};
  for (int b = level - 1; b >= 0; --b) {
    const int bit = (slot >> b) & 1;
    if (r.size <= c) {
      if (slot & ((2 << b) - 1)) r.active = 0;   // some remaining bit is set
      return r;
    }
    const int L = c * ((r.size + c) / (2 * c));
    if (bit) { r.lo += L; r.size -= L; } else { r.size = L; }
  }
  return r;
}

__device__ __forceinline__ uint32_t order_key(float x) {
  if (x == 0.0f) x = 0.0f;                       // -0 and +0 compare equal
  uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Two fp32 values in one 64-bit register and the instructions that work on both halves at once
// (each half rounded to nearest on its own: the same bits as two scalar operations).
typedef unsigned long long pair2;
__device__ __forceinline__ pair2 pair(float lo, float hi) {
  pair2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpair(pair2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ pair2 add_pair(pair2 a, pair2 b) {
  pair2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ pair2 fma_pair(pair2 a, pair2 b, pair2 c) {
  pair2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// Largest variance over the subsample of one block of 4 V coordinates of one subset, by one warp.  The estimate
// only feeds an argmax, so it is taken in float32 with a fixed operation order (reproducible bit for
// bit; every operation rounded on its own, no fused multiply-add): eight partial sums over the rows
// j = r, r+8, ... taken row after row, combined as ((p0+p1)+(p2+p3)) + ((p4+p5)+(p6+p7)); first the
// mean, then the squared deviations.  Lane 4 r + q takes the rows of residue r and V consecutive
// coordinates, and a butterfly over the lanes adds the residues in that order; a row is read once
// and kept in registers for the squares, and no barrier is needed.  Writes the largest variance of the
// block, and its coordinate (the lowest on ties) with that coordinate's mean.
// rows: the subset's rows, in shared memory, or (global) in global memory or null, then first, first + 1, ...
template <int D, int V, bool full, bool global>      // full: the subset has at least D rows
__device__ __forceinline__ void unit_variance(const float* __restrict__ Y, const int32_t* rows, int first, int sz, int block,
                                              int lane, float* best_out, int2* arg_out) {
  constexpr int PER = D / 8;                         // sample rows of a residue
  const int r = lane >> 2, t = (block * 4 + (lane & 3)) * V;
  const int m = full ? D : sz;
  // sample j stands at position floor(j sz / m): j itself where the sample is the whole subset; a
  // row beyond the sample is loaded as the last one and counts as zero
  pair2 x[PER][V / 2];
  const float* Yq = Y + t;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int pos = full ? sample_position<D>(r + 8 * k, sz) : min(r + 8 * k, m - 1);
    const unsigned row = (unsigned)(global ? (rows ? __ldg(rows + pos) : first + pos) : rows[pos]);
    const float* src = Yq + (size_t)row * D;
    if constexpr (V == 4) {
      const ulonglong2 w = __ldg(reinterpret_cast<const ulonglong2*>(src));
      x[k][0] = w.x;
      x[k][V / 2 - 1] = w.y;
    } else {
      x[k][0] = __ldg(reinterpret_cast<const unsigned long long*>(src));
    }
  }
  if (!full) {
#pragma unroll
    for (int k = 0; k < PER; ++k)
#pragma unroll
      for (int h = 0; h < V / 2; ++h) x[k][h] = r + 8 * k < m ? x[k][h] : 0ull;
  }
  // D is a power of two: the product with 1 / D rounds as the division does.  For a partial sample
  // a lane divides the value of its residue's number and the lanes of a coordinate exchange them.
  auto divide = [&](float (&v)[V]) {
    if (full) {
#pragma unroll
      for (int i = 0; i < V; ++i) v[i] = __fmul_rn(v[i], 1.0f / D);
    } else {
      float q = v[0];
#pragma unroll
      for (int i = 1; i < V; ++i) q = (r & (V - 1)) == i ? v[i] : q;
      q = __fdiv_rn(q, (float)m);
#pragma unroll
      for (int i = 0; i < V; ++i) v[i] = __shfl_sync(0xffffffffu, q, 4 * i + (lane & 3));
    }
  };
  float mean[V], var[V];
#pragma unroll
  for (int h = 0; h < V / 2; ++h) {
    pair2 acc = pair(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < PER; ++k) acc = add_pair(acc, x[k][h]);
    unpair(acc, mean[2 * h], mean[2 * h + 1]);
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1)
#pragma unroll
    for (int v = 0; v < V; ++v) mean[v] = __fadd_rn(mean[v], __shfl_xor_sync(0xffffffffu, mean[v], o));
  divide(mean);
  // All operations on two values per instruction (each half rounded on its own: the bits of two
  // scalar operations).  A multiply followed by an add would be merged into one fused multiply-add, which
  // rounds once where the definition rounds twice; the square is a fused multiply-add of its own, with
  // an addend of -0 that only the launch knows (gridDim.z is 1).
  const float minus_zero = __uint_as_float(gridDim.z << 31);
  const pair2 addend = pair(minus_zero, minus_zero);
#pragma unroll
  for (int h = 0; h < V / 2; ++h) {
    const pair2 neg = pair(-mean[2 * h], -mean[2 * h + 1]);
    pair2 acc = pair(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      pair2 dev = add_pair(x[k][h], neg);
      if (!full && r + 8 * k >= m) dev = 0ull;       // a missing row adds an exact zero
      acc = add_pair(acc, fma_pair(dev, dev, addend));
    }
    unpair(acc, var[2 * h], var[2 * h + 1]);
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1)
#pragma unroll
    for (int v = 0; v < V; ++v) var[v] = __fadd_rn(var[v], __shfl_xor_sync(0xffffffffu, var[v], o));
  divide(var);
  // a variance that is not a number (an infinity among the samples) loses against every other
#pragma unroll
  for (int v = 0; v < V; ++v) var[v] = fmaxf(var[v], -1.f);
  float best = var[0], best_mean = mean[0];
  int arg = t;
#pragma unroll
  for (int v = 1; v < V; ++v)
    if (var[v] > best) { best = var[v]; arg = t + v; best_mean = mean[v]; }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
    const float om = __shfl_xor_sync(0xffffffffu, best_mean, o);
    if (ob > best || (ob == best && oa < arg)) { best = ob; arg = oa; best_mean = om; }
  }
  if (lane == 0) {
    *best_out = best;
    *arg_out = make_int2(arg, __float_as_int(best_mean));
  }
}
// Out of line: only subsets of fewer than D rows take it, which split only where the cluster size is below D.
template <int D, int V, bool global>
__device__ __noinline__ void unit_variance_small(const float* __restrict__ Y, const int32_t* rows, int first, int sz,
                                                 int block, int lane, float* best_out, int2* arg_out) {
  unit_variance<D, V, false, global>(Y, rows, first, sz, block, lane, best_out, arg_out);
}

// 4-byte asynchronous copy global -> shared (no register held while in flight)
__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gmem_src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

struct SplitSide {
  const float* Y;          // [P][n][D]
  const float* Yt;         // [P][kSplitCols][n] the first coordinates once more, coordinate-major, or null
  const int32_t* perm_in;  // [P][n] or null (identity)
  int32_t* perm_out;       // [P][n]
  uint32_t* keybuf;        // [P][n] staging for sets larger than the shared-memory windows
  int n, c, levels, tail_level;
};

struct SplitParams {
  SplitSide side[2];
  int D, level, problems, smem_rows;
  int first_side, sides;   // the sides of this launch: queries 0, keys 1 (they can run on different streams)
};

// Scale and offset of the bins of one coordinate: `half` bins to either side of the sample's mean for two
// standard deviations; scale 0 (all rows in one bin) where that cannot be had.
__device__ __forceinline__ float2 bin_map(float variance, float mean, float half) {
  const float scale = 0.5f * half * rsqrtf(variance), shift = fmaf(-mean, scale, half);
  const bool usable = variance > 0.f && scale < 1e30f && fabsf(shift) < 1e30f;     // also false for NaN
  return usable ? make_float2(scale, shift) : make_float2(0.f, half);
}
// The bin of a value among `bins`.  It grows with the key for every value: infinities land at the ends
// (the scale is positive and finite, or zero and all bins equal), NaNs are put where their keys stand.
__device__ __forceinline__ int bin_of(float x, uint32_t key, float2 map, int bins) {
  const float last = (float)(bins - 1);
  int bin = (int)fminf(fmaxf(fmaf(x, map.x, map.y), 0.f), last);
  if (x != x) bin = (int)key < 0 ? bins - 1 : 0;
  return map.x == 0.f ? 0 : bin;
}
__device__ __forceinline__ float key_value(uint32_t key) {               // inverse of order_key
  return __uint_as_float((key & 0x80000000u) ? key & 0x7fffffffu : ~key);
}

// ---------------------------------------------------------------------------
// One level of the large sets.  grid.x = slots * cluster size.
// ---------------------------------------------------------------------------
// A cluster per set, a slice of up to 8,192 rows per CTA where eight CTAs can hold the set that way.  A CTA is
// a chain of short sweeps over its slice between barriers, bound by their latencies: two CTAs
// share an SM and small sets take more CTAs while the SMs are not all taken.  The L-th value is found from
// one count into 1,024 bins between mean - 2 s and mean + 2 s of the sample, the rows of its bin are
// collected in the first CTA's list and every CTA ranks a copy.  Where the bin holds more rows than the
// list (values repeat, far outliers) and for keys computed elsewhere (keys_in, the basic variant) the
// digits of the key are counted eight bits a pass until the candidates fit the list, or are all equal.
// Levels of both sides, against one CTA of 1,024 threads per 16,384 rows that counted two digits: 12 heads of
// 16,385 rows, d = 64: 151 -> 103 us; 8 heads of 1,531 x 23,117 rows: 66 -> 44; 8 heads of 16,384 x 131,072 rows: 191
// -> 160; 40 heads of 32,760 rows, d = 128: 214 -> 184.
template <int D, int nt, bool keys_in>
__global__ void __launch_bounds__(nt, nt == 1024 ? 1 : 2) split_level_kernel(const SplitParams prm) {
  wait_for_previous();
  cg::cluster_group cluster = cg::this_cluster();
  const int csize = (int)cluster.num_blocks();
  const int crank = (int)cluster.block_rank();
  constexpr int NW = nt / 32;
  constexpr int V = D == 64 ? 4 : 2, UNITS = D / (4 * V);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* s_keys = reinterpret_cast<uint32_t*>(smem_raw);                  // [smem_rows]
  int32_t* s_rows = reinterpret_cast<int32_t*>(s_keys + prm.smem_rows);      // [smem_rows]
  __shared__ __align__(8) int s_hist[kLevelBins];        // bins, or 256 digits for each of four passes
  __shared__ unsigned long long s_list[kLevelList];      // (key, position in the set)
  __shared__ int s_list_n;                               // counted in the cluster's first CTA
  __shared__ float s_best[UNITS];
  __shared__ int2 s_arg[UNITS];
  __shared__ float2 s_map;
  __shared__ int s_coord, s_pick[3];                     // bin, 1-based rank inside it, its rows
  __shared__ int s_warp[NW];
  __shared__ int s_total;                                // of this CTA, read by its peers
  __shared__ unsigned long long s_thr;                   // the last (key, position) that goes down

  const int which = prm.first_side + blockIdx.y / prm.problems;
  const int p = blockIdx.y % prm.problems;
  const SplitSide sd = prm.side[which];
  if (prm.level >= sd.tail_level) return;             // uniform over the cluster
  const SegmentRef seg = locate_segment(sd.n, sd.c, prm.level, blockIdx.x / csize);
  if (!seg.active) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* Y = sd.Y + (size_t)p * sd.n * D;
  const int32_t* pin = sd.perm_in ? sd.perm_in + (size_t)p * sd.n : nullptr;
  int32_t* pout = sd.perm_out + (size_t)p * sd.n;
  const int lo = seg.lo, s = seg.size;
  auto row_at = [pin, lo](int i) { return pin ? __ldg(pin + lo + i) : lo + i; };
  auto sync_all = [&]() {
    if (csize > 1) cluster.sync();
    else __syncthreads();
  };

  if (s <= sd.c) {                                   // final set: carry over
    if (crank == 0)
#pragma unroll 1
      for (int i = tid; i < s; i += nt) pout[lo + i] = row_at(i);
    return;
  }

  // ---- 1. coordinate of largest subsample variance (every CTA of the cluster computes it)
  if (tid < kLevelBins / 2) reinterpret_cast<int2*>(s_hist)[tid] = make_int2(0, 0);
  if (tid == 0) s_list_n = 0;
  if constexpr (!keys_in) {
#pragma unroll 1
    for (int unit = warp; unit < UNITS; unit += NW) {
      const int32_t* set = pin ? pin + lo : nullptr;
      if (s >= D) unit_variance<D, V, true, true>(Y, set, lo, s, unit, lane, &s_best[unit], &s_arg[unit]);
      else unit_variance_small<D, V, true>(Y, set, lo, s, unit, lane, &s_best[unit], &s_arg[unit]);
    }
    __syncthreads();
    if (warp == 0) {
      float v = s_best[lane % UNITS];
      int at = lane % UNITS;
#pragma unroll
      for (int o = 1; o < UNITS; o <<= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oa = __shfl_xor_sync(0xffffffffu, at, o);
        if (ov > v || (ov == v && oa < at)) { v = ov; at = oa; }       // later blocks hold higher coordinates
      }
      if (lane == 0) {
        const int2 am = s_arg[at];
        s_coord = am.x;
        s_map = bin_map(v, __int_as_float(am.y), kLevelBins / 2);
      }
    }
  }
  __syncthreads();

  // ---- 2. keys of this CTA's slice [c0, c1) of the set, and their bins
  const int chunk = (s + csize - 1) / csize;
  const int c0 = min(s, crank * chunk), c1 = min(s, c0 + chunk);
  const int cs = c1 - c0;
  const bool in_smem = cs <= prm.smem_rows;
  uint32_t* g_keys = sd.keybuf + (size_t)p * sd.n + lo + c0;
  auto key_at = [&](int i) { return in_smem ? s_keys[i] : g_keys[i]; };
  float2 map = make_float2(0.f, 0.f);
  if constexpr (keys_in) {
    // the projections of this level were turned into keys by another kernel, position by position
    if (in_smem) {
#pragma unroll 4
      for (int i = tid; i < cs; i += nt) {
        s_keys[i] = g_keys[i];
        s_rows[i] = row_at(c0 + i);
      }
    }
  } else {
    map = s_map;
    const int coord = s_coord;
    const bool column = sd.Yt && coord < kSplitCols;
    const float* Yc = column ? sd.Yt + ((size_t)p * kSplitCols + coord) * sd.n : Y + coord;
    const int row_stride = column ? 1 : D;
    if (in_smem) {
      // asynchronous copies: the rows, then their values in place of the keys.  (The loops are rolled: a
      // launch runs this code once, so an unrolled sweep costs more in instruction fetch than it saves.)
      if (pin) {
#pragma unroll 1
        for (int i = tid; i < cs; i += nt) cp_async4(&s_rows[i], pin + lo + c0 + i);
        cp_async_wait_all();
      } else {
#pragma unroll 1
        for (int i = tid; i < cs; i += nt) s_rows[i] = lo + c0 + i;
      }
#pragma unroll 1
      for (int i = tid; i < cs; i += nt) cp_async4(&s_keys[i], Yc + (size_t)s_rows[i] * row_stride);
      cp_async_wait_all();
    }
#pragma unroll 1
    for (int i = tid; i < cs; i += nt) {
      const float x = in_smem ? __uint_as_float(s_keys[i]) : __ldg(Yc + (size_t)row_at(c0 + i) * row_stride);
      const uint32_t key = order_key(x);
      if (in_smem) s_keys[i] = key;
      else g_keys[i] = key;
      atomicAdd(&s_hist[bin_of(x, key, map, kLevelBins)], 1);
    }
  }

  // ---- 3. the threshold.  Counts of bins [first, first + 2 w) summed over the cluster; the bin that holds the
  // row of rank `rank`.  A peer may still be reading counts after this returns, so they are
  // cleared or counted again only beyond another cluster barrier.
  auto pick = [&](int first, int w, int rank) {
    sync_all();                                        // every slice has counted
    int n0 = 0, n1 = 0;
    if (tid < w) {
#pragma unroll 1
      for (int r = 0; r < csize; ++r) {
        const int* h = csize > 1 ? cluster.map_shared_rank(s_hist, r) : s_hist;
        const int2 n = *reinterpret_cast<const int2*>(h + first + 2 * tid);
        n0 += n.x;
        n1 += n.y;
      }
    }
    int incl = n0 + n1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    const int left = rank - (int)__reduce_add_sync(0xffffffffu, lane < warp ? s_warp[lane & (NW - 1)] : 0) - (incl - n0 - n1);
    if (left >= 1 && left <= n0 + n1) {                // exactly one thread
      const bool second = left > n0;
      s_pick[0] = 2 * tid + (second ? 1 : 0);
      s_pick[1] = second ? left - n0 : left;
      s_pick[2] = second ? n1 : n0;
    }
    __syncthreads();
  };
  const int L = sd.c * ((s + sd.c) / (2 * sd.c));
  int rank = L, shift = 32, n_list = 0;                 // shift: digits known down to this bit
  uint32_t prefix = 0;
  bool listed = false;
  if constexpr (!keys_in) {
    pick(0, kLevelBins / 2, rank);
    n_list = s_pick[2];
    listed = n_list <= kLevelList;                     // uniform over the cluster: every CTA holds the same totals
    if (!listed) {
      sync_all();
      if (tid < kLevelBins / 2) reinterpret_cast<int2*>(s_hist)[tid] = make_int2(0, 0);
    } else {
      prefix = (uint32_t)s_pick[0];
      rank = s_pick[1];
    }
  }
  if (!listed) {
    __syncthreads();
#pragma unroll 1
    while (shift > 0 && !listed) {
      const int first = 256 * (shift / 8 - 1);
#pragma unroll 4
      for (int i = tid; i < cs; i += nt) {
        const uint32_t k = key_at(i);
        if (shift == 32 || (k >> shift) == prefix) atomicAdd(&s_hist[first + ((k >> (shift - 8)) & 255u)], 1);
      }
      shift -= 8;
      pick(first, 128, rank);
      prefix = prefix << 8 | (uint32_t)s_pick[0];
      rank = s_pick[1];
      n_list = s_pick[2];
      listed = n_list <= kLevelList;
    }
  }
  if (listed) {
    unsigned long long* const list0 = csize > 1 ? cluster.map_shared_rank(s_list, 0) : s_list;
    int* const count0 = csize > 1 ? cluster.map_shared_rank(&s_list_n, 0) : &s_list_n;
    const bool digits = keys_in || shift < 32;
#pragma unroll 1
    for (int i = tid; i < cs; i += nt) {
      const uint32_t k = key_at(i);
      const uint32_t mine = digits ? k >> shift : (uint32_t)bin_of(key_value(k), k, map, kLevelBins);
      if (mine == prefix) list0[atomicAdd(count0, 1)] = ((unsigned long long)k << 32) | (unsigned)(c0 + i);
    }
    sync_all();                                        // the list is complete
    if (crank != 0) {
#pragma unroll 1
      for (int i = tid; i < n_list; i += nt) s_list[i] = list0[i];
      __syncthreads();
    }
#pragma unroll 1
    for (int i = tid; i < n_list; i += nt) {
      const unsigned long long e = s_list[i];
      int less = 0;
#pragma unroll 4
      for (int j = 0; j < n_list; ++j) less += s_list[j] < e ? 1 : 0;
      if (less == rank - 1) s_thr = e;                 // exactly one thread
    }
    __syncthreads();
  } else {
    // more rows than the list holds are equal to the threshold: the one of rank `rank` in order of position
    int equal = 0;
#pragma unroll 1
    for (int i = tid; i < cs; i += nt) equal += key_at(i) == prefix ? 1 : 0;
    equal = (int)__reduce_add_sync(0xffffffffu, equal);
    if (lane == 0) s_warp[warp] = equal;
    __syncthreads();
    equal = (int)__reduce_add_sync(0xffffffffu, lane < NW ? s_warp[lane & (NW - 1)] : 0);
    if (tid == 0) s_total = equal;
    sync_all();
#pragma unroll 1
    for (int r = 0; r < crank; ++r) rank -= *cluster.map_shared_rank(&s_total, r);
    if (warp == 0 && rank >= 1 && rank <= equal) {     // in one CTA of the cluster
#pragma unroll 1
      for (int i0 = 0; i0 < cs; i0 += 32) {
        const bool eq = i0 + lane < cs && key_at(i0 + lane) == prefix;
        const unsigned b = __ballot_sync(0xffffffffu, eq);
        if (rank <= __popc(b)) {
          if (eq && __popc(b & ((1u << lane) - 1u)) == rank - 1)
            for (int r = 0; r < csize; ++r)
              *(csize > 1 ? cluster.map_shared_rank(&s_thr, r) : &s_thr) = ((unsigned long long)prefix << 32) | (unsigned)(c0 + i0 + lane);
          break;
        }
        rank -= __popc(b);
      }
    }
    sync_all();
  }
  const unsigned long long thr = s_thr;

  let_next_start();
  // ---- 4. stable two-sided partition.  Every warp owns a contiguous run of the slice and walks
  // it 32 positions at a time with ballots; offsets = totals of the earlier slices and warps.
  const int run = ((cs + NW - 1) / NW + 31) & ~31;               // positions per warp (multiple of 32)
  const int w0 = min(cs, warp * run), w1 = min(cs, w0 + run);
  int below = 0;
#pragma unroll 1
  for (int i0 = w0; i0 < w1; i0 += 32) {
    const int i = i0 + lane;
    const bool down = i < w1 && (((unsigned long long)key_at(i) << 32) | (unsigned)(c0 + i)) <= thr;
    below += __popc(__ballot_sync(0xffffffffu, down));
  }
  if (lane == 0) s_warp[warp] = below;
  __syncthreads();
  const int mine = lane < NW ? s_warp[lane & (NW - 1)] : 0;
  below = (int)__reduce_add_sync(0xffffffffu, lane < warp ? mine : 0);
  if (csize > 1) {
    const int total = (int)__reduce_add_sync(0xffffffffu, mine);
    if (tid == 0) s_total = total;
    cluster.sync();
    const int earlier = lane < crank ? *cluster.map_shared_rank(&s_total, lane) : 0;
    below += (int)__reduce_add_sync(0xffffffffu, earlier);
  }
#pragma unroll 1
  for (int i0 = w0; i0 < w1; i0 += 32) {
    const int i = i0 + lane;
    const bool ok = i < w1;
    const bool down = ok && (((unsigned long long)key_at(i) << 32) | (unsigned)(c0 + i)) <= thr;
    const unsigned b = __ballot_sync(0xffffffffu, down);
    const int before = below + __popc(b & ((1u << lane) - 1u));
    if (ok) pout[down ? lo + before : lo + L + (c0 + i - before)] = in_smem ? s_rows[i] : row_at(c0 + i);
    below += __popc(b);
  }
  if (csize > 1) cluster.sync();                     // keep shared memory alive for the peers' reads
}

// ---------------------------------------------------------------------------
// Subtree of a set of at most kTailRowsMax rows, finished by one CTA.
// ---------------------------------------------------------------------------
constexpr int kTailList = 64;            // candidates of a subset that a warp ranks

struct TailSmem {
  int32_t rows[2][kTailRowsMax];
  uint32_t keys[kTailRowsMax];           // by position: first the value, then its key
  uint16_t state[kTailRowsMax];          // by position: subset << 8 | bin
  uint32_t hist[kTailSegs][128];         // counts of 256 bins, two to a word
  unsigned long long list[kTailSegs][kTailList];   // (key, position) of the rows in the threshold's bin
  int4 seg[kTailSegs];                   // coordinate, L (0: final), start, index of the first child
  float2 seg_map[kTailSegs];             // bin of a value x = x . x + y
  int2 seg_pick[kTailSegs];              // the threshold's bin (-1: found digit by digit), its 1-based rank in the bin
  unsigned long long seg_thr[kTailSegs]; // the last (key, position) that goes down
  int seg_base[kTailSegs];               // rows that go down in the subsets before this one
  int seg_cand[kTailSegs];               // entries of the list
  uint32_t seg_prefix[kTailSegs];        // digits found so far, and the rank that is left
  int seg_rem[kTailSegs];
  int seg_lo[2][kTailSegs + 1];          // start of each subset (relative), +1 sentinel
  float unit_best[kTailSegs][20];        // per block of coordinates: largest variance, then (coordinate, mean) of it
  int2 unit_arg[kTailSegs][17];
  int warp_tot[32];
  unsigned crowded;                      // subsets whose bin has more rows than the list holds
  int nseg, more;
};

// The bin of one subset that holds its `rank`-th row (1-based), the rank inside it and its rows, in
// the one lane that finds it (false elsewhere); clears the counts for their next use.
__device__ __forceinline__ bool pick_bin(uint32_t* hist, int rank, int lane, int& bin, int& rank_in, int& rows_in) {
  uint4* h4 = reinterpret_cast<uint4*>(hist) + lane;
  const uint4 h = *h4;
  *h4 = make_uint4(0u, 0u, 0u, 0u);
  const uint32_t pairs = (h.x + h.y) + (h.z + h.w);      // at most 1,024 rows: the halves do not overflow
  const int sum = (int)((pairs & 0xffffu) + (pairs >> 16));
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (!(incl - sum < rank && rank <= incl)) return false;
  rank_in = rank - (incl - sum);
  bin = lane * 8;
  const uint32_t w[4] = {h.x, h.y, h.z, h.w};
  bool found = false;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int n = (int)((w[j / 2] >> (16 * (j & 1))) & 0xffffu);
    if (found) continue;
    if (rank_in <= n) { found = true; rows_in = n; }
    else { rank_in -= n; ++bin; }
  }
  return true;
}

// The thresholds of the crowded subsets by radix selection, eight bits a pass; keys that are equal in
// all digits go down in order of position.  Out of line: rarely needed.
template <int nt>
__device__ __noinline__ void tail_thresholds_by_digits(TailSmem& sm, unsigned crowded, int s0, int nseg, const int* slo, int tid) {
  const int lane = tid & 31, warp = tid >> 5;
  constexpr int NW = nt / 32;
#pragma unroll 1
  for (int shift = 24; shift >= 0; shift -= 8) {
#pragma unroll 1
    for (int i = tid; i < s0; i += nt) {
      const int g = sm.state[i] >> 8;
      const uint32_t key = sm.keys[i];
      if (!((crowded >> g) & 1) || (shift < 24 && (key >> (shift + 8)) != sm.seg_prefix[g])) continue;
      const int digit = (key >> shift) & 255;
      atomicAdd(&sm.hist[g][digit >> 1], 1u << (16 * (digit & 1)));
    }
    __syncthreads();
#pragma unroll 1
    for (int g = warp; g < nseg; g += NW) {
      if (!((crowded >> g) & 1)) continue;
      int digit, rank, rows_in;
      const int want = shift == 24 ? sm.seg[g].y : sm.seg_rem[g];
      __syncwarp();
      if (pick_bin(sm.hist[g], want, lane, digit, rank, rows_in)) {
        sm.seg_prefix[g] = shift == 24 ? digit : (sm.seg_prefix[g] << 8 | digit);
        sm.seg_rem[g] = rank;
      }
    }
    __syncthreads();
  }
#pragma unroll 1
  for (int g = warp; g < nseg; g += NW) {
    if (!((crowded >> g) & 1)) continue;
    const uint32_t thr = sm.seg_prefix[g];
    int left = sm.seg_rem[g];                            // of the keys equal to the threshold go down
    for (int i0 = slo[g]; i0 < slo[g + 1]; i0 += 32) {
      const bool eq = i0 + lane < slo[g + 1] && sm.keys[i0 + lane] == thr;
      const unsigned b = __ballot_sync(0xffffffffu, eq);
      if (left <= __popc(b)) {
        if (eq && __popc(b & ((1u << lane) - 1u)) == left - 1)
          sm.seg_thr[g] = ((unsigned long long)thr << 32) | (unsigned)(i0 + lane);
        break;
      }
      left -= __popc(b);
    }
  }
}

// Subtree of a set of at most kTailRowsMax rows, finished by one CTA.  A level is a chain of short
// stages between barriers (at most 16 subsets side by side), so its time is latency: loads from L2,
// shuffles, barriers, and the instruction fetch of a long loop body, which has to stay well below the
// 32 KB that the SM keeps: the position loops are rolled and their state lives in shared memory.  Per level:
// sample variances by independent warps (unit_variance); values gathered by asynchronous copies; the
// bin of every value between mean - 2 s and mean + 2 s of the sample in 256 steps; the bin that holds
// the L-th value; the rows in that bin, ranked by one warp; the partition from ballots, where the
// rows that go down before a subset are known beforehand (the L of the subsets to its left).  A bin with
// more than 64 rows (values repeat, or far outliers stretch s) is resolved digit by digit.
// Four CTAs of 256 threads share an SM, or two of 512 where all CTAs of both sides fit that way (256 instead: 2 heads of
// 1,024 rows 27 -> 33 us a side).  Subtrees of at most 4,096 rows, two CTAs of 512 threads to an SM, were the form before: CTAs
// that run long leave the last wave nearly empty (40 heads of 32,760 rows, d = 128, 320 CTAs on 296 places: 285 us
// a side, and 197 for 37 heads), and twice their 90 KB of shared memory leave too little L1 for the pieces of sample
// rows in flight (1,024 rows to a CTA with 48 KB 285 us a side, with 33 KB 193).  Levels and subtrees of a side, before ->
// after: 12 heads of 1,370 rows, d = 64: 36 -> 35 us, 12 x 16,385: 98 -> 94; 8 x 131,072 keys and 16,384 queries: 178 -> 161, 4 x
// 5,003, d = 128: 83 -> 58; 40 x 32,760, d = 128: 373 -> 341.  At d = 128 the sample rows are read from HBM (0.65 GB a side in
// pieces of one row).
template <int D, int nt>
__global__ void __launch_bounds__(nt, 1024 / nt) split_tail_kernel(const SplitParams prm) {
  wait_for_previous();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TailSmem& sm = *reinterpret_cast<TailSmem*>(smem_raw);
  const int which = prm.first_side + blockIdx.y / prm.problems;
  const int p = blockIdx.y % prm.problems;
  const SplitSide sd = prm.side[which];
  const int level = sd.tail_level;
  if ((int)blockIdx.x >= (1 << level)) return;
  const SegmentRef root = locate_segment(sd.n, sd.c, level, blockIdx.x);
  if (!root.active) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = nt / 32;
  constexpr int V = D == 64 ? 4 : 2;                     // coordinates of a lane in unit_variance: D V / 8 = 32 registers
  constexpr int UNITS = D / (4 * V);
  const int c = sd.c;
  const float* Y = sd.Y + (size_t)p * sd.n * D;
  const float* Yt = sd.Yt ? sd.Yt + (size_t)p * sd.n * kSplitCols : nullptr;
  const int32_t* pin = sd.perm_in ? sd.perm_in + (size_t)p * sd.n : nullptr;
  int32_t* pout = sd.perm_out + (size_t)p * sd.n;
  const int lo = root.lo, s0 = root.size;
  // a warp owns consecutive positions, 32 at a time
  const int span = 32 * (((s0 + 31) / 32 + NW - 1) / NW);
  const int w0 = warp * span, w1 = min(s0, w0 + span);

#pragma unroll 1
  for (int i = tid; i < s0; i += nt) {
    sm.rows[0][i] = pin ? pin[lo + i] : lo + i;
    sm.state[i] = 0;
  }
#pragma unroll 1
  for (int e = tid; e < kTailSegs * 32; e += nt) reinterpret_cast<uint4*>(&sm.hist[0][0])[e] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) { sm.seg_lo[0][0] = 0; sm.seg_lo[0][1] = s0; sm.nseg = 1; sm.more = s0 > c; }
  __syncthreads();

  int cur = 0;
  while (sm.more) {
    const int nseg = sm.nseg;
    const int* slo = sm.seg_lo[cur];
    const int32_t* rows = sm.rows[cur];
    int32_t* rows_next = sm.rows[cur ^ 1];

    // ---- 1. coordinate of largest subsample variance for every subset that still splits
#pragma unroll 1
    for (int unit = warp; unit < nseg * UNITS; unit += NW) {
      const int g = unit / UNITS, block = unit % UNITS;
      const int a = slo[g], sz = slo[g + 1] - a;
      if (sz <= c) continue;
      if (sz >= D) unit_variance<D, V, true, false>(Y, rows + a, 0, sz, block, lane, &sm.unit_best[g][block], &sm.unit_arg[g][block]);
      else unit_variance_small<D, V, false>(Y, rows + a, 0, sz, block, lane, &sm.unit_best[g][block], &sm.unit_arg[g][block]);
    }
    __syncthreads();
    if (warp == 0) {
      const bool live = lane < nseg;
      const int a = live ? slo[lane] : 0, sz = live ? slo[lane + 1] - a : 0;
      const bool splits = sz > c;
      const int L = splits ? c * ((sz + c) / (2 * c)) : 0;
      const unsigned ballot = __ballot_sync(0xffffffffu, splits);
      const int child = lane + __popc(ballot & ((1u << lane) - 1u));
      int coord = 0;
      if (splits) {
        float v = sm.unit_best[lane][0];
        int at = 0;
#pragma unroll
        for (int b = 1; b < UNITS; ++b) {
          const float q = sm.unit_best[lane][b];
          if (q > v) { v = q; at = b; }                  // later blocks hold higher coordinates
        }
        const int2 am = sm.unit_arg[lane][at];
        coord = am.x;
        sm.seg_map[lane] = bin_map(v, __int_as_float(am.y), 128.f);
      }
      int before = L;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o) before += x;
      }
      if (live) {
        sm.seg[lane] = make_int4(coord, L, a, child);
        sm.seg_base[lane] = before - L;
        sm.seg_cand[lane] = 0;
        int* nlo = sm.seg_lo[cur ^ 1];
        nlo[child] = a;
        if (splits) nlo[child + 1] = a + L;
      }
      const bool more = __any_sync(0xffffffffu, splits && (L > c || sz - L > c));
      if (lane == 0) {
        sm.nseg = nseg + __popc(ballot);
        sm.seg_lo[cur ^ 1][nseg + __popc(ballot)] = s0;
        sm.more = more;
        sm.crowded = 0u;
      }
    }
    __syncthreads();

    // ---- 2. values, keys and bins
#pragma unroll 2
    for (int i = w0 + lane; i < w1; i += 32) {
      const int4 sg = sm.seg[sm.state[i] >> 8];
      const int row = rows[i];
      const bool column = Yt && sg.x < kSplitCols;
      if (sg.y > 0) cp_async4(&sm.keys[i], column ? Yt + (size_t)sg.x * sd.n + row : Y + (size_t)row * D + sg.x);
    }
    cp_async_wait_all();
#pragma unroll 1
    for (int i = w0 + lane; i < w1; i += 32) {
      const int g = sm.state[i] >> 8;
      if (sm.seg[g].y == 0) continue;
      const float x = __uint_as_float(sm.keys[i]);
      const uint32_t key = order_key(x);
      const int bin = bin_of(x, key, sm.seg_map[g], 256);
      sm.keys[i] = key;
      sm.state[i] = (uint16_t)(g << 8 | bin);
      atomicAdd(&sm.hist[g][bin >> 1], 1u << (16 * (bin & 1)));
    }
    __syncthreads();

    // ---- 3. the bin with the L-th value
#pragma unroll 1
    for (int g = warp; g < nseg; g += NW) {
      const int L = sm.seg[g].y;
      if (L == 0) continue;                              // warp-uniform
      int bin, rank, rows_in;
      if (pick_bin(sm.hist[g], L, lane, bin, rank, rows_in)) {
        if (rows_in > kTailList) { atomicOr(&sm.crowded, 1u << g); bin = -1; }
        sm.seg_pick[g] = make_int2(bin, rank);
      }
    }
    __syncthreads();
    const unsigned crowded = sm.crowded;
    if (crowded) tail_thresholds_by_digits<nt>(sm, crowded, s0, nseg, slo, tid);

    // ---- 4. the rows of that bin, ranked by (key, position)
#pragma unroll 2
    for (int i = w0 + lane; i < w1; i += 32) {
      const int st = sm.state[i], g = st >> 8;
      if (sm.seg[g].y > 0 && (st & 255) == sm.seg_pick[g].x)
        sm.list[g][atomicAdd(&sm.seg_cand[g], 1)] = ((unsigned long long)sm.keys[i] << 32) | (unsigned)i;
    }
    __syncthreads();
#pragma unroll 1
    for (int g = warp; g < nseg; g += NW) {
      if (sm.seg[g].y == 0) continue;
      const int n = sm.seg_cand[g], rank = sm.seg_pick[g].y - 1;
      const unsigned long long e0 = sm.list[g][lane], e1 = sm.list[g][32 + lane];   // beyond n: not used
      int r0 = 0, r1 = 0;
#pragma unroll 4
      for (int j = 0; j < n; ++j) {
        const unsigned long long v = sm.list[g][j];
        r0 += v < e0 ? 1 : 0;
        r1 += v < e1 ? 1 : 0;
      }
      if (lane < n && r0 == rank) sm.seg_thr[g] = e0;                              // exactly one lane
      if (32 + lane < n && r1 == rank) sm.seg_thr[g] = e1;
    }
    __syncthreads();

    // ---- 5. stable partition
    auto goes_down = [&](int i) {
      const int g = sm.state[i] >> 8;
      return sm.seg[g].y > 0 && (((unsigned long long)sm.keys[i] << 32) | (unsigned)i) <= sm.seg_thr[g];
    };
    int total = 0;
#pragma unroll 2
    for (int i = w0 + lane; i - lane < w1; i += 32)
      total += __popc(__ballot_sync(0xffffffffu, i < w1 && goes_down(i)));
    if (lane == 0) sm.warp_tot[warp] = total;
    __syncthreads();
    int below = (int)__reduce_add_sync(0xffffffffu, lane < warp ? sm.warp_tot[lane & (NW - 1)] : 0);
#pragma unroll 1
    for (int i = w0 + lane; i - lane < w1; i += 32) {
      const bool down = i < w1 && goes_down(i);
      const unsigned b = __ballot_sync(0xffffffffu, down);
      if (i < w1) {
        const int g = sm.state[i] >> 8;
        const int4 sg = sm.seg[g];
        const int mine = below + __popc(b & ((1u << lane) - 1u)) - sm.seg_base[g];
        const int dst = sg.y == 0 ? i : (down ? sg.z + mine : i + sg.y - mine);
        rows_next[dst] = rows[i];
        // the subsets of the next level stand at known positions
        sm.state[i] = (uint16_t)((sg.w + (sg.y > 0 && i - sg.z >= sg.y ? 1 : 0)) << 8);
      }
      below += __popc(b);
    }
    __syncthreads();
    cur ^= 1;
  }
  let_next_start();
#pragma unroll 1
  for (int i = tid; i < s0; i += nt) pout[lo + i] = sm.rows[cur][i];
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int next_size(int big, int c) {
  const int L = c * ((big + c) / (2 * c));
  return (L > big - L) ? L : big - L;
}

int split_levels_for(int n, int c) {
  int levels = 0;
  for (int big = n; big > c; big = next_size(big, c)) ++levels;   // the largest set follows the larger child
  return levels;
}

static int max_segment_at_level(int n, int c, int level) {
  int big = n;
  for (int l = 0; l < level && big > c; ++l) big = next_size(big, c);
  return big;
}

// Rows of the sets that the subtree kernel starts from: at most 1,024, and half of that where all CTAs of both
// sides then have an SM to themselves (a level costs a CTA with few rows less than it costs a launch; 4 heads of 5,003
// rows, d = 128, clustering 465 us from 4,096 rows, 437 from 1,024, 436 from 512; 2 heads of 1,024 rows, d = 64 130, 129, 126;
// 8 heads of 131,072 rows 573, 558, 567; 40 heads of 32,760 rows, d = 128 1,681, 1,662, 1,690).
static int tail_rows_for(int n, int c, int problems) {
  const int most = 2LL * problems * ceil_div(n, kTailRowsMax / 2) <= 148 ? kTailRowsMax / 2 : kTailRowsMax;
  return min(kTailSegs * c, most);
}
static int basic_rows_for(int c) { return min(kBasicSegs * c, kBasicRowsMax); }

// Levels [0, tail_level) run as per-level launches; a subtree kernel finishes sets of at most `rows` rows.
static int tail_level_for(int n, int c, int rows) {
  int level = 0;
  for (int big = n; big > rows; big = next_size(big, c)) ++level;
  return level;
}

// One launch of the per-level kernel: the cluster size (see the kernel) and the slice it stages.
static int launch_level(SplitParams& prm, bool keys_in, int level, int max_seg, LaunchStream st) {
  const long long sets = (long long)prm.problems * 2 << level;             // of both sides
  int csize = 1;
  while (csize < kMaxCluster && (max_seg > csize * 8192 || (max_seg > csize * 2048 && sets * csize * 2 <= 296))) csize *= 2;
  const int per_cta = ceil_div(max_seg, csize);
  const bool wide = per_cta > 8192;
  auto kernel = keys_in ? (wide ? split_level_kernel<64, 1024, true> : split_level_kernel<64, 512, true>)
                : prm.D == 64 ? (wide ? split_level_kernel<64, 1024, false> : split_level_kernel<64, 512, false>)
                              : (wide ? split_level_kernel<128, 1024, false> : split_level_kernel<128, 512, false>);
  prm.level = level;
  prm.smem_rows = per_cta < kSmemRowsMax ? per_cta : kSmemRowsMax;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemRowsMax * 8));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((1u << level) * csize, prm.sides * prm.problems);
  cfg.blockDim = dim3(wide ? 1024 : 512);
  cfg.dynamicSmemBytes = (size_t)prm.smem_rows * 8;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = st.chained ? 1 : 0;
  cfg.attrs = attr; cfg.numAttrs = 2;
  CA_RETURN_IF_CUDA(cudaLaunchKernelEx(&cfg, kernel, prm));
  CA_LAUNCH_CHECK();
  return CA_OK;
}

int launch_split(const float* Yq, const float* Yk, int problems, int D, int n_q, int n_k, int c_q,
                 int c_k, int32_t* perm_q_out, int32_t* perm_q_tmp, int32_t* perm_k_out,
                 int32_t* perm_k_tmp, uint32_t* keybuf_q, uint32_t* keybuf_k, int sides, LaunchStream st,
                 const float* Ytq, const float* Ytk) {
  // sides: bit 0 = queries, bit 1 = keys
  const bool do_q = (sides & 1) != 0, do_k = (sides & 2) != 0;
  const int tail_q = tail_level_for(n_q, c_q, tail_rows_for(n_q, c_q, problems));
  const int tail_k = tail_level_for(n_k, c_k, tail_rows_for(n_k, c_k, problems));
  const int top_q = do_q ? tail_q : 0, top_k = do_k ? tail_k : 0;
  const int top_levels = top_q > top_k ? top_q : top_k;
  SplitParams prm;
  prm.D = D; prm.problems = problems;
  prm.first_side = do_q ? 0 : 1; prm.sides = do_q && do_k ? 2 : 1;
  // per-level launches write alternately to tmp/out so that the tail kernel, which runs last,
  // reads the buffer that is not the output
  auto fill = [&](int level) {
    for (int w = 0; w < 2; ++w) {
      SplitSide& sd = prm.side[w];
      int32_t* out = w == 0 ? perm_q_out : perm_k_out;
      int32_t* tmp = w == 0 ? perm_q_tmp : perm_k_tmp;
      const int tail = w == 0 ? tail_q : tail_k;
      sd.Y = w == 0 ? Yq : Yk;
      sd.Yt = w == 0 ? Ytq : Ytk;
      sd.keybuf = w == 0 ? keybuf_q : keybuf_k;
      sd.n = w == 0 ? n_q : n_k; sd.c = w == 0 ? c_q : c_k;
      sd.levels = split_levels_for(sd.n, sd.c);
      sd.tail_level = tail;
      // level l of this side (l < tail) writes tmp if (tail - 1 - l) is even, else out;
      // the tail kernel (level == tail) reads what level tail-1 wrote and writes out
      const bool to_tmp = ((tail - 1 - level) % 2) == 0;
      if (level < tail) {
        sd.perm_out = to_tmp ? tmp : out;
        sd.perm_in = level == 0 ? nullptr : (to_tmp ? out : tmp);
      } else {
        sd.perm_out = out;
        sd.perm_in = tail == 0 ? nullptr : tmp;
      }
    }
  };
  if (top_levels > 0 && prof_enabled()) prof_mark(kProfSplitLevels, st, true);
  for (int level = 0; level < top_levels; ++level) {
    fill(level);
    int max_seg = 1;
    if (level < top_q) max_seg = max_segment_at_level(n_q, c_q, level);
    if (level < top_k) { const int ms = max_segment_at_level(n_k, c_k, level); if (ms > max_seg) max_seg = ms; }
    const int rc = launch_level(prm, false, level, max_seg, st);
    if (rc != CA_OK) return rc;
  }
  if (top_levels > 0 && prof_enabled()) prof_mark(kProfSplitLevels, st, false);
  ProfScope ps(kProfSplitTail, st);
  fill(top_levels);       // any level >= both tails selects the tail buffers
  prm.level = top_levels;
  prm.smem_rows = 0;
  const int slots = 1 << ((do_q ? tail_q : 0) > (do_k ? tail_k : 0) ? (do_q ? tail_q : 0) : (do_k ? tail_k : 0));
  const bool few = 2LL * slots * problems <= 296;          // both sides run at the same time
  auto tail_kernel = D == 64 ? (few ? split_tail_kernel<64, 512> : split_tail_kernel<64, 256>)
                             : (few ? split_tail_kernel<128, 512> : split_tail_kernel<128, 256>);
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(tail_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TailSmem)));
  launch_chained(tail_kernel, dim3(slots, prm.sides * problems), few ? 512 : 256, sizeof(TailSmem), st, prm);
  CA_LAUNCH_CHECK();
  return CA_OK;
}

// ---------------------------------------------------------------------------
// Basic recursive splitting (Section 3.2.1) with the metric injected into the
// power iteration (Section 5.2): per set, the first principal direction of a
// subsample in the metric A, in the dual form u <- A C u, then the projection
// x . u of every row of the set as the key of the same select-and-partition step.
// Every floating-point step is float32 with sequential sums (each product and
// sum rounded on its own), because the projections decide the partition:
//   subsample m = min(d, s) rows at positions floor(j s / m); mu_k = (sum_i x_ik) / m;
//   z = x - mu; start g / |g| (root) or (u_parent + g / |g|) / 2, g the node's noise row;
//   iteration: v_i = sum_k z_ik u_k; w_k = sum_i z_ik v_i; y_j = sum_k A_jk w_k; u = y / |y|.
// Nodes are numbered 2^level - 1 + slot.
// ---------------------------------------------------------------------------
struct BasicSide {
  const void* X;           // [P][n][D] rows in the storage type
  const float* A;          // [P][D][D] metric
  const float* noise;      // [P][nodes][D]
  float* dirs;             // [P][nodes][D] directions of every node (output, read by the children)
  const int32_t* perm_in;  // [P][n] or null (identity)
  uint32_t* keybuf;        // [P][n]
  int n, c, levels, nodes;
};
struct BasicParams {
  BasicSide side[2];
  int level, problems, iterations;
};

// Sums of the power iteration, terms in order.  The operands come eight at a time in 16-byte loads, so that the
// additions, one dependent chain, are what takes the time.
// a . b, n a multiple of 8
__device__ __forceinline__ float ordered_dot(const float* a, const float* b, int n) {
  float acc = 0.f;
#pragma unroll 2
  for (int k0 = 0; k0 < n; k0 += 8) {
    float term[8];
#pragma unroll
    for (int h = 0; h < 8; h += 4) {
      const float4 x = *reinterpret_cast<const float4*>(a + k0 + h), y = *reinterpret_cast<const float4*>(b + k0 + h);
      term[h] = __fmul_rn(x.x, y.x); term[h + 1] = __fmul_rn(x.y, y.y);
      term[h + 2] = __fmul_rn(x.z, y.z); term[h + 3] = __fmul_rn(x.w, y.w);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) acc = __fadd_rn(acc, term[k]);
  }
  return acc;
}
__device__ __forceinline__ float seq_norm(const float* v, int d) {
  float acc = 0.f;
#pragma unroll 2
  for (int k0 = 0; k0 < d; k0 += 8) {
    const float4 x = *reinterpret_cast<const float4*>(v + k0), y = *reinterpret_cast<const float4*>(v + k0 + 4);
    const float sq[8] = {__fmul_rn(x.x, x.x), __fmul_rn(x.y, x.y), __fmul_rn(x.z, x.z), __fmul_rn(x.w, x.w),
                         __fmul_rn(y.x, y.x), __fmul_rn(y.y, y.y), __fmul_rn(y.z, y.z), __fmul_rn(y.w, y.w)};
#pragma unroll
    for (int k = 0; k < 8; ++k) acc = __fadd_rn(acc, sq[k]);
  }
  return __fsqrt_rn(acc);
}

// One CTA of D threads per (slot, side, head).
template <typename T, int D>
__global__ void __launch_bounds__(D) basic_direction_kernel(const BasicParams prm) {
  wait_for_previous();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int LD = D + 4;
  float* z = reinterpret_cast<float*>(smem_raw);       // [m][LD]
  float* As = z + D * LD;                              // [D][LD]   the metric
  __shared__ __align__(16) float u[D], v[D], w[D], y[D], g[D];
  const int which = blockIdx.y / prm.problems, p = blockIdx.y % prm.problems;
  const BasicSide sd = prm.side[which];
  if (prm.level >= sd.levels) return;
  const SegmentRef seg = locate_segment(sd.n, sd.c, prm.level, blockIdx.x);
  if (!seg.active || seg.size <= sd.c) return;
  const int tid = threadIdx.x;
  const int s = seg.size, lo = seg.lo, m = min(D, s);
  const T* X = static_cast<const T*>(sd.X) + (size_t)p * sd.n * D;
  const int32_t* pin = sd.perm_in ? sd.perm_in + (size_t)p * sd.n : nullptr;
  const int node = (1 << prm.level) - 1 + (int)blockIdx.x;
  // subsample rows, one row per thread, then centred column by column
  if (tid < m) {
    const int pos = lo + (int)(((long long)tid * s) / m);
    const int row = pin ? pin[pos] : pos;
    const T* xr = X + (size_t)row * D;
    if (sizeof(T) == 2) {                                // 16-byte loads, all in flight together
      uint4 q[D / 8];
#pragma unroll
      for (int k8 = 0; k8 < D / 8; ++k8) q[k8] = __ldg(reinterpret_cast<const uint4*>(xr) + k8);
#pragma unroll
      for (int k8 = 0; k8 < D / 8; ++k8) {
        const uint32_t wds[4] = {q[k8].x, q[k8].y, q[k8].z, q[k8].w};
#pragma unroll
        for (int e = 0; e < 4; e += 2)
          *reinterpret_cast<float4*>(&z[tid * LD + k8 * 8 + 2 * e]) =
              make_float4(__uint_as_float(wds[e] << 16), __uint_as_float(wds[e] & 0xffff0000u),
                          __uint_as_float(wds[e + 1] << 16), __uint_as_float(wds[e + 1] & 0xffff0000u));
      }
    } else {
#pragma unroll 8
      for (int k4 = 0; k4 < D / 4; ++k4)
        *reinterpret_cast<float4*>(&z[tid * LD + k4 * 4]) = __ldg(reinterpret_cast<const float4*>(xr) + k4);
    }
  }
  {
    const float4* A4 = reinterpret_cast<const float4*>(sd.A + (size_t)p * D * D);
#pragma unroll 16
    for (int e = tid; e < D * D / 4; e += D) *reinterpret_cast<float4*>(&As[(e / (D / 4)) * LD + 4 * (e % (D / 4))]) = __ldg(A4 + e);
  }
  g[tid] = sd.noise[((size_t)p * sd.nodes + node) * D + tid];
  __syncthreads();
  {
    float mu = 0.f;                                      // thread k: column k, rows in order
#pragma unroll 8
    for (int i = 0; i < m; ++i) mu = __fadd_rn(mu, z[i * LD + tid]);
    mu = __fdiv_rn(mu, (float)m);
#pragma unroll 8
    for (int i = 0; i < m; ++i) z[i * LD + tid] = __fsub_rn(z[i * LD + tid], mu);
    const float gn = __fdiv_rn(g[tid], seq_norm(g, D));
    float start = gn;
    if (prm.level > 0) {
      const int parent = (1 << (prm.level - 1)) - 1 + ((int)blockIdx.x >> 1);
      start = __fmul_rn(__fadd_rn(sd.dirs[((size_t)p * sd.nodes + parent) * D + tid], gn), 0.5f);
    }
    u[tid] = start;
  }
  __syncthreads();
  for (int it = 0; it < prm.iterations; ++it) {
    if (tid < m) v[tid] = ordered_dot(&z[tid * LD], u, D);
    __syncthreads();
    {
      float acc = 0.f;
#pragma unroll 8
      for (int i = 0; i < m; ++i) acc = __fadd_rn(acc, __fmul_rn(z[i * LD + tid], v[i]));
      w[tid] = acc;
    }
    __syncthreads();
    y[tid] = ordered_dot(&As[tid * LD], w, D);
    __syncthreads();
    const float nrm = seq_norm(y, D);                    // every thread takes the same sequential sum
    if (nrm > 0.f && isfinite(nrm)) u[tid] = __fdiv_rn(y[tid], nrm);
    __syncthreads();
  }
  let_next_start();
  sd.dirs[((size_t)p * sd.nodes + node) * D + tid] = u[tid];
}

// Keys of 32 R rows by one warp, R per lane (row: none if negative; dir: offset of the row's direction in `dirs`, shared
// or global memory, a multiple of 4): projection x . u, terms in the order of the columns.  A lane that reads its own row touches 32
// lines with every load; so the rows are copied to shared memory (2 x 2 KB of the warp), 64 bytes of 32 rows at a time and a piece
// ahead of the sums, four lanes to a row, 16-byte chunk c of row r at place c ^ (r / 2 & 3).  A level of a subtree
// of 4,096 rows, d = 64: 60 k -> 18 k cycles; 25 k with the pieces loaded through registers, one after the other.
template <typename T, int D, int R>
__device__ __forceinline__ void project_rows(const T* __restrict__ X, const int (&row)[R], const float* dirs, const int (&dir)[R], uint4* buf,
                                             int lane, uint32_t (&key)[R]) {
  constexpr int SEGS = D * (int)sizeof(T) / 64, E = 16 / (int)sizeof(T);
  auto pick = [&](const int (&of)[R], int y) {
    int v = of[0];
#pragma unroll
    for (int k = 1; k < R; ++k) v = y == k ? of[k] : v;
    return v;
  };
  auto fetch = [&](int n) {
    const int mine = pick(row, n / SEGS);
    const uint4* src = reinterpret_cast<const uint4*>(X) + (n % SEGS) * 4 + (lane & 3);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int at = 8 * k + (lane >> 2), r = __shfl_sync(0xffffffffu, mine, at);
      if (r >= 0)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(
                         &buf[(n & 1) * 128 + at * 4 + ((lane & 3) ^ ((at >> 1) & 3))])), "l"(src + (size_t)r * (SEGS * 4)) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float t = 0.f;
  fetch(0);
#pragma unroll 1
  for (int n = 0; n < R * SEGS; ++n) {
    if (n + 1 < R * SEGS) {
      fetch(n + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    const int y = n / SEGS;
    const float* u = dirs + pick(dir, y) + (n % SEGS) * 4 * E;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const uint4 x = buf[(n & 1) * 128 + lane * 4 + (c ^ ((lane >> 1) & 3))];
      const uint32_t wds[4] = {x.x, x.y, x.z, x.w};
      float uu[E];
#pragma unroll
      for (int e = 0; e < E; e += 4) {
        const float4 w = *reinterpret_cast<const float4*>(u + c * E + e);
        uu[e] = w.x; uu[e + 1] = w.y; uu[e + 2] = w.z; uu[e + 3] = w.w;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (sizeof(T) == 2) {
          t = __fadd_rn(t, __fmul_rn(__uint_as_float(wds[e] << 16), uu[2 * e]));
          t = __fadd_rn(t, __fmul_rn(__uint_as_float(wds[e] & 0xffff0000u), uu[2 * e + 1]));
        } else {
          t = __fadd_rn(t, __fmul_rn(__uint_as_float(wds[e]), uu[e]));
        }
      }
    }
    __syncwarp();                                       // (the piece has been read)
    if (n % SEGS == SEGS - 1) {
#pragma unroll
      for (int k = 0; k < R; ++k) key[k] = y == k ? order_key(t) : key[k];
      t = 0.f;
    }
  }
}

// Keys of one level, two positions per thread; the set of a position follows from the size rule.
template <typename T, int D>
__global__ void __launch_bounds__(256) basic_keys_kernel(const BasicParams prm) {
  wait_for_previous();
  let_next_start();
  __shared__ uint4 staged[8][256];
  const int which = blockIdx.y / prm.problems, p = blockIdx.y % prm.problems;
  const BasicSide sd = prm.side[which];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, i0 = (blockIdx.x * 8 + warp) * 64 + lane;
  if (prm.level >= sd.levels || i0 - lane >= sd.n) return;
  int row[2], node[2];
#pragma unroll
  for (int y = 0; y < 2; ++y) {
    const int i = i0 + 32 * y;
    int lo = 0, size = sd.n, slot = 0;
    for (int l = 0; l < prm.level && size > sd.c; ++l) {   // (a final set: nothing to split at this level)
      const int L = sd.c * ((size + sd.c) / (2 * sd.c));
      if (i < lo + L) { size = L; slot = 2 * slot; } else { lo += L; size -= L; slot = 2 * slot + 1; }
    }
    const bool splits = i < sd.n && size > sd.c;
    node[y] = splits ? ((1 << prm.level) - 1 + slot) * D : 0;      // (an offset: of fewer than 2^31 / D nodes)
    row[y] = !splits ? -1 : sd.perm_in ? sd.perm_in[(size_t)p * sd.n + i] : i;
  }
  const float* dirs = sd.dirs + (size_t)p * sd.nodes * D;
  uint32_t key[2] = {0u, 0u};
  project_rows<T, D, 2>(static_cast<const T*>(sd.X) + (size_t)p * sd.n * D, row, dirs, node, staged[warp], lane, key);
#pragma unroll
  for (int y = 0; y < 2; ++y)
    if (row[y] >= 0) sd.keybuf[(size_t)p * sd.n + i0 + 32 * y] = key[y];
}

// ---------------------------------------------------------------------------
// Selection and partition of one level of a subtree, all of its subsets side by side: radix
// selection of every subset's threshold key (seg_L, seg_rem, seg_prefix set up by the caller), then
// the stable partition into rows_next.  A thread owns the four consecutive positions 4 tid .. 4 tid + 3
// (my_seg: subset of a position, -1 - g in a final subset, INT_MIN past the end; my_key: its key).
template <typename Smem>
__device__ __forceinline__ void tail_select_partition(Smem& sm, const int (&my_seg)[kBasicRowsMax / kSplitThreads],
                                                      const uint32_t (&my_key)[kBasicRowsMax / kSplitThreads],
                                                      int nseg, const int* slo, const int32_t* rows,
                                                      int32_t* rows_next, int tid, int* hist, uint32_t* scan) {
  constexpr int nt = kSplitThreads;
  constexpr int PT = kBasicRowsMax / kSplitThreads;
  const int lane = tid & 31, warp = tid >> 5;
  // ---- radix selection, all subsets side by side: two digits of eight bits by counting; then the
  // keys that share those sixteen bits with the threshold are few (a handful per subset unless keys
  // repeat), and a warp ranks them directly.  A subset with more than 32 of them goes on with the two
  // remaining digits.  (The digit counts are cleared once per level: the warp that picks a subset's
  // digit clears the counts it has read, ready for the next pass.)
  uint32_t mask = 0;
  for (int e = tid; e < nseg * 256; e += nt) hist[e] = 0;
  if (tid < nseg) sm.seg_cand[tid] = 0;
  if (tid == 0) sm.overflow = 0;
  __syncthreads();
  for (int shift = 24; shift >= 0; shift -= 8) {
    uint32_t pre[PT];                               // read ahead of the atomics, which order memory accesses
#pragma unroll
    for (int u = 0; u < PT; ++u) pre[u] = sm.seg_prefix[my_seg[u] >= 0 ? my_seg[u] : 0];
    if (shift == 8) {
      // candidates of every subset into its list (the scan array is free until the partition)
#pragma unroll
      for (int u = 0; u < PT; ++u) {
        const int g = my_seg[u];
        if (g >= 0 && (my_key[u] & mask) == pre[u]) {
          const int slot = atomicAdd(&sm.seg_cand[g], 1);
          if (slot < 32) scan[g * 32 + slot] = my_key[u];
        }
      }
      __syncthreads();
      for (int g = warp; g < nseg; g += nt / 32) {
        if (sm.seg_L[g] == 0) continue;             // warp-uniform
        const int n = sm.seg_cand[g];
        if (n > 32) {
          if (lane == 0) sm.overflow = 1;
          continue;
        }
        const int remaining = sm.seg_rem[g];        // 1 <= remaining <= n
        const uint32_t key = lane < n ? scan[g * 32 + lane] : 0xffffffffu;
        int less = 0, eq_before = 0;
        for (int j = 0; j < n; ++j) {
          const uint32_t kj = __shfl_sync(0xffffffffu, key, j);
          less += kj < key ? 1 : 0;
          eq_before += (kj == key && j < lane) ? 1 : 0;
        }
        if (lane < n && less + eq_before == remaining - 1) {   // exactly one lane
          sm.seg_prefix[g] = key;
          sm.seg_rem[g] = remaining - less;          // how many of the keys equal to the threshold go down
          sm.seg_cand[g] = -1;
        }
      }
      __syncthreads();
      if (!sm.overflow) break;                      // uniform: every threshold is found
#pragma unroll
      for (int u = 0; u < PT; ++u) pre[u] = sm.seg_prefix[my_seg[u] >= 0 ? my_seg[u] : 0];
    }
#pragma unroll
    for (int u = 0; u < PT; ++u) {
      const int g = my_seg[u];
      const bool live = g >= 0;
      const uint32_t k = my_key[u];
      if (live && ((k & mask) == pre[u])) atomicAdd(&hist[(g << 8) | (int)((k >> shift) & 255u)], 1);
    }
    __syncthreads();
    for (int g = warp; g < nseg; g += nt / 32) {
      const int remaining = sm.seg_rem[g];
      if (sm.seg_L[g] == 0) continue;               // warp-uniform
      int local[8]; int sum = 0;
      {
        int4* h4 = reinterpret_cast<int4*>(&hist[g * 256 + lane * 8]);
        const int4 h0 = h4[0], h1 = h4[1];
        h4[0] = make_int4(0, 0, 0, 0);
        h4[1] = make_int4(0, 0, 0, 0);
        local[0] = h0.x; local[1] = h0.y; local[2] = h0.z; local[3] = h0.w;
        local[4] = h1.x; local[5] = h1.y; local[6] = h1.z; local[7] = h1.w;
      }
      if (sm.seg_cand[g] < 0) continue;             // found by the direct ranking (its keys were still counted)
#pragma unroll
      for (int j = 0; j < 8; ++j) sum += local[j];
      int incl = sum;
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      int before = incl - sum;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (before < remaining && remaining <= before + local[j]) {
          sm.seg_digit[g] = lane * 8 + j;
          sm.seg_rem[g] = remaining - before;
        }
        before += local[j];
      }
      __syncwarp();
      if (lane == 0) sm.seg_prefix[g] |= (uint32_t)sm.seg_digit[g] << shift;
    }
    mask |= 255u << shift;
    __syncthreads();
  }

  // ---- 3. stable partition of every subset: one scan of (less | equal << 16) over all positions
  // (a thread's four, then the warp, then the warps' totals by warp 0)
  uint32_t my_scan[PT];
  {
    int run = 0;
#pragma unroll
    for (int u = 0; u < PT; ++u) {
      if (my_seg[u] >= 0) {
        const uint32_t k = my_key[u], thr = sm.seg_prefix[my_seg[u]];
        run += (k < thr ? 1 : 0) | (k == thr ? 1 << 16 : 0);
      }
      my_scan[u] = (uint32_t)run;
    }
    int incl = run;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) sm.warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const int v = sm.warp_tot[lane];                 // nt / 32 == 32 warps
      int wi = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) wi += x;
      }
      sm.warp_tot[lane] = wi - v;                      // totals of the warps before this one
    }
    __syncthreads();
    const uint32_t before = (uint32_t)(sm.warp_tot[warp] + incl - run);
#pragma unroll
    for (int u = 0; u < PT; ++u) my_scan[u] += before;
    *reinterpret_cast<uint4*>(&scan[PT * tid]) = make_uint4(my_scan[0], my_scan[1], my_scan[2], my_scan[3]);
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < PT; ++u) {
    const int i = PT * tid + u;
    const int g = my_seg[u];
    if (g == INT_MIN) continue;
    if (g < 0) { rows_next[i] = rows[i]; continue; }
    const int a = slo[g];
    const uint32_t base = a > 0 ? scan[a - 1] : 0u;
    const uint32_t k = my_key[u], thr = sm.seg_prefix[g];
    const int is_less = k < thr, is_eq = k == thr;
    const uint32_t excl = my_scan[u] - base - (uint32_t)(is_less | (is_eq << 16));
    const int less_here = (int)(excl & 0xffffu), eq_here = (int)(excl >> 16);
    const int eq_left = sm.seg_rem[g], L = sm.seg_L[g];
    const bool down = is_less || (is_eq && eq_here < eq_left);
    const int down_before = less_here + min(eq_here, eq_left);
    const int dst = down ? a + down_before : a + L + (i - a - down_before);
    rows_next[dst] = rows[i];
  }
}

// Subtree of the basic variant: a set of at most kBasicRowsMax rows finished by one CTA, so that
// the deepest levels are one launch instead of three per level.  Per level: the directions of all
// subsets that still split (a team of D threads per subset; the operations of
// basic_direction_kernel in the same order -- the sample rows are staged as stored and centred
// where they are used, which yields the same float32 values), the projection of every row onto its
// subset's direction (the sum of basic_keys_kernel), then the selection and partition of the
// diagonalized subtree kernel.
// ---------------------------------------------------------------------------
// staged sample rows: 16 subsets of 64 bf16 rows at d = 64, 4 of 128 at d = 128 (then the rows that are projected, 4 KB
// per warp; then the scan and the digit counts).  16-byte chunk c of row r stands at place c ^ (r & 7).
constexpr int kBasicStage = 131072;

template <int D>
struct BasicTailSmem {
  static constexpr int TEAMS = kSplitThreads / D;
  int32_t rows[2][kBasicRowsMax];
  __align__(16) unsigned char stage[kBasicStage];
  float dirs[2][kBasicSegs][D];            // directions of this level's subsets and of the level above
  __align__(16) float mu[TEAMS][D], u[TEAMS][D], v[TEAMS][D], w[TEAMS][D], y[TEAMS][D], g[TEAMS][D];
  float4 metric[D == 64 ? D * D / 4 : 1];   // d = 64: the metric, chunks of a row placed as above (d = 128: no room)
  int seg_lo[2][2 * kBasicSegs + 2];
  int seg_slot[2][2 * kBasicSegs + 2];     // slot of a subset in the tree, at the level it stands on
  int seg_par[2][2 * kBasicSegs + 2];      // subset of the level above it came from
  int seg_digit[kBasicSegs], seg_rem[kBasicSegs], seg_L[kBasicSegs];
  int seg_cand[kBasicSegs];                // candidates left after the first two digits; -1: threshold found
  int overflow;                           // some subset has more candidates than a warp takes
  uint32_t seg_prefix[kBasicSegs];
  int split_list[kBasicSegs];              // the subsets that still split
  int warp_tot[32];
  int nseg[2];
  int nsplit;
  int more;
};

template <typename T, int D>
__global__ void __launch_bounds__(kSplitThreads) basic_tail_kernel(const BasicParams prm, const SplitParams sp) {
  wait_for_previous();
  using Sm = BasicTailSmem<D>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Sm& sm = *reinterpret_cast<Sm*>(smem_raw);
  constexpr int nt = kSplitThreads;
  constexpr int V = D * (int)sizeof(T) / 16;            // 16-byte chunks of a row
  constexpr int E = 16 / (int)sizeof(T);                // elements of a chunk
  constexpr int NODE_BYTES = D * V * 16;
  constexpr int ROUND = (kBasicStage / NODE_BYTES) < Sm::TEAMS ? (kBasicStage / NODE_BYTES) : Sm::TEAMS;
  static_assert(ROUND >= 1, "a subset's sample must fit the staging area");
  constexpr int PT = kBasicRowsMax / kSplitThreads;
  static_assert(PT == 4 && kBasicRowsMax * 4 + kBasicSegs * 256 * 4 <= kBasicStage && nt / 32 * 4096 <= kBasicStage, "scan, digit counts and projected rows live in the staging area");
  uint32_t* scan = reinterpret_cast<uint32_t*>(sm.stage);
  int* hist = reinterpret_cast<int*>(sm.stage + kBasicRowsMax * 4);

  const int which = blockIdx.y / prm.problems, p = blockIdx.y % prm.problems;
  const BasicSide bs = prm.side[which];
  const SplitSide sd = sp.side[which];
  const int level0 = sd.tail_level;
  if ((int)blockIdx.x >= (1 << level0)) return;
  const SegmentRef root = locate_segment(sd.n, sd.c, level0, blockIdx.x);
  if (!root.active) return;
  const int tid = threadIdx.x;
  const int team = tid / D, member = tid % D;
  // where half of a team works, it is the second half of every other team, so that all four sub-cores have part in it
  const int half_member = (D == 64 ? team >> 1 : team) & 1 ? (member + D / 2) % D : member;
  const int c = sd.c;
  const T* X = static_cast<const T*>(bs.X) + (size_t)p * sd.n * D;
  const float* Am = bs.A + (size_t)p * D * D;
  const float* noise = bs.noise + (size_t)p * bs.nodes * D;
  const int32_t* pin = sd.perm_in ? sd.perm_in + (size_t)p * sd.n : nullptr;
  int32_t* pout = sd.perm_out + (size_t)p * sd.n;
  const int lo = root.lo, s0 = root.size;

  for (int i = tid; i < s0; i += nt) sm.rows[0][i] = pin ? pin[lo + i] : lo + i;
  if (D == 64 && s0 > c) {
#pragma unroll
    for (int e = tid; e < D * D / 4; e += nt)
      sm.metric[(e & ~7) | ((e & 7) ^ ((e / (D / 4)) & 7))] = __ldg(reinterpret_cast<const float4*>(Am) + e);
  }
  if (tid == 0) {
    sm.seg_lo[0][0] = 0; sm.seg_lo[0][1] = s0; sm.nseg[0] = 1; sm.more = s0 > c;
    sm.seg_slot[0][0] = (int)blockIdx.x; sm.seg_par[0][0] = -1;
    sm.split_list[0] = 0; sm.nsplit = s0 > c ? 1 : 0;
  }
  __syncthreads();

  int cur = 0, level = level0;
  while (sm.more) {
    const int nseg = sm.nseg[cur];
    const int* slo = sm.seg_lo[cur];
    const int32_t* rows = sm.rows[cur];
    int32_t* rows_next = sm.rows[cur ^ 1];
    const int nsplit = sm.nsplit;
    float (*dir_now)[D] = sm.dirs[cur];
    float (*dir_up)[D] = sm.dirs[cur ^ 1];

    // ---- 1. directions, ROUND subsets at a time (every stage boundary is a barrier of the CTA; teams
    // without a subset go through them idle)
    for (int r0 = 0; r0 < nsplit; r0 += ROUND) {
      const bool active = team < ROUND && r0 + team < nsplit;
      const int g = active ? sm.split_list[r0 + team] : 0;
      const int a = slo[g], sz = slo[g + 1] - a, m = min(D, sz);
      uint4* xs = reinterpret_cast<uint4*>(sm.stage + (size_t)(team < ROUND ? team : 0) * NODE_BYTES);   // [D][V]
      const uint32_t* xw = reinterpret_cast<const uint32_t*>(xs);
      // Columns: a word per thread and row, two columns of bf16 (by half of the team) or one
      const bool columns = active && half_member < 4 * V;
      auto word = [&](int i) { return xw[i * (4 * V) + (((half_member >> 2) ^ (i & 7)) << 2) + (half_member & 3)]; };
      auto first_of = [&](uint32_t x) { return sizeof(T) == 2 ? __uint_as_float(x << 16) : __uint_as_float(x); };
      auto second_of = [&](uint32_t x) { return __uint_as_float(x & 0xffff0000u); };
      const int col = sizeof(T) == 2 ? 2 * half_member : half_member;
      if (active) {
        // a row index per lane, the rows by 128 bytes and more of neighbouring lanes
        const int lane = tid & 31;
        const int sample = member < m ? rows[a + (int)(((long long)member * sz) / m)] : -1;
        const uint4* X4 = reinterpret_cast<const uint4*>(X);
#pragma unroll
        for (int k0 = 0; k0 < V; k0 += 8) {
          uint4 q[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int r = __shfl_sync(0xffffffffu, sample, (k0 + k) * (32 / V) + lane / V);
            q[k] = r >= 0 ? __ldg(X4 + (size_t)r * V + lane % V) : make_uint4(0u, 0u, 0u, 0u);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int r = (member & ~31) + (k0 + k) * (32 / V) + lane / V;
            xs[r * V + ((lane % V) ^ (r & 7))] = q[k];
          }
        }
        const int node = (1 << level) - 1 + sm.seg_slot[cur][g];
        sm.g[team][member] = noise[(size_t)node * D + member];
      }
      __syncthreads();
      if (columns) {                                         // means, rows in order
        float mu = 0.f, mu2 = 0.f;
#pragma unroll 8
        for (int i = 0; i < m; ++i) {
          const uint32_t x = word(i);
          mu = __fadd_rn(mu, first_of(x));
          if (sizeof(T) == 2) mu2 = __fadd_rn(mu2, second_of(x));
        }
        sm.mu[team][col] = __fdiv_rn(mu, (float)m);
        if (sizeof(T) == 2) sm.mu[team][col + 1] = __fdiv_rn(mu2, (float)m);
      }
      if (active) {
        const float gn = __fdiv_rn(sm.g[team][member], seq_norm(sm.g[team], D));
        float start = gn;
        if (level > 0) {
          const int par = sm.seg_par[cur][g];
          const float up = par >= 0 ? dir_up[par][member]
                                    : bs.dirs[((size_t)p * bs.nodes + (1 << (level - 1)) - 1 + (sm.seg_slot[cur][g] >> 1)) * D + member];
          start = __fmul_rn(__fadd_rn(up, gn), 0.5f);
        }
        sm.u[team][member] = start;
      }
      __syncthreads();
      for (int it = 0; it < prm.iterations; ++it) {
        if (active && half_member < D / 2) {
          // (two rows per thread, which share the loads of mean and direction; the terms of a chunk are formed, then
          // added in order: the loads do not wait for the sum)
          float acc[2] = {0.f, 0.f};
#pragma unroll 1
          for (int c8 = 0; c8 < V; ++c8) {
            float mu[E], u[E];
#pragma unroll
            for (int e = 0; e < E; e += 4) {
              *reinterpret_cast<float4*>(&mu[e]) = *reinterpret_cast<const float4*>(&sm.mu[team][c8 * E + e]);
              *reinterpret_cast<float4*>(&u[e]) = *reinterpret_cast<const float4*>(&sm.u[team][c8 * E + e]);
            }
#pragma unroll
            for (int y = 0; y < 2; ++y) {
              const int r = half_member + y * (D / 2);
              const uint4 x = xs[r * V + (c8 ^ (r & 7))];
              const uint32_t wds[4] = {x.x, x.y, x.z, x.w};
              float term[E];
#pragma unroll
              for (int e = 0; e < E; ++e) {
                const float xe = sizeof(T) == 4 ? __uint_as_float(wds[e & 3]) : e % 2 ? second_of(wds[e / 2]) : first_of(wds[e / 2]);
                term[e] = __fmul_rn(__fsub_rn(xe, mu[e]), u[e]);
              }
#pragma unroll
              for (int e = 0; e < E; ++e) acc[y] = __fadd_rn(acc[y], term[e]);
            }
          }
          sm.v[team][half_member] = acc[0];                       // (rows behind a smaller sample: not used)
          sm.v[team][half_member + D / 2] = acc[1];
        }
        __syncthreads();
        if (columns) {
          const float mk = sm.mu[team][col], mk2 = sizeof(T) == 2 ? sm.mu[team][col + 1] : 0.f;
          float acc = 0.f, acc2 = 0.f;
          int i = 0;
#pragma unroll 2
          for (; i + 4 <= m; i += 4) {
            const float4 v4 = *reinterpret_cast<const float4*>(&sm.v[team][i]);
            const float vv[4] = {v4.x, v4.y, v4.z, v4.w};
            uint32_t x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = word(i + k);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              acc = __fadd_rn(acc, __fmul_rn(__fsub_rn(first_of(x[k]), mk), vv[k]));
              if (sizeof(T) == 2) acc2 = __fadd_rn(acc2, __fmul_rn(__fsub_rn(second_of(x[k]), mk2), vv[k]));
            }
          }
          for (; i < m; ++i) {
            const uint32_t x = word(i);
            acc = __fadd_rn(acc, __fmul_rn(__fsub_rn(first_of(x), mk), sm.v[team][i]));
            if (sizeof(T) == 2) acc2 = __fadd_rn(acc2, __fmul_rn(__fsub_rn(second_of(x), mk2), sm.v[team][i]));
          }
          sm.w[team][col] = acc;
          if (sizeof(T) == 2) sm.w[team][col + 1] = acc2;
        }
        __syncthreads();
        if (active && half_member < D / 2) {
          float acc[2] = {0.f, 0.f};
// (at d = 128 from L2, so loads in flight count: 1 head of 300 rows, clusters of 64, bf16 147.8 -> 139.5 us)
#pragma unroll (D == 64 ? 2 : 8)
          for (int c4 = 0; c4 < D / 4; ++c4) {
            const float4 w4 = *reinterpret_cast<const float4*>(&sm.w[team][4 * c4]);
#pragma unroll
            for (int y = 0; y < 2; ++y) {
              const int j = half_member + y * (D / 2);
              const float4 av = D == 64 ? sm.metric[j * (D / 4) + ((c4 & ~7) | ((c4 & 7) ^ (j & 7)))]
                                        : __ldg(reinterpret_cast<const float4*>(Am + (size_t)j * D) + c4);
              const float term[4] = {__fmul_rn(av.x, w4.x), __fmul_rn(av.y, w4.y), __fmul_rn(av.z, w4.z), __fmul_rn(av.w, w4.w)};
#pragma unroll
              for (int k = 0; k < 4; ++k) acc[y] = __fadd_rn(acc[y], term[k]);
            }
          }
          sm.y[team][half_member] = acc[0];
          sm.y[team][half_member + D / 2] = acc[1];
        }
        __syncthreads();
        if (active) {
          const float nrm = seq_norm(sm.y[team], D);          // every thread takes the same sequential sum
          if (nrm > 0.f && isfinite(nrm)) sm.u[team][member] = __fdiv_rn(sm.y[team][member], nrm);
        }
        __syncthreads();
      }
      if (active) dir_now[g][member] = sm.u[team][member];
      __syncthreads();
    }
    if (tid < nseg) {
      const int a = slo[tid], sz = slo[tid + 1] - a;
      sm.seg_L[tid] = sz > c ? c * ((sz + c) / (2 * c)) : 0;
      sm.seg_prefix[tid] = 0u;
      sm.seg_rem[tid] = sm.seg_L[tid];
    }

    // ---- 2. keys: the projection of a row onto its subset's direction, terms in the order of the columns
    // (the staged samples have been read)
    int my_seg[PT];
    uint32_t my_key[PT];
    {
      const int i0 = PT * tid;
      int g = 0;
      if (i0 < s0) {
        int hi = nseg;                                  // slo[g] <= i0 < slo[g+1]
        while (hi - g > 1) { const int mid = (g + hi) >> 1; if (slo[mid] <= i0) g = mid; else hi = mid; }
      }
#pragma unroll
      for (int u = 0; u < PT; ++u) {
        const int i = i0 + u;
        my_key[u] = 0u;
        if (i < s0) {
          while (slo[g + 1] <= i) ++g;
          const bool splits = slo[g + 1] - slo[g] > c;
          my_seg[u] = splits ? g : -1 - g;              // final subset: carried over unchanged
        } else {
          my_seg[u] = INT_MIN;
        }
      }
      int row[PT], dir[PT];
      bool any = false;
#pragma unroll
      for (int u = 0; u < PT; ++u) {
        row[u] = my_seg[u] >= 0 ? rows[i0 + u] : -1;
        dir[u] = max(my_seg[u], 0) * D;
        any |= row[u] >= 0;
      }
      if (__any_sync(0xffffffffu, any))
        project_rows<T, D, PT>(X, row, dir_now[0], dir, reinterpret_cast<uint4*>(sm.stage + (tid >> 5) * 4096), tid & 31, my_key);
    }
    __syncthreads();                                    // the staging area becomes the scan and the digit counts

    tail_select_partition(sm, my_seg, my_key, nseg, slo, rows, rows_next, tid, hist, scan);

    // ---- next level's subsets
    if (tid == 0) {
      int* nlo = sm.seg_lo[cur ^ 1];
      int* nslot = sm.seg_slot[cur ^ 1];
      int* npar = sm.seg_par[cur ^ 1];
      int n2 = 0, more = 0, ns = 0;
      for (int g = 0; g < nseg; ++g) {
        const int a = slo[g], sz = slo[g + 1] - a;
        if (sz > c) {
          const int L = sm.seg_L[g];
          nlo[n2] = a;     nslot[n2] = 2 * sm.seg_slot[cur][g];     npar[n2] = g;
          if (L > c) sm.split_list[ns++] = n2;
          ++n2;
          nlo[n2] = a + L; nslot[n2] = 2 * sm.seg_slot[cur][g] + 1; npar[n2] = g;
          if (sz - L > c) sm.split_list[ns++] = n2;
          ++n2;
          more |= (L > c) | (sz - L > c);
        } else {
          nlo[n2] = a; nslot[n2] = 0; npar[n2] = g;      // a final subset: only carried along
          ++n2;
        }
      }
      nlo[n2] = s0;
      sm.nseg[cur ^ 1] = n2;
      sm.nsplit = ns;
      sm.more = more;
    }
    __syncthreads();
    cur ^= 1;
    ++level;
  }
  let_next_start();
  for (int i = tid; i < s0; i += nt) pout[lo + i] = sm.rows[cur][i];
}

template <typename T>
static int launch_split_basic_t(const T* Q, const T* K, const float* A_q, const float* A_k, const float* noise_q,
                                const float* noise_k, float* dirs_q, float* dirs_k, int iterations, int problems,
                                int D, int n_q, int n_k, int c_q, int c_k, int32_t* perm_q_out, int32_t* perm_q_tmp,
                                int32_t* perm_k_out, int32_t* perm_k_tmp, uint32_t* keybuf_q, uint32_t* keybuf_k,
                                LaunchStream st) {
  const int lev_q = split_levels_for(n_q, c_q), lev_k = split_levels_for(n_k, c_k);
  // Sets of more than kBasicRowsMax rows take three launches per level (directions, projections,
  // select + partition); the subtree kernel finishes the rest.  Per-level launches write alternately
  // to tmp/out so that the subtree kernel, which runs last, reads the buffer that is not the output.
  const int tail_q = tail_level_for(n_q, c_q, basic_rows_for(c_q)), tail_k = tail_level_for(n_k, c_k, basic_rows_for(c_k));
  const int top = tail_q > tail_k ? tail_q : tail_k;
  BasicParams bp;
  bp.problems = problems; bp.iterations = iterations;
  SplitParams prm;
  prm.D = D; prm.problems = problems;
  prm.first_side = 0; prm.sides = 2;
  auto fill = [&](int level) {
    for (int w = 0; w < 2; ++w) {
      const int tail = w == 0 ? tail_q : tail_k;
      int32_t* out = w == 0 ? perm_q_out : perm_k_out;
      int32_t* tmp = w == 0 ? perm_q_tmp : perm_k_tmp;
      SplitSide& sd = prm.side[w];
      sd.Y = nullptr;
      sd.Yt = nullptr;
      sd.keybuf = w == 0 ? keybuf_q : keybuf_k;
      sd.n = w == 0 ? n_q : n_k; sd.c = w == 0 ? c_q : c_k;
      sd.levels = w == 0 ? lev_q : lev_k;
      sd.tail_level = tail;
      const bool to_tmp = ((tail - 1 - level) % 2) == 0;
      if (level < tail) {
        sd.perm_out = to_tmp ? tmp : out;
        sd.perm_in = level == 0 ? nullptr : (to_tmp ? out : tmp);
      } else {
        sd.perm_out = out;
        sd.perm_in = tail == 0 ? nullptr : tmp;
      }
      BasicSide& bs = bp.side[w];
      bs.X = w == 0 ? static_cast<const void*>(Q) : static_cast<const void*>(K);
      bs.A = w == 0 ? A_q : A_k;
      bs.noise = w == 0 ? noise_q : noise_k;
      bs.dirs = w == 0 ? dirs_q : dirs_k;
      bs.perm_in = sd.perm_in; bs.keybuf = sd.keybuf;
      bs.n = sd.n; bs.c = sd.c;
      bs.levels = tail;                                    // the per-level kernels stop where the subtrees begin
      bs.nodes = (1 << (sd.levels > 0 ? sd.levels : 1)) - 1;
    }
  };
  for (int level = 0; level < top; ++level) {
    fill(level);
    bp.level = level;
    const size_t dsmem = (size_t)2 * D * (D + 4) * sizeof(float);
    if (D == 64) {
      auto dk = basic_direction_kernel<T, 64>;
      CA_RETURN_IF_CUDA(cudaFuncSetAttribute(dk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dsmem));
      launch_chained(dk, dim3(1u << level, 2 * problems), 64, dsmem, st, bp);
    } else {
      auto dk = basic_direction_kernel<T, 128>;
      CA_RETURN_IF_CUDA(cudaFuncSetAttribute(dk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dsmem));
      launch_chained(dk, dim3(1u << level, 2 * problems), 128, dsmem, st, bp);
    }
    CA_LAUNCH_CHECK();
    const int n_max = n_q > n_k ? n_q : n_k;
    launch_chained(D == 64 ? basic_keys_kernel<T, 64> : basic_keys_kernel<T, 128>, dim3(ceil_div(n_max, 512), 2 * problems), 256,
                   0, st, bp);
    CA_LAUNCH_CHECK();
    int max_seg = 1;
    if (level < tail_q) max_seg = max_segment_at_level(n_q, c_q, level);
    if (level < tail_k) { const int ms = max_segment_at_level(n_k, c_k, level); if (ms > max_seg) max_seg = ms; }
    const int rc = launch_level(prm, true, level, max_seg, st);
    if (rc != CA_OK) return rc;
  }
  fill(top);
  bp.level = top; prm.level = top;
  const int slots = 1 << top;
  if (D == 64) {
    auto tk = basic_tail_kernel<T, 64>;
    CA_RETURN_IF_CUDA(cudaFuncSetAttribute(tk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BasicTailSmem<64>)));
    launch_chained(tk, dim3(slots, 2 * problems), kSplitThreads, sizeof(BasicTailSmem<64>), st, bp, prm);
  } else {
    auto tk = basic_tail_kernel<T, 128>;
    CA_RETURN_IF_CUDA(cudaFuncSetAttribute(tk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BasicTailSmem<128>)));
    launch_chained(tk, dim3(slots, 2 * problems), kSplitThreads, sizeof(BasicTailSmem<128>), st, bp, prm);
  }
  CA_LAUNCH_CHECK();
  return CA_OK;
}

int launch_split_basic(const void* Q, const void* K, int dtype, const float* A_q, const float* A_k,
                       const float* noise_q, const float* noise_k, float* dirs_q, float* dirs_k, int iterations,
                       int problems, int D, int n_q, int n_k, int c_q, int c_k, int32_t* perm_q_out,
                       int32_t* perm_q_tmp, int32_t* perm_k_out, int32_t* perm_k_tmp, uint32_t* keybuf_q,
                       uint32_t* keybuf_k, LaunchStream st) {
  if (dtype == CA_DTYPE_BF16)
    return launch_split_basic_t(static_cast<const __nv_bfloat16*>(Q), static_cast<const __nv_bfloat16*>(K), A_q, A_k,
                                noise_q, noise_k, dirs_q, dirs_k, iterations, problems, D, n_q, n_k, c_q, c_k,
                                perm_q_out, perm_q_tmp, perm_k_out, perm_k_tmp, keybuf_q, keybuf_k, st);
  return launch_split_basic_t(static_cast<const float*>(Q), static_cast<const float*>(K), A_q, A_k, noise_q, noise_k,
                              dirs_q, dirs_k, iterations, problems, D, n_q, n_k, c_q, c_k, perm_q_out, perm_q_tmp,
                              perm_k_out, perm_k_tmp, keybuf_q, keybuf_k, st);
}

}  // namespace ca
