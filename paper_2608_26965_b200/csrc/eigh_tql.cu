// Principal components of the transformed rows (Section 3.2.1, diagonalized
// variant), one CTA per head and side: builds the d x d covariance, decomposes
// it, and writes the projection that the split coordinates are computed with.
//
// Prologue.  Keys: the transformed keys K F (F F^T = M the query metric, Section
// 3.2.2) have covariance F^T C_K F / n_k with C_K the centred scatter of the keys,
// formed here from the Gram matrix and the column sums of K (two d x d x d
// products in shared memory, no pass over the data).  Queries: the covariance of
// the representation r(q) from its Gram matrix and column sums.
//
// Decomposition (d = 64, 128; float32: the bases only feed fp32 coordinates), in three parts.
// 1. Householder reduction to tridiagonal form.  For k = 0 .. d-3 the reflector H = I - beta v v^T of row k,
// v = x - alpha e_{k+1}, x the row right of the diagonal, takes A to H A H.  A step is a chain of latencies
// (barrier, shuffles, root), so what counts is how short the chain is and how few instructions stand in it.  With
// y = A x, row k + 1 of H A H right of its diagonal is H y / alpha: every thread forms the next x for itself from the
// published y, one barrier per step and two sums over the threads of a row, and the update of A (A - v p^T - u v^T
// with p = beta A v = beta (y - alpha A e_{k+1}), u = p - beta (v.p) v) is off the chain.  (Before: two barriers
// and three sums, the next row published behind the update; 58 k and 184 k cycles for d = 64 / 128, now 47 k and
// 160 k by itself.)  The warps that the reduction does not use apply the reflectors, a block behind, to the
// rows of the factor F (another 3 k and 25 k cycles of the reduction's time, against 12 k and 52 k for applying them to the
// eigenvectors of the tridiagonal matrix at the end, by all warps).
// 2. Divide and conquer.  The tridiagonal matrix is cut into blocks of kBase rows (a cut writes
// T = diag(T1, T2) + rho u u^T), each diagonalised by one lane with Jacobi rotations, then merged pairwise up to
// the whole.  A merge solves
// diag(d) + rho z z^T, z the eigenvectors' components at the cut: poles sorted, negligible weights and
// coinciding poles deflated, the roots of the secular equation by an iteration that treats the
// nearest pole exactly (a few threads per root; offsets from that pole keep the differences
// d_j - x accurate), the weights recomputed from the roots (Gu and Eisenstat, 1994) so that the
// eigenvectors stay orthogonal to rounding, and one product with the blocks' eigenvectors, which leaves out their zeros.
// 3. W = (F Q) S, Q the product of the reflectors and S the eigenvectors of T.
// SM cycles of a launch (12 heads, d = 64 / 40 heads, d = 128; queries): covariance 2.5 k / 11 k (keys 11 k / 60 k),
// reduction 51 k / 187 k, base blocks 5 k / 10 k, merges 50 k / 103 k, map 4.5 k / 26 k, output 4.5 k / 11 k;
// in all 120 k / 352 k, where it took 152 k / 437 k.
//
// Epilogue.  Components in order of descending eigenvalue.  With E the
// eigenvectors and F the factor that produced the transformed rows, the map from
// the original space to the coordinates is F E; component t is oriented so that
// the entry of largest magnitude (lowest row on ties) of column t of F E is
// positive -- a rule that gives the same signs whatever root of the metric F is.
// Written out: the projection matrix W (F E where rows are projected from the original
// space, the keys always and the queries of bf16 storage; E for the queries of fp32
// storage, whose representation is kept) or W^T as bf16 hi + lo parts for the
// tensor-core projection, and its bias -mean . F E, or . E where the mean is one of
// transformed rows.
#include <type_traits>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace ca {

using namespace ptx;

namespace {

__device__ __forceinline__ float sum2(f32x2 v) {
  float lo, hi;
  unpack2(v, lo, hi);
  return lo + hi;
}

__device__ __forceinline__ void named_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int count) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

constexpr int kThreads = 512;
constexpr int kBaseLog = 2, kBase = 1 << kBaseLog;   // rows of a base block of the divide and conquer
constexpr int kMaxSweeps = 12;
// The reduction multiplies up to three entries (x . A x), of which those of directions with little variance are small: it runs on
// the matrix with 2^20 as its largest diagonal entry, so that products of entries down to 1e-15 of that are normal numbers.
constexpr float kReduceScale = 1048576.f;

// Eigenvalues that are not numbers (the covariance of rows with infinities, or whose sums overflow) stand as +inf: the
// rank of a pole among the others is then a permutation for every input, and indexes stay in range.
__device__ __forceinline__ float pole_value(float x) { return fminf(x, INFINITY); }

// ---- eigen-decomposition of the 4 x 4 blocks on the diagonal of a tridiagonal matrix (de[i] = (diagonal i, coupling of
// i and i + 1); the coupling behind a block's last row is not part of it), a block per lane of one warp:
// cyclic Jacobi rotations in registers, two disjoint ones at a time.  Four sweeps or so of three rounds, against one
// dependent chain of rotations per eigenvalue with the implicit-shift QL iteration (a warp per block): 2.5 k
// cycles where that took 8-9 k at d = 64 and 14-15 k at d = 128.  Eigenvectors become rows of Qt.
__device__ __forceinline__ void jacobi_blocks(float2* de, int blocks, float* Qt, int lda, int lane) {
  static_assert(kBase == 4, "rounds of a 4 x 4 matrix");
  const bool mine = lane < blocks;
  float m[4][4], v[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 d = mine ? de[4 * lane + i] : make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] = i == j ? 1.f : 0.f;
#pragma unroll
    for (int j = i + 1; j < 4; ++j) m[i][j] = m[j][i] = j == i + 1 ? d.y : 0.f;
    m[i][i] = d.x;
  }
  // zero to rounding: of the two diagonal entries, or of the whole matrix, whose largest diagonal entry is 1
  auto negligible = [&](int p, int q) { return !(fabsf(m[p][q]) > fmaxf(1e-8f * (fabsf(m[p][p]) + fabsf(m[q][q])), 1e-18f)); };
  auto rotate = [&](int p, int q) {
    const float x = m[p][q], d = m[q][q] - m[p][p];
    float root, inv;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(root) : "f"(fmaf(d, d, 4.f * x * x)));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(fabsf(d) + root));
    const float t = negligible(p, q) ? 0.f : copysignf(2.f * inv, d) * x;          // tangent of the angle
    const float n = fmaf(t, t, 1.f);
    float c;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(n));
    c = c * fmaf(-0.5f * n, c * c, 1.5f);
    const float sn = t * c;
    m[p][p] = fmaf(-t, x, m[p][p]);
    m[q][q] = fmaf(t, x, m[q][q]);
    m[p][q] = m[q][p] = t == 0.f ? x : 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k != p && k != q) {
        const float a = m[k][p], b = m[k][q];
        m[k][p] = m[p][k] = fmaf(c, a, -sn * b);
        m[k][q] = m[q][k] = fmaf(sn, a, c * b);
      }
      const float a = v[k][p], b = v[k][q];
      v[k][p] = fmaf(c, a, -sn * b);
      v[k][q] = fmaf(sn, a, c * b);
    }
  };
#pragma unroll 1
  for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
    const bool done = negligible(0, 1) && negligible(0, 2) && negligible(0, 3) && negligible(1, 2) && negligible(1, 3) && negligible(2, 3);
    if (__all_sync(0xffffffffu, done)) break;
    rotate(0, 1); rotate(2, 3);
    rotate(0, 2); rotate(1, 3);
    rotate(0, 3); rotate(1, 2);
  }
  if (mine) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      de[4 * lane + i].x = pole_value(m[i][i]);
      *reinterpret_cast<float4*>(&Qt[(4 * lane + i) * lda + 4 * lane]) = make_float4(v[0][i], v[1][i], v[2][i], v[3][i]);
    }
  }
}

}  // namespace

// d x d x d products in shared memory, a tile of 8 x TJ of the result per thread (128 threads of 8 x 4 at d = 64, 256 of
// 8 x 8 at d = 128): a 16-byte load costs four cycles of shared memory whether its lanes read one address or eight, so
// that what counts is how many multiply-adds it feeds.  With 4 x 4 tiles the products took 4.1 k (d = 64) and
// 26-30 k cycles, all of it shared memory.  The lanes of a quarter-warp read distinct banks.
template <int D>
struct Tile {
  static constexpr int TI = 8, TJ = D == 64 ? 4 : 8, NUMBER = D * D / (TI * TJ), COLS = D / TJ;
  static_assert(NUMBER <= kThreads, "a tile per thread");
  int i, j;                                            // rows 8 i .., columns 4 j + (D / 2) c .. or j + COLS c
  bool live;
  __device__ __forceinline__ explicit Tile(int tid) : i(tid / COLS), j(tid % COLS), live(tid < NUMBER) {}
};

// Terms are added for k = 0, 1, ... in that order; column b of a tile is 4 tj + b (b < 4) or d / 2 + 4 tj + b - 4.
//   XT = false: acc[a][b] = sum_k X[(8 ti + a) lda + k] Y[k lda + column b]
//   XT = true:  acc[a][b] = sum_k X[k lda + 8 ti + a]   Y[k lda + column b]
template <int D, bool XT>
__device__ __forceinline__ void tile_product(const float* __restrict__ X, const float* __restrict__ Y, int lda, const Tile<D>& t,
                                             float (&acc)[Tile<D>::TI][Tile<D>::TJ]) {
  constexpr int TI = Tile<D>::TI, TJ = Tile<D>::TJ;
#pragma unroll
  for (int x = 0; x < TI; ++x)
#pragma unroll
    for (int y = 0; y < TJ; ++y) acc[x][y] = 0.f;
#pragma unroll 1
  for (int k0 = 0; k0 < D; k0 += 4) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float y[TJ], x[TI];
#pragma unroll
      for (int c = 0; c < TJ; c += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&Y[(k0 + e) * lda + 4 * t.j + (D / 8) * c]);
        y[c] = v.x; y[c + 1] = v.y; y[c + 2] = v.z; y[c + 3] = v.w;
      }
      if (XT) {
#pragma unroll
        for (int r = 0; r < TI; r += 4) {
          const float4 v = *reinterpret_cast<const float4*>(&X[(k0 + e) * lda + TI * t.i + r]);
          x[r] = v.x; x[r + 1] = v.y; x[r + 2] = v.z; x[r + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int r = 0; r < TI; ++r) x[r] = X[(TI * t.i + r) * lda + k0 + e];
      }
#pragma unroll
      for (int r = 0; r < TI; ++r)
#pragma unroll
        for (int c = 0; c < TJ; ++c) acc[r][c] = fmaf(x[r], y[c], acc[r][c]);
    }
  }
}

// acc[a][c] = sum_k X[(8 ti + a) lda + k] Yr[(tj + COLS c) lda + k]   (both operands by rows, terms in order)
template <int D>
__device__ __forceinline__ void tile_product_rows(const float* __restrict__ X, const float* __restrict__ Yr, int lda, const Tile<D>& t,
                                                  float (&acc)[Tile<D>::TI][Tile<D>::TJ]) {
  constexpr int TI = Tile<D>::TI, TJ = Tile<D>::TJ;
#pragma unroll
  for (int x = 0; x < TI; ++x)
#pragma unroll
    for (int y = 0; y < TJ; ++y) acc[x][y] = 0.f;
#pragma unroll 1
  for (int k0 = 0; k0 < D; k0 += 4) {
    float4 y[TJ];
#pragma unroll
    for (int c = 0; c < TJ; ++c) y[c] = *reinterpret_cast<const float4*>(&Yr[(t.j + Tile<D>::COLS * c) * lda + k0]);
#pragma unroll
    for (int r = 0; r < TI; ++r) {
      const float4 v = *reinterpret_cast<const float4*>(&X[(TI * t.i + r) * lda + k0]);
#pragma unroll
      for (int c = 0; c < TJ; ++c)
        acc[r][c] = fmaf(v.w, y[c].w, fmaf(v.z, y[c].z, fmaf(v.y, y[c].y, fmaf(v.x, y[c].x, acc[r][c]))));
    }
  }
}

// ---- merge of two adjacent blocks of the tridiagonal matrix whose eigen-decompositions are known
// (rows [b0, b0 + NB) of Qt are their eigenvectors, zero outside their block's columns, de[].x their
// eigenvalues): with the cut before row b0 + NB / 2, u = e_{cut - 1} + theta e_cut, and z = Q^T u, the
// eigen-decomposition of diag(d) + rho2 z z^T with z scaled to unit length (rho2 = 2 rho).
// Run by a group of T threads per row (lt = index in the group); the new
// rows go to rows [b0, b0 + NB) of L; every array of `scratch` is used at [b0, b0 + NB), so groups on
// disjoint blocks run side by side.
// One instance of the code serves all levels (NB = 2^lg rows): code that runs once per launch is fetched
// from L2 or beyond at 3 to 14 cycles per instruction.
template <int D>
__device__ __noinline__ void merge_blocks(float* __restrict__ Qt, float* __restrict__ L, float* __restrict__ A,
                                          float2* de, float* scratch, int lg, float rho, float theta, int lt, int grp) {
  constexpr int LDA = D + 4, T = kThreads / D;
  const int NB = 1 << lg, GT = T * NB, b0 = grp * NB;
  auto sync = [&]() {
    if (GT == 32) __syncwarp();
    else named_sync(grp + 1, GT);
  };
  const int lane = lt & 31;
  float* ds = scratch + b0;                                // poles in ascending order
  float* zs = ds + D;
  int* ord = reinterpret_cast<int*>(zs + D);               // sorted position -> row of Qt
  int* keep_row = ord + D;                                 // kept pole -> row of Qt
  float* kd = reinterpret_cast<float*>(keep_row + D);      // kept poles, weights
  float* kz = kd + D;
  int* korg = reinterpret_cast<int*>(kz + D);              // root -> pole its offset is measured from
  float* kmu = reinterpret_cast<float*>(korg + D);
  float* kzh = kmu + D;
  float* gc = kzh + D;                                     // plane rotations of the deflation
  float* gs = gc + D;
  int* ga = reinterpret_cast<int*>(gs + D);
  int* gb = ga + D;
  int* defl_row = gb + D;                                  // deflated: row of Qt, eigenvalue
  float* defl_d = reinterpret_cast<float*>(defl_row + D);
  int* counts = reinterpret_cast<int*>(scratch + 15 * D) + 8 * grp;   // kept, rotations, deflated, skip, left, right
  // The rows of the two blocks are zero in the other block's columns (but for those that a rotation has mixed): the
  // columns of the left half take the terms of one list of kept poles, those of the right half of another, which
  // grows downwards from position NB + 3, each filled up to a multiple of four.  (A rotation takes a pole away for every
  // row that it mixes, so that both fit.)
  int* place = reinterpret_cast<int*>(scratch + 16 * D) + b0;         // kept pole -> positions in the lists (16 bits each, 0xffff: none)
  int* at_row = reinterpret_cast<int*>(scratch + 17 * D) + b0 + 4 * grp;   // position -> row of Qt
  float2* pole = reinterpret_cast<float2*>(scratch + 19 * D) + b0;    // kept pole, squared weight
  int* side = reinterpret_cast<int*>(kzh);                            // kept pole -> halves of its row that are not zero
  const float rho2 = 2.f * rho;
  {
    // rank of a pole among the others, T threads to a pole
    const int i = lt / T;
    const float mine = de[b0 + i].x;
    const int cut = b0 + NB / 2;
    const float z = i < NB / 2 ? Qt[(b0 + i) * LDA + cut - 1] : theta * Qt[(b0 + i) * LDA + cut];
    int rank = 0;
#pragma unroll 4
    for (int k = lt % T; k < NB; k += T) {
      const float other = de[b0 + k].x;
      rank += (other < mine) || (other == mine && k < i);
    }
#pragma unroll
    for (int o = 1; o < T; o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (lt % T == 0) {
      ord[rank] = b0 + i;
      ds[rank] = mine;
      zs[rank] = 0.70710678f * z;
    }
  }
  sync();
  if (lt < 32) {
    float dmax = 0.f, zmax = 0.f;
    for (int j = lane; j < NB; j += 32) { dmax = fmaxf(dmax, fabsf(ds[j])); zmax = fmaxf(zmax, fabsf(zs[j])); }
    // (the bits of floats that are not negative are in their order)
    dmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(dmax)));
    zmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(zmax)));
    const float tol = 8.f * 6e-8f * fmaxf(dmax, zmax);
    const bool skip = !(rho2 * zmax > tol);                // the blocks do not couple, or not by a number: nothing to merge
    int K = 0, ng = 0, nd = 0;
    if (!skip) {
      // negligible weights, a pole per lane
#pragma unroll 1
      for (int base = 0; base < NB; base += 32) {
        const int j = base + lane;
        const bool in = j < NB;
        const float dj = in ? ds[j] : 0.f, zj = in ? zs[j] : 0.f;
        const bool keep = in && rho2 * fabsf(zj) > tol;
        const unsigned mk = __ballot_sync(0xffffffffu, keep), md = __ballot_sync(0xffffffffu, in && !keep);
        const unsigned below = (1u << lane) - 1u;
        if (keep) {
          const int at = K + __popc(mk & below);
          keep_row[at] = ord[j]; kd[at] = dj; kz[at] = zj;
          side[at] = ord[j] < b0 + NB / 2 ? 1 : 2;
        } else if (in) {
          const int at = nd + __popc(md & below);
          defl_row[at] = ord[j]; defl_d[at] = dj;
        }
        K += __popc(mk);
        nd += __popc(md);
      }
      __syncwarp();
      // two poles coincide when |t c s| <= tol, c = z_j / tau, s = -z_prev / tau, tau^2 = z_j^2 + z_prev^2;
      // the test is made without the root and the divisions, which only a deflation needs
      auto coincide = [&](int j) {
        const float zj = kz[j], zp = kz[j - 1];
        return zp != 0.f && fabsf((kd[j] - kd[j - 1]) * zj * zp) <= tol * fmaf(zj, zj, zp * zp);
      };
      unsigned* found = reinterpret_cast<unsigned*>(zs);   // (the sorted lists have been read)
      bool any = false;
#pragma unroll 1
      for (int base = 0; base < K; base += 32) {
        const int j = base + lane;
        const unsigned m = __ballot_sync(0xffffffffu, j > 0 && j < K && coincide(j));
        any = any || m != 0;
        if (lane == 0) found[base >> 5] = m;
      }
      if (any) {
        // A rotation moves the weight of pole j - 1 into pole j, and changes what pole j + 1 is compared
        // with: one thread walks over the pairs found, the poles that give way drop out afterwards.
        if (lane == 0) {
#pragma unroll 1
          for (int c = 0; c < (K + 31) >> 5; ++c) {
            unsigned m = found[c];
#pragma unroll 1
            while (m) {
              int j = 32 * c + __ffs(m) - 1;
              m &= m - 1;
              // (a pair already taken in, or parted by the rotation before, fails the test)
              float dp = kd[j - 1], zp = kz[j - 1];
              int rp = keep_row[j - 1], both = side[j - 1];
              float dj = kd[j], zj = kz[j];
#pragma unroll 1
              for (; j < K; ++j) {
                const float n2 = fmaf(zj, zj, zp * zp);
                if (zp == 0.f || !(fabsf((dj - dp) * zj * zp) <= tol * n2)) break;
                float r;
                asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(n2));
                r = r * fmaf(-0.5f * n2 * r, r, 1.5f);
                const int rj = keep_row[j];
                both |= side[j];
                side[j] = both;
                const float d_next = kd[j + 1], z_next = kz[j + 1];   // (within scratch; not used behind the last pole)
                const float cs = zj * r, sn = -zp * r, cc = cs * cs, ss = sn * sn;
                gc[ng] = cs; gs[ng] = sn; ga[ng] = rp; gb[ng] = rj; ++ng;
                defl_row[nd] = rp; defl_d[nd] = fmaf(dj, ss, dp * cc); ++nd;
                kz[j - 1] = 0.f;                           // mark of a pole that has given way
                dp = fmaf(dj, cc, dp * ss);
                zp = n2 * r;
                rp = rj;
                kd[j] = dp;
                kz[j] = zp;
                dj = d_next;
                zj = z_next;
              }
            }
          }
        }
        __syncwarp();
        int kept = 0;
#pragma unroll 1
        for (int base = 0; base < K; base += 32) {
          const int j = base + lane;
          const float dj = j < K ? kd[j] : 0.f, zj = j < K ? kz[j] : 0.f;
          const int rj = j < K ? keep_row[j] : 0, sj = j < K ? side[j] : 0;
          const unsigned mk = __ballot_sync(0xffffffffu, zj != 0.f);
          if (zj != 0.f) {
            const int at = kept + __popc(mk & ((1u << lane) - 1u));
            keep_row[at] = rj; kd[at] = dj; kz[at] = zj; side[at] = sj;
          }
          kept += __popc(mk);
          __syncwarp();
        }
        K = kept;
        ng = __shfl_sync(0xffffffffu, ng, 0);
        nd = __shfl_sync(0xffffffffu, nd, 0);
      }
      // squared weights of the kept poles; the two lists
      int nl = 0, nr = 0;
      const unsigned below = (1u << lane) - 1u;
#pragma unroll 1
      for (int base = 0; base < K; base += 32) {
        const int j = base + lane;
        const int sj = j < K ? side[j] : 0;
        const unsigned ml = __ballot_sync(0xffffffffu, sj & 1), mr = __ballot_sync(0xffffffffu, sj & 2);
        const int at = nl + __popc(ml & below), at_r = NB + 3 - nr - __popc(mr & below);
        if (j < K) {
          const float zj = kz[j];
          const int row = keep_row[j];
          pole[j] = make_float2(kd[j], zj * zj);
          place[j] = (sj & 1 ? at : 0xffff) | (sj & 2 ? at_r : 0xffff) << 16;
          if (sj & 1) at_row[at] = row;
          if (sj & 2) at_row[at_r] = row;
        }
        nl += __popc(ml);
        nr += __popc(mr);
      }
      // (any row where a list is filled up: its factor is zero)
      if (lane < (-nl & 3)) at_row[nl + lane] = b0;
      if (lane < (-nr & 3)) at_row[NB + 3 - nr - lane] = b0;
      if (lane == 0) { counts[4] = (nl + 3) & ~3; counts[5] = (nr + 3) & ~3; }
    }
    if (lane == 0) { counts[0] = K; counts[1] = ng; counts[2] = nd; counts[3] = skip; }
  }
  sync();
  if (counts[3]) {
    // nothing to merge: the rows move as they are, so that every block ends in L
#pragma unroll 1
    for (int e = lt; e < NB * NB; e += GT)
      L[(b0 + (e >> lg)) * LDA + b0 + (e & (NB - 1))] = Qt[(b0 + (e >> lg)) * LDA + b0 + (e & (NB - 1))];
    sync();
    return;
  }
  const int K = counts[0], ng = counts[1], nd = counts[2], nl = counts[4], nr = counts[5];
  // rotations of the deflation on the rows of Qt (one column per thread, in the order recorded)
  if (ng > 0) {
    if (lt < NB) {
#pragma unroll 1
      for (int g = 0; g < ng; ++g) {
        float* xr = &Qt[ga[g] * LDA + b0 + lt];
        float* yr = &Qt[gb[g] * LDA + b0 + lt];
        const float x = *xr, y = *yr;
        *xr = gc[g] * x + gs[g] * y;
        *yr = gc[g] * y - gs[g] * x;
      }
    }
    sync();
  }
  auto sum_t = [&](float x) {
#pragma unroll
    for (int o = 1; o < T; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  };
  // roots: group i = lt / T of T threads, each with the poles j = sub (mod T)
  const int gi = lt / T, sub = lt % T;
  const bool live = gi < K;
  {
    const int i = live ? gi : 0;
    // the last root lies in (d_{K-1}, d_{K-1} + rho2 |z|^2), |z| = 1 to rounding; every other one between two
    // poles, and the sign of the function half-way says next to which
    const bool last = i >= K - 1;
    const float width = last ? 1.0001f * rho2 : kd[i + 1] - kd[i];
    const float mid = 0.5f * width, d0 = kd[i];
    float acc = 0.f;
#pragma unroll 4
    for (int j = sub; j < K; j += T) {
      const float2 pj = pole[j];
      float inv;                                            // one special-function operation, no rounding fix-up
      asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"((pj.x - d0) - mid));
      acc = fmaf(pj.y, inv, acc);
    }
    const float f_mid = fmaf(rho2, sum_t(acc), 1.f);
    const bool right = !last && f_mid < 0.f;
    const int org = right ? i + 1 : i;
    const float w_org = rho2 * pole[org].y, d_org = kd[org];
    // f(m) = 1 - w_org / m + r(m), r the sum over the other poles: smooth around the root, so it is
    // replaced by its tangent and the pole is kept as it is: the root of b m^2 + a m - w_org = 0 on the
    // origin's side.  Safeguarded by the bracket; a root that has not settled after kSteps is bisected.
    constexpr int kSteps = 10;
    float lo_m = right ? -mid : 0.f, hi_m = right ? 0.f : (last ? width : mid);
    float m = right ? -mid : mid;
    bool done = false;
#pragma unroll 1
    for (int it = 0; it < kSteps + 48; ++it) {
      float r0 = 0.f, r1 = 0.f;
#pragma unroll 4
      for (int j = sub; j < K; j += T) {
        const float2 pj = pole[j];
        float inv;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"((pj.x - d_org) - m));
        const float x = j == org ? 0.f : pj.y * inv;
        r0 += x;
        r1 = fmaf(x, inv, r1);
      }
      r0 = rho2 * sum_t(r0);
      r1 = rho2 * sum_t(r1);
      const float f = (1.f + r0) - __fdividef(w_org, m);
      if (f > 0.f) hi_m = fminf(hi_m, m); else lo_m = fmaxf(lo_m, m);
      const float ca = fmaf(-r1, m, 1.f + r0);
      float disc;
      asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(disc) : "f"(fmaf(ca, ca, 4.f * r1 * w_org)));
      const float cs = right ? -ca : ca;                   // (one expression for both sides: no branches)
      const float mag = __fdividef(cs >= 0.f ? 2.f * w_org : disc - cs, cs >= 0.f ? cs + disc : 2.f * r1);
      float next = right ? -mag : mag;
      // settled: convergence is quadratic, so behind a step of 1e-4 nothing but rounding is left.  The sign of f,
      // which moves the bracket, is rounding too by then: a short step that leaves the bracket ends the search (bisecting a bracket
      // whose other end is still far away starts it again: up to 58 rounds, 14 k cycles of a merge).
      const bool inside = next > lo_m && next < hi_m;
      bool still = fabsf(next - m) <= (inside ? 1e-4f : 1e-3f) * fabsf(m);
      if (!still && (it >= kSteps || !inside)) {
        next = 0.5f * (lo_m + hi_m);
        still = next == lo_m || next == hi_m;
      }
      if (!done) m = next;
      done = done || still;
      if (__all_sync(0xffffffffu, done)) break;
    }
    if (live && sub == 0) { korg[gi] = org; kmu[gi] = m; }
  }
  sync();
  // weights recomputed from the roots: zhat_j^2 = prod_i (x_i - d_j) / (rho2 prod_{i != j} (d_i - d_j))
  {
    const int j = live ? gi : 0;
    const float dj = kd[j];
    float prod = 1.f;
#pragma unroll 2
    for (int i = sub; i < K; i += T) {
      const float num = (kd[korg[i]] - dj) + kmu[i];
      prod *= __fdividef(num, (i == j) ? rho2 : kd[i] - dj);
    }
#pragma unroll
    for (int o = 1; o < T; o <<= 1) prod *= __shfl_xor_sync(0xffffffffu, prod, o);
    if (live && sub == 0) kzh[gi] = copysignf(sqrtf(fabsf(prod)), kz[gi]);
  }
  sync();
  // eigenvector i over the kept poles, normalised, as row b0 + i of A
  {
    const int i = live ? gi : 0;
    const float d0 = K > 0 ? kd[korg[i]] : 0.f, mu = kmu[i];     // (without a kept pole there is no root, and no korg)
    float nrm = 0.f;
#pragma unroll 2
    for (int j = sub; j < K; j += T) {
      const float v = __fdividef(kzh[j], (kd[j] - d0) - mu);
      nrm = fmaf(v, v, nrm);
    }
    const float inv = rsqrtf(sum_t(nrm));
    if (live) {
      float* row = A + (b0 + gi) * LDA;
      if (sub < 4) {                                        // what fills the lists up
        if (nl > sub) row[nl - 1 - sub] = 0.f;
        if (nr > sub) row[NB + 4 - nr + sub] = 0.f;
      }
      __syncwarp(((1u << T) - 1u) << (lane & ~(T - 1)));
#pragma unroll 2
      for (int j = sub; j < K; j += T) {
        const float v = inv * __fdividef(kzh[j], (kd[j] - d0) - mu);
        const unsigned at = place[j];
        if ((at & 0xffffu) != 0xffffu) row[at & 0xffffu] = v;
        if ((at >> 16) != 0xffffu) row[at >> 16] = v;
      }
    }
  }
  sync();
  // rows of the merged basis into L: row b0 + i = sum_j A[b0 + i][place of j] Qt[keep_row[j]] (i < K), then
  // the deflated rows (a 4 x 4 tile per thread, terms in the order of j)
#pragma unroll 1
  for (int tile = lt; tile < NB * NB / 16; tile += GT) {
    const int i0 = 4 * (tile >> (lg - 2)), c = 4 * (tile & (NB / 4 - 1)), c0 = b0 + c;
    if (i0 >= K) break;
    const int first = c < NB / 2 ? 0 : NB + 4 - nr, end = c < NB / 2 ? nl : NB + 4;
    float acc[4][4];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
#pragma unroll 1
    for (int j = first; j < end; j += 4) {
      float xa[4][4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const float4 v = *reinterpret_cast<const float4*>(&A[(b0 + i0 + x) * LDA + j]);
        xa[x][0] = v.x; xa[x][1] = v.y; xa[x][2] = v.z; xa[x][3] = v.w;
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float4 y = *reinterpret_cast<const float4*>(&Qt[at_row[j + kk] * LDA + c0]);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          acc[x][0] = fmaf(xa[x][kk], y.x, acc[x][0]); acc[x][1] = fmaf(xa[x][kk], y.y, acc[x][1]);
          acc[x][2] = fmaf(xa[x][kk], y.z, acc[x][2]); acc[x][3] = fmaf(xa[x][kk], y.w, acc[x][3]);
        }
      }
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (i0 + x < K)
        *reinterpret_cast<float4*>(&L[(b0 + i0 + x) * LDA + c0]) = make_float4(acc[x][0], acc[x][1], acc[x][2], acc[x][3]);
  }
#pragma unroll 1
  for (int e = lt; e < nd * NB; e += GT)
    L[(b0 + K + (e >> lg)) * LDA + b0 + (e & (NB - 1))] = Qt[defl_row[e >> lg] * LDA + b0 + (e & (NB - 1))];
  if (lt < NB) de[b0 + lt].x = pole_value(lt < K ? kd[korg[lt]] + kmu[lt] : defl_d[lt - K]);
  sync();
}

template <int D>
__global__ void __launch_bounds__(kThreads) eigh_tql_kernel(const PcaArgs a) {
  wait_for_previous();
  constexpr int NT = kThreads, LDA = D + 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* A = reinterpret_cast<float*>(smem_raw);       // [D][LDA]
  float* Qt = A + D * LDA;                             // [D][LDA]   rows become the eigenvectors
  float* L = Qt + D * LDA;                             // [D][LDA]   the factor F (prologue, sign rule); merged bases and reflectors in between
  float* refl = A;                                     // rows: the reflectors as they come
  float* ybuf = A + 3 * D * LDA;                       // [2][D]     A times the row to be reflected
  float* abuf = ybuf + 2 * D;                          // [2][D]     the row after it
  float2* de = reinterpret_cast<float2*>(abuf + 2 * D);   // [D]     (diagonal i, sub-diagonal coupling i and i+1)
  float* beta = abuf + 4 * D;                          // [D]        factors of the reflectors
  float* mean = beta + D;                              // [D]
  float* scratch = mean + D;                           // [21 D]     arrays of the merge
  // what is multiplied by the reduction's Q on the way: the factor F, or the identity where E itself is asked for
  const bool need_e = !(a.lift && a.out_lifted);
  __shared__ double s_scale;
  __shared__ unsigned s_largest;
  __shared__ float s_rho[D / kBase], s_theta[D / kBase];   // cut before row i kBase

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t mat = (size_t)blockIdx.x * D * D;
  constexpr int TI = Tile<D>::TI, TJ = Tile<D>::TJ;
  const Tile<D> tile(tid);

  // ---- prologue: the matrix to decompose, in A
  // (16-byte loads, several in flight: the launch starts with nothing else to do)
  auto load_factor = [&]() {
    const double2* F = reinterpret_cast<const double2*>(a.lift + mat);
#pragma unroll 4
    for (int e = tid; e < D * D / 2; e += NT) {
      const double2 f = F[e];
      *reinterpret_cast<float2*>(&L[(2 * e / D) * LDA + 2 * e % D]) = make_float2((float)f.x, (float)f.y);
    }
  };
  if (a.lift) load_factor();
  if (a.mode == kPcaKeys) {
    // C = (gram - s s^T / n) c_scale, the centred scatter of the keys; then alpha F^T C F
    // (double-precision operations are scarce on this part: no division per element)
    const double* G = a.gram + mat;
    const double* sm = a.sum + (size_t)blockIdx.x * D;
    const double cs = a.c_scale, cn = a.c_scale / a.n;
#pragma unroll 4
    for (int e = tid; e < D * D / 2; e += NT) {
      const int i = 2 * e / D, j = 2 * e % D;
      const double2 g = reinterpret_cast<const double2*>(G)[e];
      const double si = -cn * sm[i];
      *reinterpret_cast<float2*>(&A[i * LDA + j]) = make_float2((float)fma(si, sm[j], g.x * cs), (float)fma(si, sm[j + 1], g.y * cs));
    }
    __syncthreads();
    float acc[TI][TJ];
    auto put_tile = [&](float* out, float f) {
#pragma unroll
      for (int x = 0; x < TI; ++x)
#pragma unroll
        for (int c = 0; c < TJ; c += 4)
          *reinterpret_cast<float4*>(&out[(TI * tile.i + x) * LDA + 4 * tile.j + (D / 8) * c]) =
              make_float4(f * acc[x][c], f * acc[x][c + 1], f * acc[x][c + 2], f * acc[x][c + 3]);
    };
    if (tile.live) {
      tile_product<D, true>(L, A, LDA, tile, acc);                                        // F^T C
      put_tile(Qt, 1.f);
    }
    __syncthreads();
    if (tile.live) {
      tile_product<D, false>(Qt, L, LDA, tile, acc);                                      // (F^T C) F
      put_tile(A, (float)a.alpha);
    }
  } else if (a.mode == kPcaQueries) {
    // covariance of the representation from its moments: gram / n - mean mean^T
    const double* G = a.gram + mat;
    const double* sm = a.sum + (size_t)blockIdx.x * D;
    const double inv_n = 1.0 / a.n, inv_n2 = inv_n * inv_n;
#pragma unroll 4
    for (int e = tid; e < D * D / 2; e += NT) {
      const int i = 2 * e / D, j = 2 * e % D;
      const double2 g = reinterpret_cast<const double2*>(G)[e];
      const double si = -inv_n2 * sm[i];
      *reinterpret_cast<float2*>(&A[i * LDA + j]) = make_float2((float)fma(si, sm[j], g.x * inv_n), (float)fma(si, sm[j + 1], g.y * inv_n));
    }
  } else {
    const double* Ain = a.A_in + mat;
    if (tid == 0) s_largest = 0u;
    __syncthreads();
    float largest = 0.f;
    for (int e = tid; e < D * D; e += NT) {
      const float v = (float)Ain[e];
      A[(e / D) * LDA + e % D] = v;
      largest = fmaxf(largest, fabsf(v));
    }
    atomicMax(&s_largest, __float_as_uint(largest));
  }
  __syncthreads();
  // scale so that the largest diagonal entry is 1 (eigenvectors unchanged, eigenvalues scaled back at the end); of a matrix
  // of the caller's, which need not be a covariance, the largest entry
  if (tid < 32) {
    float mx = 0.f;
    for (int i = tid; i < D; i += 32) mx = fmaxf(mx, fabsf(A[i * LDA + i]));
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (a.mode == kPcaMatrix) mx = fmaxf(mx, __uint_as_float(s_largest));
    if (tid == 0) s_scale = mx > 0.f ? (double)mx : 1.0;
  }
  __syncthreads();
  const double a_scale = s_scale;

  // ---- 1. reduction to tridiagonal form
  // By the first warps: one per sub-core at d = 64, two at d = 128.  A thread keeps RW rows by D / TR columns of the
  // matrix, and its columns of the row to be reflected.
  constexpr int RW = D == 64 ? 2 : 4, TR = D == 64 ? 4 : 8;
  constexpr int CH = D / (4 * TR), CW = 4 * TR;        // float4 chunks of a row per thread; columns of a chunk
  constexpr int kParties = TR * D / RW, kHelpers = NT - kParties;
  // the other warps take the reflectors over in blocks, each behind a barrier of its own
  constexpr int kBlock = D / 8, kBlockBar = 2, kHelperBar = 10;
  static_assert(CH == 4 && kParties % 128 == 0, "division of the reduction");
  if (tid < kParties) {
    const int r = RW * (tid / TR), q = tid % TR;       // first of this thread's rows
    const int warp_last = (32 * RW / TR) * (warp + 1) - 1;   // last row of this warp
    const bool publisher = warp == kParties / 32 - 1, publish = publisher && lane < TR;   // the last warp lives to the end
    float v0_prev = 0.f;
    f32x2 areg[RW][CH][2], x[CH][2];
    float d_cur;
    {
      const float inv = (float)((double)kReduceScale / a_scale);
      auto entry = [&](int i, int j) { return 0.5f * (A[i * LDA + j] + A[j * LDA + i]) * inv; };
#pragma unroll
      for (int t = 0; t < CH; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int j = 4 * (q + TR * t) + 2 * h;
#pragma unroll
          for (int y = 0; y < RW; ++y) areg[y][t][h] = pack2(entry(r + y, j), entry(r + y, j + 1));
          x[t][h] = pack2(j > 0 ? entry(0, j) : 0.f, entry(0, j + 1));
        }
      d_cur = entry(0, 0);
    }
    // row k of `refl` takes the reflector of step k
    auto put_row = [&](float* row, const f32x2 (&val)[CH][2], int t0) {
#pragma unroll
      for (int t = 0; t < CH; ++t) {
        ulonglong2 w = make_ulonglong2(0ull, 0ull);
        if (t >= t0) w = make_ulonglong2(val[t][0], val[t][1]);
        *reinterpret_cast<ulonglong2*>(&row[4 * (q + TR * t)]) = w;
      }
    };
    named_sync(1, kParties);                           // (the matrix has been read)
    if (publish) put_row(refl, x, 0);
    // Columns below T0 chunks are done in a segment: its chunks are left out without a branch per chunk
    // (a taken branch costs some 20 cycles and keeps the loads of the chunks from overlapping).
    auto segment = [&](auto t0c) {
      constexpr int T0 = decltype(t0c)::value;
      constexpr int k_first = T0 > 0 ? CW * T0 - 1 : 0, k_end = T0 + 1 < CH ? CW * (T0 + 1) - 1 : D - 2;
#pragma unroll 1
      for (int k = k_first; k < k_end; ++k) {
        const int m0 = k + 1;
        float* yk = ybuf + (k & 1) * D;
        float* ak = abuf + (k & 1) * D;
        if (warp_last < m0) {                          // rows that are done: only the barrier
          named_sync(1, kParties);
          continue;
        }
        // y = A x and |x|^2 (x is zero before m0); row m0 of A goes to the others as it is
#pragma unroll
        for (int y = 0; y < RW; ++y)
          if (r + y == m0) put_row(ak, areg[y], T0);
        float y_r[RW], sig;
        {
          f32x2 s[RW + 1][2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int y = 0; y < RW; ++y) s[y][h] = mul2(areg[y][T0][h], x[T0][h]);
            s[RW][h] = mul2(x[T0][h], x[T0][h]);
#pragma unroll
            for (int t = T0 + 1; t < CH; ++t) {
#pragma unroll
              for (int y = 0; y < RW; ++y) s[y][h] = fma2(areg[y][t][h], x[t][h], s[y][h]);
              s[RW][h] = fma2(x[t][h], x[t][h], s[RW][h]);
            }
          }
#pragma unroll
          for (int y = 0; y < RW; ++y) y_r[y] = sum2(add2(s[y][0], s[y][1]));
          sig = sum2(add2(s[RW][0], s[RW][1]));
        }
#pragma unroll
        for (int o = 1; o < TR; o <<= 1) {
#pragma unroll
          for (int y = 0; y < RW; ++y) y_r[y] += __shfl_xor_sync(0xffffffffu, y_r[y], o);
          sig += __shfl_xor_sync(0xffffffffu, sig, o);
        }
        float y_q = y_r[0];
#pragma unroll
        for (int y = 1; y < RW; ++y) y_q = q == y ? y_r[y] : y_q;
        if (q < RW) yk[r + q] = y_q;
        // approximate root and reciprocals (a unit in the last place or two): the reflector stays
        // orthogonal to the same order as the float32 updates that apply it, and they are on the
        // critical path of every one of the d - 2 steps
        float rt, irt;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(rt) : "f"(sig));
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(irt) : "f"(sig));
        named_sync(1, kParties);
        f32x2 p[CH][2];                                // first y
        float s1;
        {
          f32x2 s[2];
#pragma unroll
          for (int t = T0; t < CH; ++t) {
            // (columns before m0 may hold an older y: x is zero there, and the entries it changes are not used again)
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&yk[4 * (q + TR * t)]);
            p[t][0] = w.x; p[t][1] = w.y;
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            s[h] = mul2(x[T0][h], p[T0][h]);
#pragma unroll
            for (int t = T0 + 1; t < CH; ++t) s[h] = fma2(x[t][h], p[t][h], s[h]);
          }
          s1 = sum2(add2(s[0], s[1]));
        }
        const float* xk = refl + k * LDA;
        const float x0 = xk[m0], y0 = yk[m0], a0 = ak[m0];
        float x_own[RW], a_own[RW];
#pragma unroll
        for (int y = 0; y < RW; y += 2) {
          const float2 xo = *reinterpret_cast<const float2*>(&xk[r + y]), ao = *reinterpret_cast<const float2*>(&ak[r + y]);
          x_own[y] = xo.x; x_own[y + 1] = xo.y;
          a_own[y] = ao.x; a_own[y + 1] = ao.y;
        }
#pragma unroll
        for (int o = 1; o < TR; o <<= 1) s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        // already tridiagonal in this column otherwise, to 1e-15 of the largest diagonal entry (uniform: every
        // group has added the same numbers); beta = 0 then makes the step do nothing
        const bool reflect = sig - x0 * x0 > 1e-30f * kReduceScale * kReduceScale;
        float bn;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(bn) : "f"(fmaf(fabsf(x0), rt, sig)));
        bn = reflect ? bn : 0.f;
        const float alpha = !reflect ? x0 : (x0 >= 0.f ? -rt : rt);
        const float i_alpha = x0 >= 0.f ? -irt : irt;
        const float vy = fmaf(-alpha, y0, s1);                               // v . y, v = x - alpha e_m0
        const float k2 = bn * (bn * fmaf(-alpha, fmaf(-alpha, a0, y0), vy));   // beta^2 v^T A v
        if (publisher) {
          // the first entry of a reflector is put in its place a step later, when no thread reads the row any more
          if (lane == 0) {
            de[k] = make_float2(d_cur / kReduceScale, alpha / kReduceScale);
            beta[k] = bn;
            if (k > 0) refl[(k - 1) * LDA + k] = v0_prev;
          }
          v0_prev = x0 - alpha;
          if (k % kBlock == 0 && k > 0) { __syncwarp(); named_arrive(kBlockBar + k / kBlock - 1, 32 + kHelpers); }
        }
        d_cur = reflect ? s1 * i_alpha * i_alpha : a0;
        // p = beta A v = beta (y - alpha A e_m0);  A - x_r p - (p_r - k2 x_r) x
        const float ba = -bn * alpha;
        if (reflect) {
          const float g = -bn * vy * i_alpha;
          // two rows at a time (registers)
#pragma unroll
          for (int y0 = 0; y0 < RW; y0 += 2) {
            const f32x2 bn2 = pack2(bn, bn), ba2 = pack2(ba, ba);
            f32x2 v2[2], u2[2];
#pragma unroll
            for (int y = 0; y < 2; ++y) {
              const bool live = r + y0 + y > m0;
              const float v_r = live ? -x_own[y0 + y] : 0.f;
              const float u_r = live ? fmaf(k2, x_own[y0 + y], -fmaf(ba, a_own[y0 + y], bn * y_r[y0 + y])) : 0.f;
              v2[y] = pack2(v_r, v_r);
              u2[y] = pack2(u_r, u_r);
            }
#pragma unroll
            for (int t = T0; t < CH; ++t) {
              const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&ak[4 * (q + TR * t)]);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const f32x2 pj = fma2(ba2, h == 0 ? w.x : w.y, mul2(bn2, p[t][h]));
#pragma unroll
                for (int y = 0; y < 2; ++y) areg[y0 + y][t][h] = fma2(u2[y], x[t][h], fma2(v2[y], pj, areg[y0 + y][t][h]));
              }
            }
          }
          const f32x2 g2 = pack2(g, g), ia2 = pack2(i_alpha, i_alpha);
#pragma unroll
          for (int t = T0; t < CH; ++t)
#pragma unroll
            for (int h = 0; h < 2; ++h) x[t][h] = fma2(g2, x[t][h], mul2(ia2, p[t][h]));
        } else {
#pragma unroll
          for (int t = T0; t < CH; ++t) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&ak[4 * (q + TR * t)]);
            x[t][0] = w.x; x[t][1] = w.y;
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {                  // the chunk that holds column m0
          const int j = 4 * (q + TR * T0) + 2 * h;
          float lo, hi;
          unpack2(x[T0][h], lo, hi);
          x[T0][h] = pack2(j > m0 ? lo : 0.f, j + 1 > m0 ? hi : 0.f);
        }
        if (publish) put_row(refl + m0 * LDA, x, T0);
      }
    };
    segment(std::integral_constant<int, 0>{});
    segment(std::integral_constant<int, 1>{});
    segment(std::integral_constant<int, 2>{});
    segment(std::integral_constant<int, 3>{});
    // the last 2 x 2 block
    if (r + RW == D && q == TR - 1) {
      float lo, hi, last;
      unpack2(x[CH - 1][1], lo, hi);
      unpack2(areg[RW - 1][CH - 1][1], lo, last);
      de[D - 2] = make_float2(d_cur / kReduceScale, hi / kReduceScale);
      de[D - 1] = make_float2(last / kReduceScale, 0.f);
    }
    named_sync(1, kParties);
    if (publisher) {
      if (lane == 0) refl[(D - 3) * LDA + D - 2] = v0_prev;
      __syncwarp();
      named_arrive(kBlockBar + 7, 32 + kHelpers);
    }
  } else {
    // The other warps apply the reflectors, a block behind, to the rows of the factor (or the identity), which come
    // out as F Q, Q = H_0 H_1 ...: two rows per four threads (a row per thread group costs twice the
    // shared-memory reads, which the reduction feels); one warp to the mean as well, D / 32 entries per lane.
    constexpr int DC = D / 16;                         // float4 chunks of a row per thread
    constexpr int kMeanWarp = NT / 32 - 1;
    const int h = tid - kParties, row = 2 * (h / 4), q = h % 4;
    const bool has_row = row < D;
    f32x2 z[2][DC][2];
    float m[D / 32];
    if (has_row) {
#pragma unroll
      for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int t = 0; t < DC; ++t) {
          const int j = 4 * (q + 4 * t);
          if (need_e) {
            z[y][t][0] = pack2(j == row + y ? 1.f : 0.f, j + 1 == row + y ? 1.f : 0.f);
            z[y][t][1] = pack2(j + 2 == row + y ? 1.f : 0.f, j + 3 == row + y ? 1.f : 0.f);
          } else {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&L[(row + y) * LDA + j]);
            z[y][t][0] = w.x; z[y][t][1] = w.y;
          }
        }
    }
    if (warp == kMeanWarp) {
#pragma unroll
      for (int c = 0; c < D / 32; ++c)
        m[c] = a.mean_sum ? (float)(a.mean_sum[(size_t)blockIdx.x * D + lane * (D / 32) + c] / a.mean_n) : 0.f;
    }
    named_sync(kHelperBar, kHelpers);                  // the factor has been read
    // zero outside the blocks of the divide and conquer, in both buffers
    for (int e = 4 * h; e < D * LDA; e += 4 * kHelpers) {
      *reinterpret_cast<float4*>(&Qt[e]) = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(&L[e]) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const bool lifted_mean = !need_e && a.mean_lifted;   // (otherwise the mean is multiplied by what comes out)
    // reflectors k of two blocks, without an entry before chunk T0
    auto blocks = [&](auto t0c, int b0) {
      constexpr int T0 = decltype(t0c)::value;
#pragma unroll 1
      for (int b = b0; b < b0 + 2; ++b) {
        named_sync(kBlockBar + b, 32 + kHelpers);
        const int k_end = min(kBlock * (b + 1), D - 2);
#pragma unroll 1
        for (int k = kBlock * b; k < k_end; ++k) {
          const float* vk = refl + k * LDA;
          const float bk = -beta[k];
          if (has_row) {
            ulonglong2 v[DC];
            f32x2 s[2][2];
#pragma unroll
            for (int t = T0; t < DC; ++t) v[t] = *reinterpret_cast<const ulonglong2*>(&vk[4 * (q + 4 * t)]);
            float f[2];
#pragma unroll
            for (int y = 0; y < 2; ++y) {
              s[y][0] = mul2(v[T0].x, z[y][T0][0]);
              s[y][1] = mul2(v[T0].y, z[y][T0][1]);
#pragma unroll
              for (int t = T0 + 1; t < DC; ++t) {
                s[y][0] = fma2(v[t].x, z[y][t][0], s[y][0]);
                s[y][1] = fma2(v[t].y, z[y][t][1], s[y][1]);
              }
              f[y] = sum2(add2(s[y][0], s[y][1]));
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1)
#pragma unroll
              for (int y = 0; y < 2; ++y) f[y] += __shfl_xor_sync(0xffffffffu, f[y], o);
#pragma unroll
            for (int y = 0; y < 2; ++y) {
              const f32x2 f2 = pack2(f[y] * bk, f[y] * bk);
#pragma unroll
              for (int t = T0; t < DC; ++t) {
                z[y][t][0] = fma2(v[t].x, f2, z[y][t][0]);
                z[y][t][1] = fma2(v[t].y, f2, z[y][t][1]);
              }
            }
          }
          if (warp == kMeanWarp && lifted_mean) {
            float v[D / 32], f = 0.f;
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
              v[c] = vk[lane * (D / 32) + c];
              f = fmaf(v[c], m[c], f);
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
            f *= bk;
#pragma unroll
            for (int c = 0; c < D / 32; ++c) m[c] = fmaf(f, v[c], m[c]);
          }
        }
      }
    };
    blocks(std::integral_constant<int, 0>{}, 0);
    blocks(std::integral_constant<int, DC / 4>{}, 2);
    blocks(std::integral_constant<int, DC / 2>{}, 4);
    blocks(std::integral_constant<int, 3 * DC / 4>{}, 6);
    if (has_row) {
#pragma unroll
      for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int t = 0; t < DC; ++t)                   // (no room in shared memory at d = 128)
          *reinterpret_cast<ulonglong2*>(&a.W32[mat + (size_t)(row + y) * D + 4 * (q + 4 * t)]) = make_ulonglong2(z[y][t][0], z[y][t][1]);
    }
    if (warp == kMeanWarp) {
#pragma unroll
      for (int c = 0; c < D / 32; ++c) mean[lane * (D / 32) + c] = m[c];
    }
  }
  __syncthreads();

  // ---- 2. divide and conquer.  A cut between rows k-1 and k writes T = diag(T1, T2) + rho u u^T with
  // rho = |b|, b the coupling of the two rows, u = e_{k-1} + sign(b) e_k, and b subtracted from the
  // two diagonal entries it touches.
  if (tid > 0 && tid < D / kBase) {
    const int k = tid * kBase;
    const float bk = de[k - 1].y;
    s_rho[tid] = fabsf(bk);
    s_theta[tid] = bk < 0.f ? -1.f : 1.f;
    de[k - 1] = make_float2(de[k - 1].x - fabsf(bk), 0.f);
    de[k].x -= fabsf(bk);
  }
  __syncthreads();
  if (warp == 0) jacobi_blocks(de, D / kBase, Qt, LDA, lane);
  __syncthreads();
  // merges of a level side by side, T threads per row
#pragma unroll 1
  for (int lg = kBaseLog + 1; (1 << lg) <= D; ++lg) {
    const int grp = tid / ((NT / D) << lg), cut = ((2 * grp + 1) << (lg - 1)) / kBase;
    merge_blocks<D>(Qt, L, A, de, scratch, lg, s_rho[cut], s_theta[cut], tid - grp * ((NT / D) << lg), grp);
    __syncthreads();
    float* swap = Qt; Qt = L; L = swap;
  }

  // ---- 3. the map from the original space, W = F E = (F Q) S, into A, S the eigenvectors of T (rows of Qt); where E is
  // asked for, E = Q S first, its columns as rows of Qt, and then F E for the sign rule
  for (int e = tid; e < D * D / 4; e += NT)
    *reinterpret_cast<float4*>(&L[(4 * e / D) * LDA + 4 * e % D]) = *reinterpret_cast<const float4*>(&a.W32[mat + 4 * (size_t)e]);
  __syncthreads();
  // out[i][j] = sum_k L[i][k] Qt[j][k], or its transpose
  auto product = [&](float* out, bool transposed) {
    if (tile.live) {
      float acc[TI][TJ];
      tile_product_rows<D>(L, Qt, LDA, tile, acc);
#pragma unroll
      for (int x = 0; x < TI; ++x)
#pragma unroll
        for (int y = 0; y < TJ; ++y) {
          const int i = TI * tile.i + x, j = tile.j + Tile<D>::COLS * y;
          out[transposed ? j * LDA + i : i * LDA + j] = acc[x][y];
        }
    }
  };
  product(A, need_e);
  if (need_e) {
    float* swap = Qt; Qt = A; A = swap;
    if (a.lift) {
      __syncthreads();
      load_factor();
      __syncthreads();
      product(A, false);
    }
  }
  let_next_start();
  // ---- order, sign, bias
  double* lam = reinterpret_cast<double*>(ybuf);             // [D] doubles over ybuf's 2D floats
  int* rank_of = reinterpret_cast<int*>(abuf);
  float* sign_of = beta;
  if (tid < D) {
    lam[tid] = (double)de[tid].x * a_scale;
  }
  __syncthreads();
  const bool lifted_out = a.lift && a.out_lifted;
  if (tid < D) {
    const double mine = lam[tid];
    int rank = 0;
#pragma unroll 16
    for (int k = 0; k < D; ++k) {
      const double other = lam[k];
      rank += (other > mine) || (other == mine && k < tid);
    }
    // sign rule on column tid of F E (of E when no factor is given); bias = -mean . that column, or
    // . column tid of E where the mean is one of transformed rows (without E: of S, the mean then is in the basis Q)
    float best = -1.f, sgn = 1.f, dot = 0.f;
#pragma unroll 8
    for (int i = 0; i < D; ++i) {
      const float e_i = Qt[tid * LDA + i];
      const float w_i = a.lift ? A[i * LDA + tid] : e_i;
      if (fabsf(w_i) > best) { best = fabsf(w_i); sgn = (w_i < 0.f) ? -1.f : 1.f; }
      dot = fmaf(mean[i], a.mean_lifted ? e_i : w_i, dot);
    }
    rank_of[tid] = rank;
    sign_of[tid] = sgn;
    if (a.bias) a.bias[(size_t)blockIdx.x * D + rank] = -sgn * dot;
    if (a.evals) a.evals[(size_t)blockIdx.x * D + rank] = mine;
  }
  __syncthreads();
  // projection matrix [in i][out rank(j)] in fp32, or its transpose as bf16 hi + lo parts
  if (!a.wt_hi) {
    for (int e = tid; e < D * D; e += NT) {
      const int i = e / D, j = e % D;
      const float v = sign_of[j] * (lifted_out ? A[i * LDA + j] : Qt[j * LDA + i]);
      a.W32[mat + (size_t)i * D + rank_of[j]] = v;
    }
  } else {
#pragma unroll 4
    for (int e = tid; e < D * D; e += NT) {
      const int j = e / D, i = e % D;
      const float v = sign_of[j] * (lifted_out ? A[i * LDA + j] : Qt[j * LDA + i]);
      const __nv_bfloat16 h = __float2bfloat16_rn(v);
      a.wt_hi[mat + (size_t)rank_of[j] * D + i] = h;
      a.wt_lo[mat + (size_t)rank_of[j] * D + i] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
  }
}

int launch_pca(const PcaArgs& args, int count, int D, LaunchStream st) {
  const size_t smem = sizeof(float) * ((size_t)3 * D * (D + 4) + 8 * D + 21 * D);
  auto k = D == 64 ? eigh_tql_kernel<64> : eigh_tql_kernel<128>;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  launch_chained(k, count, kThreads, smem, st, args);
  CA_LAUNCH_CHECK();
  return CA_OK;
}

}  // namespace ca
