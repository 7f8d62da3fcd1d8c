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
// 1. Householder reduction to tridiagonal form.  For k = 0 .. d-3 the reflector H_k = I - beta v v^T
// annihilates A[k+2.., k]; the trailing block is updated as A - v w^T - w v^T with p = beta A v,
// w = p - (beta/2)(v.p) v.  A step is a chain of latencies (two barriers, shuffles, a root), so
// what counts is how short the chain is and how few instructions stand in it: a few threads per
// row keep the matrix in registers, the owners of the next row only publish it, and every thread
// derives the reflector from it for itself; rows and columns that are done drop out.  The
// reflectors are stored, not accumulated.
// 2. Divide and conquer.  The tridiagonal matrix is cut into blocks of kBase rows (a cut writes
// T = diag(T1, T2) + rho u u^T), each diagonalised by one warp with the implicit-shift QL iteration
// (the rotation chase is one dependent chain on lane 0, the lanes apply its rotations to the columns
// that they keep in registers), then merged pairwise up to the whole.  A merge solves
// diag(d) + rho z z^T, z the eigenvectors' components at the cut: poles sorted, negligible weights and
// coinciding poles deflated, the roots of the secular equation by an iteration that treats the
// nearest pole exactly (a few threads per root; offsets from that pole keep the differences
// d_j - x accurate), the weights recomputed from the roots (Gu and Eisenstat, 1994) so that the
// eigenvectors stay orthogonal to rounding, and one product with the blocks' eigenvectors.
// 3. The stored reflectors are applied to the eigenvectors of T, a few threads per vector, without a barrier.
// Two launches (keys, queries) one after the other: 8 heads, d = 64 0.27 ms and 40 heads, d = 128 0.86 ms
// with the transform accumulated during the reduction (eight threads per row, the next reflector
// built by one warp, branches around finished chunks), quarters as base blocks and bisected roots;
// now 0.185 and 0.53 ms.  SM cycles of a launch (d = 64 / d = 128): covariance 8-25 k / 12-80 k,
// reduction 58 k / 180 k (62 / 126 steps), base blocks 8 k / 15 k, merges 56-65 k / 120-135 k, reflectors
// 13 k / 55 k, map and output 9 k / 45 k.
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

namespace ca {

namespace {

__device__ __forceinline__ void named_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

constexpr int kThreads = 512;
constexpr int kBaseLog = 2, kBase = 1 << kBaseLog;   // rows of a base block of the divide and conquer
constexpr int kMaxQlIterations = 64;

// Eigenvalues that are not numbers (the covariance of rows with infinities, or whose sums overflow) stand as +inf: the
// rank of a pole among the others is then a permutation for every input, and indexes stay in range.
__device__ __forceinline__ float pole_value(float x) { return fminf(x, INFINITY); }

// ---- implicit-shift QL on rows [l0, l0 + kBase) of a tridiagonal matrix (de[i] = (diagonal i, coupling of
// i and i + 1); the coupling behind the last row is not part of the block), by one warp: the search
// for a negligible sub-diagonal entry uses all lanes, the rotation chase is one dependent chain on
// lane 0, and lane t applies the rotations of a chase (rt, in shared memory) to column t of the
// block's eigenvectors, which start as the identity and end as rows of Qt.
__device__ __forceinline__ void ql_block(float2* de, int l0, float2* rt, float* Qt, int lda, int lane) {
  const float eps = 6e-8f;
  const int l1 = l0 + kBase;
  float z[kBase];
#pragma unroll
  for (int i = 0; i < kBase; ++i) z[i] = i == lane ? 1.f : 0.f;
#pragma unroll 1
  for (int l = l0; l < l1; ++l) {
#pragma unroll 1
    for (int iter = 0; iter < kMaxQlIterations; ++iter) {
      // first m >= l whose sub-diagonal entry is negligible (m = l1 - 1 if none)
      const int idx = l + lane;
      bool small = false;
      if (idx < l1 - 1) {
        const float2 a = de[idx];
        small = fabsf(a.y) <= eps * (fabsf(a.x) + fabsf(de[idx + 1].x));
      }
      const unsigned bal = __ballot_sync(0xffffffffu, small);
      const int m = bal ? l + __ffs(bal) - 1 : l1 - 1;
      if (m == l) break;
      int lo = l;
      if (lane == 0) {
        const float2 top = de[l];
        // the shift only steers the convergence (the rotations are formed from the matrix itself), so
        // approximate division and root are enough for it
        float g = __fdividef(de[l + 1].x - top.x, 2.f * top.y);
        float rr;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(rr) : "f"(fmaf(g, g, 1.f)));
        g = de[m].x - top.x + __fdividef(top.y, g + (g >= 0.f ? rr : -rr));
        float s = 1.f, c = 1.f, p = 0.f;
        bool under = false;
        int i = m - 1;
        float2 cur = de[i];              // (d_i, e_i)
        float d_i1 = de[i + 1].x;
#pragma unroll 1
        for (; i >= l; --i) {
          // operands of the next rotation, fetched ahead of the dependent chain
          const float2 nxt = de[i > l ? i - 1 : l];
          const float f = s * cur.y, bb = c * cur.y;
          const float r2 = fmaf(f, f, g * g);
          float rinv;
          asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rinv) : "f"(r2));
          const float p_old = p, d_old = d_i1;
          s = f * rinv;
          c = g * rinv;
          g = d_i1 - p;
          rr = fmaf(c, bb + bb, (cur.x - g) * s);
          p = s * rr;
          de[i + 1] = make_float2(g + p, r2 * rinv);       // new d_{i+1}; e_{i+1} = hypot(f, g)
          g = fmaf(c, rr, -bb);
          rt[i - l0] = make_float2(c, s);
          // The chase has died out (f = g = 0): deflate here.  Tested after the rotation has been
          // formed so that the test is off the dependent chain; its results are discarded.
          if (r2 < 1e-36f) {
            de[i + 1] = make_float2(d_old - p_old, 0.f);
            de[m].y = 0.f;
            under = true;
            break;
          }
          d_i1 = cur.x;          // d_i is the next step's d_{i+1}; it has not been modified yet
          cur = nxt;
        }
        if (!under) {
          de[l] = make_float2(top.x - p, g);
          de[m].y = 0.f;
        } else {
          lo = i + 1;
        }
      }
      lo = __shfl_sync(0xffffffffu, lo, 0);
      __syncwarp();
#pragma unroll
      for (int i = kBase - 2; i >= 0; --i) {
        // (no branch: a rotation outside the chase is the identity)
        const bool in = l0 + i < m && l0 + i >= lo;
        const float2 cs = rt[i];
        const float c = in ? cs.x : 1.f, sn = in ? cs.y : 0.f;
        const float zi = z[i], zn = z[i + 1];
        z[i + 1] = fmaf(sn, zi, c * zn);
        z[i] = fmaf(c, zi, -sn * zn);
      }
      __syncwarp();
    }
  }
  if (lane < kBase) {
    de[l0 + lane].x = pole_value(de[l0 + lane].x);
#pragma unroll
    for (int i = 0; i < kBase; ++i) Qt[(l0 + i) * lda + l0 + lane] = z[i];
  }
}

}  // namespace

// d x d x d products in shared memory, a 4 x 4 tile of the result per thread (the first d^2 / 16
// threads; every shared-memory load feeds four or sixteen multiply-adds, and the lanes of a
// quarter-warp read distinct banks).  Terms are added for k = 0, 1, ... in that order.
//   XT = false: acc[a][b] = sum_k X[(4 ti + a) lda + k] Y[k lda + 4 tj + b]
//   XT = true:  acc[a][b] = sum_k X[k lda + 4 ti + a]   Y[k lda + 4 tj + b]
template <int D, bool XT>
__device__ __forceinline__ void tile_product(const float* __restrict__ X, const float* __restrict__ Y, int lda,
                                             int ti, int tj, float (&acc)[4][4]) {
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
#pragma unroll 2
  for (int k0 = 0; k0 < D; k0 += 4) {
    float xa[4][4];                                    // [row][k]
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (XT) {
        const float4 v = *reinterpret_cast<const float4*>(&X[(k0 + e) * lda + 4 * ti]);
        xa[0][e] = v.x; xa[1][e] = v.y; xa[2][e] = v.z; xa[3][e] = v.w;
      } else {
        const float4 v = *reinterpret_cast<const float4*>(&X[(4 * ti + e) * lda + k0]);
        xa[e][0] = v.x; xa[e][1] = v.y; xa[e][2] = v.z; xa[e][3] = v.w;
      }
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const float4 y = *reinterpret_cast<const float4*>(&Y[(k0 + kk) * lda + 4 * tj]);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        acc[x][0] = fmaf(xa[x][kk], y.x, acc[x][0]); acc[x][1] = fmaf(xa[x][kk], y.y, acc[x][1]);
        acc[x][2] = fmaf(xa[x][kk], y.z, acc[x][2]); acc[x][3] = fmaf(xa[x][kk], y.w, acc[x][3]);
      }
    }
  }
}

// acc[a][c] = sum_k X[(4 ti + a) lda + k] Yr[(tj + (D / 4) c) lda + k]   (both operands by rows)
template <int D>
__device__ __forceinline__ void tile_product_rows(const float* __restrict__ X, const float* __restrict__ Yr, int lda,
                                                  int ti, int tj, float (&acc)[4][4]) {
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
#pragma unroll 2
  for (int k0 = 0; k0 < D; k0 += 4) {
    float4 xv[4], yv[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      xv[e] = *reinterpret_cast<const float4*>(&X[(4 * ti + e) * lda + k0]);
      yv[e] = *reinterpret_cast<const float4*>(&Yr[(tj + (D / 4) * e) * lda + k0]);
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        acc[x][y] = fmaf(xv[x].x, yv[y].x, acc[x][y]); acc[x][y] = fmaf(xv[x].y, yv[y].y, acc[x][y]);
        acc[x][y] = fmaf(xv[x].z, yv[y].z, acc[x][y]); acc[x][y] = fmaf(xv[x].w, yv[y].w, acc[x][y]);
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
  float* kz2 = defl_d + D;                                 // squared weights of the kept poles
  int* counts = reinterpret_cast<int*>(scratch + 16 * D) + 8 * grp;   // kept, rotations, deflated, skip
  float* z2sum = reinterpret_cast<float*>(counts + 4);
  const float rho2 = 2.f * rho;
  if (lt < NB) {
    const float mine = de[b0 + lt].x;
    int rank = 0;
#pragma unroll 4
    for (int k = 0; k < NB; ++k) {
      const float other = de[b0 + k].x;
      rank += (other < mine) || (other == mine && k < lt);
    }
    const int cut = b0 + NB / 2;
    ord[rank] = b0 + lt;
    ds[rank] = mine;
    zs[rank] = 0.70710678f * (lt < NB / 2 ? Qt[(b0 + lt) * LDA + cut - 1] : theta * Qt[(b0 + lt) * LDA + cut]);
  }
  sync();
  if (lt < 32) {
    float dmax = 0.f, zmax = 0.f;
    for (int j = lane; j < NB; j += 32) { dmax = fmaxf(dmax, fabsf(ds[j])); zmax = fmaxf(zmax, fabsf(zs[j])); }
    for (int o = 16; o > 0; o >>= 1) {
      dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
      zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
    }
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
#pragma unroll 1
              for (; j < K && coincide(j); ++j) {
                const float d_prev = kd[j - 1], dj = kd[j];
                float sn = kz[j - 1], cs = kz[j];
                const float tau = sqrtf(fmaf(cs, cs, sn * sn));
                cs = __fdividef(cs, tau);
                sn = -__fdividef(sn, tau);
                gc[ng] = cs; gs[ng] = sn; ga[ng] = keep_row[j - 1]; gb[ng] = keep_row[j]; ++ng;
                kd[j] = d_prev * sn * sn + dj * cs * cs;
                kz[j] = tau;
                defl_row[nd] = keep_row[j - 1]; defl_d[nd] = d_prev * cs * cs + dj * sn * sn; ++nd;
                kz[j - 1] = 0.f;                           // mark of a pole that has given way
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
          const int rj = j < K ? keep_row[j] : 0;
          const unsigned mk = __ballot_sync(0xffffffffu, zj != 0.f);
          if (zj != 0.f) {
            const int at = kept + __popc(mk & ((1u << lane) - 1u));
            keep_row[at] = rj; kd[at] = dj; kz[at] = zj;
          }
          kept += __popc(mk);
          __syncwarp();
        }
        K = kept;
        ng = __shfl_sync(0xffffffffu, ng, 0);
        nd = __shfl_sync(0xffffffffu, nd, 0);
      }
      // squared weights of the kept poles and their sum (the last root's bracket)
      float z2 = 0.f;
      for (int j = lane; j < NB; j += 32) {
        const float w = j < K ? kz[j] * kz[j] : 0.f;
        kz2[j] = w;
        z2 += w;
      }
      for (int o = 16; o > 0; o >>= 1) z2 += __shfl_xor_sync(0xffffffffu, z2, o);
      if (lane == 0) *z2sum = z2;
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
  const int K = counts[0], ng = counts[1], nd = counts[2];
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
    // the last root lies in (d_{K-1}, d_{K-1} + rho2 |z|^2); every other one between two poles, and the
    // sign of the function half-way says next to which
    const bool last = i >= K - 1;
    const float width = last ? rho2 * *z2sum : kd[i + 1] - kd[i];
    const float mid = 0.5f * width, d0 = kd[i];
    float acc = 0.f;
#pragma unroll 4
    for (int j = sub; j < K; j += T) {
      float inv;                                            // one special-function operation, no rounding fix-up
      asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"((kd[j] - d0) - mid));
      acc = fmaf(kz2[j], inv, acc);
    }
    const float f_mid = fmaf(rho2, sum_t(acc), 1.f);
    const bool right = !last && f_mid < 0.f;
    const int org = right ? i + 1 : i;
    const float w_org = rho2 * kz2[org], d_org = kd[org];
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
        float inv;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"((kd[j] - d_org) - m));
        const float x = j == org ? 0.f : kz2[j] * inv;
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
      float next;
      if (!right) next = ca >= 0.f ? __fdividef(2.f * w_org, ca + disc) : __fdividef(disc - ca, 2.f * r1);
      else next = ca <= 0.f ? -__fdividef(2.f * w_org, disc - ca) : -__fdividef(ca + disc, 2.f * r1);
      // settled: convergence is quadratic, so behind a step of 1e-5 nothing but rounding is left (and the
      // sign of f, which moves the bracket, is rounding too: such a step may leave it)
      bool still = fabsf(next - m) <= 1e-5f * fabsf(m);
      if (!still && (it >= kSteps || !(next > lo_m && next < hi_m))) {
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
      if (live) A[(b0 + gi) * LDA + j] = v;
    }
    const float inv = rsqrtf(sum_t(nrm));
    if (live)
      for (int j = sub; j < K; j += T) A[(b0 + gi) * LDA + j] *= inv;
  }
  sync();
  // rows of the merged basis into L: row b0 + i = sum_j A[b0 + i][j] Qt[keep_row[j]] (i < K), then
  // the deflated rows (a 4 x 4 tile per thread, terms in the order of j)
#pragma unroll 1
  for (int tile = lt; tile < NB * NB / 16; tile += GT) {
    const int i0 = 4 * (tile >> (lg - 2)), c0 = b0 + 4 * (tile & (NB / 4 - 1));
    if (i0 >= K) break;
    float acc[4][4];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
    int j = 0;
#pragma unroll 1
    for (; j + 4 <= K; j += 4) {
      float xa[4][4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const float4 v = *reinterpret_cast<const float4*>(&A[(b0 + i0 + x) * LDA + j]);
        xa[x][0] = v.x; xa[x][1] = v.y; xa[x][2] = v.z; xa[x][3] = v.w;
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float4 y = *reinterpret_cast<const float4*>(&Qt[keep_row[j + kk] * LDA + c0]);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          acc[x][0] = fmaf(xa[x][kk], y.x, acc[x][0]); acc[x][1] = fmaf(xa[x][kk], y.y, acc[x][1]);
          acc[x][2] = fmaf(xa[x][kk], y.z, acc[x][2]); acc[x][3] = fmaf(xa[x][kk], y.w, acc[x][3]);
        }
      }
    }
#pragma unroll 1
    for (; j < K; ++j) {
      const float4 y = *reinterpret_cast<const float4*>(&Qt[keep_row[j] * LDA + c0]);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const float xv = A[(b0 + i0 + x) * LDA + j];
        acc[x][0] = fmaf(xv, y.x, acc[x][0]); acc[x][1] = fmaf(xv, y.y, acc[x][1]);
        acc[x][2] = fmaf(xv, y.z, acc[x][2]); acc[x][3] = fmaf(xv, y.w, acc[x][3]);
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
  float* xbuf = A + 3 * D * LDA;                       // [2][D]     the next row of the reduction
  float* pbuf = xbuf + 2 * D;                          // [D]
  float2* de = reinterpret_cast<float2*>(pbuf + D);    // [D]        (diagonal i, sub-diagonal coupling i and i+1)
  float* beta = pbuf + 3 * D;                          // [D]        factors of the reflectors
  float* rot = beta + D;                               // [2 D]      rotations of a chase, (c, s) per row
  float* scratch = rot + 2 * D;                        // [18 D]     arrays of the merge
  __shared__ double s_scale;
  __shared__ float s_rho[D / kBase], s_theta[D / kBase];   // cut before row i kBase

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t mat = (size_t)blockIdx.x * D * D;
  constexpr int TILES = D * D / 16;                    // d x d x d products: 4 x 4 tiles

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
    float acc[4][4];
#pragma unroll 1
    for (int tile = tid; tile < TILES; tile += NT) {
      const int tile_i = tile / (D / 4), tile_j = tile % (D / 4);
      tile_product<D, true>(L, A, LDA, tile_i, tile_j, acc);                              // F^T C
#pragma unroll
      for (int x = 0; x < 4; ++x)
        *reinterpret_cast<float4*>(&Qt[(4 * tile_i + x) * LDA + 4 * tile_j]) = make_float4(acc[x][0], acc[x][1], acc[x][2], acc[x][3]);
    }
    __syncthreads();
    const float al = (float)a.alpha;
#pragma unroll 1
    for (int tile = tid; tile < TILES; tile += NT) {
      const int tile_i = tile / (D / 4), tile_j = tile % (D / 4);
      tile_product<D, false>(Qt, L, LDA, tile_i, tile_j, acc);                            // (F^T C) F
#pragma unroll
      for (int x = 0; x < 4; ++x)
        *reinterpret_cast<float4*>(&A[(4 * tile_i + x) * LDA + 4 * tile_j]) =
            make_float4(al * acc[x][0], al * acc[x][1], al * acc[x][2], al * acc[x][3]);
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
    for (int e = tid; e < D * D; e += NT) A[(e / D) * LDA + e % D] = (float)Ain[e];
  }
  __syncthreads();
  // scale so that the largest diagonal entry is 1 (eigenvectors unchanged, eigenvalues scaled back at the end)
  if (tid < 32) {
    float mx = 0.f;
    for (int i = tid; i < D; i += 32) mx = fmaxf(mx, fabsf(A[i * LDA + i]));
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (tid == 0) s_scale = mx > 0.f ? (double)mx : 1.0;
  }
  // zero outside the blocks of the divide and conquer, in both buffers
  for (int e = tid; e < D * LDA; e += NT) { Qt[e] = 0.f; L[e] = 0.f; }
  __syncthreads();
  const double a_scale = s_scale;

  // ---- 1. reduction to tridiagonal form
  // A thread keeps RW rows by D / TR columns.  The vectors that a step reads back (v, then p) cost shared-memory
  // bandwidth -- every thread reads its columns -- and every halving of the columns costs another
  // shuffle in each of the three sums: one row by 32 columns at d = 64, two rows by 16 at d = 128.
  constexpr int RW = D == 64 ? 1 : 2, TR = D == 64 ? 2 : 8;
  constexpr int CH = D / (4 * TR), CW = 4 * TR;        // float4 chunks of a row per thread; columns of a chunk
  constexpr int SEG = CH / 4;                          // chunks per segment
  if (tid < TR * D / RW) {
    constexpr int kParties = TR * D / RW;
    const int r = RW * (tid / TR), q = tid % TR;       // first of this thread's rows
    const int warp_last = (32 * RW / TR) * (warp + 1) - 1;   // last row of this warp
    float areg[RW][CH][4];
    {
      const float inv = (float)(1.0 / a_scale);
#pragma unroll
      for (int x = 0; x < RW; ++x)
#pragma unroll
        for (int t = 0; t < CH; ++t)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int j = 4 * (q + TR * t) + c;
            areg[x][t][c] = 0.5f * (A[(r + x) * LDA + j] + A[j * LDA + r + x]) * inv;
          }
    }
    if (r == 0) {
#pragma unroll
      for (int t = 0; t < CH; ++t)
        *reinterpret_cast<float4*>(&xbuf[4 * (q + TR * t)]) = make_float4(areg[0][t][0], areg[0][t][1], areg[0][t][2], areg[0][t][3]);
    }
    auto sum_row = [](float x) {
#pragma unroll
      for (int o = 1; o < TR; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      return x;
    };
    // Columns below T0 chunks are done in a segment: its chunks are left out without a branch per chunk
    // (a taken branch costs some 20 cycles and keeps the loads of the chunks from overlapping).
    auto segment = [&](auto t0c) {
      constexpr int T0 = decltype(t0c)::value;
      constexpr int k_first = T0 > 0 ? CW * T0 - 1 : 0, k_end = T0 + SEG < CH ? CW * (T0 + SEG) - 1 : D - 2;
#pragma unroll 1
      for (int k = k_first; k < k_end; ++k) {
        const int m0 = k + 1;
        const float* x = xbuf + (k & 1) * D;
        named_sync(1, kParties);                       // row k has been published
        if (warp_last < k) {                           // rows that are done: only the barriers
          named_sync(1, kParties);
          continue;
        }
        // reflector of row k, the same in every thread group
        float v[CH][4];
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        const float x0 = x[m0], x_k = x[k];
        float x_r[RW];
#pragma unroll
        for (int y = 0; y < RW; ++y) x_r[y] = x[r + y];
#pragma unroll
        for (int t = T0; t < CH; ++t) {
          const float4 xx = *reinterpret_cast<const float4*>(&x[4 * (q + TR * t)]);
          v[t][0] = xx.x; v[t][1] = xx.y; v[t][2] = xx.z; v[t][3] = xx.w;
        }
#pragma unroll
        for (int t = T0; t < CH; ++t) {
          if (t <= T0 + SEG) {                         // chunks that can hold column m0
            const int j0 = 4 * (q + TR * t);
#pragma unroll
            for (int c = 0; c < 4; ++c) v[t][c] = j0 + c >= m0 ? v[t][c] : 0.f;
          }
          s0 = fmaf(v[t][0], v[t][0], s0); s1 = fmaf(v[t][1], v[t][1], s1);
          s2 = fmaf(v[t][2], v[t][2], s2); s3 = fmaf(v[t][3], v[t][3], s3);
        }
        const float sig = sum_row((s0 + s1) + (s2 + s3));
        // already tridiagonal in this column otherwise (uniform: every group has added the same numbers);
        // beta = 0 then makes the step do nothing
        const bool reflect = sig - x0 * x0 > 1e-30f;
        // approximate root and reciprocal (a unit in the last place or two): the reflector stays
        // orthogonal to the same order as the float32 updates that apply it, and they are on the
        // critical path of every one of the d - 2 steps
        float rt, bn;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(rt) : "f"(sig));
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(bn) : "f"(fmaf(fabsf(x0), rt, sig)));
        const float alpha = !reflect ? x0 : (x0 >= 0.f ? -rt : rt);
        const float v0 = x0 - alpha;
        bn = reflect ? bn : 0.f;
#pragma unroll
        for (int t = T0; t <= T0 + SEG && t < CH; ++t)
#pragma unroll
          for (int c = 0; c < 4; ++c) v[t][c] = 4 * (q + TR * t) + c == m0 ? v0 : v[t][c];
        float p[RW];
#pragma unroll
        for (int y = 0; y < RW; ++y) {
          s0 = s1 = s2 = s3 = 0.f;
#pragma unroll
          for (int t = T0; t < CH; ++t) {
            s0 = fmaf(areg[y][t][0], v[t][0], s0); s1 = fmaf(areg[y][t][1], v[t][1], s1);
            s2 = fmaf(areg[y][t][2], v[t][2], s2); s3 = fmaf(areg[y][t][3], v[t][3], s3);
          }
          p[y] = (s0 + s1) + (s2 + s3);
        }
#pragma unroll
        for (int y = 0; y < RW; ++y) p[y] = bn * sum_row(p[y]);
#pragma unroll
        for (int y = 0; y < RW; ++y)
          if (q == y) pbuf[r + y] = r + y >= m0 ? p[y] : 0.f;
        // kept for part 3 in the space of the result
        if (k - r >= 0 && k - r < RW) {
          if (q == 0) { de[k] = make_float2(x_k, alpha); beta[k] = bn; }
#pragma unroll
          for (int t = 0; t < CH; ++t)
            *reinterpret_cast<float4*>(&a.W32[mat + (size_t)k * D + 4 * (q + TR * t)]) =
                t < T0 ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(v[t][0], v[t][1], v[t][2], v[t][3]);
        }
        named_sync(1, kParties);
        float p_r[RW];
#pragma unroll
        for (int y = 0; y < RW; ++y) p_r[y] = pbuf[r + y];
        float pv[CH][4];
#pragma unroll
        for (int t = T0; t < CH; ++t) {
          // (columns below m0 may hold an older p: v is zero there, and the entries they change are not used again)
          const float4 pp = *reinterpret_cast<const float4*>(&pbuf[4 * (q + TR * t)]);
          pv[t][0] = pp.x; pv[t][1] = pp.y; pv[t][2] = pp.z; pv[t][3] = pp.w;
        }
        s0 = s1 = s2 = s3 = 0.f;
#pragma unroll
        for (int t = T0; t < CH; ++t) {
          s0 = fmaf(v[t][0], pv[t][0], s0); s1 = fmaf(v[t][1], pv[t][1], s1);
          s2 = fmaf(v[t][2], pv[t][2], s2); s3 = fmaf(v[t][3], pv[t][3], s3);
        }
        const float K = 0.5f * bn * sum_row((s0 + s1) + (s2 + s3));
#pragma unroll
        for (int y = 0; y < RW; ++y) {
          // a -= v_r (p - K v) + (p_r - K v_r) v = v_r p + (p_r - 2 K v_r) v
          const float v_r = r + y > m0 ? x_r[y] : (r + y == m0 ? v0 : 0.f);
          const float u_r = r + y >= m0 ? fmaf(-2.f * K, v_r, p_r[y]) : 0.f;
          const bool apply = reflect && r + y >= m0;
#pragma unroll
          for (int t = T0; t < CH; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float next = fmaf(-v_r, pv[t][c], fmaf(-u_r, v[t][c], areg[y][t][c]));
              areg[y][t][c] = apply ? next : areg[y][t][c];
            }
          if (r + y == m0) {
            float* xn = xbuf + ((k + 1) & 1) * D;
#pragma unroll
            for (int t = T0; t < CH; ++t)
              *reinterpret_cast<float4*>(&xn[4 * (q + TR * t)]) = make_float4(areg[y][t][0], areg[y][t][1], areg[y][t][2], areg[y][t][3]);
          }
        }
      }
    };
    segment(std::integral_constant<int, 0>{});
    segment(std::integral_constant<int, SEG>{});
    segment(std::integral_constant<int, 2 * SEG>{});
    segment(std::integral_constant<int, 3 * SEG>{});
    // the last 2 x 2 block
    if (q == TR - 1) {
#pragma unroll
      for (int y = 0; y < RW; ++y) {
        if (r + y == D - 2) de[D - 2] = make_float2(areg[y][CH - 1][2], areg[y][CH - 1][3]);
        if (r + y == D - 1) de[D - 1] = make_float2(areg[y][CH - 1][3], 0.f);
      }
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
#pragma unroll 1
  for (int w = warp; w < D / kBase; w += NT / 32) ql_block(de, w * kBase, reinterpret_cast<float2*>(rot) + w * kBase, Qt, LDA, lane);
  __syncthreads();
  // merges of a level side by side, T threads per row
#pragma unroll 1
  for (int lg = kBaseLog + 1; (1 << lg) <= D; ++lg) {
    const int grp = tid / ((NT / D) << lg), cut = ((2 * grp + 1) << (lg - 1)) / kBase;
    merge_blocks<D>(Qt, L, A, de, scratch, lg, s_rho[cut], s_theta[cut], tid - grp * ((NT / D) << lg), grp);
    __syncthreads();
    float* swap = Qt; Qt = L; L = swap;
  }

  // ---- 3. the reflectors, last one first, on the eigenvectors of T (rows of Qt)
  for (int e = tid; e < (D - 2) * D / 4; e += NT)
    *reinterpret_cast<float4*>(&L[(e / (D / 4)) * LDA + 4 * (e % (D / 4))]) = *reinterpret_cast<const float4*>(&a.W32[mat + 4 * (size_t)e]);
  __syncthreads();
  {
    // Two reflectors at a time: H_a (H_b z) needs v_a . z and v_b . z only, once v_a . v_b is known.
    constexpr int T = 8, CB = D / (4 * T);             // threads per two vectors (r, r + d / 2), float4 chunks per thread
    float* cross = pbuf;                               // [k] = v_k . v_{k+1}
    {
      constexpr int TP = NT / (D / 2);
      const int k = 2 * (tid / TP), q = tid % TP;
      float dot = 0.f;
      if (k < D - 2)
        for (int j = q; j < D; j += TP) dot = fmaf(L[k * LDA + j], L[(k + 1) * LDA + j], dot);
#pragma unroll
      for (int o = 1; o < TP; o <<= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
      if (q == 0 && k < D - 2) cross[k] = dot;
    }
    __syncthreads();
    const int r = tid / T, q = tid % T;
    if (tid < T * D / 2) {
      float z[2][CB][4];
#pragma unroll
      for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int t = 0; t < CB; ++t) {
          const float4 x = *reinterpret_cast<const float4*>(&Qt[(r + y * (D / 2)) * LDA + 4 * (q + T * t)]);
          z[y][t][0] = x.x; z[y][t][1] = x.y; z[y][t][2] = x.z; z[y][t][3] = x.w;
        }
      auto segment = [&](auto t0c, int k_first, int k_last) {  // reflectors without an entry before chunk T0
        constexpr int T0 = decltype(t0c)::value;
#pragma unroll 1
        for (int k = k_first; k >= k_last; k -= 2) {
          const float ba = beta[k], bb = beta[k + 1], cc = cross[k];
          float4 va[CB], vb[CB];
#pragma unroll
          for (int t = T0; t < CB; ++t) {
            va[t] = *reinterpret_cast<const float4*>(&L[k * LDA + 4 * (q + T * t)]);
            vb[t] = *reinterpret_cast<const float4*>(&L[(k + 1) * LDA + 4 * (q + T * t)]);
          }
          float da[2], db[2];
#pragma unroll
          for (int y = 0; y < 2; ++y) {
            float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
#pragma unroll
            for (int t = T0; t < CB; ++t) {
              a0 = fmaf(va[t].x, z[y][t][0], a0); a1 = fmaf(va[t].y, z[y][t][1], a1);
              a0 = fmaf(va[t].z, z[y][t][2], a0); a1 = fmaf(va[t].w, z[y][t][3], a1);
              b0 = fmaf(vb[t].x, z[y][t][0], b0); b1 = fmaf(vb[t].y, z[y][t][1], b1);
              b0 = fmaf(vb[t].z, z[y][t][2], b0); b1 = fmaf(vb[t].w, z[y][t][3], b1);
            }
            da[y] = a0 + a1;
            db[y] = b0 + b1;
          }
#pragma unroll
          for (int o = 1; o < T; o <<= 1)
#pragma unroll
            for (int y = 0; y < 2; ++y) {
              da[y] += __shfl_xor_sync(0xffffffffu, da[y], o);
              db[y] += __shfl_xor_sync(0xffffffffu, db[y], o);
            }
#pragma unroll
          for (int y = 0; y < 2; ++y) {
            const float fb = -bb * db[y];
            const float fa = -ba * fmaf(cc, fb, da[y]);
#pragma unroll
            for (int t = T0; t < CB; ++t) {
              z[y][t][0] = fmaf(fa, va[t].x, fmaf(fb, vb[t].x, z[y][t][0])); z[y][t][1] = fmaf(fa, va[t].y, fmaf(fb, vb[t].y, z[y][t][1]));
              z[y][t][2] = fmaf(fa, va[t].z, fmaf(fb, vb[t].z, z[y][t][2])); z[y][t][3] = fmaf(fa, va[t].w, fmaf(fb, vb[t].w, z[y][t][3]));
            }
          }
        }
      };
      // reflector k starts at entry k + 1
      segment(std::integral_constant<int, CB / 2>{}, D - 4, D / 2);
      segment(std::integral_constant<int, 0>{}, D / 2 - 2, 0);
#pragma unroll
      for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int t = 0; t < CB; ++t)
          *reinterpret_cast<float4*>(&Qt[(r + y * (D / 2)) * LDA + 4 * (q + T * t)]) =
              make_float4(z[y][t][0], z[y][t][1], z[y][t][2], z[y][t][3]);
    }
  }
  __syncthreads();
  // the factor of the sign rule (its space served the prologue, the merges and the reflectors)
  if (a.lift) load_factor();
  __syncthreads();

  // ---- the map from the original space, W = F E (W[i][j] = sum_k F[i][k] Qt[j][k]), into A
  if (a.lift) {
#pragma unroll 1
    for (int tile = tid; tile < TILES; tile += NT) {
      const int tile_i = tile / (D / 4), tile_j = tile % (D / 4);
      float acc[4][4];
      tile_product_rows<D>(L, Qt, LDA, tile_i, tile_j, acc);
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) A[(4 * tile_i + x) * LDA + tile_j + (D / 4) * y] = acc[x][y];
    }
  }
  let_next_start();
  // ---- order, sign, bias
  double* lam = reinterpret_cast<double*>(xbuf);             // [D] doubles over xbuf's 2D floats
  int* rank_of = reinterpret_cast<int*>(pbuf);
  float* sign_of = beta;
  float* mean = rot;                                         // the rotation lists are free now
  if (tid < D) {
    lam[tid] = (double)de[tid].x * a_scale;
    mean[tid] = a.mean_sum ? (float)(a.mean_sum[(size_t)blockIdx.x * D + tid] / a.mean_n) : 0.f;
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
    // . column tid of E where the mean is one of transformed rows
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
  const size_t smem = sizeof(float) * ((size_t)3 * D * (D + 4) + 8 * D + 18 * D);
  auto k = D == 64 ? eigh_tql_kernel<64> : eigh_tql_kernel<128>;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  launch_chained(k, count, kThreads, smem, st, args);
  CA_LAUNCH_CHECK();
  return CA_OK;
}

}  // namespace ca
