// potrf_tile.cuh -- Cholesky factor and inverse of one 64 x 64 diagonal tile by a CTA of 256 threads (the FP64 and the
// mixed factorization's POTRF).
#pragma once
#include "gp_internal.cuh"

namespace {

// POTRF of the 64 x 64 diagonal tiles. A tile accumulates its assembled values and every update in FP64. On the
// factorization's critical path it is eliminated in FP32 (the tile rounded once to FP32) for the FP32 inverse
// of its factor, which the FP32 TRSM of the rows below and the FP32 solves use, like every other off-diagonal
// operand of this path. The factor of the tile itself (L_11, whose diagonal gives the log-determinant) is
// computed in FP64 from the FP64 tile by one batched launch over all diagonal tiles after the last level (the
// tiles are final once their block step has run, and no later step reads L_11); with GP_OPT_DIAG_FP32 the FP32
// elimination stores its L_11 instead. Right-looking, with the tile in registers: thread (tr, tc) of a 16 x 16 grid
// holds the entries (tr + 16 p, tc + 16 q), p, q < 4, of the tile and of X = inv(U), U the unit lower factor
// (A = U diag(d) U^T, U_ik = a_ik / d_k with a_ik column k as updated through column k - 1). The pivots
// d_k = L_kk^2 stay unscaled: column k enters through s_j = a_jk / d_k as a_ij -= a_ik s_j (j > k), and the
// same step eliminates below X's row k: X_ij -= U_ik X_kj (i > k, j <= k), the forward elimination of the
// identity. Two columns per step and one barrier per step (the step's fixed costs -- barrier, shared-memory
// round trip, reciprocal -- are what a column costs here): every thread reads columns k and k + 1 and rows k,
// k + 1 of X as published by their holders, forms column k + 1's and row k + 1's updates by column k itself, and
// applies both. Then L_ik = a_ik / sqrt(d_k), inv(L)_ij = X_ij / sqrt(d_i). X is eliminated in FP32 only.
constexpr int POTRF_THREADS = 256;
constexpr int PT = GP_TILE;

// 1 / d by Newton's iteration r <- r + r (1 - d r) from the hardware's FP32 approximate reciprocal: one step in
// FP32 (within about an ulp), two in FP64 (the error squares per step: about 2^-23 -> 2^-46 -> below an FP64 ulp).
// The pivots are normal numbers well inside the FP32 range (a tile's entries are covariances of order one).
__device__ __forceinline__ float rcp_seed(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}
__device__ __forceinline__ float recip_nr(float d) {
  const float r = rcp_seed(d);
  return fmaf(r, fmaf(-d, r, 1.f), r);
}
__device__ __forceinline__ double recip_nr(double d) {
  double r = (double)rcp_seed((float)d);
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}
// The same for any normal FP64 pivot: its significand goes through the iteration, its exponent is put back after.
__device__ __forceinline__ double recip_any(double d) {
  const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff;
  const double m = __hiloint2double((hi & 0x800fffff) | 0x3ff00000, __double2loint(d));   // in [1, 2)
  return recip_nr(m) * __hiloint2double(max(1, min(2046, 2046 - e)) << 20, 0);
}
__device__ __forceinline__ float recip_any(float d) { return recip_nr(d); }
__device__ __forceinline__ float sqrt_r(float x) { return sqrtf(x); }
__device__ __forceinline__ double sqrt_r(double x) { return sqrt(x); }

// The factorization of one tile by the CTA's 256 threads in arithmetic R (the inverse in X): D the FP64 tile, entry
// (i, j) at i si + j sj (in: the accumulated entries; out, if STORE_L: L), DI its inverse tile (row-major; out, if INV),
// bw its width, first the global column of its first column (a failed pivot records the smallest such column in *flag).
template <class R, class X, bool INV, bool STORE_L>
__device__ __forceinline__ void potrf_tile(double* __restrict__ D, int64_t si, int64_t sj, X* __restrict__ DI, int bw,
                                           int32_t first, int32_t* __restrict__ flag) {
  constexpr int T = PT;
  __shared__ R col[2][2][T];      // columns k, k + 1 after the updates of columns < k (double-buffered)
  __shared__ X xrow[2][2][T]; // rows k, k + 1 of X after the eliminations of rows < k (double-buffered)
  __shared__ R piv[T];            // pivots d_k
  __shared__ R rd[T];             // 1 / d_k
  __shared__ R sc[T];             // 1 / L_kk
  const int tid = threadIdx.x, tr = tid >> 4, tc = tid & 15;
  __syncthreads();   // an earlier call's readers of the shared arrays are done
  R a[4][4];
  X x[4][4];
  uint32_t own = 0;   // bit 4 p + q: entry (tr + 16 p, tc + 16 q) is in the lower triangle of the bw x bw tile
#pragma unroll
  for (int p = 0; p < 4; p++)
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int i = tr + 16 * p, j = tc + 16 * q;
      const bool in = j <= i && i < bw;
      a[p][q] = in ? (R)D[i * si + j * sj] : R(0);
      x[p][q] = i == j ? X(1) : X(0);
      own |= (in ? 1u : 0u) << (4 * p + q);
    }
  if (tc < 2) {
#pragma unroll
    for (int p = 0; p < 4; p++) col[0][tc][tr + 16 * p] = a[p][0];
  }
  if (tr < 2) {
#pragma unroll
    for (int q = 0; q < 4; q++) xrow[0][tr][tc + 16 * q] = x[0][q];
  }
  // Four phases of 16 columns: in phase m columns below 16 m are final, so only the tile's entries of column
  // groups q >= m and row groups p >= q take part (entries above the diagonal inside a diagonal block, and rows
  // past bw, are updated but never read), and only X's entries of row groups p >= m and column groups q <= m.
#pragma unroll
  for (int m = 0; m < 4; m++) {
    const int kend = min(16 * (m + 1), bw);
    for (int k = 16 * m; k < kend; k += 2) {
      __syncthreads();
      const int buf = k & 2 ? 1 : 0;
      const R* ca = col[buf][0];       // column k
      const R* cb = col[buf][1];       // column k + 1 (not yet updated by column k)
      const X* xa = xrow[buf][0];  // row k of X (final)
      const X* xb = xrow[buf][1];  // row k + 1 of X (not yet eliminated by row k)
      const bool two = k + 1 < bw;
      R d0 = ca[k];
      if (!(d0 > R(0))) {
        if (tid == 0) atomicMin(flag, first + k);
        d0 = R(1);
      }
      const R r0 = sizeof(X) == 8 ? recip_any(d0) : recip_nr(d0);
      const R s01 = two ? ca[k + 1] * r0 : R(0);   // U_{k+1, k}
      R d1 = two ? fma(-ca[k + 1], s01, cb[k + 1]) : R(1);
      if (!(d1 > R(0))) {
        if (tid == 0) atomicMin(flag, first + k + 1);
        d1 = R(1);
      }
      const R r1 = sizeof(X) == 8 ? recip_any(d1) : recip_nr(d1);
      if (tid == 0) {
        piv[k] = d0;
        rd[k] = r0;
        if (two) {
          piv[k + 1] = d1;
          rd[k + 1] = r1;
        }
      }
      R ci0[4], ci1[4], sj0[4], sj1[4];
      X xa4[4], xb4[4];
#pragma unroll
      for (int p = m; p < 4; p++) {
        ci0[p] = ca[tr + 16 * p];
        ci1[p] = fma(-ci0[p], s01, cb[tr + 16 * p]);
      }
#pragma unroll
      for (int q = m; q < 4; q++) {
        const R v = ca[tc + 16 * q];
        sj0[q] = v * r0;
        sj1[q] = fma(-v, s01, cb[tc + 16 * q]) * r1;
      }
      const X s01f = (X)s01;
      if (INV) {
#pragma unroll
        for (int q = 0; q <= m; q++) {
          xa4[q] = xa[tc + 16 * q];
          xb4[q] = fma(-s01f, xa4[q], xb[tc + 16 * q]);   // row k + 1 of X, eliminated by row k
        }
      }
      const int jm = tc + 16 * m;   // this thread's column of group m
      const int im = tr + 16 * m;   // this thread's row of group m
#pragma unroll
      for (int q = m; q < 4; q++)
#pragma unroll
        for (int p = q; p < 4; p++) {
          if (q > m || jm > k) a[p][q] = fma(-ci0[p], sj0[q], a[p][q]);
          if (two && (q > m || jm > k + 1)) a[p][q] = fma(-ci1[p], sj1[q], a[p][q]);
        }
      if (INV) {
#pragma unroll
        for (int p = m; p < 4; p++) {
          const X u0 = (X)(ci0[p] * r0), u1 = (X)(ci1[p] * r1);   // U_ik, U_i,k+1
#pragma unroll
          for (int q = 0; q <= m; q++) {
            if (p > m || im > k) x[p][q] = fma(-u0, xa4[q], x[p][q]);
            if (two && (p > m || im > k + 1)) x[p][q] = fma(-u1, xb4[q], x[p][q]);
          }
        }
      }
      const int k2 = k + 2;
      if (k2 < bw) {
        const int qb = k2 >> 4;
        if ((tc >> 1) == ((k2 & 15) >> 1)) {   // publish columns k + 2 and k + 3
          const int h = tc & 1;
          R* cn = col[buf ^ 1][h];
#pragma unroll
          for (int p = m; p < 4; p++) {
            const int i = tr + 16 * p;
            R v = a[p][m];
            if (m < 3 && qb == m + 1) v = a[p][m < 3 ? m + 1 : m];
            if (i >= k2 + h && i < bw) cn[i] = v;
          }
        }
        if (INV && (tr >> 1) == ((k2 & 15) >> 1)) {   // publish rows k + 2 and k + 3 of X
          const int h = tr & 1;
          X* xn = xrow[buf ^ 1][h];
#pragma unroll
          for (int q = 0; q < 4; q++) {
            X v = x[m][q];
            if (m < 3 && qb == m + 1) v = x[m < 3 ? m + 1 : m][q];
            xn[tc + 16 * q] = v;
          }
        }
      }
    }
  }
  __syncthreads();
  if (tid < T) sc[tid] = tid < bw ? sqrt_r(piv[tid]) * rd[tid] : R(1);   // sqrt(d) / d = 1 / L_kk
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 4; p++)
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int i = tr + 16 * p, j = tc + 16 * q;
      X li = X(0);
      if (own >> (4 * p + q) & 1) {
        if (STORE_L) D[i * si + j * sj] = i == j ? (double)sqrt_r(piv[i]) : (double)(a[p][q] * sc[j]);
        li = x[p][q] * (X)sc[i];
      }
      if (INV) DI[i * T + j] = li;
    }
}

}  // namespace
