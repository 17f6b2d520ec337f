// extend_add.cuh -- assembly of a level's fronts from their children's update matrices, one launch per level.
//
// A front's lower triangle is cut into runs of whole rows of about equal size, one CTA each (FP64 fronts, which are
// column-major: runs of whole columns). The CTA zeroes its part of the front's own update matrix and adds, child by
// child in child order, the entries of the child's update matrix that fall into its rows: those of a run of the child's
// rows, since the child's rows keep their order in the parent. Nobody else writes those rows, so the order of the sums
// does not depend on timing. Each child entry is read once, and the front's own entries are zeroed, added to and left in
// the caches meanwhile; a pass that zeroed the matrices ahead and one launch per child slot moved them through memory
// once more each, and a level of small fronts cost as many launches as its front with the most children.
// The work of a warp is a unit of four rows (FP64: two) by 64 columns: the target columns' indices are read once for
// the unit's rows, whose pointers are the same for the whole warp. It is bounded by instructions and by loads in flight:
// decoding each entry's row and column and choosing its target one by one took 0.70 of the issue slots at 16 % of the
// memory rate. Mixed: 0.74 -> 0.18 ms of a factorization at n = 9000 (35 launches -> 9), 2.27 -> 1.30 ms at 100k, 5.1 -> 3.2
// at 200k, 19.8 -> 13.1 at 600k; FP64 (whose zeroing took one CTA per front beside that): 2.25 -> 1.21 ms at 100k, 5.9 -> 4.0
// at 200k. Four rows and four CTAs per SM (64 registers) measured 13.1 ms at 600k, two CTAs (102 registers) 19.1, eight
// rows 18.0, two rows 13.2; FP64 with two rows 4.05 ms at 200k, with four 4.2, with one 4.3.
#pragma once
#include "gp_internal.cuh"

namespace {
namespace ea {

constexpr int T = GP_TILE;
constexpr int THREADS = 256, WARPS = THREADS / 32;
constexpr int COLS = 64;   // of a unit

// Position of the first of the n ascending entries at or after `key`.
__device__ __forceinline__ int32_t lower(const int32_t* __restrict__ a, int32_t n, int32_t key) {
  int32_t lo = 0, hi = n;
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    if (a[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// The units of a CTA go round its warps; `next` counts them (the same in every warp).
struct Units {
  int next = 0;
  // first unit of this warp among n, and the count goes on
  __device__ __forceinline__ int first(int n) {
    const int u = ((int)(threadIdx.x >> 5) - next) & (WARPS - 1);
    next += n;
    return u;
  }
};

// Zeros columns [c0, c0 + 64) below `end` of row pointer p.
template <class V>
__device__ __forceinline__ void zero_strip(V* p, int64_t c0, int64_t end) {
  const int64_t c = c0 + (threadIdx.x & 31);
  if (c < end) p[c] = V(0);
  if (c + 32 < end) p[c + 32] = V(0);
}

// GP_MIXED: FP32 fronts, row-major (panel m x ldw, update matrix r x r), FP64 diagonal tiles. task: (front, first row, end
// row, -).
__global__ void __launch_bounds__(THREADS, 4) k_assemble32(const int4* __restrict__ tab, DevPlan dp,
                                                        float* __restrict__ p32, double* __restrict__ dg,
                                                        float* __restrict__ u32, int64_t P32E, int64_t DE, int64_t UE) {
  constexpr int ROWS = 4;
  __shared__ int32_t rng[3];
  const int lane = threadIdx.x & 31;
  const int4 task = tab[blockIdx.x];
  const int32_t s = task.x;
  const int32_t w = dp.w[s];
  const int64_t r = dp.r[s], ldw = dp.ldw[s];
  float* P = p32 + (int64_t)blockIdx.y * P32E + dp.loff32[s];
  double* D = dg + (int64_t)blockIdx.y * DE + dp.doff[s];
  float* ub = u32 + (int64_t)blockIdx.y * UE;
  float* U = ub + dp.uoff[s];
  Units un;
  for (int32_t i = max(w, task.y); i < task.z; i++) {   // this run's rows of the update matrix: columns up to the diagonal
    const int32_t n = i - w + 1, ns = (n + COLS - 1) / COLS;
    for (int u = un.first(ns); u < ns; u += WARPS) zero_strip(U + (int64_t)(i - w) * r, u * COLS, n);
  }
  for (int32_t q = dp.ch_ptr[s]; q < dp.ch_ptr[s + 1]; q++) {
    const int32_t c = dp.ch_idx[q];
    const int64_t rc = dp.r[c];
    const int32_t* rl = dp.relidx + dp.relidx_off[c];
    const float* Uc = ub + dp.uoff[c];
    __syncthreads();   // zeros and the previous child are in; rng is free
    if (threadIdx.x < 3) rng[threadIdx.x] = lower(rl, (int32_t)rc, threadIdx.x == 0 ? task.y : threadIdx.x == 1 ? task.z : w);
    __syncthreads();
    const int32_t a0 = rng[0], a1 = rng[1], bp = rng[2];   // the child's rows of this run; its columns in the panel
    for (int32_t a = a0; a < a1; a += ROWS) {
      const int32_t ae = min(a + ROWS, a1);                       // columns below ae
      const int np = (min(bp, ae) + COLS - 1) / COLS;             // units in the panel, then in the update matrix
      const int nu = ae > bp ? (ae - bp + COLS - 1) / COLS : 0;
      for (int u = un.first(np + nu); u < np + nu; u += WARPS) {
        const bool inU = u >= np;
        const int32_t b0 = (inU ? bp + (u - np) * COLS : u * COLS) + lane, be = inU ? ae : min(bp, ae);
        int32_t i[ROWS], j[2];
        float* t[ROWS];
        float v[ROWS][2], old[ROWS][2];
        bool ok[ROWS][2];
#pragma unroll
        for (int h = 0; h < 2; h++) j[h] = b0 + 32 * h < be ? rl[b0 + 32 * h] : 0;
#pragma unroll
        for (int k = 0; k < ROWS; k++) {
          i[k] = rl[min(a + k, a1 - 1)];
          t[k] = inU ? U + (i[k] - w) * r - w : P + i[k] * ldw;
          const float* src = Uc + (a + k) * rc + b0;
#pragma unroll
          for (int h = 0; h < 2; h++) {
            ok[k][h] = b0 + 32 * h < be && b0 + 32 * h <= a + k && a + k < a1;
            v[k][h] = ok[k][h] ? src[32 * h] : 0.f;
          }
        }
        if (!inU && i[0] < w) {   // rows of the parent's columns: entries of their FP64 diagonal tiles first
#pragma unroll
          for (int k = 0; k < ROWS; k++)
#pragma unroll
            for (int h = 0; h < 2; h++)
              if (ok[k][h] && i[k] < w && (i[k] >> 6) == (j[h] >> 6)) {
                D[(int64_t)(i[k] >> 6) * (T * T) + (i[k] & 63) * T + (j[h] & 63)] += (double)v[k][h];
                ok[k][h] = false;
              }
        }
#pragma unroll
        for (int k = 0; k < ROWS; k++)
#pragma unroll
          for (int h = 0; h < 2; h++)
            if (ok[k][h]) old[k][h] = t[k][j[h]];
#pragma unroll
        for (int k = 0; k < ROWS; k++)
#pragma unroll
          for (int h = 0; h < 2; h++)
            if (ok[k][h]) t[k][j[h]] = old[k][h] + v[k][h];
      }
    }
  }
}

// GP_FP64: FP64 fronts, column-major; "rows" of the units are columns and the other way round. The runs are counted from
// the end: (front, first, end, -) are the columns m - end .. m - 1 - first.
__global__ void __launch_bounds__(THREADS, 5) k_assemble64(const int4* __restrict__ tab, DevPlan dp,
                                                        double* __restrict__ panels, double* __restrict__ upd, int64_t PE,
                                                        int64_t UE) {
  constexpr int ROWS = 2;
  __shared__ int32_t rng[2];
  const int lane = threadIdx.x & 31;
  const int4 task = tab[blockIdx.x];
  const int32_t s = task.x;
  const int32_t w = dp.w[s];
  const int64_t r = dp.r[s], m = w + r;
  const int32_t j0 = (int32_t)m - task.z, j1 = (int32_t)m - task.y;
  double* P = panels + (int64_t)blockIdx.y * PE + dp.loff[s];
  double* ub = upd + (int64_t)blockIdx.y * UE;
  double* U = ub + dp.uoff[s];
  Units un;
  for (int32_t j = max(w, j0); j < j1; j++) {   // this run's columns of the update matrix: rows from the diagonal on
    const int ns = ((int32_t)m - j + COLS - 1) / COLS;
    for (int u = un.first(ns); u < ns; u += WARPS) zero_strip(U + (j - w) * r, j - w + u * COLS, r);
  }
  for (int32_t q = dp.ch_ptr[s]; q < dp.ch_ptr[s + 1]; q++) {
    const int32_t c = dp.ch_idx[q];
    const int32_t rc = dp.r[c];
    const int32_t* rl = dp.relidx + dp.relidx_off[c];
    const double* Uc = ub + dp.uoff[c];
    __syncthreads();   // zeros and the previous child are in; rng is free
    if (threadIdx.x < 2) rng[threadIdx.x] = lower(rl, rc, threadIdx.x == 0 ? j0 : j1);
    __syncthreads();
    const int32_t b1 = rng[1];
    for (int32_t b = rng[0]; b < b1; b += ROWS) {
      const int ns = (rc - b + COLS - 1) / COLS;
      for (int u = un.first(ns); u < ns; u += WARPS) {
        const int32_t a0 = b + u * COLS + lane;
        int32_t i[2];
        double* t[ROWS];
        double v[ROWS][2], old[ROWS][2];
        bool ok[ROWS][2];
#pragma unroll
        for (int h = 0; h < 2; h++) i[h] = a0 + 32 * h < rc ? rl[a0 + 32 * h] : 0;
#pragma unroll
        for (int k = 0; k < ROWS; k++) {
          const int32_t j = rl[min(b + k, b1 - 1)];
          t[k] = j < w ? P + j * m : U + (j - w) * r - w;   // from row 0
          const double* src = Uc + (int64_t)(b + k) * rc + a0;
#pragma unroll
          for (int h = 0; h < 2; h++) {
            ok[k][h] = a0 + 32 * h < rc && a0 + 32 * h >= b + k && b + k < b1;
            v[k][h] = ok[k][h] ? src[32 * h] : 0.0;
          }
        }
#pragma unroll
        for (int k = 0; k < ROWS; k++)
#pragma unroll
          for (int h = 0; h < 2; h++)
            if (ok[k][h]) old[k][h] = t[k][i[h]];
#pragma unroll
        for (int k = 0; k < ROWS; k++)
#pragma unroll
          for (int h = 0; h < 2; h++)
            if (ok[k][h]) t[k][i[h]] = old[k][h] + v[k][h];
      }
    }
  }
}

}  // namespace ea
}  // namespace
