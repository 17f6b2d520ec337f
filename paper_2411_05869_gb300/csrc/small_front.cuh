// small_front.cuh -- the elimination of a front of order m <= GP_SMALL_M in FP64 shared memory, one CTA of 256 threads, for
// both precisions' factors.
#pragma once
#include "gp_internal.cuh"

namespace sf {

constexpr int THREADS = 256;

// First w columns of the Cholesky of A (m x m, column-major, lower part used; its trailing part becomes the update
// matrix). A column's pivot chain bounds it (FP64 instructions depend on one another at 64 clocks each), so the chain holds
// no more than it must: warp 0 updates the next column first and forms the reciprocal root of its pivot while the other
// warps update the rest; the root itself, which nothing waits for, is the last warp's. (Root, then a division by every
// thread, and the whole update before the next pivot: 77 against 55 us a launch at n = 2000 in FP64.)
__device__ __forceinline__ void eliminate(double* A, int m, int w, int32_t first, int32_t* notpd) {
  __shared__ double inv_s[2];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    const double d = A[0];
    inv_s[0] = d > 0.0 ? rsqrt(d) : 1.0;
  }
  __syncthreads();
  for (int k = 0; k < w; k++) {
    double* ak = A + k * m;
    const double inv = inv_s[k & 1];
    for (int i = k + 1 + (int)threadIdx.x; i < m; i += THREADS) ak[i] *= inv;
    __syncthreads();
    if (ty == 0) {
      if (k + 1 < m) {
        const double ajk = ak[k + 1];
        for (int i = k + 1 + tx; i < m; i += 32) A[(k + 1) * m + i] -= ak[i] * ajk;
        __syncwarp();
        if (tx == 0 && k + 1 < w) {
          const double d = A[(k + 1) * m + k + 1];
          inv_s[(k + 1) & 1] = d > 0.0 ? rsqrt(d) : 1.0;
        }
      }
    } else {
      for (int j = k + 1 + ty; j < m; j += THREADS / 32 - 1) {
        const double ajk = ak[j];
        for (int i = j + tx; i < m; i += 32) A[j * m + i] -= ak[i] * ajk;
      }
      if (threadIdx.x == THREADS - 32) {
        const double d = ak[k];
        if (!(d > 0.0)) atomicMin(notpd, first + k);
        ak[k] = d > 0.0 ? sqrt(d) : 1.0;
      }
    }
    __syncthreads();
  }
}

}  // namespace sf
