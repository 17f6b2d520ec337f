// variance.cu -- the predictive variance (Sec. 3.2): the diagonal of the conditional covariance
//   C_{y|z} = C_y - C_{y,z} C_z^{-1} C_{z,y},   var_k = C_y(x*_k, x*_k) - |w_k|^2,   L w_k = P c_k,
// c_k = C_y(X, x*_k) the cross-covariance column of test point k (no noise term at test inputs, Sec. 3.2) and
// C_y(x*, x*) = core_var (s0 + sum_i f_i(x*)^2) (f0(0) = 1 for the core and for C_sparse).
//
// c_k is nonzero only at the training neighbours of x*_k (the core support), so w_k is nonzero only on the
// supernodes on the paths from those neighbours' supernodes to the root of the supernodal elimination tree. Test
// points go through the factor's forward sweep R = 32 at a time (a chunk; NC chunks side by side in the grid):
//   mark  (warp per test point): the prior C_y(x*, x*) into the output, and every supernode on a neighbour's path
//         marked active for the chunk;
//   zero / scatter: the active supernodes' front vectors (m_s x R) cleared, then c_k written at its neighbours'
//         rows;
//   levels ascending: children's update vectors added into the parents (in child order), fronts of order <= 96
//         eliminated by one CTA, larger fronts of the mixed factor by groups of four 64-column blocks J: one CTA
//         solves a group's X_J = inv(L_JJ) (F_J - sum of the group's L_JK X_K), then one launch applies
//         F_I -= L_IJ X_J to the later blocks' rows; a last launch applies all J to the rows below the front's
//         columns. A CTA takes two or four of the chunks that are active in its front. FP64: a block at a time, 16 rows
//         of one chunk per CTA;
//   sum: |w_k|^2 over all entries in a fixed order, var_k = prior_k - |w_k|^2.
// The arithmetic is the factor's working precision: FP64 with the FP64 factor; FP32 vectors with the mixed
// factor's FP32 panels and inverses (the variance then carries the mixed factor's ~1e-6 relative accuracy).
#include <cuda_pipeline.h>

#include <algorithm>
#include <type_traits>

#include "factor_access.cuh"
#include "gp_internal.cuh"
#include "testpoint.cuh"

namespace {

constexpr int T = GP_TILE;
constexpr int R = 32;   // test points per chunk

// Per chunk c: front vectors at F + c * cs (row i of front s at (frow_off[s] + i) * R), then the w entries of the
// n permuted columns at X + c * cs (column j at j * R).
template <class V>
struct VarWork {
  V* F;
  V* X;
  int64_t cs;             // entries per chunk (front rows x R + n x R)
  uint8_t* active;        // NC x ns
  int64_t ns;
};

__global__ void k_var_mark(const double* __restrict__ Xt, int64_t m, int64_t k0, tp::GridInfo g,
                           const double* __restrict__ X, const double* __restrict__ Us,
                           const int32_t* __restrict__ cell_perm, const int64_t* __restrict__ cell_start,
                           const double* __restrict__ theta, int n1, int n2, int bd, const double* __restrict__ F,
                           const double* __restrict__ Cpt, const int32_t* __restrict__ pinv, DevPlan dp,
                           uint8_t* __restrict__ active, int64_t ns, double* __restrict__ var) {
  __shared__ double fs[8][GP_MAX_N1];
  __shared__ double gs[8][64];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int64_t q = (int64_t)blockIdx.x * 8 + wi;   // index in the batch
  const int64_t k = k0 + q;
  if (k >= m) return;
  const tp::TestPoint p = tp::load_features(Xt, k, g, theta, n1, n2, bd, fs[wi], gs[wi]);
  uint8_t* act = active + (q / R) * ns;
  tp::for_each_neighbour(p, g, X, Us, cell_perm, cell_start, theta, n1, fs[wi], F, Cpt, [&](int32_t j, double) {
    for (int32_t s = dp.sn_of_col[pinv[j]]; s >= 0 && !act[s]; s = dp.sn_parent[s]) act[s] = 1;
  });
  if (lane == 0) {   // C_y(x*, x*) = C_core(x*, x*) (s0 + sum_i f_i(x*)^2)
    double ss = theta[TH_S0];
    for (int i = 0; i < n1; i++) ss += fs[wi][i] * fs[wi][i];
    double core = theta[TH_CORE_VAR];
    if (theta[TH_KIND] != 0.0) {
      double cs[2];
      tp::core_point(theta, p.xs, g.d, cs);
      core = tp::core_paciorek(cs, cs, p.xs, p.xs, g.d);
    }
    var[k] = core * ss;
  }
}

// A warp per (supernode, chunk): clears the active supernodes' front vectors.
template <class V>
__global__ void k_var_zero(DevPlan dp, int64_t ns, VarWork<V> vw) {
  const int64_t s = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int c = blockIdx.y, lane = threadIdx.x & 31;
  if (s >= ns || !vw.active[c * ns + s]) return;
  V* f = vw.F + c * vw.cs + dp.frow_off[s] * R;
  const int64_t cnt = ((int64_t)dp.w[s] + dp.r[s]) * R;
  for (int64_t e = lane; e < cnt; e += 32) f[e] = V(0);
}

template <class V>
__global__ void k_var_scatter(const double* __restrict__ Xt, int64_t m, int64_t k0, tp::GridInfo g,
                              const double* __restrict__ X, const double* __restrict__ Us,
                              const int32_t* __restrict__ cell_perm, const int64_t* __restrict__ cell_start,
                              const double* __restrict__ theta, int n1, int n2, int bd, const double* __restrict__ F,
                              const double* __restrict__ Cpt, const int32_t* __restrict__ pinv, DevPlan dp,
                              VarWork<V> vw) {
  __shared__ double fs[8][GP_MAX_N1];
  __shared__ double gs[8][64];
  const int wi = threadIdx.x >> 5;
  const int64_t q = (int64_t)blockIdx.x * 8 + wi;
  const int64_t k = k0 + q;
  if (k >= m) return;
  const tp::TestPoint p = tp::load_features(Xt, k, g, theta, n1, n2, bd, fs[wi], gs[wi]);
  V* base = vw.F + (q / R) * vw.cs;
  const int r = (int)(q % R);
  tp::for_each_neighbour(p, g, X, Us, cell_perm, cell_start, theta, n1, fs[wi], F, Cpt, [&](int32_t j, double cy) {
    const int32_t pj = pinv[j];
    const int32_t s = dp.sn_of_col[pj];
    base[(dp.frow_off[s] + (pj - dp.sn_first[s])) * R + r] = (V)cy;
  });
}

// Children's update vectors into the front vectors of the level's supernodes (children in order): CTA (x, y, z) takes
// rows [GROWS z, GROWS (z + 1)) of front list[x] for chunk y.
constexpr int GROWS = 256;
template <class V>
__global__ void k_var_gather(const int32_t* __restrict__ list, DevPlan dp, VarWork<V> vw) {
  const int32_t s = list[blockIdx.x];
  const int c = blockIdx.y;
  const uint8_t* act = vw.active + c * vw.ns;
  const int32_t lo = (int32_t)blockIdx.z * GROWS;
  if (lo >= dp.w[s] + dp.r[s] || !act[s]) return;
  __shared__ int32_t rng[2];
  V* W = vw.F + c * vw.cs;
  V* fv = W + dp.frow_off[s] * R;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int32_t qc = dp.ch_ptr[s]; qc < dp.ch_ptr[s + 1]; qc++) {
    const int32_t ch = dp.ch_idx[qc];
    if (!act[ch]) continue;
    const V* uc = W + ((int64_t)dp.frow_off[ch] + dp.w[ch]) * R;
    const int32_t* rel = dp.relidx + dp.relidx_off[ch];
    if (threadIdx.x < 2) {   // the child's rows that fall into this CTA's: rel is increasing
      const int32_t key = lo + (threadIdx.x == 0 ? 0 : GROWS);
      int32_t x = 0, y = dp.r[ch];
      while (x < y) {
        const int32_t mid = (x + y) >> 1;
        if (rel[mid] < key) x = mid + 1;
        else y = mid;
      }
      rng[threadIdx.x] = x;
    }
    __syncthreads();
    for (int32_t a = rng[0] + warp; a < rng[1]; a += nw) fv[(int64_t)rel[a] * R + lane] += uc[(int64_t)a * R + lane];
    __syncthreads();   // this child's rows land before the next child's, and rng is free again
  }
}

// Fronts of order <= GP_SMALL_M: forward elimination of the whole front, R right-hand sides, one CTA.
template <class St>
__global__ void k_var_small(const int32_t* __restrict__ list, DevPlan dp, St store, int b,
                            VarWork<typename St::V> vw) {
  using V = typename St::V;
  __shared__ V Fs[GP_SMALL_M][R];
  __shared__ V xr[R];
  const int32_t s = list[blockIdx.x];
  const int c = blockIdx.y;
  if (!vw.active[c * vw.ns + s]) return;
  auto A = store.acc(dp, s, b);
  V* fv = vw.F + c * vw.cs + dp.frow_off[s] * R;
  V* xv = vw.X + c * vw.cs + (int64_t)dp.sn_first[s] * R;
  const int w = dp.w[s], m = w + dp.r[s];
  for (int e = threadIdx.x; e < m * R; e += blockDim.x) Fs[e / R][e % R] = fv[e];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int j = 0; j < w; j++) {
    if (warp == 0) {
      const V x = Fs[j][lane] / A.L(j, j);
      xr[lane] = x;
      xv[(int64_t)j * R + lane] = x;
    }
    __syncthreads();
    for (int i = j + 1 + warp; i < m; i += nw) Fs[i][lane] -= A.L(i, j) * xr[lane];
    __syncthreads();
  }
  for (int e = threadIdx.x; e < (m - w) * R; e += blockDim.x) fv[(int64_t)w * R + e] = Fs[w + e / R][e % R];
}

// The large fronts of a level with the mixed factor. A CTA of 256 threads takes CH of the chunks that are active in its
// front (32 CH right-hand sides) and a 64-row tile, a thread four rows by 2 CH right-hand sides in groups of four: per
// step of the products it reads 1 + CH / 2 16-byte vectors from shared memory, a step ahead, for 8 CH multiply-adds. The
// products bound it: FP32 multiply-adds, at about 60% of their rate on the wide levels, and one CTA's latency on the
// narrow ones. The front vectors move through memory once per group of blocks, not once per block. 2048 test points of
// the 100k workload: 48 ms with one chunk per CTA, eight entries of one row per thread and X_J formed anew by every tile
// of a block column; 22 ms with two chunks and X_J formed once; 16.5 ms with the rows below the columns in one launch,
// groups of four blocks and every load on its way before the first wait; 14.1 ms with the products' reads a step ahead.
// Every entry's sum runs over a block's columns in order, and the blocks' sums are subtracted in order.
constexpr int MS = T + 4;   // row stride of the matrix tile in shared memory (16-byte vectors)
constexpr size_t var_smem(int bufs, int ch) { return (size_t)(T * MS + bufs * T * ch * R) * sizeof(float); }

__device__ __forceinline__ void ld4(const float* p, float* d) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  d[0] = u.x, d[1] = u.y, d[2] = u.z, d[3] = u.w;
}
__device__ __forceinline__ void st4(float* p, const float* d) {
  *reinterpret_cast<float4*>(p) = make_float4(d[0], d[1], d[2], d[3]);
}
__device__ __forceinline__ void ld4_or_zero(bool on, const float* p, float* d) {
  if (on) ld4(p, d);
  else d[0] = d[1] = d[2] = d[3] = 0.f;
}

// acc[e][f] = sum_l Mt[l][tr + e] Fb[l][tc + 64 (f / 4) + f % 4].
template <int CH>
__device__ __forceinline__ void var_product(const float* Mt, const float* Fb, int tr, int tc, float (&acc)[4][2 * CH]) {
#pragma unroll
  for (int e = 0; e < 4; e++)
#pragma unroll
    for (int f = 0; f < 2 * CH; f++) acc[e][f] = 0.f;
  float a[2][4], x[2][2 * CH];   // step l's and step l + 1's entries
  auto fetch = [&](int l, int h) {
    ld4(Mt + l * MS + tr, a[h]);
#pragma unroll
    for (int g = 0; g < CH / 2; g++) ld4(Fb + l * (CH * R) + tc + 64 * g, x[h] + 4 * g);
  };
  fetch(0, 0);
#pragma unroll 8
  for (int l = 0; l < T; l++) {
    const int h = l & 1;
    fetch(min(l + 1, T - 1), h ^ 1);
#pragma unroll
    for (int e = 0; e < 4; e++)
#pragma unroll
      for (int f = 0; f < 2 * CH; f++) acc[e][f] += a[h][e] * x[h][f];
  }
}

// This thread's rows tr.. +3 and columns tc + 64 g.. +3 of the CTA's CH chunks, the blockIdx.y-th CH of those active in
// front s: chunk c[g] (-1: none), right-hand sides r.. +3.
template <int CH>
struct VarLane {
  int tr, tc, r, c[CH / 2];
  bool any;   // of the CTA
  __device__ __forceinline__ VarLane(const VarWork<float>& vw, int32_t s, int nc)
      : tr((threadIdx.x >> 4) * 4), tc((threadIdx.x & 15) * 4), r(tc & 31) {
    const int lane = threadIdx.x & 31;   // nc <= 64
    const unsigned lo = __ballot_sync(~0u, lane < nc && vw.active[lane * vw.ns + s]);
    const unsigned hi = __ballot_sync(~0u, lane + 32 < nc && vw.active[(lane + 32) * vw.ns + s]);
    unsigned long long set = (unsigned long long)hi << 32 | lo;
    for (int q = CH * blockIdx.y; q > 0 && set; q--) set &= set - 1;
    any = set != 0;
#pragma unroll
    for (int g = 0; g < CH / 2; g++) {
      unsigned long long x = (tc >> 5) ? set & (set - 1) : set;
      c[g] = x ? __ffsll((long long)x) - 1 : -1;
      set &= set - 1;
      set &= set - 1;
    }
  }
};

// Blocks g0.. + VG of the large fronts of a step: X_J = inv(L_JJ) (F_J - sum_K L_JK X_K) over the group's blocks K < J.
// The group's X stay in shared memory; the next 64 x 64 tile is on its way to registers during each product.
constexpr int VG = 4;   // blocks per group
__global__ void __launch_bounds__(256, 2)
    k_var_group(const int32_t* __restrict__ fronts, int g0, int nc, DevPlan dp, fa::StoreMix store, int b,
                VarWork<float> vw) {
  constexpr int CH = 2, N = T * T / 256;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* Mt = reinterpret_cast<float*>(smem_raw);   // Mt[l][i]: the product's matrix, row i, column l
  float* Xb = Mt + T * MS;                      // per block [l][r]: F_J, then X_J
  const int32_t s = fronts[blockIdx.x];
  const VarLane<CH> t(vw, s, nc);
  if (!t.any) return;
  auto A = store.acc(dp, s, b);
  const float* inv = store.inv(dp, s, b);
  const int w = dp.w[s], nb = min(VG, (w - g0 * T + T - 1) / T);
  const bool on = t.c[0] >= 0;
  float* xv = vw.X + (on ? t.c[0] : 0) * vw.cs + ((int64_t)dp.sn_first[s] + t.tr) * R + t.r;
  const float* fv = vw.F + (on ? t.c[0] : 0) * vw.cs + (dp.frow_off[s] + t.tr) * R + t.r;
  float v[4][4], lt[N], acc[4][4];
  auto load = [&](int j, int k) {   // L_JK; the inverse of L_JJ (zero past w)
    const int r0 = (g0 + j) * T, c0 = (g0 + k) * T;
#pragma unroll
    for (int q = 0; q < N; q++) {
      const int e = (int)threadIdx.x + 256 * q, i = e >> 6, l = e & 63;
      if (k == j) lt[q] = inv[(int64_t)(g0 + j) * T * T + e];
      else lt[q] = r0 + i < w ? A.off(r0 + i, c0 + l) : 0.f;
    }
  };
  load(0, 0);
  for (int j = 0; j < nb; j++) {
    const int r0 = (g0 + j) * T;
    float* Xj = Xb + j * (T * CH * R) + t.tr * (CH * R) + t.tc;   // this thread's entries
#pragma unroll
    for (int e = 0; e < 4; e++) ld4_or_zero(on && r0 + t.tr + e < w, fv + (int64_t)(r0 + e) * R, v[e]);
    for (int k = 0; k <= j; k++) {
#pragma unroll
      for (int q = 0; q < N; q++) {
        const int e = (int)threadIdx.x + 256 * q;
        Mt[(e & 63) * MS + (e >> 6)] = lt[q];
      }
      if (k == j) {
#pragma unroll
        for (int e = 0; e < 4; e++) st4(Xj + e * (CH * R), v[e]);
      }
      __syncthreads();
      if (k < j) load(j, k + 1);
      else if (j + 1 < nb) load(j + 1, 0);
      var_product<CH>(Mt, Xb + k * (T * CH * R), t.tr, t.tc, acc);
      __syncthreads();   // the matrix tile and F_J are free
      if (k < j) {
#pragma unroll
        for (int e = 0; e < 4; e++)
#pragma unroll
          for (int f = 0; f < 4; f++) v[e][f] -= acc[e][f];
      }
    }
#pragma unroll
    for (int e = 0; e < 4; e++) {   // the next product's barrier makes it everyone's
      st4(Xj + e * (CH * R), acc[e]);
      if (on && r0 + t.tr + e < w) st4(xv + (int64_t)(r0 + e) * R, acc[e]);
    }
  }
}

// F_I -= sum_J L_IJ X_J on 64-row tile blockIdx.z of the later blocks' rows, J over the group of blocks g0.. + VG;
// g0 < 0: of the rows below the large fronts' columns, J over all blocks.
__global__ void __launch_bounds__(256, 2)
    k_var_rest(const int32_t* __restrict__ fronts, int g0, int nc, DevPlan dp, fa::StoreMix store, int b,
               VarWork<float> vw) {
  constexpr int CH = 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* Mt = reinterpret_cast<float*>(smem_raw);   // Mt[l][i]: L[r0 + i][c0 + l]
  float* Fb0 = Mt + T * MS;                     // two buffers of [l][r]: X_J
  const int32_t s = fronts[blockIdx.x];
  const int w = dp.w[s], b0 = max(g0, 0), b1 = g0 < 0 ? (w + T - 1) / T : g0 + VG;   // blocks [b0, b1)
  const int r0 = (g0 < 0 ? w : b1 * T) + (int)blockIdx.z * T, nr = min(T, (g0 < 0 ? w + dp.r[s] : w) - r0);
  if (nr <= 0) return;
  const VarLane<CH> t(vw, s, nc);
  if (!t.any) return;
  auto A = store.acc(dp, s, b);
  float* row = vw.F + (dp.frow_off[s] + r0 + t.tr) * R + t.r;
  const float* xs = vw.X + ((int64_t)dp.sn_first[s] + t.tr) * R + t.r;
  float v[4][2 * CH], lt[T * T / 256];
#pragma unroll
  for (int e = 0; e < 4; e++)
#pragma unroll
    for (int g = 0; g < CH / 2; g++)
      ld4_or_zero(t.c[g] >= 0 && t.tr + e < nr, row + t.c[g] * vw.cs + e * R, v[e] + 4 * g);
  auto load = [&](int kb) {   // block kb: the tile's entries to registers, X to its buffer (asynchronously)
    const int c0 = kb * T, bw = min(T, w - c0);
    float* Fb = Fb0 + (kb & 1) * T * CH * R;
#pragma unroll
    for (int q = 0; q < T * T / 256; q++) {
      const int e = (int)threadIdx.x + 256 * q, i = e >> 6, l = e & 63;
      lt[q] = i < nr && l < bw ? A.off(r0 + i, c0 + l) : 0.f;
    }
#pragma unroll
    for (int e = 0; e < 4; e++)
#pragma unroll
      for (int g = 0; g < CH / 2; g++) {   // one 16-byte vector
          float* d = Fb + (t.tr + e) * (CH * R) + t.tc + 64 * g;
          if (t.c[g] >= 0 && t.tr + e < bw)
            __pipeline_memcpy_async(d, xs + t.c[g] * vw.cs + (int64_t)(c0 + e) * R, 16);
          else
            d[0] = d[1] = d[2] = d[3] = 0.f;
        }
    __pipeline_commit();
  };
  load(b0);
  for (int kb = b0; kb < b1; kb++) {
#pragma unroll
    for (int q = 0; q < T * T / 256; q++) {
      const int e = (int)threadIdx.x + 256 * q;
      Mt[(e & 63) * MS + (e >> 6)] = lt[q];
    }
    __pipeline_wait_prior(0);
    __syncthreads();
    if (kb + 1 < b1) load(kb + 1);
    float acc[4][2 * CH];
    var_product<CH>(Mt, Fb0 + (kb & 1) * T * CH * R, t.tr, t.tc, acc);   // zeros past w
#pragma unroll
    for (int e = 0; e < 4; e++)
#pragma unroll
      for (int f = 0; f < 2 * CH; f++) v[e][f] -= acc[e][f];
    __syncthreads();   // the tile and this block's buffer are free again
  }
#pragma unroll
  for (int e = 0; e < 4; e++)
#pragma unroll
    for (int g = 0; g < CH / 2; g++)
      if (t.c[g] >= 0 && t.tr + e < nr) st4(row + t.c[g] * vw.cs + e * R, v[e] + 4 * g);
}

// The large fronts of a level in FP64. A warp's FP64 multiply-add takes 64 clocks of its scheduler, so a 64 x 64 by
// 64 x 32 product would hold an SM for 32 us: a CTA takes 16 rows of one chunk (two right-hand sides per thread), which
// spreads the narrow levels' products over the SMs; shared memory and latency do not show.
// what = VX: X_J = inv(L_JJ) F_J, rows 16 z of block J = jb; VSTEP: F_I -= L_IJ X_J, rows 16 z of the block columns' rows
// after block J; VREST: F_I -= sum_J L_IJ X_J, rows 16 z below the front's columns. 2048 (70) test points of a
// 20,000-point space-time factor: 86 (10.0) ms with 64-row tiles
// that each formed X_J anew, 66 (27) ms with the mixed factor's kernels above, 48 (5.2) ms here.
enum { VX, VSTEP, VREST };
__global__ void __launch_bounds__(256)
    k_var_rows64(const int32_t* __restrict__ fronts, int what, int jb, DevPlan dp, fa::StoreF64 store, int b,
                 VarWork<double> vw) {
  __shared__ double Mt[T][17];   // Mt[l][i]
  __shared__ __align__(16) double Xs[T][R];
  const int32_t s = fronts[blockIdx.x];
  const int c = blockIdx.y;
  if (!vw.active[c * vw.ns + s]) return;
  const int w = dp.w[s];
  const int r0 = (what == VREST ? w : what == VSTEP ? (jb + 1) * T : jb * T) + 16 * (int)blockIdx.z;
  const int nr = min(16, (what == VREST ? w + dp.r[s] : what == VSTEP ? w : min(w, (jb + 1) * T)) - r0);
  if (nr <= 0) return;
  const int b0 = what == VREST ? 0 : jb, b1 = what == VREST ? (w + T - 1) / T : jb + 1;
  const fa::AccF64 A = store.acc(dp, s, b);
  const double* inv = store.inv(dp, s, b) + (int64_t)jb * T * T;
  double* F = vw.F + c * vw.cs + dp.frow_off[s] * R;
  double* X = vw.X + c * vw.cs + (int64_t)dp.sn_first[s] * R;
  const double* src = what == VX ? F : X;
  const int i = threadIdx.x >> 4, r = (threadIdx.x & 15) * 2;
  double v[2] = {0.0, 0.0};
  if (what != VX && i < nr) {
    v[0] = F[(int64_t)(r0 + i) * R + r];
    v[1] = F[(int64_t)(r0 + i) * R + r + 1];
  }
  for (int kb = b0; kb < b1; kb++) {
    const int c0 = kb * T, bw = min(T, w - c0);
    for (int e = threadIdx.x; e < T * R; e += 256) Xs[e / R][e % R] = e / R < bw ? src[(int64_t)c0 * R + e] : 0.0;
    if (what == VX) {
      for (int e = threadIdx.x; e < T * 16; e += 256) Mt[e & 63][e >> 6] = inv[(r0 - c0) * T + e];   // zero past bw
    } else {
      for (int e = threadIdx.x; e < T * 16; e += 256)
        Mt[e >> 4][e & 15] = (e & 15) < nr && (e >> 4) < bw ? A.off(r0 + (e & 15), c0 + (e >> 4)) : 0.0;
    }
    __syncthreads();
    double a0 = 0.0, a1 = 0.0;
#pragma unroll 8
    for (int l = 0; l < T; l++) {
      const double2 x = *reinterpret_cast<const double2*>(&Xs[l][r]);
      a0 += Mt[l][i] * x.x;
      a1 += Mt[l][i] * x.y;
    }
    __syncthreads();
    if (what == VX) v[0] = a0, v[1] = a1;
    else v[0] -= a0, v[1] -= a1;
  }
  double* dst = what == VX ? X : F;
  if (i < nr) {
    dst[(int64_t)(r0 + i) * R + r] = v[0];
    dst[(int64_t)(r0 + i) * R + r + 1] = v[1];
  }
}

// Partial sums of w^2 per (chunk, right-hand side) over column slices, in a fixed order: CTA g of chunk c sums
// columns j = 8 g' + (t >> 5) for its slice, lanes = right-hand sides.
constexpr int SUM_CTAS = 64;
template <class V>
__global__ void k_var_sumsq(int64_t n, VarWork<V> vw, double* __restrict__ part) {
  __shared__ double sp[8][R];
  const int c = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const V* x = vw.X + c * vw.cs;
  double acc = 0.0;
#pragma unroll 8
  for (int64_t j = (int64_t)blockIdx.x * 8 + warp; j < n; j += (int64_t)gridDim.x * 8) {
    const double v = (double)x[j * R + lane];
    acc += v * v;
  }
  sp[warp][lane] = acc;
  __syncthreads();
  if (warp == 0) {
    double a = 0.0;
    for (int q = 0; q < 8; q++) a += sp[q][lane];
    part[((int64_t)c * gridDim.x + blockIdx.x) * R + lane] = a;
  }
}

__global__ void k_var_final(const double* __restrict__ part, int nparts, int64_t m, int64_t k0,
                            double* __restrict__ var) {
  const int c = blockIdx.x, r = threadIdx.x;
  const int64_t k = k0 + (int64_t)c * R + r;
  if (k >= m) return;
  double a = 0.0;
  for (int q = 0; q < nparts; q++) a += part[((int64_t)c * nparts + q) * R + r];
  var[k] -= a;
}

template <class St>
void variance_impl(gp_ctx* ctx, gp_factor_t* f, const St& store, int b, const double* d_Xt, int64_t m,
                   double* d_var) {
  using V = typename St::V;
  gp_pointset* ps = f->ps;
  const SymPlan& sp = ps->sp;
  const DevPlan& dp = ps->dp;
  cudaStream_t st = ctx->stream;
  const int64_t n = ps->n, ns = sp.ns, FR = sp.sn_frow[ns];
  const int64_t cs = (FR + n) * R;
  const int64_t per_chunk = cs * (int64_t)sizeof(V) + ns + SUM_CTAS * R * 8;
  const int64_t want = (m + R - 1) / R;
  if (!f->var_work) {   // workspace for NC chunks, allocated once per factor
    size_t freeb = 0, totb = 0;
    GP_CUDA(cudaMemGetInfo(&freeb, &totb));
    const int64_t cap = std::min<int64_t>((int64_t)4 << 30, (int64_t)(freeb / 4));
    int64_t nc = std::max<int64_t>(1, std::min<int64_t>(64, cap / per_chunk));
    if (ctx->budget) nc = std::max<int64_t>(1, std::min<int64_t>(nc, (int64_t)(ctx->budget - std::min(ctx->budget, ctx->held.load())) / per_chunk));
    f->var_nc = (int)nc;
    f->var_work = dalloc<uint8_t>(ctx, f->bufs, (size_t)(nc * per_chunk) + 256);
  }
  const int NC = (int)std::min<int64_t>(f->var_nc, want);
  VarWork<V> vw;
  vw.F = reinterpret_cast<V*>(f->var_work);
  vw.X = vw.F + FR * R;
  vw.cs = cs;
  vw.active = f->var_work + (size_t)f->var_nc * cs * sizeof(V);
  vw.ns = ns;
  double* part = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(vw.active + (size_t)f->var_nc * ns) + 15) &
                                           ~(uintptr_t)15);
  const tp::GridInfo g = tp::grid_of(ps);
  const gp_hyper& h0 = f->thetas_host[0];
  const double* theta = f->theta_dev + (int64_t)b * f->theta_stride;
  const double* Fb = f->F + (int64_t)b * n * h0.n1;
  const double* Cb = f->Cpt ? f->Cpt + (int64_t)b * n * 2 : nullptr;
  constexpr bool fp64 = std::is_same_v<St, fa::StoreF64>;
  const size_t rest_smem = var_smem(2, 4);
  if constexpr (!fp64) {
    GP_CUDA(cudaFuncSetAttribute(k_var_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)var_smem(VG, 2)));
    GP_CUDA(cudaFuncSetAttribute(k_var_rest, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rest_smem));
  }
  ProfScope ps_(ctx, KC_PREDICT);
  for (int64_t k0 = 0; k0 < m; k0 += (int64_t)NC * R) {
    const int64_t cnt = std::min<int64_t>(m - k0, (int64_t)NC * R);
    const int nc = (int)((cnt + R - 1) / R);
    GP_CUDA(cudaMemsetAsync(vw.active, 0, (size_t)nc * ns, st));
    for (int c = 0; c < nc; c++)
      GP_CUDA(cudaMemsetAsync(vw.X + c * cs, 0, (size_t)n * R * sizeof(V), st));
    k_var_mark<<<grid_for(cnt, 8), 256, 0, st>>>(d_Xt, m, k0, g, ps->X, ps->Us, ps->cell_perm, ps->cell_start, theta,
                                                h0.n1, h0.n2, h0.bump_dims, Fb, Cb, ps->pinv, dp, vw.active, ns,
                                                d_var);
    GP_CHECK_LAUNCH(ctx);
    k_var_zero<V><<<dim3(grid_for(ns, 8), nc), 256, 0, st>>>(dp, ns, vw);
    GP_CHECK_LAUNCH(ctx);
    k_var_scatter<V><<<grid_for(cnt, 8), 256, 0, st>>>(d_Xt, m, k0, g, ps->X, ps->Us, ps->cell_perm, ps->cell_start,
                                                       theta, h0.n1, h0.n2, h0.bump_dims, Fb, Cb, ps->pinv, dp, vw);
    GP_CHECK_LAUNCH(ctx);
    for (int32_t L = 0; L < sp.nlevels; L++) {
      const SymPlan::Level& lv = sp.levels[L];
      const int32_t nl = sp.lev_ptr[L + 1] - sp.lev_ptr[L];
      if (L > 0) {
        int32_t mmax = 1;   // the level's largest front
        for (int32_t q = sp.lev_ptr[L]; q < sp.lev_ptr[L + 1]; q++)
          mmax = std::max(mmax, sp.sn_w[sp.lev_sn[q]] + sp.sn_r[sp.lev_sn[q]]);
        k_var_gather<V><<<dim3(nl, nc, (mmax + GROWS - 1) / GROWS), 256, 0, st>>>(dp.lev_sn + sp.lev_ptr[L], dp, vw);
        GP_CHECK_LAUNCH(ctx);
      }
      if (lv.nsmall > 0) {
        k_var_small<St><<<dim3(lv.nsmall, nc), 256, 0, st>>>(dp.small_list + lv.small_off, dp, store, b, vw);
        GP_CHECK_LAUNCH(ctx);
      }
      if (lv.steps.empty()) continue;
      // The level's large fronts, widest first (nb blocks).
      const int nb = (int)lv.steps.size();
      const auto& s0 = lv.steps[0];
      const auto list = [&](int k) { return dp.large_fronts + lv.steps[k].fr_off; };   // the fronts that have block k
      int32_t rmax = 0;
      for (int32_t q = 0; q < s0.nfront; q++) rmax = std::max(rmax, sp.sn_r[sp.large_fronts[s0.fr_off + q]]);
      if constexpr (fp64) {
        for (int k = 0; k < nb; k++) {
          k_var_rows64<<<dim3(lv.steps[k].nfront, nc, T / 16), 256, 0, st>>>(list(k), VX, k, dp, store, b, vw);
          GP_CHECK_LAUNCH(ctx);
          if (k + 1 == nb) break;
          k_var_rows64<<<dim3(lv.steps[k + 1].nfront, nc, (nb - 1 - k) * (T / 16)), 256, 0, st>>>(list(k + 1), VSTEP, k,
                                                                                              dp, store, b, vw);
          GP_CHECK_LAUNCH(ctx);
        }
        if (rmax > 0) {
          k_var_rows64<<<dim3(s0.nfront, nc, (rmax + 15) / 16), 256, 0, st>>>(list(0), VREST, 0, dp, store, b, vw);
          GP_CHECK_LAUNCH(ctx);
        }
      } else {
        const unsigned n2 = (unsigned)((nc + 1) / 2), n4 = (unsigned)((nc + 3) / 4);
        for (int g0 = 0; g0 < nb; g0 += VG) {
          k_var_group<<<dim3(lv.steps[g0].nfront, n2), 256, var_smem(std::min(VG, nb - g0), 2), st>>>(list(g0), g0, nc, dp, store, b, vw);
          GP_CHECK_LAUNCH(ctx);
          const int b1 = g0 + VG;
          if (b1 >= nb) break;
          k_var_rest<<<dim3(lv.steps[b1].nfront, n4, nb - b1), 256, rest_smem, st>>>(list(b1), g0, nc, dp, store, b, vw);
          GP_CHECK_LAUNCH(ctx);
        }
        if (rmax > 0) {
          k_var_rest<<<dim3(s0.nfront, n4, (rmax + T - 1) / T), 256, rest_smem, st>>>(list(0), -1, nc, dp, store, b, vw);
          GP_CHECK_LAUNCH(ctx);
        }
      }
    }
    k_var_sumsq<V><<<dim3(SUM_CTAS, nc), 256, 0, st>>>(n, vw, part);
    GP_CHECK_LAUNCH(ctx);
    k_var_final<<<nc, R, 0, st>>>(part, SUM_CTAS, m, k0, d_var);
    GP_CHECK_LAUNCH(ctx);
  }
}

}  // namespace

void variance_run(gp_ctx* ctx, gp_factor_t* f, int b, const double* d_Xt, int64_t m, double* d_var) {
  const SymPlan& sp = f->ps->sp;
  if (f->prec == GP_FP64) {
    fa::StoreF64 store{f->panels, sp.panel_entries, f->dinv, sp.diag_entries};
    variance_impl(ctx, f, store, b, d_Xt, m, d_var);
  } else {
    fa::StoreMix store{f->panels32, f->diag, sp.panel32_entries, sp.diag_entries, f->dinv32};
    variance_impl(ctx, f, store, b, d_Xt, m, d_var);
  }
}
