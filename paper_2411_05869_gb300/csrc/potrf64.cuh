// potrf64.cuh -- Cholesky factor and inverse of one 64 x 64 FP64 diagonal tile (the FP64 factorization's POTRF).
//
// The tile is one link of the factorization's chain of dependent steps, so its latency counts. GB300's FP64 pipe takes
// 64 clocks for each warp instruction of a scheduler (0.5 lanes per clock); the integer pipe's 32 x 32 + 64 multiply-add
// takes 2. The elimination with its inverse in FP64 registers took 133 us per tile, this takes 44. Here both run in 60-bit fixed
// point on the integer pipe, on a cluster of two CTAs: the first eliminates the tile a column at a time, the second forms
// the inverse of the factor a column or two behind, from the columns that the first writes into its shared memory. (On
// one CTA the two together keep the integer pipe busy for about 700 clocks per column; apart, each is bounded by its chain
// of dependent steps.)
//
// The factor: row i is scaled by 2^-sigma_i, sqrt(a_ii) <= 2^(sigma_i - 1), so that every entry |a_ij| <= 1/4 and every
// |l_ij| <= 1/2; an entry is an integer in units of 2^-60. With l = lh 2^30 + ll (signed halves of 30 bits), a_ij -= l_ik
// l_jk is kept in two 64-bit sums, H -= lh lh' (units 2^-60) and C -= lh ll' + ll lh' (units 2^-90; below 2^63 over 64
// columns by Cauchy-Schwarz); ll ll' (2^-61, either sign) is dropped. Three multiply-adds per entry and column, absolute
// error 2^-60 of the rows' scales: smaller than the rounding of FP64 (2^-53 of a_ii on a_ii >= 2^-4). 1 / sqrt(pivot)
// comes from the FP32 approximation by one cubic step in 64-bit integers.
// The inverse: forward elimination of the identity, R_i -= l_ik X_k, X_k = R_k / l_kk, in the same halves, every row with
// an exponent of its own: its terms are kept at 2^-3 of the row's scale, so that the 63 of them in H cannot overflow 64
// bits, and a row whose next term is larger is shifted first (at 2^-5 the solves' residuals came out 1.5 times larger).
// The cross terms of C are below 2^59 + 2^56 each (the low half of l is not bounded by the shift), so C's whole units of
// 2^-60 are added to H after every eight columns: low halves that all have one sign would otherwise wrap it.
// A step is a chain of dependent instructions (pivot, reciprocal root, scaling, one hand-over), so nothing else waits
// for anything: every column of the factor and row of the inverse has a place and an mbarrier of its own, and the warp
// that holds the next one updates and publishes it before it does the rest of its updates.
// A pivot that is not positive, a diagonal that has fallen below zero before its turn or an entry larger than its diagonals
// allow (each means that the tile is not positive definite at or before that row) records its row, and the elimination
// goes on with any value. The smallest recorded column is the first failing one: what comes before it is positive
// definite and within the ranges (an infinite variance is taken as 2^1024, and its root written as infinite), and its own row either keeps to them, so that its pivot comes out right and not
// positive, or is recorded where it leaves them.
#pragma once
#include "f64_digits.cuh"
#include "gp_internal.cuh"
#include "tc_gemm.cuh"

namespace {
namespace p64 {

constexpr int PT = GP_TILE;
constexpr int THREADS = 256;   // per CTA
constexpr int PLANE = PT * 128;                       // bytes of one digit plane of the inverse (64 rows of 64 FP16)
constexpr int TILE_BYTES = 2 * f64d::NS * PLANE + 2 * PT * 4;   // the inverse's planes, the factor's, the inverse's rows'
                                                                // exponents and its columns' (the factor's rows') sigma

struct Smem {               // of either CTA; the factor's CTA writes its columns into both
  int2 lc[PT][PT];          // column k of the factor: (lh, ll) of every row
  int2 xr[PT][PT];          // row k of the inverse: (xh, xl) of every column
  int64_t R[PT];            // 1 / sqrt of the pivots (r 2^61) and their exponents
  int2 rs[PT];
  int xe[PT];               // exponents of the inverse's rows
  int sigma[PT];
  uint64_t lready[PT], rready[PT], xready[PT];   // mbarriers: lc[k]; R[k] and rs[k]; xr[k] and xe[k] are in
};

// A row's sigma for an infinite variance (an exponent field of 0x7ff).
constexpr int SIGMA_INF = ((0x7ff - 1021) >> 1) + 1;
__device__ __forceinline__ bool finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// x 2^(60 - e) to within a unit, |x| <= 2^(e - 2) in a positive definite tile; at least 2^60 in magnitude for |x| >= 2^e.
__device__ __forceinline__ int64_t double2fix60(double x, int e) {
  int f;
  const uint64_t man = f64d::significand(x, f);
  const int n = min(max(1025 + e - f, 0), 63);   // right shift
  return (int64_t)(man >> n) ^ (int64_t)(__double2hiint(x) >> 31);
}

// The reciprocal root of a pivot 0 < d < 2^60 (units of 2^-60): d 2^-60 = m 4^(1 - s), 1/4 <= m < 1, 1 / sqrt(d) = r
// 2^(s - 1), r = 1 / sqrt(m) = R0 2^-23 (1 + c 2^-70): R0 from the FP32 approximation, c one cubic step.
struct Root {
  int s;
  uint32_t R0;
  int64_t c;
};
__device__ __forceinline__ Root root_of(int64_t d) {
  Root o;
  const float f = __fmaf_rz(__uint2float_rz((uint32_t)(d >> 32)), 0x1p32f, __uint2float_rz((uint32_t)d));   // <= d
  const int ex = (__float_as_int(f) >> 23) - 127;
  const int s2 = (61 - ex) & ~1;
  o.s = s2 >> 1;
  const uint64_t M = (uint64_t)d << s2;                               // m 2^62
  float r0;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(__int_as_float(__float_as_int(f) + ((s2 - 62) << 23))));
  const int rb = __float_as_int(r0);
  o.R0 = (uint32_t)(((rb & 0x7fffff) | 0x800000) << 1) >> (128 - (rb >> 23));
  const uint64_t Q = (uint64_t)o.R0 * o.R0;
  const uint32_t Qh = (uint32_t)(Q >> 24), Ql = (uint32_t)Q & 0xffffffu;
  const uint32_t Mh = (uint32_t)(M >> 31), Ml = (uint32_t)M & 0x7fffffffu;
  // 1 - m r0^2 in units of 2^-70 (its leading bits are gone modulo 2^64)
  const int64_t e = -(int64_t)((((uint64_t)Mh * Qh) << 17) + (((uint64_t)Mh * Ql) >> 7) + (((uint64_t)Ml * Qh) >> 14) +
                               (((uint64_t)Ml * Ql) >> 38));
  const int es = (int)(e >> 24);                                      // units of 2^-46
  o.c = (e >> 1) + ((3 * ((int64_t)es * es)) >> 25);                  // e / 2 + 3 e^2 / 8
  return o;
}
// r 2^61, below 2^62.
__device__ __forceinline__ int64_t root_fix(const Root& o) {
  return ((int64_t)o.R0 << 38) + (((o.c >> 10) * (int64_t)o.R0) >> 22) - 2;
}
// a / sqrt(d) (both in units of 2^-60, below 2^60) as halves of 30 bits: a 2^(s + 2) times R0, then times 1 + c 2^-70.
__device__ __forceinline__ int2 scale_by(const Root& o, int64_t a) {
  const int64_t as = (int64_t)((uint64_t)a << (o.s + 2));             // below 2^62
  const int64_t y0 = (((as >> 31) * (int64_t)o.R0) << 7) +
                     (int64_t)(((uint64_t)((uint32_t)as & 0x7fffffffu) * o.R0) >> 24);   // four times the result
  const int yh = (int)(y0 >> 31), yl = (int)((uint32_t)y0 & 0x7fffffffu);
  const int ch = (int)(o.c >> 17), cl = (int)((uint32_t)o.c & 0x1ffffu);
  const int64_t t = (int64_t)yh * ch + (((int64_t)yh * cl) >> 17) + (((int64_t)yl * ch) >> 31);
  const int64_t y = y0 + (t >> 22);
  const int lh = (int)((y + 0x80000002LL) >> 32);
  return make_int2(lh, (int)((uint32_t)((y + 2) >> 2) - ((uint32_t)lh << 30)));
}

// (a r) / 2^64 for |a| < 2^62, 0 < r < 2^62, rounded, to about a unit, as halves of 30 bits.
__device__ __forceinline__ int2 mulfix(int64_t a, int64_t r) {
  const int ah = (int)(a >> 31), al = (int)((uint32_t)a & 0x7fffffffu);
  const int rh = (int)(r >> 31), rl = (int)((uint32_t)r & 0x7fffffffu);
  int64_t t = (int64_t)ah * rl;
  t += (int64_t)al * rh;
  const int64_t y = (int64_t)ah * rh + (t >> 31);
  const int lh = (int)((y + 0x80000002LL) >> 32);
  return make_int2(lh, (int)((uint32_t)((y + 2) >> 2) - ((uint32_t)lh << 30)));
}
__device__ __forceinline__ int64_t join30(int2 v) { return (int64_t)v.x * (1LL << 30) + v.y; }

// acc + a b, 32 x 32 + 64 bits.
__device__ __forceinline__ void mad(int64_t& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

__device__ __forceinline__ int2 split30(int64_t v) {
  const int h = (int)((v + (1LL << 29)) >> 30);
  return make_int2(h, (int)(v - ((int64_t)h << 30)));
}

__device__ __forceinline__ void st_cluster(uint32_t addr, int2 v) {
  asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(v.x), "r"(v.y) : "memory");
}

// A warp's wait for a phase-0 mbarrier (bounded; one that runs out is recorded and the tile comes out wrong).
__device__ __forceinline__ void wait(uint64_t* bar, int32_t* err) {
  if (!tcg::mbar_wait(bar, 0)) atomicExch(err, 1);
  __syncwarp();
}
// The same across the cluster (what the other CTA wrote before its arrival is seen).
__device__ __forceinline__ void wait_cluster(uint64_t* bar, int32_t* err) {
  if (!tcg::mbar_wait_cluster(bar, 0)) atomicExch(err, 1);
  __syncwarp();
}

// The elimination (the cluster's first CTA): P points at the tile's entry (0, 0), column stride ld; L replaces it, and its
// digit planes go to `planes`, row i at scale 2^(sigma_i - 2) (128-byte-swizzled tiles of 64 rows x 64 FP16). Warp w holds
// the columns w + 8 q, lane l the rows l (H0, C0; columns below 32 only) and l + 32 (H1, C1) of them; a finished column
// is shifted out, so that entry 0 is always the warp's next column.
__device__ __forceinline__ void factor(Smem& sm, double* __restrict__ P, int64_t ld, uint8_t* __restrict__ planes, int bw,
                                       int32_t first, int32_t* __restrict__ flag, int32_t* __restrict__ err) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t H0[4], C0[4], H1[8], C1[8];
  {
    double x0[4], x1[8];
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int j = w + 8 * q;
      if (q < 4) x0[q] = j <= lane && lane < bw ? P[j * ld + lane] : 0.0;
      x1[q] = j <= lane + 32 && lane + 32 < bw ? P[j * ld + lane + 32] : 0.0;
    }
    // the rows' scales, from the diagonal
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int j = w + 8 * q;
      if ((j & 31) == lane) {
        const double d = j < bw ? (q < 4 ? x0[q & 3] : x1[q]) : 1.0;
        if (!(d > 0.0)) atomicMin(flag, first + j);
        sm.sigma[j] = ((((__double2hiint(d) >> 20) & 0x7ff) - 1021) >> 1) + 1;   // 2^e <= d < 2^(e + 1): (e + 2) / 2 + 1
      }
    }
    __syncthreads();
    if (threadIdx.x < PT) {
      const uint32_t a = tcg::mapa_shared(tcg::smem_u32(&sm.sigma[threadIdx.x]), 1);
      asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(sm.sigma[threadIdx.x]) : "memory");
    }
    __syncthreads();   // before the first column's hand-over
    const int s0 = sm.sigma[lane], s1 = sm.sigma[lane + 32];
    bool bad0 = false, bad1 = false;
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int sj = sm.sigma[w + 8 * q];
      if (q < 4) {
        H0[q] = double2fix60(x0[q], s0 + sj);
        bad0 = bad0 || H0[q] >= 1LL << 60 || H0[q] < -(1LL << 60) || (!finite(x0[q]) && w + 8 * q != lane);
        C0[q] = 0;
      }
      H1[q] = double2fix60(x1[q], s1 + sj);
      bad1 = bad1 || H1[q] >= 1LL << 60 || H1[q] < -(1LL << 60) || (!finite(x1[q]) && w + 8 * q != lane + 32);
      C1[q] = 0;
    }
    if (bad0) atomicMin(flag, first + lane);
    if (bad1) atomicMin(flag, first + lane + 32);
  }
  // the same places in the inverse's CTA
  const uint32_t r_lc = tcg::mapa_shared(tcg::smem_u32(sm.lc), 1), r_R = tcg::mapa_shared(tcg::smem_u32(sm.R), 1),
                 r_rs = tcg::mapa_shared(tcg::smem_u32(sm.rs), 1), r_ready = tcg::mapa_shared(tcg::smem_u32(sm.rready), 1);
  // Column k (entry 0 of its warp, all earlier columns applied): pivot, scaling, out to the other warps.
  auto publish = [&](int k) {
    const int64_t a0 = H0[0] + (C0[0] >> 30), a1 = H1[0] + (C1[0] >> 30);
    const int64_t d0 = __shfl_sync(0xffffffffu, k < 32 ? a0 : a1, k & 31);
    const Root o = root_of(d0 <= 0 ? 1LL << 58 : d0);
    const int2 c0 = scale_by(o, a0), c1 = scale_by(o, a1);   // rows above the diagonal: read by nobody who uses them
    sm.lc[k][lane] = c0;
    sm.lc[k][lane + 32] = c1;
    __syncwarp();
    if (lane == 0) tcg::mbar_arrive(&sm.lready[k]);
    const uint32_t ro = (uint32_t)(k * PT + lane) * sizeof(int2);
    st_cluster(r_lc + ro, c0);
    st_cluster(r_lc + ro + 32 * sizeof(int2), c1);
    if (lane == 0) {
      const int64_t r = root_fix(o);
      st_cluster(r_R + k * 8, make_int2((int)(uint32_t)r, (int)(r >> 32)));
      st_cluster(r_rs + k * 8, make_int2(o.s, 0));
      if (d0 <= 0) atomicMin(flag, first + k);
    }
    __syncwarp();
    if (lane == 0) tcg::mbar_arrive_cluster(r_ready + k * 8);
    // what the diagonals allow: |a_ik| < sqrt(d) / 2 <= 2^-s, |l_ik| < 1/2
    const int64_t lim = 1LL << (60 - o.s);
    constexpr int half = (1 << 29) + 1;
    if ((a0 >= lim || a0 <= -lim || abs(c0.x) > half) && lane > k) atomicMin(flag, first + lane);
    if ((a1 >= lim || a1 <= -lim || abs(c1.x) > half) && lane + 32 > k) atomicMin(flag, first + lane + 32);
#pragma unroll
    for (int q = 0; q < 3; q++) {
      H0[q] = H0[q + 1];
      C0[q] = C0[q + 1];
    }
#pragma unroll
    for (int q = 0; q < 7; q++) {
      H1[q] = H1[q + 1];
      C1[q] = C1[q + 1];
    }
  };
  int jn = w;   // this warp's next column
  if (w == 0) {
    publish(0);
    jn = 8;
  }
#pragma unroll 1
  for (int k = 0; k < bw; k++) {
    wait(&sm.lready[k], err);
    const int2* lc = sm.lc[k];
    const int2 l0 = lc[lane], l1 = lc[lane + 32];
    if (jn == k + 1 && jn < bw) {
      const int2 v = lc[jn];
      mad(H0[0], l0.x, -v.x);
      mad(C0[0], l0.x, -v.y);
      mad(C0[0], l0.y, -v.x);
      mad(H1[0], l1.x, -v.x);
      mad(C1[0], l1.x, -v.y);
      mad(C1[0], l1.y, -v.x);
      publish(k + 1);
      jn += 8;
    }
    int2 v[8];
#pragma unroll
    for (int q = 0; q < 8; q++) v[q] = lc[min(jn + 8 * q, PT - 1)];   // past the tile: some row, into unused sums
    if (k < 32) {
#pragma unroll
      for (int q = 0; q < 4; q++) {
        mad(H0[q], l0.x, -v[q].x);
        mad(C0[q], l0.x, -v[q].y);
        mad(C0[q], l0.y, -v[q].x);
      }
#pragma unroll
      for (int q = 4; q < 8; q++) {
        mad(H1[q], l1.x, -v[q].x);
        mad(C1[q], l1.x, -v[q].y);
        mad(C1[q], l1.y, -v[q].x);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
      mad(H1[q], l1.x, -v[q].x);
      mad(C1[q], l1.x, -v[q].y);
      mad(C1[q], l1.y, -v[q].x);
    }
    if ((k & 15) == 15) {   // a diagonal below zero is seen before it can wrap: 16 columns take at most 4 of it
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int j = jn + 8 * q;
        const int64_t d = j < 32 ? H0[q & 3] + (C0[q & 3] >> 30) : H1[q] + (C1[q] >> 30);
        if (j < bw && lane == (j & 31) && d < 0) atomicMin(flag, first + j);
      }
    }
  }
  // L in FP64 (warp w the columns w + 8 q; every column has been waited for)
#pragma unroll 1
  for (int j = w; j < bw; j += 8)
#pragma unroll
    for (int p = 0; p < 2; p++) {
      const int i = lane + 32 * p;
      if (j <= i && i < bw) {
        const double l = f64d::fix2double(join30(sm.lc[j][i]), sm.sigma[i] - 60);
        P[j * ld + i] = i == j && sm.sigma[i] == SIGMA_INF ? __longlong_as_double(0x7ff0000000000000LL) : l;
      }
    }
#pragma unroll 1
  for (int e = threadIdx.x; e < PT * PT / 8; e += THREADS) {   // eight columns of a row
    const int i = e & (PT - 1), g = e / PT;
    int64_t v[8];
#pragma unroll
    for (int c = 0; c < 8; c++) {
      const int j = 8 * g + c;
      v[c] = (j <= i && i < bw ? 8 * join30(sm.lc[j][i]) : 0) + f64d::BIAS;
    }
    f64d::store8(planes + i * 128 + ((g ^ (i & 7)) << 4), PLANE, v);
  }
}

// The inverse (the cluster's second CTA): warp w holds the rows w + 8 r, lane l the columns l and l + 32; a finished row is
// shifted out. Row k leaves as FP64 (DI, row-major), as six digit planes at scale 2^xe (128-byte-swizzled tiles of 64
// rows x 64 FP16, the TRSM's operand; without the columns' 2^-sigma, which the TRSM applies to the other operand) and
// its exponent.
__device__ __forceinline__ void inverse(Smem& sm, double* __restrict__ DI, uint8_t* __restrict__ tile, int bw,
                                        int32_t* __restrict__ err) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t H[8][2], C[8][2];
  int E = 0;   // lane r < 8: the exponent of row w + 8 r
#pragma unroll
  for (int r = 0; r < 8; r++)
#pragma unroll
    for (int c = 0; c < 2; c++) {
      H[r][c] = w + 8 * r == lane + 32 * c ? 1LL << 60 : 0;
      C[r][c] = 0;
    }
  wait_cluster(&sm.rready[0], err);   // the scales are in, too
  const int sj[2] = {sm.sigma[lane], sm.sigma[lane + 32]};
  int32_t* ex = reinterpret_cast<int32_t*>(tile + 2 * f64d::NS * PLANE);
  int64_t x[2] = {0, 0};
  int xe = 0;
  // Row k (entry 0 of its warp, all earlier rows applied), scaled and out to the other warps; R, rs: its pivot's root.
  auto publish = [&](int k, int64_t R, int rs) {
    uint64_t m = 0;
    const int e0 = __shfl_sync(0xffffffffu, E, k >> 3);
#pragma unroll
    for (int c = 0; c < 2; c++) {
      x[c] = H[0][c] + (C[0][c] >> 30);
      m |= (uint64_t)(x[c] ^ (x[c] >> 63));
    }
    const uint32_t mh = __reduce_or_sync(0xffffffffu, (uint32_t)(m >> 32));
    int z = __clz((int)mh);
    if (mh == 0) z = 32 + __clz((int)__reduce_or_sync(0xffffffffu, (uint32_t)m));
    z = min(z - 2, 60);   // -1 for a sum of 2^62 or more
    xe = e0 + rs + 2 - z;
#pragma unroll
    for (int c = 0; c < 2; c++) {
      const int2 v = mulfix(z < 0 ? x[c] >> 1 : (int64_t)((uint64_t)x[c] << z), R);
      sm.xr[k][lane + 32 * c] = v;
      x[c] = join30(v);
    }
    if (lane == 0) sm.xe[k] = xe;
    __syncwarp();
    if (lane == 0) tcg::mbar_arrive(&sm.xready[k]);
#pragma unroll
    for (int r = 0; r < 7; r++)
#pragma unroll
      for (int c = 0; c < 2; c++) {
        H[r][c] = H[r + 1][c];
        C[r][c] = C[r + 1][c];
      }
  };
  // Row k's results (its warp, off the chain).
  auto store = [&](int k) {
    if (lane == 0) ex[k] = xe;
#pragma unroll 1
    for (int c = 0; c < 2; c++) {
      const int j = lane + 32 * c;
      const int64_t xc = c == 0 ? x[0] : x[1];
      DI[k * PT + j] = j <= k ? f64d::fix2double(xc, xe - 60 - (c == 0 ? sj[0] : sj[1])) : 0.0;
      const int64_t v = 2 * xc + f64d::BIAS, vn = __shfl_down_sync(0xffffffffu, v, 1);
      if ((lane & 1) == 0) {   // the digits of columns j and j + 1
        uint8_t* o = tile + k * 128 + (((j >> 3) ^ (k & 7)) << 4) + (j & 7) * 2;
        *reinterpret_cast<uint32_t*>(o) = f64d::digit_pair<0>(v, vn);
        *reinterpret_cast<uint32_t*>(o + PLANE) = f64d::digit_pair<1>(v, vn);
        *reinterpret_cast<uint32_t*>(o + 2 * PLANE) = f64d::digit_pair<2>(v, vn);
        *reinterpret_cast<uint32_t*>(o + 3 * PLANE) = f64d::digit_pair<3>(v, vn);
        *reinterpret_cast<uint32_t*>(o + 4 * PLANE) = f64d::digit_pair<4>(v, vn);
        *reinterpret_cast<uint32_t*>(o + 5 * PLANE) = f64d::digit_pair<5>(v, vn);
      }
    }
  };
  // Row r of the warp minus l (its halves negated) times row k of the inverse.
  auto elim = [&](int64_t (&Hr)[2], int64_t (&Cr)[2], int2 l, const int2& x0, const int2& x1, int k) {
    mad(Hr[0], l.x, x0.x);
    mad(Cr[0], l.x, x0.y);
    mad(Cr[0], l.y, x0.x);
    if (k >= 32) {   // columns from 32 on enter with row 32
      mad(Hr[1], l.x, x1.x);
      mad(Cr[1], l.x, x1.y);
      mad(Cr[1], l.y, x1.x);
    }
  };
  int rn = w;   // this warp's next row
  bool mine = false;
  if (w == 0) {
    publish(0, sm.R[0], sm.rs[0].x);
    rn = 8;
    mine = true;
  }
#pragma unroll 1
  for (int k = 0; k < bw; k++) {
    const bool next = rn == k + 1 && rn < bw;
    int64_t Rn = 0;
    int rsn = 0;
    if (next) {
      wait_cluster(&sm.rready[k + 1], err);
      Rn = sm.R[k + 1];
      rsn = sm.rs[k + 1].x;
    }
    wait(&sm.xready[k], err);   // row k of the inverse; its warp has seen column k of the factor
    // lane r: l of row w + 8 r at the row's scale
    const bool act = lane < 8 && w + 8 * lane > k && w + 8 * lane < bw;
    const int2 lk = sm.lc[k][(w + 8 * lane) & (PT - 1)];
    const int ek = sm.xe[k];
    const int2 x0 = sm.xr[k][lane], x1 = sm.xr[k][lane + 32];
    int64_t l = act ? join30(lk) : 0;
    const int nb = act ? 30 + max((__float_as_int(__int2float_rz(abs(lk.x))) >> 23) - 126, 0) : -4096;   // |l| <= 2^nb
    int sh = E - ek;
    const int delta = max(nb - sh - 57, 0);   // the row's scale has to grow
    E += delta;
    sh += delta;
    l = sh >= 0 ? l >> min(sh, 63) : (int64_t)((uint64_t)l << min(-sh, 63));
    int2 lp = split30(l);
    lp.x = -lp.x;
    lp.y = -lp.y;
    const uint32_t big = __ballot_sync(0xffffffffu, delta > 0);
    if (big) {
      const int base = rn >> 3;
#pragma unroll
      for (int r = 0; r < 8; r++) {
        const int dl = min(__shfl_sync(0xffffffffu, delta, (base + r) & 31), 63);
#pragma unroll
        for (int c = 0; c < 2; c++) {
          H[r][c] >>= dl;
          C[r][c] >>= dl;
        }
      }
    }
    if (next) {
      elim(H[0], C[0], make_int2(__shfl_sync(0xffffffffu, lp.x, rn >> 3), __shfl_sync(0xffffffffu, lp.y, rn >> 3)), x0,
           x1, k);
      publish(k + 1, Rn, rsn);
      rn += 8;
    } else if (mine) {
      store(k);
    }
    mine = next;
    const int base = rn >> 3;   // past the tile: finished rows' values, into unused sums
    int2 lr[8];
#pragma unroll
    for (int r = 0; r < 8; r++)
      lr[r] = make_int2(__shfl_sync(0xffffffffu, lp.x, (base + r) & 31), __shfl_sync(0xffffffffu, lp.y, (base + r) & 31));
#pragma unroll
    for (int r = 0; r < 8; r++) {
      mad(H[r][0], lr[r].x, x0.x);
      mad(C[r][0], lr[r].x, x0.y);
      mad(C[r][0], lr[r].y, x0.x);
    }
    if (k >= 32) {   // columns from 32 on enter with row 32; four rows of the warp are left
#pragma unroll
      for (int r = 0; r < 4; r++) {
        mad(H[r][1], lr[r].x, x1.x);
        mad(C[r][1], lr[r].x, x1.y);
        mad(C[r][1], lr[r].y, x1.x);
      }
    }
    if ((k & 7) == 7) {   // the cross sums' whole units go over
#pragma unroll
      for (int r = 0; r < 8; r++)
#pragma unroll
        for (int c = 0; c < 2; c++) {
          H[r][c] += C[r][c] >> 30;
          C[r][c] &= (1LL << 30) - 1;
        }
    }
  }
  // rows past the tile's width: zero
  for (int i = bw + w; i < PT; i += 8) {
    if (lane == 0) ex[i] = 0;
    DI[i * PT + lane] = 0.0;
    DI[i * PT + lane + 32] = 0.0;
    for (int s = 0; s < f64d::NS; s++) *reinterpret_cast<uint32_t*>(tile + s * PLANE + i * 128 + lane * 4) = 0u;
  }
  if (w == 0) {
    ex[PT + lane] = sj[0];
    ex[PT + lane + 32] = sj[1];
  }
}

}  // namespace p64

// POTRF of the diagonal tile of block column kb, its inverse in FP64 (row-major, for the solves) and the inverse's digit
// planes for the step's TRSM, a cluster of two CTAs per large front.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(p64::THREADS, 1)
    k_potrf64(const int32_t* __restrict__ fronts, int kb, DevPlan dp, double* __restrict__ panels, int64_t PE,
              int32_t* __restrict__ notpd, double* __restrict__ dinv, int64_t DE, uint8_t* __restrict__ itile,
              int64_t IE, int32_t* __restrict__ err) {
  extern __shared__ __align__(16) uint8_t potrf_raw[];
  p64::Smem& sm = *reinterpret_cast<p64::Smem*>(potrf_raw);
  const int fi = blockIdx.x >> 1;
  const int32_t s = fronts[fi];
  const int b = blockIdx.y;
  const int w = dp.w[s];
  const int64_t m = (int64_t)w + dp.r[s];
  const int c0 = kb * p64::PT, bw = min(p64::PT, w - c0);
  const int32_t first = dp.sn_first[s] + c0;
  double* P = panels + (int64_t)b * PE + dp.loff[s] + (int64_t)c0 * m + c0;
  if (threadIdx.x < 3 * p64::PT) tcg::mbar_init(&sm.lready[threadIdx.x], 1);   // the three arrays
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  tcg::cluster_sync();
  uint8_t* tile = itile + (int64_t)b * IE + (int64_t)fi * p64::TILE_BYTES;
  if (tcg::cluster_ctarank() == 0)
    p64::factor(sm, P, m, tile + f64d::NS * p64::PLANE, bw, first, notpd + b, err);
  else
    p64::inverse(sm, dinv + (int64_t)b * DE + dp.doff[s] + (int64_t)kb * p64::PT * p64::PT, tile, bw, err);
  tcg::cluster_sync();   // no CTA leaves while the other may write into it
}

}  // namespace
