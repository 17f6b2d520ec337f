// trsm64.cuh -- the rows below a 64 x 64 diagonal tile times its inverse in FP64 precision (the FP64 factorization's TRSM), on
// the FP16 tensor cores (f64_digits.cuh).
#pragma once
#include "f64_digits.cuh"
#include "factor_access.cuh"
#include "gp_internal.cuh"
#include "potrf64.cuh"
#include "tc_gemm.cuh"

namespace {

// Four consecutive columns (this thread's lane) of the accumulators of the levels 0..3, ld columns apart, and of the levels
// 4..6 where `deep` (zero otherwise).
__device__ __forceinline__ void tmem_ld_levels4(uint32_t ta, int ld, bool deep, float (&a)[f64d::NL][4]) {
  uint32_t r[16], q[12];
#pragma unroll
  for (int l = 0; l < 4; l++)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[4 * l]), "=r"(r[4 * l + 1]), "=r"(r[4 * l + 2]), "=r"(r[4 * l + 3])
                 : "r"(ta + l * ld));
  if (deep) {
#pragma unroll
    for (int l = 0; l < 3; l++)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                   : "=r"(q[4 * l]), "=r"(q[4 * l + 1]), "=r"(q[4 * l + 2]), "=r"(q[4 * l + 3])
                   : "r"(ta + (4 + l) * ld));
  } else {
#pragma unroll
    for (int k = 0; k < 12; k++) q[k] = 0u;
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]), "+r"(q[6]),
                 "+r"(q[7]), "+r"(q[8]), "+r"(q[9]), "+r"(q[10]), "+r"(q[11])
               :
               : "memory");
#pragma unroll
  for (int c = 0; c < 4; c++) {
#pragma unroll
    for (int l = 0; l < 4; l++) a[l][c] = __uint_as_float(r[4 * l + c]);
#pragma unroll
    for (int l = 0; l < 3; l++) a[4 + l][c] = __uint_as_float(q[4 * l + c]);
  }
}

// TRSM of the rows below diagonal tile kb, X L_11^T = B, on the tensor cores: one CTA of 512 threads per 128-row tile,
// thread (row, part) holding 16 of the row's 64 entries, in three products:
//   X_0 = B inv(L_11)^T: the rows of B (times the 2^-sigma of the inverse's columns) are cut into digits at the exponent of
//     their largest entry, straight into 128-byte-swizzled operand tiles, while the planes of the inverse and of L arrive by
//     one bulk copy; the digit products follow, one TMEM accumulator per level. X_0 alone is not backward stable:
//     |B - X_0 L_11^T| grows with the condition of L_11. In units of 2^-53 sqrt(C_ii a_jj), for a noise of 1, 1e-2, 1e-4 and
//     1e-8 of the variance, it measured 2, 28, 150 and 11,000 with six digits, where an FP64 substitution column by
//     column has 1.2 to 3.5;
//   R = B - X_0 L_11^T in 64-bit integers, from X_0 as its digits say and the digits of the tile's L: nothing is rounded
//     above 2^-60 of the row's largest entry;
//   X = X_0 + R inv(L_11)^T: 0.3 to 1.4 units at any noise down to 1e-12 of the variance.
// Each product with the inverse leaves about 2^-35 cond(L_11) of what it is to remove with four digits on either side (10
// products, levels 0..3), 2^-53 with six (26, levels 0..6): four where the inverse's entries, scaled, are below
// 2^TRSM_DEEP, so that the two of them reach 2^-60.
// Each thread then rounds its row's entries of X to FP64 for the panel and cuts them into the digits the updates read (at
// the row's scale rho), which leave through shared memory by TMA (a thread's own 16-byte stores would touch one line
// each). A row whose entries are more than its variance allows (|L_ij| <= sqrt(C_ii) <= 2^(rho + 1)) is not positive
// definite at or before its own column and records it: its digits may have wrapped.
// Bounded by latency: load, then cut, multiply and read three times, store (a launch of few tiles: 32 us, 117 us as an FP64
// substitution). The 16 warps' integer chains take two thirds of it, the products a sixth.
constexpr int TRSM_ROWS = 128, TRSM_THREADS = 512;
constexpr int TRSM_COLS = 64 * TRSM_ROWS / TRSM_THREADS;   // of a thread
constexpr int TRSM_PLANE_A = TRSM_ROWS * 128;   // bytes of one digit plane of B
constexpr int TRSM_DEEP = 6;
constexpr int TRSM_SMEM = f64d::NS * TRSM_PLANE_A + p64::TILE_BYTES + 1024;

// The digit products of A's planes (128 rows) with those at sb into the levels' accumulators. Plane d of A times
// consecutive planes of B is one instruction with N = 64 per plane: the planes lie behind one another as rows of B, and the
// levels they go to behind one another in tensor memory. (Plane by plane each instruction reads 6 KB of shared memory for 64
// columns: 5400 clocks for the 26 products, 3400 so.) The descriptors' offsets are constants, since one thread issues
// them all.
struct DigitProducts {
  uint32_t tmem;
  uint64_t da, db;   // descriptors, addresses in units of 16 bytes
  __device__ __forceinline__ DigitProducts(uint32_t tm, uint32_t sa, uint32_t sb)
      : tmem(tm), da(tcg::smem_desc_sw128(sa)), db(tcg::smem_desc_sw128(sb)) {}
  // plane D with the W planes from T0 on; the first products of a level do not accumulate
  template <int D, int T0, int W, bool FIRST = false>
  __device__ __forceinline__ void add() const {
#pragma unroll
    for (int kk = 0; kk < 4; kk++)
      tcg::mma_f16(tmem + (D + T0) * p64::PT, da + (D * TRSM_PLANE_A + kk * 32) / 16, db + (T0 * p64::PLANE + kk * 32) / 16,
                   tcg::idesc_f16(TRSM_ROWS, W * p64::PT), !FIRST || kk > 0);
  }
  __device__ __forceinline__ void four_levels() const {   // 10 products, levels 0..3
    add<0, 0, 4, true>();
    add<1, 0, 3>();
    add<2, 0, 2>();
    add<3, 0, 1>();
  }
  __device__ __forceinline__ void seven_levels(bool six_planes) const {   // 26 products, 21 of four planes of A
    static_assert(f64d::NS == 6 && f64d::NL == 7, "six planes and seven levels");
    add<0, 0, 4, true>();
    add<0, 4, 2, true>();
    add<1, 0, 4>();
    add<1, 4, 1>();
    add<1, 5, 1, true>();
    add<2, 0, 4>();
    add<2, 4, 1>();
    add<3, 0, 4>();
    if (six_planes) {
      add<4, 0, 3>();
      add<5, 0, 2>();
    }
  }
};

// Digit planes of eight consecutive entries: four, or all six.
__device__ __forceinline__ void store_planes(uint8_t* dst, const int64_t (&v)[8], bool six) {
  using f64d::pack8;
  *reinterpret_cast<uint4*>(dst) = pack8<0>(v);
  *reinterpret_cast<uint4*>(dst + TRSM_PLANE_A) = pack8<1>(v);
  *reinterpret_cast<uint4*>(dst + 2 * TRSM_PLANE_A) = pack8<2>(v);
  *reinterpret_cast<uint4*>(dst + 3 * TRSM_PLANE_A) = pack8<3>(v);
  if (six) {
    *reinterpret_cast<uint4*>(dst + 4 * TRSM_PLANE_A) = pack8<4>(v);
    *reinterpret_cast<uint4*>(dst + 5 * TRSM_PLANE_A) = pack8<5>(v);
  }
}

__global__ void __launch_bounds__(TRSM_THREADS, 1)
    k_trsm64(const int32_t* __restrict__ fronts, const int64_t* __restrict__ pre, int nfront, int kb, DevPlan dp,
             double* __restrict__ panels, int64_t PE, const uint8_t* __restrict__ itile, int64_t IE,
             const int32_t* __restrict__ rho, int64_t n, const uint8_t* __restrict__ tmaps,
             const int32_t* __restrict__ slot_of, int32_t* __restrict__ notpd, int32_t* __restrict__ err,
             tcg::WaitLimit lim) {
  using namespace f64d;
  constexpr int PT = p64::PT;
  extern __shared__ __align__(1024) uint8_t trsm_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)trsm_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* inv = sm + NS * TRSM_PLANE_A;   // the inverse's planes, then the planes of L, then exponents
  const int32_t* einv = reinterpret_cast<const int32_t*>(inv + 2 * NS * p64::PLANE);   // rows' exponents, columns' sigma
  __shared__ uint64_t bar, ibar;
  __shared__ uint32_t tslot;
  __shared__ int emax_s[TRSM_THREADS / TRSM_ROWS][TRSM_ROWS], skip_s;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int row = tid & 127, part = tid >> 7, c16 = TRSM_COLS * part;   // columns c16 ..
  const int64_t t = blockIdx.x;
  const int fi = fa::find_front(pre, nfront, t);
  const int b = blockIdx.y;
  if (tid == 0) {
    tcg::mbar_init(&bar, 1);
    tcg::mbar_init(&ibar, 1);
    skip_s = *(volatile int32_t*)err;   // an earlier launch of this factorization ran out of a wait
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    tcg::mbar_arrive_expect_tx(&ibar, p64::TILE_BYTES);
    tcg::bulk_load(tcg::smem_u32(inv), itile + (int64_t)b * IE + (int64_t)fi * p64::TILE_BYTES, p64::TILE_BYTES, &ibar);
  }
  if (warp == 0) tcg::tmem_alloc(&tslot, 512);
  const int32_t s = fronts[fi];
  const int w = dp.w[s], r = dp.r[s];
  const int64_t m = (int64_t)w + r;
  const int c0 = kb * PT, bw = min(PT, w - c0), c1 = c0 + bw;
  const int64_t r0 = c1 + (t - pre[fi]) * TRSM_ROWS;
  const int nr = (int)imin64(TRSM_ROWS, m - r0);
  const bool rok = row < nr;
  double* P = panels + (int64_t)b * PE + dp.loff[s] + (int64_t)(c0 + c16) * m + r0 + row;   // this thread's entries
  const int nc = min(max(bw - c16, 0), rok ? TRSM_COLS : 0);
  const int32_t col = rok ? dp.frows[dp.frow_off[s] + r0 + row] : 0;   // the row's own (permuted) column
  const int32_t rr = rok ? rho[(int64_t)b * n + col] : 0;
  // this thread's 16-byte chunks of its row in digit plane 0
  auto chunk = [&](int g) { return sm + row * 128 + (((TRSM_COLS / 8 * part + g) ^ (row & 7)) << 4); };
  int rx, xmax;   // exponents of the row of B, of the inverse
  bool deep;
  bool over = false;   // more than the row's variance allows
  {
    double x[TRSM_COLS];
    const double* p = P;
#pragma unroll
    for (int c = 0; c < TRSM_COLS; c++, p += m) x[c] = c < nc ? *p : 0.0;
    __syncthreads();   // ibar is initialised
    if (!tcg::mbar_wait(&ibar, 0, lim)) {
      atomicExch(err, 1);
      tcg::mbar_wait(&ibar, 0);   // the copy must land before the CTA ends
    }
    int ex = -4096;
#pragma unroll
    for (int c = 0; c < TRSM_COLS; c++) {
      const int e = (__double2hiint(x[c]) >> 20) & 0x7ff;
      ex = max(ex, max(e, 1) - einv[PT + c16 + c]);
      over = over || e == 0x7ff;
    }
    emax_s[part][row] = ex;
    xmax = __reduce_max_sync(0xffffffffu, max(einv[tid & 31], einv[(tid & 31) + 32]));
    deep = xmax > TRSM_DEEP;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < TRSM_THREADS / TRSM_ROWS; q++) ex = max(ex, emax_s[q][row]);
    rx = ex - 1022;   // |x| 2^-sigma < 2^rx
#pragma unroll 1
    for (int g = 0; g < 2; g++) {
      int64_t v[8];
#pragma unroll
      for (int c = 0; c < 8; c++) v[c] = to_biased(g == 0 ? x[c] : x[8 + c], rx + einv[PT + c16 + 8 * g + c]);
      store_planes(chunk(g), v, deep);
    }
  }
  const uint32_t sa = tcg::smem_u32(sm), sinv = tcg::smem_u32(inv), sl = sinv + NS * p64::PLANE;
  const uint32_t ta = (uint32_t)((warp & 3) * 32) << 16;   // this warp's lanes of tensor memory
  uint32_t phase = 0;
  bool ok = true;
  // The operand tiles' products with the planes at sb, awaited by everyone. One barrier per CTA and one at a time in flight.
  auto multiply = [&](uint32_t sb, bool seven) {
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // the operand tiles are visible to the tensor core
    tcg::tc_fence_before();
    __syncthreads();
    tcg::tc_fence_after();
    if (tid == 0 && !skip_s) {
      const DigitProducts pr(tslot, sa, sb);
      if (seven) pr.seven_levels(deep);
      else pr.four_levels();
      tcg::mma_commit(&bar);
    }
    __syncwarp();
    if (skip_s) ok = false;
    else if (!tcg::mbar_wait_warp(&bar, phase, lim)) {   // record it, then wait for the MMAs issued all the same
      ok = false;
      atomicExch(err, 1);
      tcg::mbar_wait(&bar, phase);
    }
    __syncwarp();
    tcg::tc_fence_after();
    phase ^= 1;
  };
  multiply(sinv, deep);
  const uint32_t tmem = tslot + ta + c16;
  over = over || rx > rr + 1;   // |B_c| 2^-sigma_c < 2^rr in a positive definite matrix
  // X_0 in fixed point at scale rho, or less where B is small (64 terms below 2^rx times the inverse's largest), and then
  // cut into digits at the scale of the row's largest, which R shares: X_0 in units of 2^(re - 61), |X_0| < 2^60 of them
  const int e0 = min(rr, rx + xmax + 5);
  int64_t xa[8], xb[8], big = 0;   // the thread's first and last eight (loops over them are not unrolled: instructions
                                   // have to be fetched, and each is executed by a CTA's 16 warps once)
#pragma unroll 1
  for (int g = 0; g < 2; g++) {
    float a[NL][4];
#pragma unroll
    for (int c = 0; c < 8; c++) {
      const int h = c & 3;
      if (h == 0) tmem_ld_levels4(tmem + 8 * g + c, PT, deep, a);
      const float al[NL] = {a[0][h], a[1][h], a[2][h], a[3][h], a[4][h], a[5][h], a[6][h]};
      const int64_t v = product_fixed(al, rx + einv[c16 + 8 * g + c], e0, deep, over);
      big |= v ^ (v >> 63);
      if (g == 0) xa[c] = v;
      else xb[c] = v;
    }
  }
  const int z = __clzll(big);
  emax_s[part][row] = -z;   // last read before the products
  __syncthreads();
  int zrow = -z;
#pragma unroll
  for (int q = 0; q < TRSM_THREADS / TRSM_ROWS; q++) zrow = max(zrow, emax_s[q][row]);
  const int up = -zrow - 4, re = e0 - up;   // -3 .. 60
#pragma unroll 1
  for (int g = 0; g < 2; g++) {
    int64_t v[8];
#pragma unroll
    for (int c = 0; c < 8; c++) {
      const int64_t x = g == 0 ? xa[c] : xb[c];
      v[c] = (up >= 0 ? x << up : x >> -up) + BIAS;
      if (g == 0) xa[c] = digits_of(v[c], deep);
      else xb[c] = digits_of(v[c], deep);
    }
    store_planes(chunk(g), v, deep);
  }
  double x[TRSM_COLS];   // B once more
  {
    const double* p = P;
#pragma unroll
    for (int c = 0; c < TRSM_COLS; c++, p += m) x[c] = c < nc ? *p : 0.0;
  }
  multiply(sl, true);
  {
#pragma unroll 1
    for (int g = 0; g < 2; g++) {
      float a[NL][4];
      int64_t v[8];
#pragma unroll
      for (int c = 0; c < 8; c++) {
        const int h = c & 3;
        if (h == 0) tmem_ld_levels4(tmem + 8 * g + c, PT, true, a);
        const float al[NL] = {a[0][h], a[1][h], a[2][h], a[3][h], a[4][h], a[5][h], a[6][h]};
        // R in units of 2^-72 of the product of the row's scale and 2^(sigma - 2), modulo 2^64 (below 2^50 of them)
        int64_t d = (int64_t)(fixed_mod(g == 0 ? x[c] : x[8 + c], re + einv[PT + c16 + 8 * g + c] - 2 - 72) - product_mod72(al));
        d = (int64_t)((uint64_t)(uint32_t)min(max((int)(d >> 32), -(1 << 18)), (1 << 18) - 1) << 32 | (uint32_t)d);
        v[c] = (d << 11) + BIAS;   // at scale 2^(re - 24), times 2^-sigma
      }
      store_planes(chunk(g), v, deep);
    }
  }
  multiply(sinv, deep);
  {
    double* p = P;
#pragma unroll 1
    for (int g = 0; g < 2; g++) {
      float a[NL][4];
      int64_t v[8];
#pragma unroll
      for (int c = 0; c < 8; c++, p += m) {
        const int h = c & 3;
        if (h == 0) tmem_ld_levels4(tmem + 8 * g + c, PT, deep, a);
        const float al[NL] = {a[0][h], a[1][h], a[2][h], a[3][h], a[4][h], a[5][h], a[6][h]};
        const int64_t x = (g == 0 ? xa[c] : xb[c]) + product_fixed(al, re - 24 + einv[c16 + 8 * g + c], re, deep, over);
        if (ok && 8 * g + c < nc) *p = fix2double(x, re - 61);
        v[c] = (re < rr ? x >> min(rr - re, 63) : x << (re - rr)) + BIAS;
      }
      store_planes(chunk(g), v, true);
    }
  }
  if (ok && rok && over) atomicMin(notpd + b, col);
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  tcg::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tcg::tc_fence_after();
    tcg::tmem_dealloc(tslot, 512);
  }
  if (tid == 0 && ok) {   // the digits of X: 64-row boxes, rows past the front are not written
    const uint8_t* map = tmaps + (int64_t)slot_of[s] * 128;
    tcg::tmap_acquire(map);
    for (int h = 0; h < 2 && h * PT < nr; h++)
      for (int d = 0; d < NS; d++)
        tcg::tma_store_4d(map, kb % (KG / PT) * PT, (int)r0 + h * PT, d, b, tcg::smem_u32(sm) + d * TRSM_PLANE_A + h * PT * 128);
    tcg::bulk_store_wait();
  }
}

}  // namespace
