// trsm64.cuh -- the rows below a 64 x 64 diagonal tile times its inverse in FP64 precision (the FP64 factorization's TRSM), on
// the FP16 tensor cores (f64_digits.cuh).
#pragma once
#include "f64_digits.cuh"
#include "factor_access.cuh"
#include "gp_internal.cuh"
#include "potrf64.cuh"
#include "tc_gemm.cuh"

namespace {

// Eight consecutive columns of the seven level accumulators (ld columns apart) of this thread's lane.
__device__ __forceinline__ void tmem_ld_levels(uint32_t ta, int ld, float (&a)[f64d::NL][8]) {
  uint32_t r[f64d::NL * 8];
  static_assert(f64d::NL == 7, "the wait below takes seven levels");
#pragma unroll
  for (int l = 0; l < f64d::NL; l++)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[8 * l]), "=r"(r[8 * l + 1]), "=r"(r[8 * l + 2]), "=r"(r[8 * l + 3]), "=r"(r[8 * l + 4]),
                   "=r"(r[8 * l + 5]), "=r"(r[8 * l + 6]), "=r"(r[8 * l + 7])
                 : "r"(ta + l * ld));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31]), "+r"(r[32]), "+r"(r[33]), "+r"(r[34]), "+r"(r[35]),
                 "+r"(r[36]), "+r"(r[37]), "+r"(r[38]), "+r"(r[39]), "+r"(r[40]), "+r"(r[41]), "+r"(r[42]),
                 "+r"(r[43]), "+r"(r[44]), "+r"(r[45]), "+r"(r[46]), "+r"(r[47]), "+r"(r[48]), "+r"(r[49]),
                 "+r"(r[50]), "+r"(r[51]), "+r"(r[52]), "+r"(r[53]), "+r"(r[54]), "+r"(r[55])
               :
               : "memory");
#pragma unroll
  for (int l = 0; l < f64d::NL; l++)
#pragma unroll
    for (int c = 0; c < 8; c++) a[l][c] = __uint_as_float(r[8 * l + c]);
}

// TRSM of the rows below diagonal tile kb as X = B inv(L_11)^T on the tensor cores: one CTA of 256 threads per 128-row
// tile, thread (row, half) holding 32 of the row's 64 entries. The rows of B (times the 2^-sigma of the inverse's columns)
// are cut into digits at the exponent of their largest entry, straight into 128-byte-swizzled operand tiles, while the
// inverse's planes arrive by one bulk copy; 26 digit products of 128 x 64 x 64 follow, one TMEM accumulator per level;
// each thread then rounds its row's entries of X to FP64 for the panel and cuts them into the digits the updates read (at
// the row's scale rho), which leave through shared memory by TMA (a thread's own 16-byte stores would touch one line
// each). A row whose entries are more than its variance allows (|L_ij| <= sqrt(C_ii) <= 2^(rho + 1)) is not positive
// definite at or before its own column and records it: its digits may have wrapped. Bounded by latency at the top levels (one wave of CTAs: load, cut, multiply, store in turn): 21 us a launch with
// one tile, 117 us as an FP64 substitution column by column.
constexpr int TRSM_ROWS = 128;
constexpr int TRSM_PLANE_A = TRSM_ROWS * 128;   // bytes of one digit plane of B
constexpr int TRSM_SMEM = f64d::NS * TRSM_PLANE_A + p64::TILE_BYTES + 1024;

__global__ void __launch_bounds__(256, 1)
    k_trsm64(const int32_t* __restrict__ fronts, const int64_t* __restrict__ pre, int nfront, int kb, DevPlan dp,
             double* __restrict__ panels, int64_t PE, const uint8_t* __restrict__ itile, int64_t IE,
             const int32_t* __restrict__ rho, int64_t n, const uint8_t* __restrict__ tmaps,
             const int32_t* __restrict__ slot_of, int32_t* __restrict__ notpd, int32_t* __restrict__ err,
             tcg::WaitLimit lim) {
  using namespace f64d;
  extern __shared__ __align__(1024) uint8_t trsm_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)trsm_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* inv = sm + NS * TRSM_PLANE_A;
  const int32_t* einv = reinterpret_cast<const int32_t*>(inv + NS * p64::PLANE);   // rows' exponents, columns' sigma
  __shared__ uint64_t bar, ibar;
  __shared__ uint32_t tslot;
  __shared__ int emax_s[2][TRSM_ROWS], skip_s;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int row = tid & 127, half = tid >> 7;
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
  const int c0 = kb * p64::PT, bw = min(p64::PT, w - c0), c1 = c0 + bw;
  const int64_t r0 = c1 + (t - pre[fi]) * TRSM_ROWS;
  const int nr = (int)imin64(TRSM_ROWS, m - r0);
  const bool rok = row < nr;
  double* P = panels + (int64_t)b * PE + dp.loff[s] + (int64_t)(c0 + 32 * half) * m + r0 + row;   // this thread's entries
  const int nc = min(max(bw - 32 * half, 0), rok ? 32 : 0);
  const int32_t col = rok ? dp.frows[dp.frow_off[s] + r0 + row] : 0;   // the row's own (permuted) column
  const int32_t rr = rok ? rho[(int64_t)b * n + col] : 0;
  int rx;
  bool over = false;   // more than the row's variance allows
  {
    double x[32];
    const double* p = P;
#pragma unroll
    for (int c = 0; c < 32; c++, p += m) x[c] = c < nc ? *p : 0.0;
    __syncthreads();   // ibar is initialised
    if (!tcg::mbar_wait(&ibar, 0, lim)) {
      atomicExch(err, 1);
      tcg::mbar_wait(&ibar, 0);   // the copy must land before the CTA ends
    }
    int ex = -4096;
#pragma unroll
    for (int c = 0; c < 32; c++) {
      const int e = (__double2hiint(x[c]) >> 20) & 0x7ff;
      ex = max(ex, max(e, 1) - einv[p64::PT + 32 * half + c]);
      over = over || e == 0x7ff;
    }
    emax_s[half][row] = ex;
    __syncthreads();
    rx = max(ex, emax_s[half ^ 1][row]) - 1022;   // |x| 2^-sigma < 2^rx
#pragma unroll
    for (int g = 0; g < 4; g++) {
      int64_t v[8];
#pragma unroll
      for (int c = 0; c < 8; c++) v[c] = to_biased(x[8 * g + c], rx + einv[p64::PT + 32 * half + 8 * g + c]);
      store8(sm + row * 128 + (((4 * half + g) ^ (row & 7)) << 4), TRSM_PLANE_A, v);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // the operand tiles are visible to the tensor core
  tcg::tc_fence_before();
  __syncthreads();
  tcg::tc_fence_after();
  const uint32_t tmem = tslot;
  const bool skip = skip_s != 0;
  if (tid == 0 && !skip) {
    const uint32_t sa = tcg::smem_u32(sm), sb = tcg::smem_u32(inv);
    const uint32_t idesc = tcg::idesc_f16(TRSM_ROWS, p64::PT);
#pragma unroll 1
    for (int l = 0; l < NL; l++)
      for (int d = max(0, l - NS + 1); d <= min(l, NS - 1); d++)
#pragma unroll
        for (int kk = 0; kk < 4; kk++)
          tcg::mma_f16(tmem + l * p64::PT, tcg::smem_desc_sw128(sa + d * TRSM_PLANE_A + kk * 32),
                       tcg::smem_desc_sw128(sb + (l - d) * p64::PLANE + kk * 32), idesc,
                       d > max(0, l - NS + 1) || kk > 0);
    tcg::mma_commit(&bar);
  }
  __syncwarp();
  bool ok = skip || tcg::mbar_wait_warp(&bar, 0, lim);
  if (!ok) {   // record it, then wait for the MMAs issued before tensor memory is given back
    atomicExch(err, 1);
    tcg::mbar_wait(&bar, 0);
  }
  ok = ok && !skip;
  __syncwarp();
  tcg::tc_fence_after();
  over = over || rx > rr + 1;   // |B_c| 2^-sigma_c < 2^rr in a positive definite matrix
  {
    double* p = P;
#pragma unroll 1
    for (int g = 0; g < 4; g++) {
      float a[NL][8];
      tmem_ld_levels(tmem + ((uint32_t)((warp & 3) * 32) << 16) + 32 * half + 8 * g, p64::PT, a);
      int64_t v[8];
#pragma unroll
      for (int c = 0; c < 8; c++, p += m) {
        const float al[NL] = {a[0][c], a[1][c], a[2][c], a[3][c], a[4][c], a[5][c], a[6][c]};
        const Norm x = product_any(al, rx + einv[32 * half + 8 * g + c], rr + 1, over);
        if (ok && 8 * g + c < nc) *p = to_double(x);
        v[c] = to_biased(x, rr);
      }
      store8(sm + row * 128 + (((4 * half + g) ^ (row & 7)) << 4), TRSM_PLANE_A, v);
    }
  }
  if (ok && rok && over) atomicMin(notpd + b, col);
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  tcg::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tcg::tc_fence_after();
    tcg::tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && ok) {   // the digits of X: 64-row boxes, rows past the front are not written
    const uint8_t* map = tmaps + (int64_t)slot_of[s] * 128;
    tcg::tmap_acquire(map);
    for (int h = 0; h < 2 && h * p64::PT < nr; h++)
      for (int d = 0; d < NS; d++)
        tcg::tma_store_4d(map, kb % (KG / p64::PT) * p64::PT, (int)r0 + h * p64::PT, d, b, tcg::smem_u32(sm) + d * TRSM_PLANE_A + h * p64::PT * 128);
    tcg::bulk_store_wait();
  }
}

}  // namespace
