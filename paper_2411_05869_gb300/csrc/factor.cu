// factor.cu -- step A7: multifrontal supernodal Cholesky of P C_z P^T, level by level over the supernodal
// elimination tree, every launch batched over the B proposals (grid y).
//
// Front of supernode s: order m = w + r, rows = its w columns then the r rows below it. Its first w columns
// are the panel (stored column-major, ld m, in the factor); the trailing r x r block is the update matrix U_s
// (column-major, ld r, in the update workspace). Per level:
//   1. assembly: the update matrices are zeroed and every child's update matrix is added into its parent's front
//      through the child's relative indices, in child order (extend_add.cuh);
//   2. partial factorization of each front: POTRF of the w x w diagonal block, TRSM of the r rows below,
//      SYRK of U_s -= L21 L21^T. Fronts of order <= 96 are factored by one CTA in shared memory; the larger ones
//      advance together 64 columns (a block) at a time, in groups of 4 blocks: the block's columns receive the
//      updates of the group's earlier blocks, POTRF of the 64 x 64 diagonal tile with its inverse, the rows below
//      times the inverse, and at a group's end the rows and columns after it receive the group's updates at once
//      (K = 256). The products of the last three run on the FP16 tensor cores, on six 9-bit digits per FP64 entry
//      (f64_digits.cuh), since GB300's FP64 pipe gives 1 TFLOP/s.
// A non-positive pivot records the smallest failing permuted column of that proposal and the factorization continues
// (small fronts with a unit pivot, diagonal tiles of large fronts with any value), so the launch sequence is fixed and no
// kernel traps. Large fronts also record a row whose entries are larger than positive definiteness allows, before they
// can leave the range of their digits.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <climits>
#include <cstring>

#include "extend_add.cuh"
#include "f64_digits.cuh"
#include "gp_internal.cuh"
#include "potrf64.cuh"
#include "small_front.cuh"
#include "tc_gemm.cuh"
#include "trsm64.cuh"

void values_run(gp_ctx* ctx, gp_factor_t* f);

namespace {

constexpr int T = GP_TILE;
using fa::find_front;

struct FrontRef {
  int32_t w, r;
  int64_t m;
  double* P;   // panel
  double* Uu;  // update matrix
};

__device__ __forceinline__ FrontRef front_of(const DevPlan& dp, int32_t s, double* panels, double* upd) {
  FrontRef fr;
  fr.w = dp.w[s];
  fr.r = dp.r[s];
  fr.m = (int64_t)fr.w + fr.r;
  fr.P = panels + dp.loff[s];
  fr.Uu = upd + dp.uoff[s];
  return fr;
}

// Address of front entry (i, j), i >= j, in panel or update storage.
__device__ __forceinline__ double* front_at(const FrontRef& fr, int64_t i, int64_t j) {
  return j < fr.w ? fr.P + j * fr.m + i : fr.Uu + (j - fr.w) * fr.r + (i - fr.w);
}

// Whole partial factorization of a front of order <= GP_SMALL_M in shared memory.
__global__ void __launch_bounds__(sf::THREADS)
    k_small_front(const int32_t* __restrict__ list, DevPlan dp, double* __restrict__ panels, double* __restrict__ upd,
                  int64_t PE, int64_t UE, int32_t* __restrict__ notpd) {
  extern __shared__ double A[];   // m x m, column-major, lower part used
  int32_t s = list[blockIdx.x];
  int b = blockIdx.y;
  FrontRef fr = front_of(dp, s, panels + (int64_t)b * PE, upd + (int64_t)b * UE);
  const int m = (int)fr.m, w = fr.w;
  const int32_t first = dp.sn_first[s];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // a warp per column: along the storage
  for (int j = ty; j < m; j += sf::THREADS / 32)
    for (int i = j + tx; i < m; i += 32) A[j * m + i] = *front_at(fr, i, j);
  __syncthreads();
  sf::eliminate(A, m, w, first, notpd + b);
  for (int j = ty; j < m; j += sf::THREADS / 32)
    for (int i = j + tx; i < m; i += 32) *front_at(fr, i, j) = A[j * m + i];
}

// rho of every row of L (permuted order): sqrt(C_jj) <= 2^(rho + 1), from the exponent of the assembled diagonal;
// |L_ji| <= sqrt(C_jj) makes it a scale for the digits of the whole row.
__global__ void __launch_bounds__(256) k_row_scale(DevPlan dp, int64_t n, const double* __restrict__ panels, int64_t PE,
                                                   int32_t* __restrict__ rho) {
  const int b = blockIdx.y;
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int32_t s = dp.sn_of_col[j];
  const int64_t i = j - dp.sn_first[s], m = (int64_t)dp.w[s] + dp.r[s];
  const double d = panels[(int64_t)b * PE + dp.loff[s] + i * m + i];
  const int e = ((__double2hiint(d) >> 20) & 0x7ff) - 1023;   // 2^e <= C_jj < 2^(e + 1)
  rho[(int64_t)b * n + j] = ((e + 2) >> 1) - 1;
}

constexpr int KB = f64d::KG / T;   // blocks per group
static_assert(KB == GP_GROUP64 && f64d::NS == GP_DIGITS64 && p64::TILE_BYTES == GP_TILE_BYTES64, "the plan's layout");

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

// The updates F[i, j] -= sum_{l in K} L[i, l] L[j, l] on 128 x 64 tiles, j <= i, from the digit planes:
//   LEFT: the columns of block kb (rows >= c0), K = the group's earlier blocks, before the block's POTRF;
//   GROUP: rows and columns after the group, tiles on and below the diagonal, K = the whole group.
// One persistent CTA per SM, as in the mixed path's update kernel: warp 0 loads operand planes (A 128 rows and B 64
// rows of 64 FP16, 24 KB per slot) into a ring of 9 slots, warp 1 issues the MMAs of a plane with the planes before
// it as it lands (26 products of 4 instructions per 64 columns of K, into one accumulator per level: 7 x 64 TMEM
// columns), warps 2-9 put the levels together in 64-bit integers and subtract from the front in FP64 -- lanes are rows,
// so the column-major front is read and written in whole 256-byte segments. The seven accumulators fill the tensor
// memory, so a tile's epilogue does not overlap the next tile's MMAs (its operand loads do): the tensor pipe is busy 60 % of
// the time, and with N = 64 an instruction (6 KB of shared memory read in 48 clocks) uses half of its rate. A group end of 5744
// rows: 326 us, tensor cycles 30 %, DRAM 9 % (counters of one launch), 0.35 of the measured FP16 rate in digit products.
// Against FP64 multiply-adds (64-column updates of the whole trailing matrix at the FP64 pipe's 1 TFLOP/s) the updates
// of one factorization went from 101.8 to 10.3 ms at n = 100k (1.1e11 flops) and from 725 to 47 ms at n = 200k (8.3e11
// flops), left-looking strips included; residuals |r - C alpha| / |r| stayed the same.
constexpr int U64_THREADS = 320, U64_SLOTS = 9, U64_SLOT = (128 + T) * 128;
constexpr int U64_SMEM = U64_SLOTS * U64_SLOT + 256 + 1024;

struct Tile64 {
  int32_t s, slot;
  int b, w, r, K;
  int64_t m, i0, j0, jlim;
};

template <bool GROUP>
__device__ __forceinline__ Tile64 decode_tile64(const int32_t* __restrict__ fronts, const int64_t* __restrict__ pre,
                                                int nfront, int64_t total, int kb, const DevPlan& dp,
                                                const int32_t* __restrict__ slot_of, int64_t tt) {
  Tile64 u;
  u.b = (int)(tt / total);
  const int64_t t = tt - (int64_t)u.b * total;
  const int fi = find_front(pre, nfront, t);
  u.s = fronts[fi];
  u.slot = slot_of[u.s];
  u.w = dp.w[u.s];
  u.r = dp.r[u.s];
  u.m = (int64_t)u.w + u.r;
  const int64_t loc = t - pre[fi];
  const int c0 = kb * T, g0 = kb / KB * f64d::KG;
  if (!GROUP) {
    u.i0 = c0 + loc * 128;
    u.j0 = c0;
    u.jlim = min(c0 + T, u.w);
    u.K = c0 - g0;
  } else {   // tile row I (128 rows) holds 2 I + 2 tiles of 64 columns
    int64_t I = (int64_t)((sqrtf(4.f * (float)loc + 1.f) - 1.f) * 0.5f);
    while ((I + 1) * (I + 2) <= loc) I++;
    while (I * (I + 1) > loc) I--;
    const int gend = min(g0 + f64d::KG, u.w);
    u.i0 = gend + I * 128;
    u.j0 = gend + (loc - I * (I + 1)) * T;
    u.jlim = u.m;
    u.K = gend - g0;
  }
  return u;
}

template <bool GROUP>
__global__ void __launch_bounds__(U64_THREADS, 1)
    k_update64(const int32_t* __restrict__ fronts, const int64_t* __restrict__ pre, int nfront, int64_t total,
               int64_t ntiles, int kb, DevPlan dp, const uint8_t* __restrict__ tmaps,
               const int32_t* __restrict__ slot_of, const int32_t* __restrict__ rho, int64_t n,
               double* __restrict__ panels, double* __restrict__ upd, int64_t PE, int64_t UE, int32_t* __restrict__ err,
               tcg::WaitLimit lim) {
  using namespace f64d;
  extern __shared__ __align__(1024) uint8_t u64_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)u64_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + U64_SLOTS * U64_SLOT);
  uint64_t* full = bars;                   // [9] plane landed
  uint64_t* empty = bars + U64_SLOTS;      // [9] plane's MMAs done
  uint64_t* tfull = bars + 2 * U64_SLOTS;  // accumulators complete
  uint64_t* tempty = tfull + 1;            // accumulators drained
  uint64_t* drain = tfull + 2;             // the MMA issuer's last commit (winding down)
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tfull + 3);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  uint32_t* issued_s = tslot + 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = tcg::smem_u32(smem);
  if (threadIdx.x == 0) {
    for (int q = 0; q < U64_SLOTS; q++) {
      tcg::mbar_init(&full[q], 1);
      tcg::mbar_init(&empty[q], 1);
    }
    tcg::mbar_init(tfull, 1);
    tcg::mbar_init(tempty, 8);
    tcg::mbar_init(drain, 1);
    *issued_s = 0;
    *abort_flag = *(volatile int32_t*)err != 0;   // an earlier launch of this factorization failed: skip the tiles
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) tcg::tmem_alloc(tslot, 512);
  tcg::tc_fence_before();
  __syncthreads();
  tcg::tc_fence_after();
  const uint32_t tmem = *tslot;
  auto fail = [&]() {
    *abort_flag = 1;
    atomicExch(err, 1);
  };
  if (warp == 0) {
    if (lane == 0) {   // TMA producer: planes in order, slots round robin
      uint32_t slot = 0, ph = 0, issued = 0;
      for (int64_t tt = blockIdx.x; tt < ntiles && !*abort_flag; tt += gridDim.x) {
        const Tile64 u = decode_tile64<GROUP>(fronts, pre, nfront, total, kb, dp, slot_of, tt);
        const uint8_t* map = tmaps + (int64_t)u.slot * 128;
        tcg::tmap_acquire(map);
        const int np = (u.K + T - 1) / T * NS;
        for (int p = 0; p < np; p++) {
          if (!tcg::mbar_wait(&empty[slot], ph ^ 1, lim)) {
            fail();
            break;
          }
          const uint32_t sa = sbase + slot * U64_SLOT;
          const int x = p / NS * T, z = p % NS;
          tcg::mbar_arrive_expect_tx(&full[slot], U64_SLOT);
          tcg::tma_load_4d(sa, map, x, (int)u.i0, z, u.b, &full[slot]);
          tcg::tma_load_4d(sa + T * 128, map, x, (int)u.i0 + T, z, u.b, &full[slot]);
          tcg::tma_load_4d(sa + 2 * T * 128, map, x, (int)u.j0, z, u.b, &full[slot]);
          ++issued;
          if (++slot == U64_SLOTS) {
            slot = 0;
            ph ^= 1;
          }
        }
      }
      *issued_s = issued;
    }
  } else if (warp == 1) {
    if (lane == 0) {   // MMA issuer
      const uint32_t idesc = tcg::idesc_f16(128, T);
      uint32_t slot = 0, ph = 0, aph = 0;
      for (int64_t tt = blockIdx.x; tt < ntiles && !*abort_flag; tt += gridDim.x) {
        const Tile64 u = decode_tile64<GROUP>(fronts, pre, nfront, total, kb, dp, slot_of, tt);
        const int nch = (u.K + T - 1) / T;
        if (!tcg::mbar_wait(tempty, aph ^ 1, lim)) {
          fail();
          break;
        }
        tcg::tc_fence_after();
        bool ok = true;
        for (int c = 0; c < nch && ok; c++) {
          uint32_t base[NS];
          uint32_t sl[NS];
#pragma unroll
          for (int d = 0; d < NS; d++) {   // plane d with the planes 0..min(d, 6 - d)
            if (ok && !tcg::mbar_wait(&full[slot], ph, lim)) ok = false;
            if (ok) {
              tcg::tc_fence_after();
              sl[d] = slot;
              base[d] = sbase + slot * U64_SLOT;
              if (++slot == U64_SLOTS) {
                slot = 0;
                ph ^= 1;
              }
#pragma unroll
              for (int e = 0; e <= d; e++) {
                if (d + e >= NL) continue;
                const uint32_t acc = tmem + (d + e) * T;
                // the first product of a level: (d, e) with the largest d it starts from, i.e. e = d or e = d - 1
                const bool first = c == 0 && (e == d || e == d - 1);
#pragma unroll
                for (int kk = 0; kk < 4; kk++) {
                  const uint64_t ad = tcg::smem_desc_sw128(base[d] + kk * 32);
                  const uint64_t be = tcg::smem_desc_sw128(base[e] + 2 * T * 128 + kk * 32);
                  tcg::mma_f16(acc, ad, be, idesc, first && kk == 0 ? 0u : 1u);
                  if (e < d)
                    tcg::mma_f16(acc, tcg::smem_desc_sw128(base[e] + kk * 32),
                                 tcg::smem_desc_sw128(base[d] + 2 * T * 128 + kk * 32), idesc, 1u);
                }
              }
              // planes no later plane of this chunk multiplies any more: d once d + (d + 1) > 6, and e whose last
              // partner is d (d + e = 6)
              if (2 * d + 1 >= NL) tcg::mma_commit(&empty[sl[d]]);
              if (NL - 1 - d >= 0 && NL - 1 - d < d && NL - 1 - d > 1) tcg::mma_commit(&empty[sl[NL - 1 - d]]);
              if (d == NS - 1) {
                tcg::mma_commit(&empty[sl[0]]);
                tcg::mma_commit(&empty[sl[1]]);
              }
            }
          }
        }
        if (!ok) {
          fail();
          break;
        }
        tcg::mma_commit(tfull);
        aph ^= 1;
      }
    }
  } else {   // epilogue: warp reads TMEM lanes 32 (warp % 4) .. + 31, columns [32 h, 32 h + 32) of each level
    const int q = warp & 3, h = (warp - 2) >> 2;
    uint32_t aph = 0;
    for (int64_t tt = blockIdx.x; tt < ntiles && !__any_sync(0xffffffffu, *abort_flag); tt += gridDim.x) {
      const Tile64 u = decode_tile64<GROUP>(fronts, pre, nfront, total, kb, dp, slot_of, tt);
      double* P = panels + (int64_t)u.b * PE + dp.loff[u.s];
      double* U = upd + (int64_t)u.b * UE + dp.uoff[u.s];
      const int32_t* rows = dp.frows + dp.frow_off[u.s];
      const int32_t* rb = rho + (int64_t)u.b * n;
      const int64_t ib = u.i0 + q * 32, i = ib + lane, jb = u.j0 + 32 * h;
      // column j of the front from row 0: P or U storage
      auto colp = [&](int64_t j) { return j < u.w ? P + j * u.m : U + (j - u.w) * u.r - u.w; };
      {   // while the tile's MMAs run: pull the target columns (256 bytes each, one column per lane) into L2
        const int64_t j = jb + lane;
        const int64_t i1 = j > ib ? j : ib;
        if (j < u.jlim && i1 < imin64(u.m, ib + 32)) {
          const double* pa = colp(j) + i1;
          asm volatile("prefetch.global.L2 [%0];" ::"l"(pa));
          if (i1 + 16 < imin64(u.m, ib + 32)) asm volatile("prefetch.global.L2 [%0];" ::"l"(pa + 16));
        }
      }
      const int ri = i < u.m ? rb[rows[i]] : 0;
      const int rjl = jb + lane < u.jlim ? rb[rows[jb + lane]] : 0;   // lane l: column jb + l
      const int nv = i < u.m ? (int)imin64(32, imin64(i + 1, u.jlim) - jb) : 0;   // this row's entries: the first nv columns
      double* p = colp(jb) + i;   // dereferenced only below nv
      int wl = (int)imin64(64, u.w - jb);   // columns from wl on lie in the update matrix
      if (!tcg::mbar_wait_warp(tfull, aph, lim)) {
        fail();
        break;
      }
      tcg::tc_fence_after();
#pragma unroll 1
      for (int g = 0; g < 4; g++) {
        double old[8];
        double* pc[8];
#pragma unroll
        for (int c = 0; c < 8; c++) {
          const int j = 8 * g + c;
          pc[c] = p;
          old[c] = j < nv ? *p : 0.0;
          p = j + 1 == wl ? U + (i - u.w) : p + (j < wl ? u.m : (int64_t)u.r);
        }
        float a[NL][8];
        tmem_ld_levels(tmem + ((uint32_t)(q * 32) << 16) + 32 * h + 8 * g, T, a);
        if (g == 3) {   // this warp's part of the accumulators has been read
          tcg::tc_fence_before();
          __syncwarp();
          if (lane == 0) tcg::mbar_arrive(tempty);
        }
#pragma unroll
        for (int c = 0; c < 8; c++) {
          const float al[NL] = {a[0][c], a[1][c], a[2][c], a[3][c], a[4][c], a[5][c], a[6][c]};
          const int rj = __shfl_sync(0xffffffffu, rjl, 8 * g + c);
          const double v = to_double(product_rows(al, ri + rj));
          if (8 * g + c < nv) *pc[c] = old[c] - v;
        }
      }
      aph ^= 1;
    }
  }
  // Winding down (waits that return at once after a normal run): before tensor memory is freed, wait for every
  // plane copy issued and for every MMA issued.
  tcg::tc_fence_before();
  __syncthreads();
  if (warp == 0 && lane == 0) {
    const uint32_t nq = *issued_s;
    for (uint32_t c = nq > (uint32_t)U64_SLOTS ? nq - U64_SLOTS : 0; c < nq; c++)
      if (!tcg::mbar_wait(&full[c % U64_SLOTS], (c / U64_SLOTS) & 1)) fail();
  }
  if (warp == 1 && lane == 0) {
    tcg::mma_commit(drain);
    if (!tcg::mbar_wait(drain, 0)) fail();
  }
  tcg::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tcg::tc_fence_after();
    tcg::tmem_dealloc(tmem, 512);
  }
}

std::once_flag g_attrs_once;
void set_attrs() {   // once per process (contexts may run on several host threads)
  std::call_once(g_attrs_once, [] {
    GP_CUDA(cudaFuncSetAttribute(k_small_front, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 GP_SMALL_M * GP_SMALL_M * (int)sizeof(double)));
    GP_CUDA(cudaFuncSetAttribute(k_potrf64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(p64::Smem)));
    GP_CUDA(cudaFuncSetAttribute(k_trsm64, cudaFuncAttributeMaxDynamicSharedMemorySize, TRSM_SMEM));
    GP_CUDA(cudaFuncSetAttribute(k_update64<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, U64_SMEM));
    GP_CUDA(cudaFuncSetAttribute(k_update64<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, U64_SMEM));
  });
}

__global__ void k_fill_i32(int32_t* p, int n, int32_t v) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

}  // namespace

void factor_run_mixed(gp_ctx* ctx, gp_factor_t* f);
void set_attrs_mixed();
static void factor_body(gp_ctx* ctx, gp_factor_t* f);

// A3, A4, A7: the launch sequence is fixed by the plan, so it is captured once per factor as a CUDA graph
// and replayed (theta only changes the device-side parameter block).
void factor_run(gp_ctx* ctx, gp_factor_t* f) {
  set_attrs();
  set_attrs_mixed();
  if (!use_graphs(ctx)) {
    factor_body(ctx, f);
    return;
  }
  if (!f->gx_factor) f->gx_factor = capture_graph(ctx, [&] { factor_body(ctx, f); }, &f->n_factor);
  replay_graph(ctx, f->gx_factor, f->n_factor);
}

static void factor_body(gp_ctx* ctx, gp_factor_t* f) {
  if (f->prec == GP_MIXED) {
    factor_run_mixed(ctx, f);
    return;
  }
  gp_pointset* ps = f->ps;
  const SymPlan& sp = ps->sp;
  const DevPlan& dp = ps->dp;
  cudaStream_t st = ctx->stream;
  set_attrs();
  const int B = f->B;
  const int64_t PE = sp.panel_entries, UE = sp.update64_entries, IE = UE * (int64_t)sizeof(double);
  int32_t* rho = reinterpret_cast<int32_t*>(f->work);   // the scale exponent of every row of L, B x n (the solves come later)
  values_run(ctx, f);   // A3, A4 (zeroes and fills the panels)
  k_fill_i32<<<grid_for(B, 128), 128, 0, st>>>(f->notpd, B, INT_MAX);
  GP_CHECK_LAUNCH(ctx);
  GP_CUDA(cudaMemsetAsync(f->tiles_err, 0, sizeof(int32_t), st));
  k_row_scale<<<dim3(grid_for(ps->n, 256), B), 256, 0, st>>>(dp, ps->n, f->panels, PE, rho);
  GP_CHECK_LAUNCH(ctx);
  ProfLevelScope pls_(ctx);
  for (int32_t L = 0; L < sp.nlevels; L++) {
    const SymPlan::Level& lv = sp.levels[L];
    ctx->prof_level = L;
    uint8_t* itile = reinterpret_cast<uint8_t*>(f->upd + lv.tile64_off);   // the step's tiles
    if (lv.asm_n > 0) {
      ProfScope ps_(ctx, KC_EXTEND_ADD);
      ea::k_assemble64<<<dim3((unsigned)lv.asm_n, B), ea::THREADS, 0, st>>>(dp.asm_tab + lv.asm_off, dp, f->panels,
                                                                           f->upd, PE, UE);
      GP_CHECK_LAUNCH(ctx);
    }
    if (lv.nsmall > 0) {
      // the largest small front of this level sets the shared memory size
      int32_t mmax = 1;
      for (int32_t q = 0; q < lv.nsmall; q++) {
        int32_t s = sp.small_list[lv.small_off + q];
        mmax = std::max(mmax, sp.sn_w[s] + sp.sn_r[s]);
      }
      ProfScope ps_(ctx, KC_FRONT_SMALL);
      k_small_front<<<dim3(lv.nsmall, B), sf::THREADS, (size_t)mmax * mmax * sizeof(double), st>>>(
          dp.small_list + lv.small_off, dp, f->panels, f->upd, PE, UE, f->notpd);
      GP_CHECK_LAUNCH(ctx);
    }
    auto update = [&](const SymPlan::Upd64& u, int32_t kb, bool group) {
      const int64_t ntiles = u.total * B;
      const unsigned grid = (unsigned)std::min<int64_t>(ntiles, ctx->nsm);
      ProfScope ps_(ctx, group ? KC_UPDATE : KC_UPDATE_LEFT, B * u.flops);
      auto k = group ? k_update64<true> : k_update64<false>;
      k<<<grid, U64_THREADS, U64_SMEM, st>>>(dp.upd64_fronts + u.off, dp.upd64_pre + u.pre_off, u.n, u.total, ntiles,
                                             kb, dp, f->op_maps, f->op_slot, rho, ps->n, f->panels, f->upd, PE, UE,
                                             f->tiles_err, f->wait_lim);
      GP_CHECK_LAUNCH(ctx);
    };
    for (const auto& stp : lv.steps) {
      const int32_t* fronts = dp.large_fronts + stp.fr_off;
      if (stp.left64.total > 0) update(stp.left64, stp.kb, false);
      {
        ProfScope ps_(ctx, KC_POTRF, B * stp.potrf_flops);
        k_potrf64<<<dim3(2 * stp.nfront, B), p64::THREADS, sizeof(p64::Smem), st>>>(
            fronts, stp.kb, dp, f->panels, PE, f->notpd, f->dinv, sp.diag_entries, itile, IE, f->tiles_err);
        GP_CHECK_LAUNCH(ctx);
      }
      if (stp.trsm128_total > 0) {
        ProfScope ps_(ctx, KC_TRSM, B * stp.trsm_flops);
        k_trsm64<<<dim3((unsigned)stp.trsm128_total, B), TRSM_THREADS, TRSM_SMEM, st>>>(
            fronts, dp.step_pre + stp.pre_off + stp.nfront + 1, stp.nfront, stp.kb, dp, f->panels, PE, itile, IE,
            rho, ps->n, f->op_maps, f->op_slot, f->notpd, f->tiles_err, f->wait_lim);
        GP_CHECK_LAUNCH(ctx);
      }
      if (stp.group64.total > 0) update(stp.group64, stp.kb, true);
    }
  }
}

// The tensor maps of the FP64 path's digit planes, one per large front: 4-D (columns of a group x rows x digit planes x
// proposals), boxes of 64 columns x 64 rows with the 128-byte swizzle; rows past the front read as zeros.
void build_digit_maps(gp_ctx* ctx, gp_factor_t* f) {
  const SymPlan& sp = f->ps->sp;
  std::vector<int32_t> slot(sp.ns, -1), order;
  for (int32_t s : sp.large_fronts)
    if (slot[s] < 0) {
      slot[s] = (int32_t)order.size();
      order.push_back(s);
    }
  std::vector<CUtensorMap> maps(std::max<size_t>(order.size(), 1));
  std::memset(maps.data(), 0, maps.size() * sizeof(CUtensorMap));
  auto enc = tensor_map_encoder();
  for (size_t k = 0; k < order.size(); k++) {
    const int32_t s = order[k];
    const int64_t m = (int64_t)sp.sn_w[s] + sp.sn_r[s], ldk = sp.op64_ldk(s);
    cuuint64_t dims[4] = {(cuuint64_t)ldk, (cuuint64_t)m, (cuuint64_t)f64d::NS, (cuuint64_t)f->B};
    cuuint64_t strides[3] = {(cuuint64_t)ldk * 2, (cuuint64_t)(m * ldk) * 2, (cuuint64_t)sp.update64_entries * 8};
    cuuint32_t box[4] = {T, T, 1, 1}, es[4] = {1, 1, 1, 1};
    CUresult r = enc(&maps[k], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, f->upd + sp.sn_op64_off[s], dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    GP_REQUIRE(r == CUDA_SUCCESS, "cuTensorMapEncodeTiled rejected a digit map");
  }
  f->op_maps = dalloc<uint8_t>(ctx, f->bufs, maps.size() * sizeof(CUtensorMap));
  f->op_slot = dalloc<int32_t>(ctx, f->bufs, (size_t)sp.ns + 1);
  GP_CUDA(cudaMemcpyAsync(f->op_maps, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice,
                          ctx->stream));
  GP_CUDA(cudaMemcpyAsync(f->op_slot, slot.data(), (size_t)sp.ns * sizeof(int32_t), cudaMemcpyHostToDevice,
                          ctx->stream));
  GP_CUDA(cudaStreamSynchronize(ctx->stream));   // the host vectors go out of scope
}
