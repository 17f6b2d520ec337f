// f64_digits.cuh -- FP64 products on the FP16 tensor cores: an FP64 entry as six signed 9-bit digits.
//
// GB300's FP64 pipe runs at about 1 TFLOP/s (0.5 lanes per clock and scheduler), its FP16 tensor cores at 1.7
// PFLOP/s. An entry x with |x| <= 2^(rho + 1) is the fixed-point number x = 2^rho sum_{s < 6} d_s 2^(-9 (s + 1)) + e
// with |d_0| <= 1024, |d_s| <= 256 for s > 0 and |e| <= 2^(rho - 55): every digit is exact in FP16, every product of
// two digits exact in FP32, and a dot product's sum over one level l = s + t, A_l = sum_k sum_{s + t = l} d_s d'_t, is
// an integer, which the FP32 accumulator holds exactly below 2^24. For two rows of a Cholesky factor with 2^(rho + 1)
// >= sqrt(C_ii), the rows' squared norms are at most C_ii, so over K = 256 level 0 is below 2^21 and level 1 below 2^23
// (Cauchy-Schwarz); the lower levels' digits are noise-like, and even the sum of 256 squares of them is at most 2^24.
// Two general operands take |x| <= 2^rho (|d_0| <= 512) and K = 64. The 26 digit products of the levels 0..6 are kept;
// the dropped ones (l >= 7) and the remainders e leave a relative error of about 2^-58 sqrt(C_ii C_jj), below the
// rounding of a chain of K FP64 multiply-adds (2^-53 of the running sum per step). The levels are put together in 64-bit
// integers and rounded to FP64 once.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

namespace f64d {

constexpr int NS = 6;     // digits of an entry
constexpr int NL = 7;     // levels s + t kept
constexpr int KG = 256;   // columns of a deferred-update group: the longest sum of one accumulation

// The smallest rho with |x| <= 2^rho from the exponent field (a NaN or an infinity gives some value: its factorization
// is reported as not positive definite).
__device__ __forceinline__ int rho_of(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e == 0 ? -1022 : e - 1022;   // |x| < 2^(e - 1022)
}

// The fixed-point form of x at scale 2^rho: round(x 2^(54 - rho)) for |x| <= 2^(rho + 1) (larger |x|, which only a failed
// factorization has, saturate).
__device__ __forceinline__ int64_t to_fixed(double x, int rho) {
  const int64_t bits = __double_as_longlong(x);
  const int e = (int)(bits >> 52) & 0x7ff;
  const int64_t man = (bits & 0xfffffffffffffLL) | 0x10000000000000LL;
  const int sh = 1021 + rho - e;   // right shift of the 53-bit significand
  int64_t y;
  if (sh <= 0) y = man << (sh < -3 ? 3 : -sh);
  else y = sh > 54 ? 0 : (man + (1LL << (sh - 1))) >> sh;
  if (e == 0) y = 0;
  return bits < 0 ? -y : y;
}

// The six digits of fixed-point y (2^-54 units): d_s + 256 sit in 9-bit fields of y plus the bias 256 (2^9 + ... +
// 2^36 + 1); u[s] receives the field, u[0] the digit itself (taken modulo 2^12, which only a failed factorization
// exceeds).
__device__ __forceinline__ void digit_fields(int64_t y, uint32_t (&u)[NS]) {
  constexpr int64_t bias = 256LL * (1 + (1LL << 9) + (1LL << 18) + (1LL << 27) + (1LL << 36));
  const int64_t v = y + bias;
#pragma unroll
  for (int s = 1; s < NS; s++) u[s] = (uint32_t)((uint64_t)v >> (9 * (NS - 1 - s))) & 0x1ffu;
  u[0] = (uint32_t)(((int32_t)(v >> 45) << 20) >> 20);
}

// Two digit fields as a pair of FP16 digits: 0x6400 + u is the FP16 number 1024 + u, and d = (1024 + u) - 1280.
__device__ __forceinline__ uint32_t digits_half2(uint32_t ulo, uint32_t uhi) {
  const uint32_t p = 0x64006400u + (ulo | (uhi << 16));
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&p), __half2half2(__ushort_as_half(0x6500)));
  return *reinterpret_cast<const uint32_t*>(&d);
}

__device__ __forceinline__ uint32_t digits0_half2(uint32_t lo, uint32_t hi) {
  const __half2 d = __halves2half2(__short2half_rn((short)lo), __short2half_rn((short)hi));
  return *reinterpret_cast<const uint32_t*>(&d);
}

// Eight consecutive entries' digits s as 16 bytes.
__device__ __forceinline__ uint4 pack8(const uint32_t (&u)[8][NS], int s) {
  if (s == 0)
    return make_uint4(digits0_half2(u[0][0], u[1][0]), digits0_half2(u[2][0], u[3][0]), digits0_half2(u[4][0], u[5][0]),
                      digits0_half2(u[6][0], u[7][0]));
  return make_uint4(digits_half2(u[0][s], u[1][s]), digits_half2(u[2][s], u[3][s]), digits_half2(u[4][s], u[5][s]),
                    digits_half2(u[6][s], u[7][s]));
}

constexpr int UB = 59;   // products come out in units of 2^-59 of their scale

// The levels' sums (level l weighs 2^(-18 - 9 l)) as a fixed-point number in units of 2^-q; what the caller knows to
// be below 2^(63 - q) comes out right whatever the size of the single levels (integer arithmetic modulo 2^64).
__device__ __forceinline__ int64_t combine_at(const float (&a)[NL], int q) {
  int64_t t1 = (int64_t)__float2int_rn(a[0]) * (1LL << 27);
  t1 += (int64_t)__float2int_rn(a[1]) * (1LL << 18);
  t1 += (int64_t)__float2int_rn(a[2]) * (1LL << 9);
  t1 += (int64_t)__float2int_rn(a[3]);                       // levels 0..3 in units of 2^-45
  int64_t t0 = (int64_t)__float2int_rn(a[4]) * (1LL << 18);
  t0 += (int64_t)__float2int_rn(a[5]) * (1LL << 9);
  t0 += (int64_t)__float2int_rn(a[6]);                       // levels 4..6 in units of 2^-72
  const int s1 = q - 45, s0 = 72 - q;
  t1 = s1 >= 0 ? (s1 > 63 ? 0 : (int64_t)((uint64_t)t1 << s1)) : t1 >> min(63, -s1);
  t0 = s0 > 0 ? (t0 + (1LL << min(62, s0 - 1))) >> min(63, s0) : (s0 < -63 ? 0 : (int64_t)((uint64_t)t0 << -s0));
  return t1 + t0;
}

// The same at q = UB for the dot product of two rows of a Cholesky factor (at most 4).
__device__ __forceinline__ int64_t combine(const float (&a)[NL]) {
  constexpr int S = UB - 18;   // shift of level 0
  const float low = fmaf(a[6], 0x1p-13f, a[5] * 0x1p-4f);   // levels 5 and 6, rounded to a unit
  int64_t v = (int64_t)__float2int_rn(a[0]) * (1LL << S);
  v += (int64_t)__float2int_rn(a[1]) * (1LL << (S - 9));
  v += (int64_t)__float2int_rn(a[2]) * (1LL << (S - 18));
  v += (int64_t)__float2int_rn(a[3]) * (1LL << (S - 27));
  v += (int64_t)__float2int_rn(a[4]) * (1LL << (S - 36));
  return v + (int64_t)__float2int_rn(low);
}

// v 2^(rho - UB) rounded to FP64 (half away from zero), in integers: the FP64 pipe is the slow one here.
__device__ __forceinline__ double to_double(int64_t v, int rho) {
  if (v == 0) return 0.0;
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  const int z = __clzll((long long)a);
  const uint64_t nrm = a << z;
  const uint64_t man = (nrm >> 11) + ((nrm >> 10) & 1);    // 2^52 <= man <= 2^53
  const int E = 1023 + 62 - UB + 1 - z + rho;              // biased exponent of man / 2^52
  if (E <= 0) return 0.0;                                  // below the normal range
  const uint64_t bits = ((uint64_t)(E < 2046 ? E - 1 : 2045) << 52) + man;
  return __longlong_as_double((long long)(bits | ((uint64_t)v & 0x8000000000000000ull)));
}

// Fixed-point form in 2^-54 units (to_fixed's) of v in 2^-UB units.
__device__ __forceinline__ int64_t refix(int64_t v) { return (v + (1LL << (UB - 55))) >> (UB - 54); }

}  // namespace f64d
