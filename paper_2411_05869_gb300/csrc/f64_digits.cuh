// f64_digits.cuh -- FP64 products on the FP16 tensor cores: an FP64 entry as six signed 9-bit digits (the error-free
// splitting of matrix products of Ozaki, Ogita, Oishi and Rump, on fixed-point rows).
//
// GB300's FP64 pipe runs at about 1 TFLOP/s (0.5 lanes per clock and scheduler), its FP16 tensor cores at 1.7
// PFLOP/s. An entry x with |x| <= 2^(rho + 1) is the fixed-point number x = 2^rho sum_{s < 6} d_s 2^(-9 (s + 1)) + e
// with |d_0| <= 1024, |d_s| <= 256 for s > 0 and |e| <= 2^(rho - 55): every digit is exact in FP16, every product of
// two digits exact in FP32, and a dot product's sum over one level l = s + t, A_l = sum_k sum_{s + t = l} d_s d'_t, is
// an integer, which the FP32 accumulator holds exactly up to 2^24. For two rows of a Cholesky factor with 2^(rho + 1)
// >= sqrt(C_ii), the rows' squared norms are at most C_ii, so over K = 256 level 0 is at most 2^20 and level 1 2^23
// (Cauchy-Schwarz). The lower levels have no such bound: level l adds up l + 1 digit products, each at most 2^24 (2^22 with
// digit 0). Their digits are noise-like, so that only squares of the same digits add up: on covariances of uniform points,
// lattices, duplicates and points of common bumps the largest sums measured 0.5 times 2^24, 0.99 at the most (32 bump
// families of points without any other covariance). More takes some 150 columns of a group with entries equal to 2^-18 of
// the scale in two rows, that is, columns with the same covariance to both rows and nearly none among themselves (replicates
// at the foot of one bump, without a core term): an arrow matrix of 256 such columns reached 2.5 times 2^24, at level 6. A sum beyond 2^24 is rounded to even numbers, to a
// unit of its level, 2^(-18 - 9 l) of the scales: 2^-45 at level 3, less than FP64's rounding from level 4 on.
// The 26 digit products of the levels 0..6 are kept; the dropped ones (l >= 7) and the remainders e leave an error of about
// 2^-58 sqrt(C_ii C_jj), below the rounding of a chain of K FP64 multiply-adds of rows of that length (2^-53 of the running
// sum per step); a row's entries far below its scale keep fewer than 53 bits. The levels are put together in 64-bit integers
// and rounded to FP64 once.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

namespace f64d {

constexpr int NS = 6;     // digits of an entry
constexpr int NL = 7;     // levels s + t kept
constexpr int KG = 256;   // columns of a deferred-update group: the longest sum of one accumulation

// A fixed-point entry is kept in units of 2^-61 of its scale 2^rho, seven bits below the last digit. Digit s > 0 plus
// 256 is the 9-bit field at bit 7 + 9 (5 - s) of the entry plus BIAS (256 in every field, and half a digit unit, so that
// the digits are the entry rounded); digit 0 is what is left above bit 52.
constexpr int64_t BIAS = 64 + ((256LL << 7) | (256LL << 16) | (256LL << 25) | (256LL << 34) | (256LL << 43));

// The significand of x at bit 62 and the exponent field that goes with it, zeros and numbers below the normal range as they
// are: |x| = man 2^(e - 1085).
__device__ __forceinline__ uint64_t significand(double x, int& e) {
  const int hi = __double2hiint(x), f = (hi >> 20) & 0x7ff;
  const uint32_t mh = (uint32_t)(hi & 0xfffff) | (uint32_t)min(f, 1) << 20, ml = (uint32_t)__double2loint(x);
  e = max(f, 1);
  return ((uint64_t)__funnelshift_l(ml, mh, 10) << 32) | (ml << 10);
}

// x at scale 2^rho, |x| <= 2^(rho + 1), plus BIAS (larger |x|, which only a failed factorization has, come out wrong).
// The sign is applied as a complement: one unit of 2^-61 off for negative x.
__device__ __forceinline__ int64_t to_biased(double x, int rho) {
  int e;
  const uint64_t man = significand(x, e);
  const int n = min(max(1024 + rho - e, 0), 63);   // right shift
  return ((int64_t)(man >> n) ^ (int64_t)(__double2hiint(x) >> 31)) + BIAS;
}

// Digits s of two biased entries as a pair of FP16 numbers: 0x6400 + u is the FP16 number 1024 + u, u = d + 256.
template <int S>
__device__ __forceinline__ uint32_t digit_pair(int64_t va, int64_t vb) {
  if (S == 0) {   // up to +-1024
    uint32_t d;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"((float)(int)(vb >> 52)), "f"((float)(int)(va >> 52)));
    return d;
  }
  constexpr int SH = 7 + 9 * (NS - 1 - S);
  const uint32_t ta = (uint32_t)((uint64_t)va >> SH);
  const uint32_t tb = SH >= 16 ? (uint32_t)((uint64_t)vb >> (SH >= 16 ? SH - 16 : 0)) : (uint32_t)vb << (SH >= 16 ? 0 : 16 - SH);
  const uint32_t p = ((ta & 0x1ffu) | 0x64006400u) | (tb & 0x1ff0000u);
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&p), __half2half2(__ushort_as_half(0x6500)));
  return *reinterpret_cast<const uint32_t*>(&d);
}

// Eight consecutive entries' digits S as 16 bytes.
template <int S>
__device__ __forceinline__ uint4 pack8(const int64_t (&v)[8]) {
  return make_uint4(digit_pair<S>(v[0], v[1]), digit_pair<S>(v[2], v[3]), digit_pair<S>(v[4], v[5]),
                    digit_pair<S>(v[6], v[7]));
}

// All six digits of eight consecutive entries, plane s at dst + s * plane (bytes).
__device__ __forceinline__ void store8(uint8_t* dst, int plane, const int64_t (&v)[8]) {
  *reinterpret_cast<uint4*>(dst) = pack8<0>(v);
  *reinterpret_cast<uint4*>(dst + plane) = pack8<1>(v);
  *reinterpret_cast<uint4*>(dst + 2 * plane) = pack8<2>(v);
  *reinterpret_cast<uint4*>(dst + 3 * plane) = pack8<3>(v);
  *reinterpret_cast<uint4*>(dst + 4 * plane) = pack8<4>(v);
  *reinterpret_cast<uint4*>(dst + 5 * plane) = pack8<5>(v);
}

// A number in floating form: sign, significand n (leading bit 62, or 0) and the exponent e of its value n 2^(e - 62).
struct Norm {
  uint64_t n;
  int32_t sg;   // 0 or -1
  int e;
};
// v 2^(e0 - 62) for |v| < 2^63.
__device__ __forceinline__ Norm normalise(int64_t v, int e0) {
  Norm r;
  r.sg = (int32_t)(v >> 63);
  const int64_t s64 = (int64_t)r.sg;
  const uint64_t a = (uint64_t)((v ^ s64) - s64);
  const int z = __clzll((long long)a) - 1;   // 0..62 (63 for v = 0)
  r.n = a << z;
  r.e = e0 - z;
  return r;
}
// Rounded to FP64 (half away from zero), in integers: the FP64 pipe is the slow one here.
__device__ __forceinline__ double to_double(const Norm& r) {
  uint64_t man = (r.n + 512) >> 10;   // 2^52 <= man <= 2^53
  int E = 1022 + r.e;                 // the biased exponent less one: man brings the other one
  if (E < 0) {                        // below the normal range: man in units of 2^-1074, without a leading one of its own
    const int n = 10 - max(E, -53);
    man = (r.n + (1ull << (n - 1))) >> n;
    E = 0;
  }
  uint32_t hi = (uint32_t)(man >> 32) + ((uint32_t)min(E, 2045) << 20), lo = (uint32_t)man;
  const bool zero = r.n == 0;
  hi = zero ? 0u : hi | ((uint32_t)r.sg & 0x80000000u);
  lo = zero ? 0u : lo;
  return __hiloint2double((int)hi, (int)lo);
}
__device__ __forceinline__ double fix2double(int64_t v, int e) { return to_double(normalise(v, e + 62)); }   // v 2^e

// The levels' sums (level l weighs 2^(-18 - 9 l) of the product of the two scales, 2^e) as one number.
__device__ __forceinline__ int64_t high_levels(float a0, float a1, float a2, float a3) {   // levels 0..3 in units of 2^-45
  int64_t t = (int64_t)__float2int_rn(a0) * (1 << 27);
  t += (int64_t)__float2int_rn(a1) * (1 << 18);
  t += (int64_t)__float2int_rn(a2) * (1 << 9);
  return t + (int64_t)__float2int_rn(a3);
}
// The dot product of two rows of a Cholesky factor (at most 4): units of 2^-59. Levels 4 to 6 are added in FP32 before
// the conversion (at most 2^30 units, and the sum's rounding matters only where the diagonal's squares make it large).
// A row that is longer than its variance allows (it is not a row of a Cholesky factor: no positive definite covariance)
// must not wrap: level 0 is held at twice its bound (8, and the other levels add or take less than 2), so that the row's
// diagonal comes out below zero.
__device__ __forceinline__ Norm product_rows(const float (&a)[NL], int e) {
  const float low = fmaf(a[6], 0x1p-13f, fmaf(a[5], 0x1p-4f, a[4] * 0x1p5f));
  const float a0 = fminf(fmaxf(a[0], -0x1p21f), 0x1p21f);
  return normalise(high_levels(a0, a[1], a[2], a[3]) * (1LL << 14) + (int64_t)__float2int_rn(low), e + 3);
}
// A dot product of 64 terms of at most 2^e each, cut to units of 2^(rho - 61), from all levels or from the levels 0..3. Sets
// `over` where it is more than 1.5 times 2^(rho + 1) (levels 0 and 1 tell, to 2^-12); the result is then any number.
__device__ __forceinline__ int64_t product_fixed(const float (&a)[NL], int e, int rho, bool all, bool& over) {
  const int S = 15 - max(min(rho - e, 5), -9);   // bits kept below levels 0..3: at most 62 in all
  over = over || fabsf(fmaf(a[1], 0x1p-9f, a[0])) > 1.5f * __int_as_float((127 + 34 - S) << 23);
  int64_t v = high_levels(a[0], a[1], a[2], a[3]) << S;
  if (all) {
    const float low = fmaf(a[6], 0x1p-27f, a[5] * 0x1p-18f) * __int_as_float((127 + S) << 23);
    v += (int64_t)__float2int_rn(a[4]) * (int64_t)(1 << (S - 9)) + (int64_t)__float2int_rn(low);
  }
  const int n = rho - 61 - (e - 45 - S);   // from units of 2^(e - 45 - S)
  return n >= 0 ? v >> min(n, 63) : v << min(-n, 63);
}

// For a residual in 64-bit integers modulo 2^64, which is right wherever the residual itself is small: a dot product in
// units of 2^-72 of its scales, and x in units of 2^u.
__device__ __forceinline__ uint64_t product_mod72(const float (&a)[NL]) {
  int64_t low = (int64_t)__float2int_rn(a[4]) * (1 << 18);
  low += (int64_t)__float2int_rn(a[5]) * (1 << 9);
  low += (int64_t)__float2int_rn(a[6]);
  return ((uint64_t)high_levels(a[0], a[1], a[2], a[3]) << 27) + (uint64_t)low;
}
__device__ __forceinline__ uint64_t fixed_mod(double x, int u) {
  int e;
  const uint64_t man = significand(x, e) >> 10;   // |x| = man 2^(e - 1075)
  const int n = e - 1075 - u;
  const uint64_t v = n >= 0 ? (n < 64 ? man << n : 0) : man >> min(-n, 63);
  return __double2hiint(x) < 0 ? 0 - v : v;
}
// What the first six or four digits of a biased entry say: the entry in units of 2^-61 of its scale, cut to 2^-54 or 2^-36.
__device__ __forceinline__ int64_t digits_of(int64_t v, bool six) {
  constexpr int64_t OFF = BIAS - 64;   // 256 in every field
  return six ? (v & ~((1LL << 7) - 1)) - OFF : (v & ~((1LL << 25) - 1)) - (OFF & ~((1LL << 25) - 1));
}

}  // namespace f64d
