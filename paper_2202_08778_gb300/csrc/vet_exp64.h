// vet_exp64.h -- the FP64 segment weight of the ray march, e^-x or
// e^-x - 1 for a segment of optical depth x, with the double arithmetic cut
// to three operations.
//
// Why: GB300 executes two FP64 operations per clock per SM against 128 FP32
// or 64 integer ones, so a warp's FP64 instruction holds the SM's pipe for 16
// clocks, the time of 64 issue slots.  The CUDA library's expm1 and exp2,
// which a select between the two forms needs both of, cost about 40 FP64
// operations a segment; here only what has to be rounded to 53 bits in
// floating point is FP64 and the rest is integer arithmetic beside it.
//
// Method (table-driven exponential after Tang, ACM TOMS 15 (1989) 144 and 18
// (1992) 211): with y = kappa len = -x log2(e) <= 0 (event lengths are stored
// pre-scaled by -h log2(e)), n = round(-1024 y) from FP32 copies of kappa and
// len, and r = y + n/1024, exact up to one rounding of the product (one FMA),
//   2^y - 1 = (E_j 2^-i - 1) + E_j 2^-i (2^r - 1),   n = 1024 i + j,
//   2^r - 1 = r ln2 F(r),  F = (1 - e^-u)/u = 1 - u/2 + u^2/6 - u^3/24 + ...,
//   u = -r ln2,  |u| < 2^-11.03 (|r| < 2^-10.5, checked: half a step is 2^-11,
//   the FP32 estimate of n is up to 0.2 steps further off at large depths).
// F differs from 1 by less than 2^-12, so its bits come from a 64-bit
// fixed-point evaluation (below 2^-55 of error over the whole range).  The
// tables hold E_j ln2, E_j = 2^(-j/1024) and T_j = E_j - 1, each rounded
// once.  thin (x < 1/2, n < kThinN): w = e^-x - 1 = T_j + (E_j ln2) (r F);
// else w = e^-x = E + (E ln2) (r F) with both scaled by 2^-i.
//
// The evaluation checks its own premise: r, whose value does not depend on
// the FP32 estimate's quality once n is chosen, must lie within 2^-10.5, and
// n below 1000 * 1024; everything else (a NaN, an infinity, a depth beyond 690,
// a kappa below 0 by more than rounding, operands outside FP32's range) returns
// false, and the caller takes the library's functions.  (kappa < 0 with |r| within
// the bound has n = 0 and is evaluated like any other r.)
//
// Error against the exact weight of kappa and len, as a fraction of it, beside
// expm1 and exp2 of the rounded product (on the host): depths below 1e-3 at most
// 3.5e-16 and 3.2e-16 (RMS 9.2e-17 and 8.4e-17), 1e-3 to 0.5 2.4e-16 and 3.1e-16,
// 0.5 to 1 2.2e-16 and 1.5e-16, 1 to 2 2.2e-16 and 2.6e-16, 10 to 50 2.2e-16 and
// 5.0e-15 (the product's own rounding, which r does not have).
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

namespace vet {

constexpr int kExp64Steps = 1024;             // table steps per factor of two
constexpr uint32_t kThinN = 739;              // n below: x < 1/2 (739/1024 = 0.5003 log2(e))
constexpr uint32_t kExp64MaxN = 1000u * 1024u;

// Device copy of the tables: rec[j] = (E_j ln2, E_j), then t[j] = E_j - 1 for
// j < kThinN, as one array of doubles.
constexpr int kExp64TableDoubles = 2 * kExp64Steps + (int)kThinN + 1;

inline void exp64_fill_table(double *tab) {
  const long double ln2 = 0.693147180559945309417232121458176568L;
  for (int j = 0; j < kExp64Steps; ++j) {
    const long double e = std::exp2(-(long double)j / kExp64Steps);
    tab[2 * j] = (double)(e * ln2);
    tab[2 * j + 1] = (double)e;
  }
  for (int j = 0; j <= (int)kThinN; ++j)
    tab[2 * kExp64Steps + j] = (double)std::expm1(-(long double)j / kExp64Steps * ln2);
}

namespace exp64 {
__host__ __device__ __forceinline__ uint64_t bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
__host__ __device__ __forceinline__ uint32_t fbits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}
__host__ __device__ __forceinline__ float from_fbits(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}
__host__ __device__ __forceinline__ uint32_t mulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
}  // namespace exp64

// w and its form for kappa and one event (len, and lens = (float)(1024 len));
// false (w unset) where the premise does not hold.
__host__ __device__ __forceinline__ bool exp64_weight(double kappa, double len, float lens, const double *tab,
                                                      double &w, bool &thin) {
  using namespace exp64;
  // FP32 value of kappa >= 0 from its bits (truncated; below FP32's range 0; above
  // it, and of a kappa < 0, 0 or meaningless, which the check on r catches)
  const uint64_t kb = bits(kappa);
  const int32_t kh = (int32_t)((uint32_t)(kb >> 32) - 0x38000000u);
  const uint32_t khc = kh > 0 ? (uint32_t)kh : 0u;
  const float k32 = from_fbits((khc << 3) | ((uint32_t)kb >> 29));
  constexpr float kMagic = 12582912.f;  // 1.5 * 2^23: the sum's low bits are round(1024 y)
  const float t = fmaf(k32, lens, kMagic);
  const uint32_t n = fbits(kMagic) - fbits(t);
  const uint32_t nb = fbits(kMagic - t);  // n as an FP32 value, exact
  // n / 1024 as a double, from the FP32 bits (n < 2^20: the low word is 0)
  const double nd = from_bits((uint64_t)(n ? (nb >> 3) + (0x38000000u - (10u << 20)) : 0u) << 32);
  const double r = fma(kappa, len, nd);
  const uint64_t rb = bits(r);
  const uint32_t rh = (uint32_t)(rb >> 32), mh = rh & 0x7fffffffu;
  if (mh >= 0x3F46A09Eu || n >= kExp64MaxN) return false;  // |r| >= 2^-10.5 (or NaN)
  // |r| 2^63 as an integer (its low bits below 2^-63 dropped)
  const uint32_t sh = 1012u - (mh >> 20);
  const uint64_t m = ((uint64_t)((mh & 0xfffffu) | 0x100000u) << 32) | (uint32_t)rb;
  const uint64_t R = m >> (sh < 63u ? sh : 63u);
  const uint32_t Rh = (uint32_t)(R >> 21), Rl = (uint32_t)R & 0x1fffffu;  // Rh = |r| 2^42
  // P = |u|/2 2^75: times ln2/2 = (kC + kCl 2^-32) 2^-33
  constexpr uint32_t kC = 2977044471u, kCl = 3520035243u;
  const uint64_t P = (uint64_t)Rh * kC + mulhi(Rh, kCl) + mulhi(Rl << 11, kC);
  // H = u^2/6 - u^3/24 + u^4/120 (coefficients of |r|, at 2^35, 2^25, 2^15)
  constexpr uint32_t kC2 = 2751373309u, kC3 = 465602u, kC4 = 63u;
  const bool neg = (int32_t)rh < 0;  // r < 0: u > 0
  const uint32_t S = (uint32_t)(((uint64_t)Rh * Rh) >> 31);  // r^2 2^53
  const uint32_t q4 = mulhi(Rh, kC4), W = neg ? kC3 - q4 : kC3 + q4;
  const uint32_t q3 = mulhi(Rh, W), V = neg ? kC2 - q3 : kC2 + q3;
  const int64_t H = (int64_t)(((uint64_t)S * V) >> 13);  // at 2^75
  // F = 1 - D: below 1 in units of 2^-53, above it of 2^-52
  const int64_t D = (neg ? (int64_t)P : -(int64_t)P) - H;
  const int64_t one = 0x3FF0000000000000LL;
  const double F = from_bits((uint64_t)(D >= 0 ? one - ((D + (1LL << 21)) >> 22) : one - ((D + (1LL << 22)) >> 23)));
  const double q = r * F;
  const uint32_t j = n & (kExp64Steps - 1), scale = (n >> 10) << 20;
  thin = n < kThinN;
#ifdef __CUDA_ARCH__
  const double2 e = __ldg(reinterpret_cast<const double2 *>(tab) + j);
  const double ex = e.x, ey = e.y;
  double c = ey;
  if (thin) c = __ldg(tab + 2 * kExp64Steps + j);
#else
  const double ex = tab[2 * j], ey = tab[2 * j + 1];
  double c = thin ? tab[2 * kExp64Steps + j] : ey;
#endif
  const double el = from_bits(bits(ex) - ((uint64_t)scale << 32));
  c = from_bits(bits(c) - ((uint64_t)scale << 32));  // scale is 0 where thin
  w = fma(el, q, c);
  return true;
}

}  // namespace vet
