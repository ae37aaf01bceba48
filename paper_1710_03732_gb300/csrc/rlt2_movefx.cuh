// The folded z move of one symmetry class with its pool in 64-bit integers (host
// and device).
//
//   s_b  = (D_b - xi_b) - psi_b     b = 0..5, psi already less the tile term
//   S    = s_0 + ... + s_5
//   D'_b = D_b + (phi (S - s_b) - s_b)
//
// GB300 retires FP64 operations at about 1.7 lanes per clock per SM and 32-bit
// integer operations at about 128.  Of the FP64 form's 29 operations a class, the
// twelve that form the s_b and six that add to the D_b stay in FP64: no input or
// result is held in fewer bits than there, however far apart the members'
// magnitudes are.  What lies between is summed on one grid per class, 2^L with
// L = emax - 1081 in biased exponents, emax the largest exponent field of the s_b:
//   - |s_b| < 2^59 steps; those within 2^6 of the largest are exact, smaller ones
//     are cut toward zero by less than one step, 2^-59 to 2^-58 of the largest,
//     where the FP64 form rounds every partial sum at up to 2^-53 of it;
//   - |S| < 2^61.6, |phi (S - s_b) - s_b| < 2^60 (phi = 1/5): no overflow, and the
//     sums are exact;
//   - phi (S - s_b) is cut by less than three steps (see fx_scale);
//   - the change of D_b is rounded once to a double, and D_b + change once.
// The root mean square error against the exact move is no larger than the FP64
// form's, over a class and member by member, also for classes with members 10^9
// apart; a single entry can lie further off than there by a rounding unit of its
// change (tests/test_movefx_pool.py compares both).  Exponents at the ends of the
// range, infinities and NaN take the FP64 form.
#pragma once
#include <cstdint>
#include <cstring>

#if !defined(RLT2_HD)
#if defined(__CUDACC__)
#define RLT2_HD __host__ __device__ __forceinline__
#else
#define RLT2_HD inline
#endif
#endif

namespace rlt2 {

constexpr uint32_t kFxExpMask = 0x7ff00000u;  // exponent field in a double's high word
// Classes whose largest exponent field lies outside [64, 2040] take the FP64 form.
constexpr uint32_t kFxExpLow = 64u << 20, kFxExpHigh = 2040u << 20;

RLT2_HD uint64_t fx_bits(double x) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, sizeof b);
  return b;
#endif
}
RLT2_HD double fx_double(uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, sizeof x);
  return x;
#endif
}
RLT2_HD uint32_t fx_exp(double x) { return (uint32_t)(fx_bits(x) >> 32) & kFxExpMask; }

// x on the class's grid, cut toward zero.  A zero or subnormal x gets a hidden
// bit it does not have, but its shift is then at least 64 and the result 0.
RLT2_HD int64_t fx_align(double x, uint32_t emax) {
  const uint64_t b = fx_bits(x);
  const uint32_t hi = (uint32_t)(b >> 32);
  const uint32_t sh = (emax - (hi & kFxExpMask)) >> 20;
  const uint64_t m = (((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | (uint32_t)b) << 6;
  uint64_t q;
#if defined(__CUDA_ARCH__)
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(m), "r"(sh));  // shifts of 64 and more give 0
#else
  q = sh < 64 ? m >> sh : 0;
#endif
  const int64_t neg = (int64_t)((int32_t)hi >> 31);
  return ((int64_t)q ^ neg) - neg;
}

// q grid steps as a double, rounded to nearest (ties away from zero), |q| < 2^62.
// Integer operations only: a conversion instruction would cost the FP64 pipe as
// much as an addition.
RLT2_HD double fx_unalign(int64_t q, uint32_t emax) {
  const uint64_t neg = (uint64_t)(q >> 63);
  const uint64_t a = ((uint64_t)q ^ neg) - neg;
#if defined(__CUDA_ARCH__)
  const uint32_t z = (uint32_t)__clzll((long long)a);
#else
  const uint32_t z = a ? (uint32_t)__builtin_clzll(a) : 64u;
#endif
  // the leading bit at bit 62, half a unit added, then the unit at bit 0: a carry
  // out of the significand raises the exponent
  const uint64_t r = ((a << ((z - 1) & 63u)) + 0x200) >> 10;
  const uint32_t e = emax + ((4u - z) << 20);  // less one: the leading bit, at bit 52 of r, adds it
  return fx_double(a ? (((uint64_t)e << 32) + r) | (neg << 63) : 0);
}

// phi as hi 2^-32 + lo 2^-64 with lo signed, and phi x within three steps.
struct FxFactor {
  int32_t hi, lo;
};
RLT2_HD FxFactor fx_factor(double phi) {  // 0 <= phi < 1/2
  const int64_t f = (int64_t)(phi * 18446744073709551616.0);
  const int32_t lo = (int32_t)(uint32_t)(uint64_t)f;
  return FxFactor{(int32_t)((f - lo) >> 32), lo};
}
RLT2_HD int64_t fx_scale(FxFactor f, int64_t x) {
  const int32_t xh = (int32_t)(x >> 32);
  const uint32_t xl = (uint32_t)x;
  return (int64_t)xh * f.hi + (int64_t)(((uint64_t)xl * (uint32_t)f.hi) >> 32) + (((int64_t)xh * f.lo) >> 32);
}

// The pool of one class on its grid: s_b in grid steps and phi (S - s_b), cut;
// false where the exponents call for the FP64 form.
RLT2_HD bool class_pool_fx(const double s[6], FxFactor phi, int64_t q[6], int64_t pool[6], uint32_t& emax) {
  emax = 0;
  for (int b = 0; b < 6; ++b) {
    const uint32_t e = fx_exp(s[b]);
    emax = emax > e ? emax : e;
  }
  if (emax < kFxExpLow || emax > kFxExpHigh) return false;
  int64_t S = 0;
  for (int b = 0; b < 6; ++b) {
    q[b] = fx_align(s[b], emax);
    S += q[b];
  }
  for (int b = 0; b < 6; ++b) pool[b] = fx_scale(phi, S - q[b]);
  return true;
}

// The move of one class, in place on D, s_b = (D_b - xi_b) - psi_b; false (D
// untouched) where the exponents call for the FP64 form.
RLT2_HD bool pool_class_fx(double D[6], const double s[6], FxFactor phi) {
  int64_t q[6], pool[6];
  uint32_t emax;
  if (!class_pool_fx(s, phi, q, pool, emax)) return false;
  for (int b = 0; b < 6; ++b) D[b] += fx_unalign(pool[b] - q[b], emax);
  return true;
}

// The same move for a host program that holds the sums w_b = xi_b + psi_b:
// D'_b = w_b + phi (S - s_b), s_b = D_b - w_b, so that the result keeps what the
// sum has where s_b cancels most of D_b.  A class without slack stays as it is.
inline bool move_class_fx(double D[6], const double w[6], FxFactor phi) {
  double s[6];
  int64_t q[6], pool[6];
  uint32_t emax;
  bool rest = true, zero = true;
  for (int b = 0; b < 6; ++b) {
    s[b] = D[b] - w[b];
    rest = rest && s[b] == 0.0;
    zero = zero && D[b] == 0.0;
  }
  if (rest && !zero) return true;
  if (!class_pool_fx(s, phi, q, pool, emax)) return false;
  for (int b = 0; b < 6; ++b) D[b] = w[b] + fx_unalign(pool[b], emax);
  return true;
}

}  // namespace rlt2
