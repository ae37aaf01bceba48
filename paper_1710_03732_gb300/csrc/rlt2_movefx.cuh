// The folded z move of one symmetry class in 64-bit integers (host and device).
//
//   w_b  = xi_b + psi_b          b = 0..5, psi already less the tile term
//   s_b  = D_b - w_b,  S = s_0 + ... + s_5
//   D'_b = D_b - s_b + phi (S - s_b) = w_b + phi (S - s_b)
//
// GB300 retires FP64 operations at about 1.7 lanes per clock per SM and 32-bit
// integer operations at about 128, so the 29 FP64 operations of a class cost
// more than these sums in integers on one grid per class.  w_b is one FP64
// addition (the FP64 pipe has room for six, and six integer conversions are
// saved); D_b and w_b are cut onto the grid 2^L, L = emax - 1081 in biased
// exponents, emax the largest exponent field among the class's D_b and w_b:
//   - an input is |x| < 2^59 steps; those within 2^6 of the largest are exact,
//     smaller ones are cut toward zero by less than one step;
//   - |s_b| < 2^60, |S| < 2^62.6, |D'_b| < 2^61 (phi = 1/5): no overflow, and
//     the sums are exact;
//   - phi (S - s_b) is cut by less than three steps (see fx_scale);
//   - D'_b is rounded once, to nearest, when it is stored as a double.
// A step is 2^-6 of the rounding unit (2^-53) of the class's largest input,
// where the FP64 form rounds two differences per entry and every sum at up to
// that unit, so the result is at least as close to the exact move
// (tests/test_movefx.py).  Exponents at the ends of the range, and infinities
// or NaN, take the FP64 form.
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

// q grid steps as a double (rounded to nearest).
RLT2_HD double fx_unalign(int64_t q, uint32_t emax) {
#if defined(__CUDA_ARCH__)
  const uint64_t b = fx_bits(__ll2double_rn(q));
#else
  const uint64_t b = fx_bits((double)q);
#endif
  const uint32_t hi = (uint32_t)(b >> 32);  // 0 only for q = 0
  return fx_double(((uint64_t)(hi ? hi + (emax - (1081u << 20)) : 0u) << 32) | (uint32_t)b);
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

// The move of one class, in place on D, w_b = xi_b + psi_b; false (D untouched)
// where the class's exponents call for the FP64 form.
RLT2_HD bool move_class_fx(double D[6], const double w[6], FxFactor phi) {
  uint32_t emax = 0;
  for (int b = 0; b < 6; ++b) {
    const uint32_t a = fx_exp(D[b]), c = fx_exp(w[b]);
    emax = emax > a ? emax : a;
    emax = emax > c ? emax : c;
  }
  if (emax < kFxExpLow || emax > kFxExpHigh) return false;
  int64_t s[6], q[6], S = 0;
  for (int b = 0; b < 6; ++b) {
    q[b] = fx_align(w[b], emax);
    s[b] = fx_align(D[b], emax) - q[b];
    S += s[b];
  }
  for (int b = 0; b < 6; ++b) D[b] = fx_unalign(q[b] + fx_scale(phi, S - s[b]), emax);
  return true;
}

}  // namespace rlt2
