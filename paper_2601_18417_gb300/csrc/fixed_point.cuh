// fixed_point.cuh -- coefficients and values of the fixed-point sums as two
// limbs each, and the sums' way back to FP64 (residual.cu says what they are for).
// Plain integer code that a host compiler takes too, so that a test without a
// GPU runs these very lines.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define HOFV_HD __host__ __device__ __forceinline__
#else
#define HOFV_HD inline
#endif

namespace hofv {

constexpr int kFxMin = 555, kFxMax = 1560;  // biased exponents: the scales stay normal numbers
constexpr int kFxZero = kFxMin - 1;         // exponent of a row or a stencil of zeros
constexpr uint16_t kFxPlain = 0xffff;       // row exponent of a row to be summed by FMAs
// A sum is taken as exact enough where some of its products, the nearest cells'
// with the largest coefficients among them, add up to this in magnitude, in units
// of 2^32 of the high limbs' products: 2^55 of those in 2-D, 2^54 in 3-D, where four
// times the slots make FMAs err more (residual.cu has the figures).
HOFV_HD constexpr uint32_t fx_sure(int dim) { return dim == 2 ? 1u << 23 : 1u << 22; }

struct FxLimbs {
  int hi, lo;
};

HOFV_HD int64_t fx_bits(double c) {
#if defined(__CUDA_ARCH__)
  return __double_as_longlong(c);
#else
  int64_t b;
  memcpy(&b, &c, sizeof(b));
  return b;
#endif
}
HOFV_HD double fx_double(int64_t b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double(b);
#else
  double c;
  memcpy(&c, &b, sizeof(c));
  return c;
#endif
}
HOFV_HD int fx_min(int a, int b) { return a < b ? a : b; }

// x >> n, zero for n of 32 and more
HOFV_HD uint32_t fx_shr(uint32_t x, int n) {
#if defined(__CUDA_ARCH__)
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
#else
  return n < 32 ? x >> n : 0;
#endif
}

// Exponent E that scales a row of coefficients, mx the largest biased exponent
// among them and sum their magnitudes' sum: 2^(E - 1022) is above each, and 15
// times it is no less than the sum.
HOFV_HD uint16_t fx_row_exponent(int mx, bool zero, double sum) {
  if (zero) return (uint16_t)kFxZero;
  if (mx < kFxMin || mx > kFxMax) return kFxPlain;
  int E = mx;
  while (sum > 15.0 * fx_double((int64_t)(E + 1) << 52)) ++E;
  return (uint16_t)E;
}

// |c| 2^(1081 - E) rounded, at most 2^59, as limbs: hi 2^28 + lo with hi < 2^31
// and lo <= 2^28, both with c's sign
HOFV_HD FxLimbs fx_coef(double c, int E) {
  const int64_t b = fx_bits(c);
  const int h = (int)(b >> 32);
  const uint32_t l = (uint32_t)b;
  const int sh = fx_min(E - ((h >> 20) & 0x7ff), 60);  // 60, which leaves nothing, for zero: kFxZero
  // the significand at the top of 63 bits
  const uint32_t mh = (((uint32_t)h << 10 | l >> 22) & 0x7fffffff) | 0x40000000u;
  const uint64_t m = (uint64_t)mh << 32 | (l << 10);
  const int hi = (int)fx_shr(mh, sh);
  const int lo = (int)((((uint32_t)(m >> (sh + 3)) & 0x1fffffffu) + 1) >> 1);
  return h < 0 ? FxLimbs{-hi, -lo} : FxLimbs{hi, lo};
}

// u 2^(1077 - E) rounded, at most 2^55, as 28-bit limbs (hi, lo), the low one
// in [-2^27, 2^27); h and l the words of u
HOFV_HD FxLimbs fx_value(int h, int l, int E) {
  const int sh = fx_min(E - ((h >> 20) & 0x7ff), 63);  // 63 for zero
  const uint64_t mant = (uint64_t)(uint32_t)((h & 0xfffff) | 0x100000) << 32 | (uint32_t)l;
  int64_t v = (int64_t)((((mant << 3) >> sh) + 1) >> 1);
  if (h < 0) v = -v;
  const int64_t hi = (v + (1 << 27)) >> 28;
  return {(int)hi, (int)((uint32_t)v - ((uint32_t)hi << 28))};
}

// a sum h 2^56 + l 2^28, l >= 0
struct FxTotal {
  int64_t h;
  uint32_t l;
};

// t in units of 2^(Ec - 1081 + Eu - 1077), rounded once
HOFV_HD double fx_scale(FxTotal t, int Ec, int Eu) {
  const double h = (double)t.h;
  const int64_t rest = (t.h - (int64_t)h) * (1 << 28) + t.l;  // what h lost, and l: exact in FP64
  return fma(h, 268435456.0, (double)rest) * fx_double((int64_t)(1023 + Ec + Eu - 2130) << 52);
}

// sums of products of one component: the high limbs' (2^56) and the mixed (2^28)
struct FxSum {
  int64_t hh = 0, x = 0;
  HOFV_HD void mac(FxLimbs q, int uh, int ul) {
    hh += (int64_t)q.hi * uh;
    x += (int64_t)q.hi * ul;
    x += (int64_t)q.lo * uh;
  }
  HOFV_HD FxTotal total() const { return {hh + (x >> 28), (uint32_t)x & 0xfffffffu}; }
};

// magnitude of a product, as fx_sure counts: below 2^26
HOFV_HD uint32_t fx_size(FxLimbs q, int uh) {
  return (uint32_t)((uint64_t)(uint32_t)(q.hi < 0 ? -q.hi : q.hi) * (uint32_t)(uh < 0 ? -uh : uh) >> 32);
}

}  // namespace hofv
