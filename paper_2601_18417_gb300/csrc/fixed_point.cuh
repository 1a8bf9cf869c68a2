// fixed_point.cuh -- coefficients and values of the fixed-point sums as 28-bit
// limbs, and the sums' way back to FP64 (residual.cu says what they are for).
// Plain integer code that a host compiler takes too, so that a test without a
// GPU runs these very lines.
#pragma once
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define HOFV_HD __host__ __device__ __forceinline__
#else
#define HOFV_HD inline
#endif

namespace hofv {

constexpr int kFxMin = 540, kFxMax = 1560;  // biased exponents: the scales stay normal numbers
constexpr uint16_t kFxPlain = 0xffff;       // row exponent of a row to be summed by FMAs

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

// |c| 2^(1078 - E) truncated, below 2^56, as 28-bit limbs (hi, lo) with c's sign
HOFV_HD FxLimbs fx_coef(double c, int E) {
  const int64_t b = fx_bits(c);
  const int h = (int)(b >> 32);
  const uint32_t l = (uint32_t)b;
  const int sh = fx_min(E - ((h >> 20) & 0x7ff), 56);  // 56, which leaves nothing, for zero: kFxMin
  // the significand at the top of 63 bits
  const uint32_t mh = (((uint32_t)h << 10 | l >> 22) & 0x7fffffff) | 0x40000000u;
  const uint64_t m = (uint64_t)mh << 32 | (l << 10);
  const int hi = (int)fx_shr(mh, sh + 3);
  const int lo = (int)((uint32_t)(m >> (sh + 7)) & 0xfffffffu);
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

// t in units of 2^56 2^(Ec - 1078 + Eu - 1077)
HOFV_HD double fx_scale(int64_t t, int Ec, int Eu) {
  return (double)t * fx_double((int64_t)(1023 + Ec + Eu - 2099) << 52);
}

// sums of products of one component: the high limbs' (2^56) and the mixed (2^28)
struct FxSum {
  int64_t hh = 0, x = 0;
  HOFV_HD void mac(FxLimbs q, int uh, int ul) {
    hh += (int64_t)q.hi * uh;
    x += (int64_t)q.hi * ul;
    x += (int64_t)q.lo * uh;
  }
  HOFV_HD int64_t total() const { return hh + ((x + (1 << 27)) >> 28); }
};

}  // namespace hofv
