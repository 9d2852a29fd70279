// 64-bit fixed-point products from 32-bit multiply-adds, for device and host.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#define LSMS_HD __host__ __device__ __forceinline__

namespace {

LSMS_HD int32_t mulhi_s32(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int32_t)(((int64_t)a * b) >> 32);
#endif
}
// a b + c with 32-bit factors: written out, because a factor known to be non-negative makes the
// compiler widen both to a 64-bit multiplication.
LSMS_HD int64_t mad_wide(int32_t a, int32_t b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (int64_t)a * b + c;
#endif
}
LSMS_HD int64_t mul_wide(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (int64_t)a * b;
#endif
}
LSMS_HD int32_t hi_s32(int64_t a) { return (int32_t)(a >> 32); }

// A 64-bit number as a factor: high word and a quarter of the low word (signed 32-bit factors, and
// four cross products fit 64 bits).
struct Factor {
  int32_t h, l;
};
LSMS_HD Factor factor(int64_t a) { return {hi_s32(a), (int32_t)((uint32_t)a >> 2)}; }
// a b / 2^64 + c, and (a b + d e) / 2^64, a few units low: the leading partial products, by 32-bit
// multiply-adds with 64-bit sums.
LSMS_HD int64_t madq(Factor a, Factor b, int64_t c) {
  const int64_t x = mad_wide(a.l, b.h, mul_wide(a.h, b.l));
  return mad_wide(hi_s32(x), 4, mad_wide(a.h, b.h, c));
}
LSMS_HD int64_t mulq2(Factor a, Factor b, Factor d, Factor e) {
  const int64_t x = mad_wide(d.l, e.h, mad_wide(d.h, e.l, mad_wide(a.l, b.h, mul_wide(a.h, b.l))));
  return mad_wide(hi_s32(x), 4, mad_wide(d.h, e.h, mul_wide(a.h, b.h)));
}
LSMS_HD int64_t mulq(int64_t a, int64_t b) { return madq(factor(a), factor(b), 0); }
LSMS_HD int64_t mulq2(int64_t a, int64_t b, int64_t d, int64_t e) {
  return mulq2(factor(a), factor(b), factor(d), factor(e));
}
LSMS_HD int64_t shl(int64_t a, int n) { return (int64_t)((uint64_t)a << n); }

}  // namespace
