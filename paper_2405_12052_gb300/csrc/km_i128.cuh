// Arithmetic of the mean calculation: 128-bit integer sums (two's complement in
// a low and a high 64-bit word), their correctly rounded conversion to FP64,
// and an upward-rounded root for the centroids' moves.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace km {
namespace {

__device__ __forceinline__ double i128_to_double(long long lo_s, long long hi_s) {
  // value = hi * 2^64 + (unsigned)lo, two's complement; correctly rounded.
  unsigned long long lo = (unsigned long long)lo_s, hi = (unsigned long long)hi_s;
  bool neg = (long long)hi < 0;
  if (neg) {  // negate the 128-bit value
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0ull ? 1ull : 0ull);
  }
  double r;
  if (hi == 0ull) {
    r = __ull2double_rn(lo);
  } else {
    int sh = 64 - __clzll((long long)hi);  // bits used in hi
    unsigned long long top = (hi << (64 - sh)) | (lo >> sh);
    unsigned long long rest = lo << (64 - sh);
    if (rest) top |= 1ull;  // sticky bit, 11 places below the rounding point
    r = __ull2double_rn(top) * __hiloint2double((1023 + sh) << 20, 0);  // 2^sh: exact
  }
  return neg ? -r : r;
}

__device__ __forceinline__ void add128(unsigned long long& lo, long long& hi, long long v) {
  unsigned long long nl = lo + (unsigned long long)v;
  hi += (v < 0 ? -1ll : 0ll) + (nl < lo ? 1ll : 0ll);
  lo = nl;
}
__device__ __forceinline__ void add128p(unsigned long long& lo, long long& hi, unsigned long long vl,
                                        long long vh) {
  unsigned long long nl = lo + vl;
  hi += vh + (nl < lo ? 1ll : 0ll);
  lo = nl;
}

// sqrt(t), rounded up, for t >= 0: the FP32 root of t's significand and half
// its exponent (an FP64 root is a long chain); at least 2^-120.
__device__ __forceinline__ float sqrt_up(double t) {
  if (!(t > 0.0)) return 0.f;
  const int hi = __double2hiint(t), e = ((hi >> 20) - 1023) & ~1;
  if (e < -240) return 0x1p-120f;
  const float m = __double2float_ru(__hiloint2double(hi - (e << 20), __double2loint(t)));
  return __fmul_ru(__fsqrt_ru(m), e > 252 ? __uint_as_float(0x7f800000u) : __uint_as_float((uint32_t)(127 + e / 2) << 23));
}

}  // namespace
}  // namespace km
