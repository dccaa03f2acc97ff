// residual_key.h -- residual norms of the FP32 SCDM selection as 64-bit integers that are at once floating-point
// numbers and their own order keys: 9 bits of exponent above 54 bits of fraction (55 with the implicit one, two
// more than FP64), rounded down, exponents from 2^-382 on (a square of the smallest FP32 number is 2^-298).
//
// The update v - p^2 is exact but for bits of p^2 below 2^-54 of v, so each step loses at most what an FP64
// multiply-add may lose (2^-53 of the result) whatever the size of v against other points' norms.  It takes
// about thirty integer instructions: FP64 ones issue once per 64 cycles and scheduler, and a chain of
// dependent FP64 updates took 200 cycles a step.  The result of a step depends on v and p only, so a residual is
// the same in whatever runs of steps it is brought up to date.
//
// 0 is zero; negative values mark points that cannot be chosen (-1: chosen already, kNone: not a number).
#pragma once

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define ACE_KEY_FN __host__ __device__ __forceinline__
#else
#define ACE_KEY_FN inline
#endif

namespace ace {

constexpr long long kNone = (long long)0x8000000000000000ull;
constexpr int kKeyFrac = 54;                             // bits of fraction
constexpr int kKeyBias = 383;                            // a key of exponent field e: [2^(e - 383), 2^(e - 382))
constexpr long long kKeyInf = 511ll << kKeyFrac;

ACE_KEY_FN int key_clz(unsigned long long x) {  // x != 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}

// Key of an FP32 number given by its bits (exact).  A sum of squares is never negative; a set sign bit and NaN
// give kNone.
ACE_KEY_FN long long key_of_bits(unsigned b) {
  if (b > 0x7f800000u) return kNone;
  if (b == 0x7f800000u) return kKeyInf;
  if (b == 0) return 0;
  if (b < 0x800000u) {  // denormal: b 2^-149
    const int lz = key_clz(b);
    return ((long long)(63 - lz - 149 + kKeyBias) << kKeyFrac) |
           (long long)(((unsigned long long)b << (lz - 9)) & ((1ull << kKeyFrac) - 1));
  }
  return ((long long)((int)(b >> 23) - 127 + kKeyBias) << kKeyFrac) | (long long)(b & 0x7fffffu) << (kKeyFrac - 23);
}

// The key of v - p^2, p given by its FP32 bits: not below 0, and 0 when p is not finite; v < 0 stays.
ACE_KEY_FN long long key_downdate(long long v, unsigned p) {
  if (v <= 0) return v;
  p &= 0x7fffffffu;
  if (p >= 0x7f800000u) return 0;
  if (v >= kKeyInf) return v;
  const int pe = (int)(p >> 23);
  const unsigned long long pm = (p & 0x7fffffu) | (pe ? 0x800000u : 0u), sq = pm * pm;  // p = pm 2^(max(pe, 1) - 150)
  int e = (int)(v >> kKeyFrac);
  const unsigned long long m = (unsigned long long)(v & ((1ll << kKeyFrac) - 1)) | (1ull << kKeyFrac);
  // p^2 = sq 2^t in units of m's last bit
  const int t = 2 * ((pe ? pe : 1) - 150) + kKeyBias + kKeyFrac - e;
  unsigned long long r;
  if (t <= 9) {
    const int sh = 9 - t;  // sq < 2^48: no bit is lost on the left
    const unsigned long long s = (sq << 9) >> (sh < 63 ? sh : 63);
    r = s < m ? m - s : 0;
  } else {  // a normal p is larger than v here; a denormal one need not be
    const int sh = t < 63 ? t : 63;
    r = sq <= (m >> sh) ? m - (sq << sh) : 0;
  }
  if (r == 0) return 0;
  const int lz = key_clz(r) - (63 - kKeyFrac);
  e -= lz;
  return e < 1 ? 0 : ((long long)e << kKeyFrac) | (long long)((r << lz) & ((1ull << kKeyFrac) - 1));
}

// A key about 0.8 of v's value or a little more (a third of an octave below), not below 0.
ACE_KEY_FN long long key_somewhat_below(long long v) {
  const long long w = v - (1ll << kKeyFrac) / 3;
  return w > 0 ? w : 0;
}

}  // namespace ace
