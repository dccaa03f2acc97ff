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

// A key taken apart: m 2^(e - kKeyBias - kKeyFrac) with the leading bit of m at kKeyFrac, or m = 0 (zero and
// the marks); e from 2^20 on: infinite.
struct KeyNum {
  unsigned long long m;
  int e;
};
ACE_KEY_FN KeyNum key_open(long long v) {
  if (v <= 0) return {0, 0};
  return {(unsigned long long)(v & ((1ll << kKeyFrac) - 1)) | (1ull << kKeyFrac), v >= kKeyInf ? 1 << 20 : (int)(v >> kKeyFrac)};
}
// The key of x, for a point whose key was v before (marks stay)
ACE_KEY_FN long long key_close(KeyNum x, long long v) {
  if (v <= 0) return v;
  if (x.m == 0 || x.e < 1) return 0;
  return x.e >= 511 ? kKeyInf : ((long long)x.e << kKeyFrac) | (long long)(x.m & ((1ull << kKeyFrac) - 1));
}

// p^2 of an FP32 number given by its bits, as sq 2^t in units of the last bit of a KeyNum with exponent field 0; a p
// that is not finite has a t above every e.
struct KeySquare {
  unsigned long long sq;  // below 2^48
  int t;
};
ACE_KEY_FN KeySquare key_square(unsigned p) {
  p &= 0x7fffffffu;
  const int pe = (int)(p >> 23);  // p = pm 2^(max(pe, 1) - 150)
  const unsigned long long pm = (p & 0x7fffffu) | (pe ? 0x800000u : 0u);
  return {pm * pm, pe == 255 ? 1 << 24 : 2 * ((pe ? pe : 1) - 150) + kKeyBias + kKeyFrac};
}
// Whole units of x in p^2 (at least what x is worth where p^2 is larger)
ACE_KEY_FN unsigned long long key_units(KeyNum x, KeySquare p) {
  const int sh = x.e + 9 - p.t;
  if (sh >= 0) return (p.sq << 9) >> (sh < 63 ? sh : 63);
  // a normal p is larger than x here; a denormal one need not be
  return p.t < (1 << 23) && sh > -54 && (p.sq << 9) <= (x.m >> -sh) ? (p.sq << 9) << -sh : x.m;
}

// x - p^2: not below 0, and 0 when p is not finite; an infinite x stays for a finite p.
ACE_KEY_FN KeyNum key_less(KeyNum x, KeySquare p) {
  const unsigned long long s = key_units(x, p), r = s < x.m ? x.m - s : 0;
  const int lz = r ? key_clz(r) - (63 - kKeyFrac) : 0;
  return {r << lz, x.e - lz};
}

// x - p_0^2 - p_1^2 - ... in this order for the first `count` of R.  Where the leading bit stays in its place, which a
// look at the end tells, every step subtracts whole units of one and the same size, and their sum, taken in any order,
// goes off at once: a chain of R updates takes 70 cycles each.
template <int R>
ACE_KEY_FN KeyNum key_less_all(KeyNum x, const KeySquare (&p)[R], int count) {
  if (x.m == 0) return x;
  unsigned long long u[R];
  bool small = true;
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int sh = x.e + 9 - p[q].t;
    small = small && (q >= count || sh >= 0);
    u[q] = q < count ? (p[q].sq << 9) >> (sh < 0 ? 0 : sh < 63 ? sh : 63) : 0;
  }
#pragma unroll
  for (int w = R / 2; w > 0; w /= 2)
    for (int q = 0; q < w; ++q) u[q] += u[q + w];
  if (small && x.m >= u[0] + (1ull << kKeyFrac)) return {x.m - u[0], x.e};
  for (int q = 0; q < R; ++q)
    if (q < count) x = key_less(x, p[q]);
  return x;
}

// The key of v - p^2 for the key v
ACE_KEY_FN long long key_downdate(long long v, unsigned p) { return key_close(key_less(key_open(v), key_square(p)), v); }

// A key about 0.8 of v's value or a little more (a third of an octave below), not below 0.
ACE_KEY_FN long long key_somewhat_below(long long v) {
  const long long w = v - (1ll << kKeyFrac) / 3;
  return w > 0 ? w : 0;
}

}  // namespace ace
