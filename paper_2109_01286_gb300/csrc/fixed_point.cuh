// Fixed-point dot products for the FP64 divergence and 5-node sums.
//
// GB300 issues FP64 multiply-adds at 2 lanes per clock and SM, and 32x32+64-bit integer
// multiply-adds at 64 (measured; FP32 at 128).  A divergence row is a sum of products with one
// magnitude: its coefficients share a scale and so do the fluxes its stencil reads, so the sum
// needs no floating point.  Both factors are integers of up to 2 L - 1 bits and a sign relative to
// a power of two, split in limbs of L = 29 bits,
// a = ah 2^L + al with |ah|, |al| <= 2^(L-1), b = bh 2^L + bl with |bh| <= 2^(L-1), 0 <= bl < 2^L:
//   sum a b = 2^(2 L) sum ah bh + 2^L sum (ah bl + al bh)     (+ sum al bl, left out: below
//                                                              2^(1-2L) of the scale per product)
// is three integer multiply-adds per product instead of one DFMA: 3/64 against 1/2 clock.
// The sums of the three are exact, so they do not depend on the order of the entries or on how lanes share
// them.  The factors are rounded to 2^-57 of their row's scale and the fourth product is left out, against one
// rounding of 2^-53 of the running sum per product in FP64: over random rows of 60 to 110 products the rms
// error is 0.15 to 0.35 of the FP64 sum's, and 0.2 to 0.7 where the fluxes vary by a factor e to e^2.
// Values far below the scale lose bits: the scale has to be that of values that are added (see
// sides_in_range).
//
// Bounds: a row's coefficients take a scale of which they add up to kFxCoefSum = 127 at most, which for rows
// of up to 127 products is the largest one's; with |bh| <= 2^(L-1) the high products then add up to
// 127 2^(2L-2) and K 2^(L-1) for the roundings of K coefficients, below 2^63 = 128 2^(2L-2) for K up to
// 2^27.  A lane's cross sum takes at most 3 2^(2L-2) per product, which is below 2^63 for 42 products: a
// lane carries it over after kFxCarry.
#pragma once
#include <cuda_runtime.h>

namespace hfd {

constexpr int kSms = 152;          // SMs of a GB300, for the grids and block sizes of the kernels that use these sums
constexpr int kFxBits = 29;        // L
constexpr int kFxCoefSum = 127, kFxCarry = 40;
constexpr int kFxRaw = 0x7ff;      // code of a group stored as raw FP64 values

// A group of values with one scale has a code E: the FP64 exponent field of the largest (at least
// 1), so that |x| < 2^(E - 1022).  Groups with a value that is not finite have the code kFxRaw.
__device__ __forceinline__ int fx_code(double x) {
  const int e = (int)((unsigned)__double2hiint(x) >> 20) & 0x7ff;
  return e > 1 ? e : 1;
}

// Balanced limbs of v (coefficients).
__device__ __forceinline__ int2 fx_split(long long v, int L) {
  const long long h = (v + (1ll << (L - 1))) >> L;
  return make_int2((int)h, (int)(v - (h << L)));
}

// Exponent e with |x| < 2^e (0 for x = 0), from a double's field.
__device__ __forceinline__ int exp_above(double x) { return x == 0.0 ? -10000 : ilogb(x) + 1; }

__device__ __forceinline__ int2 coef_limbs(double c, int e, int L) {
  return fx_split(llrint(scalbn(c, 2 * L - 1 - e)), L);
}

// x at the scale of code E, as stored: the 64-bit integer x 2^(1022 - E + L - 1 + 32), truncated
// toward zero; the upper word is the high limb, the lower one the low limb and 32 - L more bits.
__device__ __forceinline__ int2 fx_encode(double x, int E, int L) {
  const int h = __double2hiint(x);
  if (E == kFxRaw) return make_int2(h, __double2loint(x));
  const int f = (h >> 20) & 0x7ff;
  unsigned long long m = ((unsigned long long)((unsigned)(h & 0xfffff) | (f ? 0x100000u : 0u)) << 32) |
                         (unsigned)__double2loint(x);
  const int s = E - (f > 1 ? f : 1);             // >= 0
  m = s < 64 ? (m << (L - 22)) >> s : 0ull;
  const long long v = h < 0 ? -(long long)m : (long long)m;
  return make_int2((int)(v >> 32), (int)(unsigned)(unsigned long long)v);
}

// The FP64 value of a stored pair (fallback rows).
__device__ __forceinline__ double fx_decode(int2 p, int E, int L) {
  if (E == kFxRaw) return __hiloint2double(p.x, p.y);
  return scalbn((double)(((long long)p.x << 32) | (unsigned)p.y), E - 1022 - (L - 1) - 32);
}

// The limbs of a stored pair at a scale d codes above its own, 0 <= d < 32.
__device__ __forceinline__ void fx_limbs(int& hi, int& lo, int d, int L) {
  lo = (int)(__funnelshift_r((unsigned)lo, (unsigned)hi, (unsigned)d) >> (32 - L));
  hi >>= d;
}

// A stored pair and its shift, for shifts of 32 or more (a value, or a zero, far below the row's).
__device__ __forceinline__ void fx_far(int& hi, int& lo, int& d) {
  if (d >= 32) {
    lo = hi;
    hi >>= 31;
    d = d - 32 < 31 ? d - 32 : 31;
  }
}

// acc += a b
__device__ __forceinline__ void fx_fma(long long& hh, long long& x, int ah, int al, int bh, int bl) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(hh) : "r"(ah), "r"(bh));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(x) : "r"(ah), "r"(bl));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(x) : "r"(al), "r"(bh));
}

// Normal form of a sum: hh 2^L + x  ->  hh' 2^L + lo with 0 <= lo < 2^L (the lo of up to 8 lanes
// then add up in 32 bits).
__device__ __forceinline__ unsigned fx_carry(long long& hh, long long x, int L) {
  hh += x >> L;
  return (unsigned)x & ((1u << L) - 1u);
}

// (hh 2^L + lo) 2^s as the nearest double (ties to even), by integer operations: GB300 converts at
// its FP64 rate.  Results outside the normal range go through scalbn.
__device__ __forceinline__ double fx_to_double(long long hh, unsigned lo, int s, int L) {
  hh += lo >> L;
  lo &= (1u << L) - 1u;
  // the leading 64 bits, with a sticky last bit for what is cut off
  const int r = __clzll(hh ^ (hh >> 63)) - 1;    // redundant sign bits of hh
  long long v;
  if (r >= L) {
    v = hh * (1ll << L) + lo;
  } else {
    const int t = L - r;
    v = hh * (1ll << r) + (lo >> t);
    v |= (lo & ((1u << t) - 1u)) ? 1ll : 0ll;
    s += t;
  }
  if (v == 0) return 0.0;
  const unsigned sign = v < 0 ? 0x80000000u : 0u;
  unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int z = __clzll((long long)m);
  m <<= z;                                       // leading bit at 63
  const unsigned rem = (unsigned)m & 0x7ffu;
  m >>= 11;                                      // 53 bits
  m += (rem > 0x400u || (rem == 0x400u && ((unsigned)m & 1u))) ? 1u : 0u;
  const int e = 63 - z + s + 1023;               // exponent field of the leading bit
  if (e < 1 || e > 2045) {
    const double d = scalbn((double)m, s + 11 - z);
    return sign ? -d : d;
  }
  // the leading bit adds one to the field (and a rounding carry one more)
  m += (unsigned long long)(unsigned)(e - 1) << 52;
  return __hiloint2double((int)((unsigned)(m >> 32) | sign), (int)(unsigned)m);
}

}  // namespace hfd
