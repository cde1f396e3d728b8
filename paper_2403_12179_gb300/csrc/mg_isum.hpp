// The FP64 arithmetic of the stencils on the integer units, bit for bit.
//
// GB300 issues FP64 instructions at 1.68 lanes per clock and SM (measured: 528 G lane
// operations/s), so one warp-wide FP64 addition holds the FP64 pipe as long as about 76 issue
// slots of each SM quarter.  An exact integer form of the same rounded operation costs 20 to 30
// instructions, and the two kinds run side by side: the stencil kernels give some of their
// operations to the integer units.  Every function states when it applies and returns false
// otherwise; the caller then uses the FP64 instruction, whose result the integer form equals
// bit for bit wherever it applies.  The header also compiles for the host (a C++ test checks it
// against the host compiler's own arithmetic).
#pragma once

#include "mg_bits.hpp"

namespace gbmg {
namespace isum {

using bits::d2u;
using bits::u2d;

GB_HD int msb32(uint32_t x) {  // index of the highest set bit, -1 for 0
#ifdef __CUDA_ARCH__
  int r;
  asm("bfind.u32 %0, %1;" : "=r"(r) : "r"(x));
  return r;
#else
  return x ? 31 - __builtin_clz(x) : -1;
#endif
}
GB_HD uint32_t umax(uint32_t a, uint32_t b) { return a > b ? a : b; }
GB_HD uint32_t umin(uint32_t a, uint32_t b) { return a < b ? a : b; }
GB_HD uint32_t mulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

// The sum of six addends, ((((v0 + v1) + v2) + v3) + v4) + v5, each addition rounded to nearest
// even, as one fixed-point sum: the mantissas are placed relative to the largest exponent (its
// leading one at bit 52 + kGuard, which with 3 bits of growth and the sign fills 63 bits), so an
// addition is one integer addition, and its rounding drops the bits below the 53rd from the sum's
// leading one.
constexpr int kGuard = 7;
GB_HD uint32_t shr_pair(uint32_t lo, uint32_t hi, uint32_t d) {  // low word of (hi:lo) >> (d mod 32)
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, d);
#else
  return (uint32_t)(((uint64_t)hi << 32 | lo) >> (d & 31u));
#endif
}
GB_HD uint32_t shl_pair(uint32_t lo, uint32_t hi, uint32_t d) {  // high word of (hi:lo) << (d mod 32)
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, d);
#else
  return (uint32_t)(((uint64_t)hi << 32 | lo) << (d & 31u) >> 32);
#endif
}

// What the six values allow, from their high words.
struct Six {
  uint32_t a[6];    // magnitudes' high words
  uint32_t em;      // the largest one's exponent field, in place
  uint32_t mn;      // the smallest of a
  uint32_t signs;   // bit 31 set: not all of one sign
  bool range;       // the largest exponent is away from the ends of the range
  GB_HD bool close() const { return mn + ((uint32_t)(kGuard - 1) << 20) >= em; }
};
GB_HD Six six_of(const double (&v)[6]) {
  Six q;
  uint32_t h[6];
  for (int i = 0; i < 6; ++i) {
    h[i] = (uint32_t)(d2u(v[i]) >> 32);
    q.a[i] = h[i] & 0x7FFFFFFFu;
  }
  const uint32_t mx = umax(umax(umax(q.a[0], q.a[1]), q.a[2]), umax(umax(q.a[3], q.a[4]), q.a[5]));
  q.mn = umin(umin(umin(q.a[0], q.a[1]), q.a[2]), umin(umin(q.a[3], q.a[4]), q.a[5]));
  q.em = mx & 0x7FF00000u;
  q.signs = (h[0] ^ h[1]) | (h[0] ^ h[2]) | (h[0] ^ h[3]) | (h[0] ^ h[4]) | (h[0] ^ h[5]);
  q.range = (q.em - (128u << 20)) < (1912u << 20);
  return q;
}

// Six addends of one sign within kGuard - 1 binary orders of each other (and so normal): the sum
// of magnitudes, about half the instructions of the general form.  Always exact.
GB_HD bool six_simple(const Six& q) { return q.range && q.close() && (int32_t)q.signs >= 0; }
GB_HD double sum6_simple(const double (&v)[6], const Six& q) {
  const uint32_t base = ((uint32_t)kGuard << 20) - q.em;
  uint64_t p = 0;
  int k = 1;
  for (int i = 0; i < 6; ++i) {
    const uint64_t u = d2u(v[i]);
    const uint32_t s = (q.a[i] + base) >> 20;  // 1 .. kGuard
    const uint32_t mh = ((uint32_t)(u >> 32) & 0xFFFFFu) | 0x100000u, ml = (uint32_t)u;
    p += (uint64_t)shl_pair(ml, mh, s) << 32 | (uint32_t)(ml << (s & 31u));
    if (i == 0) continue;
    // round to nearest even at bit k (bit 0 is always clear, so k = 1 changes nothing)
    const int f = msb32((uint32_t)(p >> 32)) - 20;
    k = f > 1 ? f : 1;
    const uint32_t one = 1u << k, pl = (uint32_t)p;
    p += (one >> 1) - 1u + ((pl >> k) & 1u);
    p &= ~(uint64_t)(one - 1u);
  }
  p >>= k;  // 53 bits (2^53 after a carry)
  const uint32_t h = ((uint32_t)(d2u(v[0]) >> 32) & 0x80000000u) |
                     (q.em + ((uint32_t)(k - (kGuard + 1)) << 20) + (uint32_t)(p >> 32));
  return u2d((uint64_t)h << 32 | (uint32_t)p);
}

// Addends of any sign up to 31 binary orders below the largest.  One kGuard or more orders below
// it loses bits off the bottom; they are kept as one sticky bit, which decides the rounding
// rightly as long as at least two bits are dropped.  False (and *out not set to the sum) unless all are
// normal, the result is at least the largest addend times 2^-kGuard (no deep cancellation, no
// zero), and, where an addend is kGuard or more orders below the largest, every partial sum is
// at least the largest times 2^(2 - kGuard).
GB_HD bool sum6(const double (&v)[6], const Six& q, double* out) {
  const uint32_t top = q.em | 0xFFFFFu;
  bool ok = q.range && q.mn + (31u << 20) >= q.em;
  int64_t p = 0;
  int k = 1, f = 0, fmin = 64;
  for (int i = 0; i < 6; ++i) {
    const uint64_t u = d2u(v[i]);
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
    const uint32_t d = (top - q.a[i]) >> 20;  // binary orders below the largest
    const uint32_t mh = (hi & 0xFFFFFu) | 0x100000u;
    const uint32_t xh = shl_pair(lo, mh, kGuard), xl = lo << kGuard;
    const uint32_t lost = shr_pair(0u, xl, d);  // the bits below bit 0, left-aligned
    const uint32_t sl = shr_pair(xl, xh, d) | umin(lost, 1u), sh = shr_pair(xh, 0u, d);
    const int64_t sg = (int64_t)((int32_t)hi >> 31);
    p += (int64_t)(((uint64_t)sh << 32 | sl) ^ (uint64_t)sg) - sg;
    if (i == 0) continue;
    // round to nearest even at bit k; where bit 0 is the lowest kept one it is clear (no addend
    // reaches it), so k = 1 changes nothing
    const uint32_t ph = (uint32_t)((uint64_t)p >> 32);
    f = msb32(ph ^ (uint32_t)((int32_t)ph >> 31)) - 20;
    fmin = f < fmin ? f : fmin;
    k = f > 1 ? f : 1;
    const uint32_t pl = (uint32_t)p, one = 1u << k;
    p += (int64_t)(uint64_t)((one >> 1) - 1u + ((pl >> k) & 1u));
    p = (int64_t)((uint64_t)p & ~(uint64_t)(one - 1u));
  }
  ok = ok && f >= 1 && (q.close() || fmin >= 2);
  const int64_t sg = p >> 63;
  const uint64_t r = (uint64_t)((p ^ sg) - sg) >> k;  // 53 bits (2^53 after a carry)
  const uint32_t h = ((uint32_t)sg & 0x80000000u) |
                     (q.em + ((uint32_t)(k - (kGuard + 1)) << 20) + (uint32_t)(r >> 32));
  *out = u2d((uint64_t)h << 32 | (uint32_t)r);
  return ok;
}

// t * (1/6 rounded to binary64), rounded to nearest even.  That constant is
// (2^54 - 1) / 3 * 2^-55, so with t's 53-bit mantissa m the exact product's mantissa is
// (4m - m / 2^52) / 3 or half of it, which rounds to floor(4m / 3), or to half of that rounded
// down where it needs 54 bits: with d = m / 2^52 in [1, 2) and 4m = 3q + r, (r - d) / 3 lies in
// [-1/2, 1/3] for m <= 3 * 2^51 (the one tie, at 3 * 2^51, rounds to the even q = 2^53), and
// with 2m = 3q + r, (r - d/2) / 3 lies in (-1/3, 1/2) for larger m (there d >= 3/2).  Applies when t
// and the product are normal.
GB_HD bool mul_sixth(double t, double* out) {
  const uint64_t u = d2u(t);
  const uint32_t hi = (uint32_t)(u >> 32), ml = (uint32_t)u;
  const uint32_t mh = (hi & 0xFFFFFu) | 0x100000u;
  // m / 3, from 2^32 = 3 * 0x55555555 + 1
  const uint32_t qh = mulhi(mh, 0x55555556u);
  const uint32_t b = mh - 3u * qh;
  const uint32_t a = mulhi(ml, 0xAAAAAAABu) >> 1;
  const uint32_t r = ml - 3u * a;
  const uint32_t ql = b * 0x55555555u + a + (b + r >= 3u ? 1u : 0u);
  const uint64_t q = ((uint64_t)mh << 32 | ml) + ((uint64_t)qh << 32 | ql);  // floor(4m / 3)
  const uint32_t c = (uint32_t)(q >> 53);                                   // 54 bits: 1
  const uint64_t s = q >> c;
  const uint32_t e = hi & 0x7FF00000u;
  // biased exponent - 3 (+ 1 with c); the mantissa's leading one adds 1
  const uint32_t h = (hi & 0x80000000u) | (e + (c << 20) - (4u << 20) + (uint32_t)(s >> 32));
  *out = u2d((uint64_t)h << 32 | (uint32_t)s);
  return (e - (4u << 20)) < (0x7FFu - 4u) << 20;
}

}  // namespace isum
}  // namespace gbmg
