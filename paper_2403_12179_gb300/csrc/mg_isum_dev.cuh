// Device side of mg_isum.hpp: the FP64 sum of six and Gauss-Seidel update with their fallbacks.
#pragma once

#include "mg_isum.hpp"

namespace gbmg {

__device__ __forceinline__ double flip(double v, unsigned n) {  // -v if n is 1
  unsigned lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(v));
  double r;
  asm("mov.b64 %0, {%1, %2};" : "=d"(r) : "r"(lo), "r"(hi ^ (n << 31)));
  return r;
}
// f(x), in a block of its own: a loop over blockDim.y (1 in every launch here, which the compiler
// does not know), each turn of which would take the last one's result.  Written as a plain
// condition, the few FP64 instructions of a rare case are predicated instead of branched around,
// and instructions that are off in all lanes hold the FP64 pipe like any others.
template <class F>
__device__ __forceinline__ double rarely(double x, F&& f) {
  int n = blockDim.y;
#pragma unroll 1
  do x = f(x);
  while (--n > 0);
  return x;
}
__device__ __forceinline__ double sum6_f64(const double (&v)[6]) {
  double s = __dadd_rn(v[0], v[1]);
  s = __dadd_rn(s, v[2]);
  s = __dadd_rn(s, v[3]);
  s = __dadd_rn(s, v[4]);
  return __dadd_rn(s, v[5]);
}
// The six-addend sum on the integer units (every lane of mask calls it together).
__device__ __forceinline__ double sum6_int(const double (&v)[6], unsigned mask) {
  const isum::Six q = isum::six_of(v);
  if (__all_sync(mask, isum::six_simple(q))) return isum::sum6_simple(v, q);
  double s;
  if (!isum::sum6(v, q, &s))
    s = rarely(v[0], [&](double x) {
      const double w[6] = {x, v[1], v[2], v[3], v[4], v[5]};
      return sum6_f64(w);
    });
  return s;
}
template <bool INT>
__device__ __forceinline__ double sum6(const double (&v)[6], unsigned mask) {
  return INT ? sum6_int(v, mask) : sum6_f64(v);
}
template <bool INT>
__device__ __forceinline__ double gs_update(double s, double rhs, double mh2) {
  const double t = __fma_rn(mh2, rhs, s);
  double u;
  if (!INT) return __dmul_rn(t, 1.0 / 6.0);
  if (!isum::mul_sixth(t, &u)) u = rarely(t, [&](double x) { return __dmul_rn(x, 1.0 / 6.0); });
  return u;
}

}  // namespace gbmg
