// FP64 half-sweep and residual that march through the planes of a box (sm_103a).
//
// What bounds these kernels is the FP64 pipe: GB300 issues 1.68 FP64 lanes per clock and SM, so 7
// FP64 instructions a cell at 100% of it take 111 us for a half-sweep and 222 us for a residual of
// 256^3 cells, against 56 us and 60 us for their bytes at the copy rate.  Two things take them below
// that:
//   * a thread owns a pair of cells in x and marches in z, so that a plane costs one load for the
//     column above (z neighbours and the pair's inner x neighbour stay in registers, the outer x
//     neighbour comes by shuffle from the next lane), one for each y neighbour and one for rhs, all
//     issued a plane ahead; rows at box faces read the neighbouring box (or image, or negated
//     boundary cell) through DRow::nbd / nbf, as the row kernels do;
//   * every second cell's six-addend sum, and every update's product with 1/6, is computed on the
//     integer units (mg_isum.hpp), which run beside the FP64 pipe; results are the same bit for bit.
// Measured on GB300 at 256^3 (64 boxes of 64^3; row kernels of mg_kernels.cu before): half-sweep 130
// -> 88 us (marching alone 121), residual 238 -> 182 us; at 128^3 in boxes of 32^3 21 -> 13.5 and
// 36 -> 30 us; 256^3 FP64 solve 19.5 -> 15.1 ms.  Now FP64 pipe (57%), integer ALU (60%) and
// load latency share the time.  All sums in integers: 114 us; two rows a thread (96 registers): 88
// us, slower on small levels; 256 threads at 64 registers: 92 us; the norm and residual-storing
// half-sweeps run best at 5 blocks an SM (no spills), the residual at 4.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "mg_isum_dev.cuh"
#include "mg_kernels.hpp"

namespace gbmg {

namespace {

constexpr int kMarchThreads = 128;

__device__ __forceinline__ unsigned long long abskey(double a) {
  unsigned lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(a));
  return ((unsigned long long)(hi & 0x7FFFFFFFu) << 32) | lo;
}
__device__ __forceinline__ double residual_of(double s, double phi, double rhs, double mih2) {
  return __fma_rn(mih2, __fma_rn(-6.0, phi, s), rhs);
}

template <int V>
struct Int {
  static constexpr int value = V;
};

// Max over the block's threads into *norm.
__device__ __forceinline__ void block_max(unsigned long long mx, unsigned long long* norm) {
  __shared__ unsigned long long sm[kMarchThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = w > mx ? w : mx;
  }
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kMarchThreads / 32; ++w) mx = sm[w] > mx ? sm[w] : mx;
    if (mx) atomicMax(norm, mx);
  }
}

template <class T>
__device__ __forceinline__ T* at(T* p, long long bytes) {
  return (T*)((uintptr_t)p + bytes);
}

// Box b of the launch; *slot: its segment's norm slot.  MULTI: the launch has several segments.
template <bool MULTI>
__device__ __forceinline__ const DRow& box_row(const SegList& L, int b, int* slot) {
  if (!MULTI) {
    *slot = L.one.slot;
    return L.one.rows[b];
  }
  Seg S;
  {
    int lo = 0, hi = L.n - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (L.segs[mid].box_begin <= b) lo = mid; else hi = mid - 1;
    }
    S = L.segs[lo];
    b -= S.box_begin;
  }
  *slot = S.slot;
  return S.rows[b];
}

// The half-sweep (x extents even).  MODE as in k_rbgs_half: 0 plain; 1 max-norm of each updated
// cell's residual after its update; 2 before it, saving the value before to v[2]; 3 the residual
// after the update stored to v[2] (one-colour views).
template <int MODE, bool INT, bool MULTI = false>
__global__ void __launch_bounds__(kMarchThreads, MODE ? 5 : 7)
    k_half_march(SegList L, int zc, int color, unsigned long long* norms) {
  pdl_begin();
  int slot;
  const DRow& R = box_row<MULTI>(L, blockIdx.y, &slot);
  const int nx = R.n[0], ny = R.n[1], nz = R.n[2];
  const int pp = nx >> 1, rb = kMarchThreads / pp;
  const int nty = (ny + rb - 1) / rb, ntz = (nz + zc - 1) / zc;
  const int tile = blockIdx.x;
  if (tile >= nty * ntz) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int ry = tid / pp, i = tid - ry * pp;
  const int y = (tile % nty) * rb + ry;
  const int z0 = (tile / nty) * zc, z1 = min(z0 + zc, nz);
  const bool active = ry < rb && y < ny;
  const unsigned mask = __ballot_sync(0xffffffffu, active);
  unsigned long long mx = 0;
  if (active) {
    const int pitch = R.v[0].pitch;
    const long long plane = R.v[0].plane;
    const unsigned nbf = (unsigned)R.nbf;
    const double mh2 = flip(R.h2, 1u), mih2 = flip(R.ih2, 1u);
    // place in the pair of the updated cell: pe in planes z0, z0 + 2, ..., pe ^ 1 in the others
    const int pe = (color + R.lo[0] + R.lo[1] + R.lo[2] + y + z0) & 1, po = pe ^ 1;
    double* own = (double*)R.v[0].p + z0 * plane + (long long)y * pitch + 2 * i + pe;
    // byte steps from an even plane's cell to the next plane's, and from an odd one's
    const int swap = (po - pe) * 8;
    const long long ie = plane * 8 + swap, io = plane * 8 - swap;
    const long long re = R.v[1].plane * 8 + swap, ro = R.v[1].plane * 8 - swap;
    const double* pn = own + plane;  // the other colour's cell above
    const double* pym = own - pitch + (y == 0 ? R.nbd[2] : 0);
    const double* pyp = own + pitch + (y == ny - 1 ? R.nbd[3] : 0);
    const double* pf = (const double*)R.v[1].p + z0 * R.v[1].plane + (long long)y * R.v[1].pitch + 2 * i + pe;
    const unsigned nym = y == 0 ? (nbf >> 2) & 1u : 0u, nyp = y == ny - 1 ? (nbf >> 3) & 1u : 0u;
    double* sv = nullptr;
    long long is = 0;
    if (MODE == 2 || MODE == 3) {
      is = R.v[2].plane * 8;
      sv = (double*)R.v[2].p + z0 * R.v[2].plane + (long long)y * R.v[2].pitch + i;
    }
    // outer x neighbour: the next pair's cell from its lane, or loaded at row ends and warp ends
    const bool exl = i == 0, exr = i == pp - 1;
    const bool lde = pe ? exr || lane == 31 : exl || lane == 0, ldo = pe ? exl || lane == 0 : exr || lane == 31;
    const unsigned nxl = exl ? nbf & 1u : 0u, nxr = exr ? (nbf >> 1) & 1u : 0u;
    const unsigned nxe = pe ? nxr : nxl, nxo = pe ? nxl : nxr;
    const int srce = pe ? lane + 1 : lane - 1, srco = pe ? lane - 1 : lane + 1;
    const long long dl = (exl ? R.nbd[0] : 0) - 1, dr = (exr ? R.nbd[1] : 0) + 1;  // from the updated cell
    const long long dxe = (pe ? dr : dl) * 8, dxo = (pe ? dl : dr) * 8;
    const double* px = own;  // updated cell of the step being loaded
    const unsigned nzm = (nbf >> 4) & 1u, nzp = (nbf >> 5) & 1u;
    const long long dz1 = R.nbd[5] * 8;
    // the other colour's cell of the column below and beside the updated one
    double cm = flip(own[-plane + (z0 == 0 ? R.nbd[4] : 0)], z0 == 0 ? nzm : 0u);
    double cc = own[po - pe];
    struct In {
      double n, ym, yp, f, x, o;
    };
    auto load = [&](auto Ec, int z, In& v) {  // inputs of step z; the pointers move on to z + 1
      constexpr int E = decltype(Ec)::value;  // 0: even step
      if (z == nz - 1) pn = at(pn, dz1);
      v.n = *pn;
      v.ym = *pym;
      v.yp = *pyp;
      v.f = *pf;
      if (E ? ldo : lde) v.x = *at(px, E ? dxo : dxe);
      if (MODE == 2) v.o = *px;
      pn = at(pn, E ? io : ie);
      pym = at(pym, E ? io : ie);
      pyp = at(pyp, E ? io : ie);
      pf = at(pf, E ? ro : re);
      px = at(px, E ? io : ie);
    };
    auto step = [&](auto Ec, int z, const In& v) {
      constexpr int E = decltype(Ec)::value;
      double xo = __shfl_sync(mask, cc, E ? srco : srce);
      if (E ? ldo : lde) xo = flip(v.x, E ? nxo : nxe);
      const double cn = z == nz - 1 ? flip(v.n, nzp) : v.n;
      double w[6] = {xo, cc, flip(v.ym, nym), flip(v.yp, nyp), cm, cn};
      const double s = sum6<INT && E>(w, mask);
      const double un = gs_update<INT>(s, v.f, mh2);
      if (MODE == 2) {
        const unsigned long long k = abskey(residual_of(s, v.o, v.f, mih2));
        mx = k > mx ? k : mx;
        *sv = v.o;
      }
      *own = un;
      if (MODE == 1 || MODE == 3) {
        double s2 = s;
        const unsigned sx = (E ? ldo : lde) ? (E ? nxo : nxe) : 0u;
        const unsigned sm = z == 0 ? nzm : 0u, sp = z == nz - 1 ? nzp : 0u;
        if (sx | nym | nyp | sm | sp) {  // reads of its own value, negated
          const double m = flip(un, 1u);
          if (sx) w[0] = m;
          if (nym) w[2] = m;
          if (nyp) w[3] = m;
          if (sm) w[4] = m;
          if (sp) w[5] = m;
          s2 = rarely(w[0], [&](double x) {
            const double q[6] = {x, w[1], w[2], w[3], w[4], w[5]};
            return sum6_f64(q);
          });
        }
        const double r = residual_of(s2, un, v.f, mih2);
        if (MODE == 3) *sv = r;
        if (MODE == 1) {
          const unsigned long long k = abskey(r);
          mx = k > mx ? k : mx;
        }
      }
      if (MODE == 2 || MODE == 3) sv = at(sv, is);
      own = at(own, E ? io : ie);
      cm = cc;
      cc = cn;
    };
    In a, b;
    load(Int<0>{}, z0, a);
    for (int z = z0; z < z1; z += 2) {
      if (z + 1 < z1) load(Int<1>{}, z + 1, b);
      step(Int<0>{}, z, a);
      if (z + 1 < z1) {
        if (z + 2 < z1) load(Int<0>{}, z + 2, a);
        step(Int<1>{}, z + 1, b);
      }
    }
  }
  if (MODE == 1 || MODE == 2) block_max(mx, &norms[slot + R.solve]);
}

// Residual of every cell (stored if v[2] is set) and its max-norm into norms (if set); any x extent.
template <bool INT, bool MULTI>
__global__ void __launch_bounds__(kMarchThreads, 4)
    k_residual_march(SegList L, int zc, unsigned long long* norms) {
  pdl_begin();
  int slot;
  const DRow& R = box_row<MULTI>(L, blockIdx.y, &slot);
  const int nx = R.n[0], ny = R.n[1], nz = R.n[2];
  const int pp = (nx + 1) >> 1, rb = kMarchThreads / pp;
  const int nty = (ny + rb - 1) / rb, ntz = (nz + zc - 1) / zc;
  const int tile = blockIdx.x;
  if (tile >= nty * ntz) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int ry = tid / pp, i = tid - ry * pp;
  const int y = (tile % nty) * rb + ry;
  const int z0 = (tile / nty) * zc, z1 = min(z0 + zc, nz);
  const bool active = ry < rb && y < ny;
  const unsigned mask = __ballot_sync(0xffffffffu, active);
  unsigned long long mx = 0;
  if (active) {
    const bool two = 2 * i + 1 < nx;  // the pair's second cell exists
    const int pitch = R.v[0].pitch;
    const long long plane = R.v[0].plane, ip = plane * 8, ir = R.v[1].plane * 8, io = R.v[2].plane * 8;
    const unsigned nbf = (unsigned)R.nbf;
    const double mih2 = flip(R.ih2, 1u);
    const double* own = (const double*)R.v[0].p + z0 * plane + (long long)y * pitch + 2 * i;
    const double* pn = own + plane;
    const double* pym = own - pitch + (y == 0 ? R.nbd[2] : 0);
    const double* pyp = own + pitch + (y == ny - 1 ? R.nbd[3] : 0);
    const double* pf = (const double*)R.v[1].p + z0 * R.v[1].plane + (long long)y * R.v[1].pitch + 2 * i;
    double* out = R.v[2].p ? (double*)R.v[2].p + z0 * R.v[2].plane + (long long)y * R.v[2].pitch + 2 * i : nullptr;
    const unsigned nym = y == 0 ? (nbf >> 2) & 1u : 0u, nyp = y == ny - 1 ? (nbf >> 3) & 1u : 0u;
    // outer x neighbours: the next pairs' cells from their lanes, or loaded at row and warp ends
    const bool exl = i == 0, exr = i == pp - 1, ldl = exl || lane == 0, ldr = exr || lane == 31;
    const unsigned nxl = exl ? nbf & 1u : 0u, nxr = exr ? (nbf >> 1) & 1u : 0u;
    const double* pxl = own - 1 + (exl ? R.nbd[0] : 0);
    const double* pxr = own + (two ? 2 : 1) + (exr ? R.nbd[1] : 0);
    const unsigned nzm = (nbf >> 4) & 1u, nzp = (nbf >> 5) & 1u;
    const long long dz1 = R.nbd[5] * 8;
    const double* below = own - plane + (z0 == 0 ? R.nbd[4] : 0);
    const unsigned nb = z0 == 0 ? nzm : 0u;
    double m0 = flip(below[0], nb), m1 = flip(below[1], nb);
    double c0 = own[0], c1 = own[1];
    struct In {
      double n0, n1, ym0, ym1, yp0, yp1, f0, f1, xl, xr;
    };
    auto load = [&](int z, In& v) {
      if (z == nz - 1) pn = at(pn, dz1);
      v.n0 = pn[0];
      v.n1 = pn[1];
      v.ym0 = pym[0];
      v.ym1 = pym[1];
      v.yp0 = pyp[0];
      v.yp1 = pyp[1];
      v.f0 = pf[0];
      v.f1 = two ? pf[1] : 0.0;
      if (ldl) v.xl = *pxl;
      if (ldr) v.xr = *pxr;
      pn = at(pn, ip);
      pym = at(pym, ip);
      pyp = at(pyp, ip);
      pxl = at(pxl, ip);
      pxr = at(pxr, ip);
      pf = at(pf, ir);
    };
    auto step = [&](int z, const In& v) {
      double xl = __shfl_sync(mask, c1, lane - 1), xr = __shfl_sync(mask, c0, lane + 1);
      if (ldl) xl = flip(v.xl, nxl);
      if (ldr) xr = flip(v.xr, nxr);
      const bool zend = z == nz - 1;
      const double n0 = zend ? flip(v.n0, nzp) : v.n0, n1 = zend ? flip(v.n1, nzp) : v.n1;
      const double w0[6] = {xl, two ? c1 : xr, flip(v.ym0, nym), flip(v.yp0, nyp), m0, n0};
      const double w1[6] = {c0, xr, flip(v.ym1, nym), flip(v.yp1, nyp), m1, n1};
      const double s0 = sum6<false>(w0, mask), s1 = sum6<INT>(w1, mask);
      const double r0 = residual_of(s0, c0, v.f0, mih2), r1 = residual_of(s1, c1, v.f1, mih2);
      unsigned long long k = abskey(r0);
      mx = k > mx ? k : mx;
      k = abskey(r1);
      if (two) mx = k > mx ? k : mx;
      if (out) {
        out[0] = r0;
        if (two) out[1] = r1;
        out = at(out, io);
      }
      m0 = c0;
      m1 = c1;
      c0 = n0;
      c1 = n1;
    };
    In a, b;
    load(z0, a);
    for (int z = z0; z < z1; z += 2) {
      if (z + 1 < z1) load(z + 1, b);
      step(z, a);
      if (z + 1 < z1) {
        if (z + 2 < z1) load(z + 2, a);
        step(z + 1, b);
      }
    }
  }
  if (norms) block_max(mx, &norms[slot + R.solve]);
}

// Residual + restriction (even extents and box corners): a thread owns a coarse column, i.e. a pair of
// cells in rows 2Y (A) and 2Y + 1 (B), and marches through planes; crhs = (sum of the 8 children's
// residuals, x fastest) / 8, cphi = 0 (if c[1] is set).  STORED: the black children's residuals are
// read from v[2] (one-colour view), only the red ones computed.  Row B's sums run on the integer
// units.  FP64-pipe bound like the kernels above: 256^3 level of the FP64 solve (STORED) 186 -> 133 us
// against a lane per coarse cell, 128^3 level 45 -> 37 us, 16^3 level 10.5 -> 7.1 us (ncu, cold); the
// 256^3 solve 15.1 -> 14.0 ms.
template <bool STORED, bool INT, bool MULTI>
__global__ void __launch_bounds__(kMarchThreads, 4) k_restrict_march(SegList L, int zc) {
  pdl_begin();
  int slot;
  const DRow& R = box_row<MULTI>(L, blockIdx.y, &slot);
  const int pp = R.n[0] >> 1, ny = R.n[1], nz = R.n[2], nc1 = ny >> 1, rb = kMarchThreads / pp;
  const int nty = (nc1 + rb - 1) / rb, ntz = (nz + zc - 1) / zc;
  const int tile = blockIdx.x;
  if (tile >= nty * ntz) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int ry = tid / pp, i = tid - ry * pp, Y = (tile % nty) * rb + ry, y = 2 * Y;
  const int z0 = (tile / nty) * zc, z1 = min(z0 + zc, nz);  // (zc even)
  const bool active = ry < rb && Y < nc1;
  const unsigned mask = __ballot_sync(0xffffffffu, active);
  if (!active) return;
  const int pitch = R.v[0].pitch;
  const long long ip = R.v[0].plane * 8, ir = R.v[1].plane * 8, dB = (long long)pitch * 8,
                  dfB = (long long)R.v[1].pitch * 8;
  const unsigned nbf = (unsigned)R.nbf;
  const double mih2 = flip(R.ih2, 1u);
  const double* own = (const double*)R.v[0].p + z0 * R.v[0].plane + (long long)y * pitch + 2 * i;
  const double* pf = (const double*)R.v[1].p + z0 * R.v[1].plane + (long long)y * R.v[1].pitch + 2 * i;
  const double* pym = own - pitch + (y == 0 ? R.nbd[2] : 0);
  const double* pyp = own + 2 * pitch + (y == ny - 2 ? R.nbd[3] : 0);
  const unsigned nym = y == 0 ? (nbf >> 2) & 1u : 0u, nyp = y == ny - 2 ? (nbf >> 3) & 1u : 0u;
  const double* st = nullptr;
  long long is = 0, dsB = 0;
  if (STORED) {
    is = R.v[2].plane * 8;
    dsB = R.v[2].pitch * 8;
    st = (const double*)R.v[2].p + z0 * R.v[2].plane + (long long)y * R.v[2].pitch + i;
  }
  double* cr = (double*)R.c[0].p + (z0 >> 1) * R.c[0].plane + (long long)Y * R.c[0].pitch + i;
  double* cp = R.c[1].p ? (double*)R.c[1].p + (z0 >> 1) * R.c[1].plane + (long long)Y * R.c[1].pitch + i : nullptr;
  const bool exl = i == 0, exr = i == pp - 1, ldl = exl || lane == 0, ldr = exr || lane == 31;
  const unsigned nxl = exl ? nbf & 1u : 0u, nxr = exr ? (nbf >> 1) & 1u : 0u;
  const double* pxl = own - 1 + (exl ? R.nbd[0] : 0);
  const double* pxr = own + 2 + (exr ? R.nbd[1] : 0);
  const unsigned nzm = (nbf >> 4) & 1u, nzp = (nbf >> 5) & 1u;
  const long long dz1 = R.nbd[5] * 8;
  const double* below = own - R.v[0].plane + (z0 == 0 ? R.nbd[4] : 0);
  const unsigned nb = z0 == 0 ? nzm : 0u;
  double acc = 0.0;
  if constexpr (STORED) {
    // box corners are even: the red cell of row A sits at place 0 of the pair in even planes, at 1 in odd
    // ones, row B's at the other place; mX / cX: the black cells below and beside them
    double mA = flip(below[0], nb), mB = flip(at(below, dB)[1], nb);
    double cA = own[1], cB = at(own, dB)[0];
    struct In {
      double nA, nB, ym, yp, fA, fB, oA, oB, sA, sB, xA, xB;
    };
    auto load = [&](auto Kc, int z, In& v) {
      constexpr int K = decltype(Kc)::value;
      const long long o = (long long)(z - z0) * ip;
      const double* up = at(own, o + ip + (z == nz - 1 ? dz1 : 0));
      const double* c = at(own, o);
      const double* f = at(pf, (long long)(z - z0) * ir);
      const double* t = at(st, (long long)(z - z0) * is);
      v.nA = up[K];
      v.nB = at(up, dB)[K ^ 1];
      v.ym = at(pym, o)[K];
      v.yp = at(pyp, o)[K ^ 1];
      v.fA = f[K];
      v.fB = at(f, dfB)[K ^ 1];
      v.oA = c[K];
      v.oB = at(c, dB)[K ^ 1];
      v.sA = *t;
      v.sB = *at(t, dsB);
      if (K ? ldr : ldl) v.xA = *at(K ? pxr : pxl, o);
      if (K ? ldl : ldr) v.xB = *at(K ? pxl : pxr, o + dB);
    };
    auto step = [&](auto Kc, int z, const In& v) {
      constexpr int K = decltype(Kc)::value;
      double xA = __shfl_sync(mask, cA, K ? lane + 1 : lane - 1), xB = __shfl_sync(mask, cB, K ? lane - 1 : lane + 1);
      if (K ? ldr : ldl) xA = flip(v.xA, K ? nxr : nxl);
      if (K ? ldl : ldr) xB = flip(v.xB, K ? nxl : nxr);
      const unsigned e = z == nz - 1 ? nzp : 0u;
      const double nA = flip(v.nA, e), nB = flip(v.nB, e);
      const double wA[6] = {xA, cA, flip(v.ym, nym), cB, mA, nA}, wB[6] = {xB, cB, cA, flip(v.yp, nyp), mB, nB};
      const double rA = residual_of(sum6<false>(wA, mask), v.oA, v.fA, mih2);
      const double rB = residual_of(sum6<INT>(wB, mask), v.oB, v.fB, mih2);
      acc = K ? __dadd_rn(acc, v.sA) : __dadd_rn(rA, v.sA);
      if (K) acc = __dadd_rn(acc, rA);
      acc = __dadd_rn(acc, K ? rB : v.sB);
      acc = __dadd_rn(acc, K ? v.sB : rB);
      mA = cA;
      cA = nA;
      mB = cB;
      cB = nB;
    };
    In a, b;
    load(Int<0>{}, z0, a);
    for (int z = z0; z < z1; z += 2) {
      load(Int<1>{}, z + 1, b);
      step(Int<0>{}, z, a);
      if (z + 2 < z1) load(Int<0>{}, z + 2, a);
      step(Int<1>{}, z + 1, b);
      *cr = __dmul_rn(acc, 0.125);
      cr += R.c[0].plane;
      if (cp) {
        *cp = 0.0;
        cp += R.c[1].plane;
      }
    }
  } else {
    double mA0 = flip(below[0], nb), mA1 = flip(below[1], nb);
    double mB0 = flip(at(below, dB)[0], nb), mB1 = flip(at(below, dB)[1], nb);
    double cA0 = own[0], cA1 = own[1], cB0 = at(own, dB)[0], cB1 = at(own, dB)[1];
    struct In {
      double nA0, nA1, nB0, nB1, ym0, ym1, yp0, yp1, fA0, fA1, fB0, fB1, lA, lB, rA, rB;
    };
    auto load = [&](int z, In& v) {
      const long long o = (long long)(z - z0) * ip;
      const double* up = at(own, o + ip + (z == nz - 1 ? dz1 : 0));
      const double* f = at(pf, (long long)(z - z0) * ir);
      v.nA0 = up[0];
      v.nA1 = up[1];
      v.nB0 = at(up, dB)[0];
      v.nB1 = at(up, dB)[1];
      v.ym0 = at(pym, o)[0];
      v.ym1 = at(pym, o)[1];
      v.yp0 = at(pyp, o)[0];
      v.yp1 = at(pyp, o)[1];
      v.fA0 = f[0];
      v.fA1 = f[1];
      v.fB0 = at(f, dfB)[0];
      v.fB1 = at(f, dfB)[1];
      if (ldl) {
        v.lA = *at(pxl, o);
        v.lB = *at(pxl, o + dB);
      }
      if (ldr) {
        v.rA = *at(pxr, o);
        v.rB = *at(pxr, o + dB);
      }
    };
    auto step = [&](int z, const In& v) {
      double lA = __shfl_sync(mask, cA1, lane - 1), lB = __shfl_sync(mask, cB1, lane - 1);
      double rA = __shfl_sync(mask, cA0, lane + 1), rB = __shfl_sync(mask, cB0, lane + 1);
      if (ldl) {
        lA = flip(v.lA, nxl);
        lB = flip(v.lB, nxl);
      }
      if (ldr) {
        rA = flip(v.rA, nxr);
        rB = flip(v.rB, nxr);
      }
      const unsigned e = z == nz - 1 ? nzp : 0u;
      const double nA0 = flip(v.nA0, e), nA1 = flip(v.nA1, e), nB0 = flip(v.nB0, e), nB1 = flip(v.nB1, e);
      const double a0[6] = {lA, cA1, flip(v.ym0, nym), cB0, mA0, nA0}, a1[6] = {cA0, rA, flip(v.ym1, nym), cB1, mA1, nA1};
      const double b0[6] = {lB, cB1, cA0, flip(v.yp0, nyp), mB0, nB0}, b1[6] = {cB0, rB, cA1, flip(v.yp1, nyp), mB1, nB1};
      const double r0 = residual_of(sum6<false>(a0, mask), cA0, v.fA0, mih2);
      acc = z & 1 ? __dadd_rn(acc, r0) : r0;
      acc = __dadd_rn(acc, residual_of(sum6<false>(a1, mask), cA1, v.fA1, mih2));
      acc = __dadd_rn(acc, residual_of(sum6<INT>(b0, mask), cB0, v.fB0, mih2));
      acc = __dadd_rn(acc, residual_of(sum6<INT>(b1, mask), cB1, v.fB1, mih2));
      mA0 = cA0, mA1 = cA1, mB0 = cB0, mB1 = cB1;
      cA0 = nA0, cA1 = nA1, cB0 = nB0, cB1 = nB1;
    };
    In a, b;
    load(z0, a);
    for (int z = z0; z < z1; z += 2) {
      load(z + 1, b);
      step(z, a);
      if (z + 2 < z1) load(z + 2, a);
      step(z + 1, b);
      *cr = __dmul_rn(acc, 0.125);
      cr += R.c[0].plane;
      if (cp) {
        *cp = 0.0;
        cp += R.c[1].plane;
      }
    }
  }
}

// Blocks over (rows of a box x chunks of *zc planes, boxes); chunks are halved until about six
// blocks an SM are there (4 and 16 instead: within 2% at 256^3, slower at 128^3 and below).
dim3 march_grid(const SegList& L, int* zc, int rows = 1) {  // rows of a thread
  const int* ext = L.ext.n;
  const int rb = kMarchThreads / ((ext[0] + 1) / 2);
  const int ty = ((ext[1] + rows - 1) / rows + rb - 1) / rb;
  *zc = 32;
  while (*zc > 2 && (long long)L.nbox * ty * ((ext[2] + *zc - 1) / *zc) < 6ll * num_sms()) *zc /= 2;
  return dim3((unsigned)(ty * ((ext[2] + *zc - 1) / *zc)), (unsigned)L.nbox);
}
// Launches over fewer cells leave the FP64 pipe idle most of the time and are bound by latency,
// where the integer sums' longer chains cost more than they save (64^3 FP64 solve: 1.70 ms with
// integer sums on every level, 1.62 ms with this line).
bool use_int(const SegList& L) {
  return (long long)L.nbox * L.ext.n[0] * L.ext.n[1] * L.ext.n[2] >= 1ll << 15;
}

}  // namespace

// The marching kernels give a thread a pair of cells and a block whole rows of one box, so small boxes
// leave lanes idle and blocks with one or two warps at work; the row kernels pack rows of many boxes
// into a block, but leave lanes of narrow rows idle.  Counted per plane of a box: 32 lanes a warp at
// work, twice for the residual (a thread takes both cells), against the lanes of the rows; blocks of
// one or two warps hide less latency and count more (one: a half-sweep of rows of 16 cells and more
// 1.3 times, restriction 1.6, residual 2.1; two: restriction and residual 1.15), the rows against
// blocks of three or four 1.25 times.  Measured on GB300, row kernels / marching, us (the faster one is
// taken): half-sweep of 64^3 in boxes of 4^3 9.2 / 14.3, 8 x 4 x 4 6.2 / 8.1, 8 x 2 x 64 6.2 / 12.6, 4 x 8 x 8 9.3 / 7.3, 8^3
// 6.2 / 4.9; residual of 32^3 in 2^3 14.5 / 24.7, 128^3 in 32 x 2 x 128 37 / 64, 8^3 123 / 63; restriction of
// 64^3 in 4^3 21 / 55, 128^3 in 8^3 67 / 82, 16^3 35 / 41, 8 x 16 x 8 67 / 49.
void MarchWork::add_box(const int n[3]) {
  auto lanes = [](int width, int cells, int lo, int hi) {  // of a row's group in the row kernels
    int g = lo;
    while (g < hi && g * cells < width) g *= 2;
    return g;
  };
  const int pp = (n[0] + 1) / 2;
  if (pp > kMarchThreads) return;
  const int rb = kMarchThreads / pp;
  auto warps = [&](int rows) { return rows / rb * ((pp * rb + 31) / 32) + (pp * (rows % rb) + 31) / 32; };
  auto busy = [&](int rows) { return (pp * std::min(rows, rb) + 31) / 32; };  // warps of a block at work
  auto up = [](int a, int b) { return (a + b - 1) / b * b; };
  const float nz = (float)n[2];
  const int one = busy(n[1]), two = busy(n[1] / 2);
  march[MARCH_HALF] += nz * 32 * warps(n[1]) * (one == 1 && pp >= 8 ? 1.3f : 1.f);
  rows[MARCH_HALF] += nz * n[1] * up(pp, lanes(n[0], 4, 4, 16)) * (one > 2 ? 1.25f : 1.f);
  march[MARCH_RESIDUAL] += nz * 64 * warps(n[1]) * (one == 1 ? 2.1f : one == 2 ? 1.15f : 1.f);
  rows[MARCH_RESIDUAL] += nz * n[1] * up(n[0], 32) * (one > 2 ? 1.25f : 1.f);
  march[MARCH_RESTRICT] += nz * 32 * warps(n[1] / 2) * (two == 1 ? 1.6f : two == 2 ? 1.15f : 1.f);
  rows[MARCH_RESTRICT] += nz * (n[1] / 2) * up(pp, lanes(n[0], 2, 8, 32)) * (two > 2 ? 1.25f : 1.f);
}

// Where the work is against them, the marching kernels still win while their blocks are few and short
// enough to run at once (7 blocks an SM of the half-sweep, 4 of the restriction; rows that read their ghosts
// start faster), and in the restriction with direct reads up to 1.4 times the work, whose row form spends more
// on its neighbours' places: half-sweep with direct reads of 32^3 in 32 x 2 x 2 3.1 us, rows 4.6; 64^3 solve
// in boxes of 32^3 with stages down to the bottom 1.09 ms, 1.29 without this line.  Solves, with the
// marching kernels throughout / with this rule: 64^3 in 4^3 2.20 / 1.48 ms, 128^3 in 8^3 4.70 / 3.87, six of 64^3 in
// 8^3 4.06 / 3.37, four of 128^3 in 16^3 8.72 / 8.21.
bool march_pays(const SegList& L, int op, bool direct) {
  const BoxExtents& e = L.ext;
  if (!e.ok || (op != MARCH_RESIDUAL && !e.even)) return false;
  if (!e.work[op]) return true;
  if (op == MARCH_RESIDUAL) return false;
  int zc;
  const dim3 g = march_grid(L, &zc, op == MARCH_RESTRICT ? 2 : 1);
  const long long blocks = (long long)g.x * g.y, sms = num_sms();
  if (op == MARCH_HALF) return std::min(zc, e.n[2]) <= 4 && blocks <= (direct ? 7 : 2) * sms;
  return blocks <= (direct ? 4 : 2) * sms || (direct && e.work[op] == 1);
}

cudaError_t launch_half_march(const SegList& L, int mode, int color, unsigned long long* norms,
                              cudaStream_t s) {
  int zc;
  const dim3 grid = march_grid(L, &zc);
  auto go = [&](auto k) { launch_k(k, grid, kMarchThreads, 0, s, L, zc, color, norms); };
  if (mode && L.n != 1) return cudaErrorInvalidValue;
  if (use_int(L)) {
    if (mode == 0 && L.n > 1) go(k_half_march<0, true, true>);
    else if (mode == 0) go(k_half_march<0, true>);
    else if (mode == 1) go(k_half_march<1, true>);
    else if (mode == 2) go(k_half_march<2, true>);
    else go(k_half_march<3, true>);
  } else {
    if (mode == 0 && L.n > 1) go(k_half_march<0, false, true>);
    else if (mode == 0) go(k_half_march<0, false>);
    else if (mode == 1) go(k_half_march<1, false>);
    else if (mode == 2) go(k_half_march<2, false>);
    else go(k_half_march<3, false>);
  }
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_residual_march(const SegList& L, unsigned long long* norms, cudaStream_t s) {
  int zc;
  const dim3 grid = march_grid(L, &zc);
  auto go = [&](auto k) { launch_k(k, grid, kMarchThreads, 0, s, L, zc, norms); };
  if (use_int(L)) {
    if (L.n > 1) go(k_residual_march<true, true>);
    else go(k_residual_march<true, false>);
  } else {
    if (L.n > 1) go(k_residual_march<false, true>);
    else go(k_residual_march<false, false>);
  }
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_restrict_march(const SegList& L, bool stored, cudaStream_t s) {
  int zc;
  const dim3 grid = march_grid(L, &zc, 2);
  auto go = [&](auto k) { launch_k(k, grid, kMarchThreads, 0, s, L, zc); };
  const bool ints = use_int(L);
  if (stored && L.n != 1) return cudaErrorInvalidValue;
  if (stored) {
    if (ints) go(k_restrict_march<true, true, false>);
    else go(k_restrict_march<true, false, false>);
  } else if (L.n > 1) {
    if (ints) go(k_restrict_march<false, true, true>);
    else go(k_restrict_march<false, false, true>);
  } else {
    if (ints) go(k_restrict_march<false, true, false>);
    else go(k_restrict_march<false, false, false>);
  }
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace gbmg
