// Red + black Gauss-Seidel sweep of FP32 levels on regular box grids (sm_103a), one launch.
//
// Equal, bit for bit, to: red half-sweep, black half-sweep, each reading box-face neighbours
// directly.  What bounds it is HBM: 12 bytes a cell (phi and rhs read, phi written) against 24
// for two half-sweeps, which read and write every sector of both colours twice; so the work is
// laid out to need few instructions and shared-memory wavefronts per cell:
//   * a block owns S strips of 4 cells x TY rows of the level's domain (not of a box: the boxes
//     are a lattice, so the place of a cell is two divisions once per thread) and marches
//     through ZC planes; a thread owns one strip in two neighbouring rows and loads whole
//     strips (16 bytes);
//   * the two colours are separated in registers: a red pair's y and z neighbours are the black
//     pairs at the same places of the neighbouring rows and planes (the colour pattern shifts by
//     one from row to row), so one 8-byte value serves two cells.  z neighbours stay in
//     registers as the thread marches, the pair's rows are each other's y neighbour, and only
//     the outer rows and one cell in x come from the other threads through shared memory;
//   * stage k updates the red cells of plane s and the black cells of plane s - 1 from the
//     values published in the stage before: one barrier a plane;
//   * strips around the tile (hx = 1) and rows (hy = 2) are loaded and updated redundantly, as
//     are the planes before and after the chunk.  Outside a Dirichlet face those rows and planes
//     are the mirrored ones, negated and never updated, which is what the ghost cells hold;
//   * planes are loaded kDepth ahead by cp.async into a ring that each thread reads back itself
//     (no barrier for it).
// Measured on GB300 (CUDA events, 12 bytes a cell): 512^3 in boxes of 128^3 316 us (5.1 TB/s, 75%
// of the copy rate; the TMA sweep of mg_fused.cu took 389 us plus two fills of two layers), 60
// periodic 96^3 levels in boxes of 32^3 121 us (two half-sweeps 324 us); inside the 512^3 mixed solve
// 265 us (ncu; 90% of the copy rate), 172 us starting from zero (phi not read), 334 us adding the
// prolongation (whose own kernel took 214).  One row a thread took
// 352 us at 512^3 (62% of the shared-memory wavefronts, 54% more instructions a cell in
// barriers and addresses); selecting colours at run time instead of by the unrolled plane
// parity took 441 us (100 instructions a cell against 38).
#include "mg_sweep.hpp"

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "mg_kernels.hpp"

namespace gbmg {

namespace {

constexpr int kDepth = 3;        // planes in flight
constexpr int kMaxChunk = 128;   // planes of a tile
constexpr int kMaxPlanes = kMaxChunk + 4 + kDepth;  // of the plane offset table
constexpr int kMaxThreads = 320, kBlocksPerSM = 2;  // 96 registers a thread

__device__ __forceinline__ void cpa16(uint32_t d, const void* s) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(s) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ float lds1(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float2 lds2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ void sts2(uint32_t a, float2 v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
// v with its sign bit flipped where m has it set
__device__ __forceinline__ float flip1(float v, uint32_t m) {
  return __uint_as_float(__float_as_uint(v) ^ m);
}
__device__ __forceinline__ float4 flip4(float4 v, uint32_t m) {
  return make_float4(flip1(v.x, m), flip1(v.y, m), flip1(v.z, m), flip1(v.w, m));
}
__device__ __forceinline__ float2 even2(const float4& v) { return make_float2(v.x, v.z); }
__device__ __forceinline__ float2 odd2(const float4& v) { return make_float2(v.y, v.w); }

// The grid of this block's tile to shared memory, a word a thread.
template <class G>
__device__ __forceinline__ void load_grid(G* to, const G* __restrict__ grids, int ng) {
  int lo = 0, hi = ng - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (grids[mid].tile_begin <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  static_assert(sizeof(G) % 8 == 0, "");
  for (int i = threadIdx.x; i < (int)(sizeof(G) / 8); i += blockDim.x)
    reinterpret_cast<long long*>(to)[i] = reinterpret_cast<const long long*>(grids + lo)[i];
}

template <int V>
struct Int {
  static constexpr int value = V;
};

__device__ __forceinline__ void cpa4(uint32_t d, const void* s) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(s) : "memory");
}
__device__ __forceinline__ float4 add_pairs(const float4& v, const float2& c) {  // c: one value a pair
  return make_float4(__fadd_rn(v.x, c.x), __fadd_rn(v.y, c.x), __fadd_rn(v.z, c.y), __fadd_rn(v.w, c.y));
}

__device__ __forceinline__ void cpa8(uint32_t d, const void* s) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(s) : "memory");
}
// A strip of 16 bytes whose source is aligned to AL.
template <int AL>
__device__ __forceinline__ void cpa_strip(uint32_t d, const char* s) {
  if (AL == 16) {
    cpa16(d, s);
  } else if (AL == 8) {
    cpa8(d, s);
    cpa8(d + 8, s + 8);
  } else {
#pragma unroll
    for (int i = 0; i < 16; i += 4) cpa4(d + i, s + i);
  }
}
template <int AL>
__device__ __forceinline__ float4 ld_strip(const char* s) {
  if (AL == 16) return *reinterpret_cast<const float4*>(s);
  const float* f = reinterpret_cast<const float*>(s);
  return make_float4(f[0], f[1], f[2], f[3]);
}

// PAL, RAL: alignment of the strips of phi and rhs; below 16 the three fields have layouts of their own.
template <int START, int PAL = 16, int RAL = 16>
__global__ void __launch_bounds__(kMaxThreads, kBlocksPerSM)
    k_sweep_f32(const SweepGrid* __restrict__ grids, int ng) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool kOne = PAL == 16 && RAL == 16;  // one layout
  __shared__ long long zoff[kMaxPlanes], czoff[START == SWEEP_PROLONG ? kMaxPlanes : 1];
  __shared__ long long rzoff_[kOne ? 1 : kMaxPlanes], dzoff_[kOne ? 1 : kMaxPlanes];
  const long long* const rzoff = kOne ? zoff : rzoff_;
  const long long* const dzoff = kOne ? zoff : dzoff_;
  __shared__ SweepGrid Gs;
  load_grid(&Gs, grids, ng);
  __syncthreads();
  const SweepGrid& G = Gs;
  const int t = blockIdx.x - G.tile_begin;
  const int tx = t % G.nt[0], ty = (t / G.nt[0]) % G.nt[1], tz = t / (G.nt[0] * G.nt[1]);
  const int hx = G.hx, hy = G.hy;
  const int W = G.S + 2 * hx, HM = (G.TY + 2 * hy) >> 1;  // strips, row pairs
  const int tid = threadIdx.x, nth = blockDim.x;
  const bool pad = tid / W >= HM;  // threads past the tile repeat its first one and own nothing
  const int m = pad ? 0 : tid / W, i = pad ? 0 : tid % W, j = 2 * m;
  const int N0 = G.N[0], N1 = G.N[1], N2 = G.N[2];
  const bool px = G.periodic & 1, py = G.periodic & 2, pz = G.periodic & 4;
  int gx = (tx * G.S + i - hx) * 4, gy = ty * G.TY + j - hy;
  const bool own = !pad && i >= hx && i < hx + G.S && j >= hy && j < hy + G.TY && gx < N0 && gy < N1;
  const int parc = (G.par0 + gy) & 1;  // colour parity of row gy (tiles begin at even rows)
  // the rows' places: the periodic image, or outside a Dirichlet face the mirrored rows, negated
  // and not updated
  bool upd = true;
  uint32_t neg = 0;
  if (px) {
    gx %= N0;
    if (gx < 0) gx += N0;
  } else {
    gx = min(max(gx, 0), N0 - 4);
  }
  int gyB = gy + 1;
  if (py) {
    gy %= N1;
    if (gy < 0) gy += N1;
    gyB = gy + 1;
  } else if (gy < 0 || gy >= N1) {
    const int q = gy < 0 ? -1 - gy : 2 * N1 - 1 - gy;
    gy = min(max(q, 0), N1 - 1);
    gyB = min(max(q - 1, 0), N1 - 1);
    neg = 0x80000000u;
    upd = false;
  }
  const bool fxm = !px && gx == 0, fxp = !px && gx + 4 == N0;
  // published pairs of colour kind (0 black, 1 red) of row A or B: (((stage & 1) * 2 + kind) * 2 + row) * kst
  const int il = i > 0 ? i - 1 : (hx == 0 ? W - 1 : 0), ir = i < W - 1 ? i + 1 : (hx == 0 ? 0 : i);
  const int md = m > 0 ? m - 1 : (hy == 0 ? HM - 1 : 0), mu = m < HM - 1 ? m + 1 : (hy == 0 ? 0 : m);
  const uint32_t sb = (uint32_t)__cvta_generic_to_shared(smem), kst = (uint32_t)nth * 8;
  const uint32_t me = sb + tid * 8;
  const uint32_t al = sb + (m * W + il) * 8 + 4, ar = sb + (m * W + ir) * 8;  // cell left / right of the strip
  const uint32_t ad = sb + (md * W + i) * 8 + kst, au = sb + (mu * W + i) * 8;  // row B below, row A above
  const uint32_t ring = sb + 8 * kst + tid * 16, rst = (uint32_t)nth * 16;
  // byte offsets of planes z0 - 2 ... (those past the domain's ends: images, or mirrored planes)
  const int z0 = tz * G.ZC, z1 = min(z0 + G.ZC, N2);
  const int np = z1 - z0 + 4 + kDepth;
  for (int q = tid; q < np; q += nth) {
    int p = z0 - 2 + q;
    if (pz) {
      p %= N2;
      if (p < 0) p += N2;
    } else {
      p = p < 0 ? -1 - p : p >= N2 ? 2 * N2 - 1 - p : p;
      p = min(max(p, 0), N2 - 1);
    }
    const int bz = p / G.E[2];
    zoff[q] = ((long long)bz * G.nb[0] * G.nb[1] * G.bstride + (long long)(p - bz * G.E[2]) * G.plane) * 4;
    if (!kOne) {
      const long long col = (long long)bz * G.nb[0] * G.nb[1], pl = p - bz * G.E[2];
      rzoff_[q] = (col * G.rstride + pl * G.rplane) * 4;
      dzoff_[q] = (col * G.dstride + pl * G.dplane) * 4;
    }
    if (START == SWEEP_PROLONG) {
      const CoarseField& C = G.coarse;
      const int Z = p >> 1, cz = Z / C.E[2];
      czoff[q] = ((long long)cz * C.nb[0] * C.nb[1] * C.bstride + (long long)(Z - cz * C.E[2]) * C.plane) * 4;
    }
  }
  __syncthreads();
  const int bx = gx / G.E[0], by = gy / G.E[1], byB = gyB / G.E[1];
  // place of the thread's strip in row A, and from there to row B, in a field's plane 0
  auto place = [&](long long stride, int pitch) {
    return ((long long)(by * G.nb[0] + bx) * stride + (long long)(gy - by * G.E[1]) * pitch + (gx - bx * G.E[0])) * 4;
  };
  auto to_b = [&](long long stride, int pitch) {
    return ((long long)(byB - by) * G.nb[0] * stride + (long long)((gyB - byB * G.E[1]) - (gy - by * G.E[1])) * pitch) * 4;
  };
  const long long tcol = place(G.bstride, G.pitch), dB = to_b(G.bstride, G.pitch);
  const char* src = (const char*)G.src + tcol;
  const char* rhs = (const char*)G.rhs + (kOne ? tcol : place(G.rstride, G.rpitch));
  char* dst = (char*)G.dst + (kOne ? tcol : place(G.dstride, G.dpitch));
  const long long rdB = kOne ? dB : to_b(G.rstride, G.rpitch), ddB = kOne ? dB : to_b(G.dstride, G.dpitch);
  // the strip's two parents (rows A and B share them), and their slots in the ring
  const char* crs = nullptr;
  const uint32_t cring = ring + 4 * kDepth * rst - tid * 8, cst = kst;
  if (START == SWEEP_PROLONG) {
    const CoarseField& C = G.coarse;
    const int X = gx >> 1, Y = gy >> 1, cx = X / C.E[0], cy = Y / C.E[1];
    crs = (const char*)C.base + ((long long)(cy * C.nb[0] + cx) * C.bstride +
                                 (long long)(Y - cy * C.E[1]) * C.pitch + (X - cx * C.E[0])) * 4;
  }
  const float mh2 = G.mh2;
  constexpr float inv6 = 1.0f / 6.0f;
  const int s_first = z0 - 1, nit = z1 - z0 + 2;  // stages: red of planes z0 - 1 ... z1
  const int P0 = (parc + s_first) & 1;
  auto plane_neg = [&](int p) -> uint32_t { return !pz && (p < 0 || p >= N2) ? 0x80000000u : 0u; };
  // Per row, entering stage k (plane s = s_first + k): black of planes s - 1 and s, old red of s,
  // new red of s - 2 and s - 1, rhs of the black cells of s - 1.
  struct Row {
    float2 bm, bc, ro, r1a, r1b, rb1;
  };
  Row RA, RB;
  {
    const uint32_t n0 = neg ^ plane_neg(s_first - 1), n1 = neg ^ plane_neg(s_first);
    auto first = [&](long long dy, int q) {  // phi of plane z0 - 2 + q
      if (START == SWEEP_ZERO) return make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 v = ld_strip<PAL>(src + dy + zoff[q]);
      if (START == SWEEP_SOURCE) return v;
      const float* c = reinterpret_cast<const float*>(crs + czoff[q]);
      return add_pairs(v, make_float2(c[0], c[1]));
    };
    const float4 A0 = flip4(first(0, 0), n0), A1 = flip4(first(0, 1), n1);
    const float4 B0 = flip4(first(dB, 0), n0), B1 = flip4(first(dB, 1), n1);
#pragma unroll
    for (int d = 0; d < kDepth; ++d) {
      if (START != SWEEP_ZERO) {
        cpa_strip<PAL>(ring + (4 * d) * rst, src + zoff[2 + d]);
        cpa_strip<PAL>(ring + (4 * d + 1) * rst, src + dB + zoff[2 + d]);
      }
      cpa_strip<RAL>(ring + (4 * d + 2) * rst, rhs + rzoff[1 + d]);
      cpa_strip<RAL>(ring + (4 * d + 3) * rst, rhs + rdB + rzoff[1 + d]);
      if (START == SWEEP_PROLONG) {
        cpa4(cring + d * cst, crs + czoff[2 + d]);
        cpa4(cring + d * cst + 4, crs + czoff[2 + d] + 4);
      }
      cpa_commit();
    }
    // row A at plane s_first has parity P0 (red at odd places if 1), row B the other
    const float2 zero = make_float2(0.f, 0.f);
    if (P0) {
      RA = Row{odd2(A0), even2(A1), odd2(A1), zero, zero, zero};
      RB = Row{even2(B0), odd2(B1), even2(B1), zero, zero, zero};
    } else {
      RA = Row{even2(A0), odd2(A1), even2(A1), zero, zero, zero};
      RB = Row{odd2(B0), even2(B1), odd2(B1), zero, zero, zero};
    }
    sts2(me, RA.bc);
    sts2(me + kst, RB.bc);
    sts2(me + 2 * kst, zero);
    sts2(me + 3 * kst, zero);
  }
  uint32_t slot = ring, cslot = cring;
  const uint32_t slot_end = ring + 4 * kDepth * rst;
  __syncthreads();
  auto stage = [&](auto Pc, auto Kc, int k) {
    constexpr int P = decltype(Pc)::value, cur = decltype(Kc)::value, nxt = cur ^ 1;
    const int s = s_first + k;
    asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
    const uint32_t n1 = neg ^ plane_neg(s + 1);
    float4 pA = make_float4(0.f, 0.f, 0.f, 0.f), pB = pA;  // phi of s + 1
    if (START != SWEEP_ZERO) {
      pA = lds4(slot);
      pB = lds4(slot + rst);
    }
    if (START == SWEEP_PROLONG) {
      const float2 c = lds2(cslot);
      pA = add_pairs(pA, c);
      pB = add_pairs(pB, c);
    }
    pA = flip4(pA, n1);
    pB = flip4(pB, n1);
    const float4 fA = lds4(slot + 2 * rst), fB = lds4(slot + 3 * rst);  // rhs of s
    {
      const int q = k + 2 + kDepth;
      const long long o = zoff[q], o1 = rzoff[q - 1];
      if (START != SWEEP_ZERO) {
        cpa_strip<PAL>(slot, src + o);
        cpa_strip<PAL>(slot + rst, src + dB + o);
      }
      cpa_strip<RAL>(slot + 2 * rst, rhs + o1);
      cpa_strip<RAL>(slot + 3 * rst, rhs + rdB + o1);
      if (START == SWEEP_PROLONG) {
        cpa4(cslot, crs + czoff[q]);
        cpa4(cslot + 4, crs + czoff[q] + 4);
        cslot = cslot == cring + (kDepth - 1) * cst ? cring : cslot + cst;
      }
      cpa_commit();
    }
    slot = slot + 4 * rst == slot_end ? ring : slot + 4 * rst;
    // row A of plane s has parity P; row B, and row A of plane s + 1, the other
    const float2 bnA = P ? odd2(pA) : even2(pA), ronA = P ? even2(pA) : odd2(pA);
    const float2 bnB = P ? even2(pB) : odd2(pB), ronB = P ? odd2(pB) : even2(pB);
    const float2 rqA = P ? odd2(fA) : even2(fA), bqA = P ? even2(fA) : odd2(fA);
    const float2 rqB = P ? even2(fB) : odd2(fB), bqB = P ? odd2(fB) : even2(fB);
    // One colour of both rows: o their own old values, n the rows' other colour, zm / zp the other
    // colour below and above, q the rhs.  Row A's cells of this colour sit at parity P (red of
    // plane s as well as black of plane s - 1), row B's at the other.
    auto update = [&](uint32_t kb, const float2& oA, const float2& oB, const float2& nA, const float2& nB,
                      const float2& zmA, const float2& zpA, const float2& zmB, const float2& zpB,
                      const float2& qA, const float2& qB, float2& uA, float2& uB) {
      const float2 ym = lds2(ad + kb), yp = lds2(au + kb);
      float XA = lds1((P ? ar : al) + kb), XB = lds1((P ? al : ar) + kb + kst);
      if (P ? fxp : fxm) XA = -(P ? oA.y : oA.x);
      if (P ? fxm : fxp) XB = -(P ? oB.x : oB.y);
      float a0 = __fadd_rn(P ? nA.x : XA, P ? nA.y : nA.x), a1 = __fadd_rn(P ? nA.y : nA.x, P ? XA : nA.y);
      float b0 = __fadd_rn(P ? XB : nB.x, P ? nB.x : nB.y), b1 = __fadd_rn(P ? nB.x : nB.y, P ? nB.y : XB);
      a0 = __fadd_rn(a0, ym.x), a1 = __fadd_rn(a1, ym.y), b0 = __fadd_rn(b0, nA.x), b1 = __fadd_rn(b1, nA.y);
      a0 = __fadd_rn(a0, nB.x), a1 = __fadd_rn(a1, nB.y), b0 = __fadd_rn(b0, yp.x), b1 = __fadd_rn(b1, yp.y);
      a0 = __fadd_rn(a0, zmA.x), a1 = __fadd_rn(a1, zmA.y), b0 = __fadd_rn(b0, zmB.x), b1 = __fadd_rn(b1, zmB.y);
      a0 = __fadd_rn(a0, zpA.x), a1 = __fadd_rn(a1, zpA.y), b0 = __fadd_rn(b0, zpB.x), b1 = __fadd_rn(b1, zpB.y);
      uA = make_float2(__fmul_rn(__fmaf_rn(mh2, qA.x, a0), inv6), __fmul_rn(__fmaf_rn(mh2, qA.y, a1), inv6));
      uB = make_float2(__fmul_rn(__fmaf_rn(mh2, qB.x, b0), inv6), __fmul_rn(__fmaf_rn(mh2, qB.y, b1), inv6));
    };
    float2 rA, rB, bA, bB;
    update((cur * 4) * kst, RA.ro, RB.ro, RA.bc, RB.bc, RA.bm, bnA, RB.bm, bnB, rqA, rqB, rA, rB);
    if (!(upd && plane_neg(s) == 0)) {  // mirrored cells hold what was there before the half-sweep
      rA = RA.ro;
      rB = RB.ro;
    }
    update((cur * 4 + 2) * kst, RA.bm, RB.bm, RA.r1b, RB.r1b, RA.r1a, rA, RB.r1a, rB, RA.rb1, RB.rb1, bA, bB);
    if (own && k >= 2) {  // plane s - 1 is final; its row A has parity P ^ 1
      const float2 xA = RA.r1b, xB = RB.r1b;
      char* d = dst + dzoff[k];
      *reinterpret_cast<float4*>(d) = P ? make_float4(xA.x, bA.x, xA.y, bA.y) : make_float4(bA.x, xA.x, bA.y, xA.y);
      *reinterpret_cast<float4*>(d + ddB) = P ? make_float4(bB.x, xB.x, bB.y, xB.y) : make_float4(xB.x, bB.x, xB.y, bB.y);
    }
    sts2(me + (nxt * 4) * kst, bnA);
    sts2(me + (nxt * 4 + 1) * kst, bnB);
    sts2(me + (nxt * 4 + 2) * kst, rA);
    sts2(me + (nxt * 4 + 3) * kst, rB);
    asm volatile("bar.sync 0;" ::: "memory");
    RA = Row{RA.bc, bnA, ronA, RA.r1b, rA, bqA};
    RB = Row{RB.bc, bnB, ronB, RB.r1b, rB, bqB};
  };
  // (P0 is the same in every thread of the block)
  if (P0) {
    for (int k = 0; k < nit; k += 2) {
      stage(Int<1>{}, Int<0>{}, k);
      if (k + 1 < nit) stage(Int<0>{}, Int<1>{}, k + 1);
    }
  } else {
    for (int k = 0; k < nit; k += 2) {
      stage(Int<0>{}, Int<0>{}, k);
      if (k + 1 < nit) stage(Int<1>{}, Int<1>{}, k + 1);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Residual + restriction.  A thread owns a strip of 4 cells in two rows (2Y, 2Y + 1), i.e. two
// coarse cells, and marches through planes; z neighbours stay in registers, the rest is loaded a
// plane ahead (neighbouring strips and rows mostly from L1, where the threads owning them put
// them).  Arithmetic and order as k_residual_restrict.  HBM bounds it (phi and rhs read once, 8
// bytes a cell); measured at 512^3: 959 us by k_residual_restrict reading neighbours directly (128-wide
// rows, scalar loads, 4 children rows a lane), 196 us here (5.5 TB/s, 81% of the copy rate); 256^3 112
// -> 38 us.  3, 4 or 5 blocks an SM: within 1%.
constexpr int kRestrictThreads = 128, kRestrictChunk = 32;
__global__ void __launch_bounds__(kRestrictThreads, 4)
    k_restrict_f32(const RestrictGrid* __restrict__ grids, int ng) {
  pdl_begin();
  __shared__ long long zoff[kRestrictChunk + 3], coff[2][kRestrictChunk / 2];
  __shared__ RestrictGrid Gs;
  load_grid(&Gs, grids, ng);
  __syncthreads();
  const RestrictGrid& Q = Gs;
  const SweepGrid& G = Q.g;
  const int t = blockIdx.x - Q.tile_begin;
  const int tz = t / Q.tiles_xy, col = (t - tz * Q.tiles_xy) * kRestrictThreads + threadIdx.x;
  const int N0 = G.N[0], N1 = G.N[1], N2 = G.N[2], strips = N0 >> 2;
  const bool px = G.periodic & 1, py = G.periodic & 2, pz = G.periodic & 4;
  const int z0 = tz * Q.ZC, z1 = min(z0 + Q.ZC, N2);
  for (int q = threadIdx.x; q < z1 - z0 + 2; q += kRestrictThreads) {  // planes z0 - 1 ... z1
    int p = z0 - 1 + q;
    if (pz) p = p < 0 ? p + N2 : p >= N2 ? p - N2 : p;
    else p = min(max(p, 0), N2 - 1);  // the mirrored plane
    const int bz = p / G.E[2];
    zoff[q] = ((long long)bz * G.nb[0] * G.nb[1] * G.bstride + (long long)(p - bz * G.E[2]) * G.plane) * 4;
  }
  for (int q = threadIdx.x; q < z1 - z0; q += kRestrictThreads) {  // coarse planes, rhs and phi
    const CoarseField& C = q & 1 ? Q.cphi : Q.crhs;
    const int Z = (z0 + q) >> 1, bz = Z / C.E[2];
    coff[q & 1][q >> 1] = ((long long)bz * C.nb[0] * C.nb[1] * C.bstride + (long long)(Z - bz * C.E[2]) * C.plane) * 4;
  }
  __syncthreads();
  if (col >= strips * (N1 >> 1)) return;
  const int m = col / strips, gx = (col - m * strips) * 4, gy = 2 * m;
  // place of cell (x, y) in plane 0 of the lattice, bytes
  auto place = [&](int x, int y) {
    const int bx = x / G.E[0], by = y / G.E[1];
    return ((long long)(by * G.nb[0] + bx) * G.bstride + (long long)(y - by * G.E[1]) * G.pitch + (x - bx * G.E[0])) * 4;
  };
  const long long pA = place(gx, gy), pB = place(gx, gy + 1);
  // outside a Dirichlet face: the cell's own value, negated
  const bool ylo = gy == 0, yhi = gy + 2 == N1, xlo = gx == 0, xhi = gx + 4 == N0;
  const long long pym = ylo ? (py ? place(gx, N1 - 1) : pA) : place(gx, gy - 1);
  const long long pyp = yhi ? (py ? place(gx, 0) : pB) : place(gx, gy + 2);
  const int xl = xlo ? (px ? N0 - 1 : 0) : gx - 1, xr = xhi ? (px ? 0 : N0 - 1) : gx + 4;
  const long long plA = place(xl, gy), plB = place(xl, gy + 1), prA = place(xr, gy), prB = place(xr, gy + 1);
  const uint32_t nym = ylo && !py ? 0x80000000u : 0u, nyp = yhi && !py ? 0x80000000u : 0u;
  const uint32_t nxl = xlo && !px ? 0x80000000u : 0u, nxr = xhi && !px ? 0x80000000u : 0u;
  const char* src = (const char*)G.src;
  const char* rhs = (const char*)G.rhs;
  const float mih2 = Q.mih2;
  const int X = gx >> 1, Y = m;
  auto cplace = [&](const CoarseField& C) {
    const int bx = X / C.E[0], by = Y / C.E[1];  // (a strip's two coarse cells share a box)
    return (char*)C.base + ((long long)(by * C.nb[0] + bx) * C.bstride + (long long)(Y - by * C.E[1]) * C.pitch + (X - bx * C.E[0])) * 4;
  };
  char* cr = cplace(Q.crhs);
  char* cp = Q.cphi.base ? cplace(Q.cphi) : nullptr;
  struct In {
    float4 nA, nB, ym, yp, fA, fB;
    float lA, lB, rA, rB;
  };
  auto ld4 = [](const char* q) { return __ldg(reinterpret_cast<const float4*>(q)); };
  auto ld1 = [](const char* q) { return __ldg(reinterpret_cast<const float*>(q)); };
  auto load = [&](int z, In& v) {  // inputs of plane z: its surroundings, and the plane above
    const char* s = src + zoff[z - z0 + 1];
    const char* u = src + zoff[z - z0 + 2];
    const char* f = rhs + zoff[z - z0 + 1];
    v.nA = ld4(u + pA);
    v.nB = ld4(u + pB);
    v.ym = ld4(s + pym);
    v.yp = ld4(s + pyp);
    v.fA = ld4(f + pA);
    v.fB = ld4(f + pB);
    v.lA = ld1(s + plA);
    v.lB = ld1(s + plB);
    v.rA = ld1(s + prA);
    v.rB = ld1(s + prB);
  };
  const uint32_t nz0 = !pz && z0 == 0 ? 0x80000000u : 0u;
  float4 mA = flip4(ld4(src + zoff[0] + pA), nz0), mB = flip4(ld4(src + zoff[0] + pB), nz0);
  float4 cA = ld4(src + zoff[1] + pA), cB = ld4(src + zoff[1] + pB);
  float acc0 = 0.f, acc1 = 0.f;
  auto res = [&](float xm, float xp, float ym, float yp, float zm, float zp, float c, float f) {
    float s = __fadd_rn(xm, xp);
    s = __fadd_rn(s, ym);
    s = __fadd_rn(s, yp);
    s = __fadd_rn(s, zm);
    s = __fadd_rn(s, zp);
    return __fmaf_rn(mih2, __fmaf_rn(-6.f, c, s), f);
  };
  auto step = [&](auto Kc, int z, const In& v) {
    constexpr int K = decltype(Kc)::value;  // plane of the pair
    const uint32_t nz = !pz && z == N2 - 1 ? 0x80000000u : 0u;
    const float4 nA = flip4(v.nA, nz), nB = flip4(v.nB, nz), ym = flip4(v.ym, nym), yp = flip4(v.yp, nyp);
    const float lA = flip1(v.lA, nxl), lB = flip1(v.lB, nxl), rA = flip1(v.rA, nxr), rB = flip1(v.rB, nxr);
    const float a0 = res(lA, cA.y, ym.x, cB.x, mA.x, nA.x, cA.x, v.fA.x);
    const float a1 = res(cA.x, cA.z, ym.y, cB.y, mA.y, nA.y, cA.y, v.fA.y);
    const float a2 = res(cA.y, cA.w, ym.z, cB.z, mA.z, nA.z, cA.z, v.fA.z);
    const float a3 = res(cA.z, rA, ym.w, cB.w, mA.w, nA.w, cA.w, v.fA.w);
    const float b0 = res(lB, cB.y, cA.x, yp.x, mB.x, nB.x, cB.x, v.fB.x);
    const float b1 = res(cB.x, cB.z, cA.y, yp.y, mB.y, nB.y, cB.y, v.fB.y);
    const float b2 = res(cB.y, cB.w, cA.z, yp.z, mB.z, nB.z, cB.z, v.fB.z);
    const float b3 = res(cB.z, rB, cA.w, yp.w, mB.w, nB.w, cB.w, v.fB.w);
    acc0 = K ? __fadd_rn(acc0, a0) : a0;
    acc1 = K ? __fadd_rn(acc1, a2) : a2;
    acc0 = __fadd_rn(__fadd_rn(__fadd_rn(acc0, a1), b0), b1);
    acc1 = __fadd_rn(__fadd_rn(__fadd_rn(acc1, a3), b2), b3);
    if (K) {
      const int q = (z - z0) >> 1;
      float* c = reinterpret_cast<float*>(cr + coff[0][q]);
      c[0] = __fmul_rn(acc0, 0.125f);
      c[1] = __fmul_rn(acc1, 0.125f);
      if (cp) {
        float* e = reinterpret_cast<float*>(cp + coff[1][q]);
        e[0] = 0.f;
        e[1] = 0.f;
      }
    }
    mA = cA;
    mB = cB;
    cA = nA;
    cB = nB;
  };
  In a, b;
  load(z0, a);
  for (int z = z0; z < z1; z += 2) {
    load(z + 1, b);
    step(Int<0>{}, z, a);
    if (z + 2 < z1) load(z + 2, a);
    step(Int<1>{}, z + 1, b);
  }
}

int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Threads of a tile, rounded to warps.
int tile_threads(int S, int TY, int hx, int hy) { return (((S + 2 * hx) * (TY / 2 + hy)) + 31) / 32 * 32; }

}  // namespace

const long long kSweepMinCells = 1ll << 14, kSweepMinCellsBatch = 1ll << 18;

bool lattice_of(const BoxArray& ba, const FabLayout& lay, Lattice* out) {
  if (ba.boxes.empty()) return false;
  Lattice G{};
  for (int d = 0; d < 3; ++d) {
    G.N[d] = ba.dom.len(d);
    G.E[d] = ba.boxes[0].len(d);
    if (G.N[d] % G.E[d] != 0) return false;
    G.nb[d] = G.N[d] / G.E[d];
  }
  const size_t nb = ba.boxes.size();
  if ((long long)nb != (long long)G.nb[0] * G.nb[1] * G.nb[2] || lay.plane[0] > (1ll << 30)) return false;
  G.pitch = lay.pitch[0];
  G.plane = (int)lay.plane[0];
  G.first = lay.off[0] + lay.g * (lay.plane[0] + lay.pitch[0] + 1);
  G.bstride = nb > 1 ? lay.off[1] - lay.off[0] : lay.cstride[0];
  size_t b = 0;
  for (int z = 0; z < G.nb[2]; ++z)
    for (int y = 0; y < G.nb[1]; ++y)
      for (int x = 0; x < G.nb[0]; ++x, ++b) {
        const int at[3] = {x, y, z};
        for (int d = 0; d < 3; ++d)
          if (ba.boxes[b].lo[d] != ba.dom.lo[d] + at[d] * G.E[d] || ba.boxes[b].len(d) != G.E[d]) return false;
        if (lay.off[b] != lay.off[0] + (long long)b * G.bstride || lay.pitch[b] != G.pitch ||
            lay.plane[b] != G.plane)
          return false;
      }
  *out = G;
  return true;
}

bool sweep_geometry(const BoxArray& ba, const FabLayout& lay, const int periodic[3], double h,
                    SweepGrid* out) {
  Lattice T;
  if (lay.g != 0 || lay.ncomp != 1 || lay.esize != 4 || !lattice_of(ba, lay, &T)) return false;
  if (T.E[0] % 4 != 0 || (T.N[1] & 1) || T.pitch % 4 != 0 || T.first != 0 || T.bstride % 4 != 0) return false;
  SweepGrid G{};
  for (int d = 0; d < 3; ++d) {
    if (periodic[d] && (T.N[d] & 1)) return false;
    G.N[d] = T.N[d];
    G.E[d] = T.E[d];
    G.nb[d] = T.nb[d];
    G.periodic |= periodic[d] ? 1 << d : 0;
  }
  G.pitch = T.pitch;
  G.plane = T.plane;
  G.bstride = T.bstride;
  G.par0 = (ba.dom.lo[0] + ba.dom.lo[1] + ba.dom.lo[2]) & 1;
  G.mh2 = -(float)(h * h);
  *out = G;
  return true;
}

bool sweep_fabs_geometry(const BoxArray& ba, const FabLayout& phi, const FabLayout& rhs,
                         const FabLayout& dst, const int periodic[3], double h, SweepGrid* out) {
  Lattice P, R;
  if (phi.ncomp != 1 || rhs.ncomp != 1 || phi.esize != 4 || rhs.esize != 4) return false;
  if (!sweep_geometry(ba, dst, periodic, h, out) || !lattice_of(ba, phi, &P) || !lattice_of(ba, rhs, &R))
    return false;
  out->dpitch = out->pitch;
  out->dplane = out->plane;
  out->dstride = out->bstride;
  out->pitch = P.pitch;
  out->plane = P.plane;
  out->bstride = P.bstride;
  out->rpitch = R.pitch;
  out->rplane = R.plane;
  out->rstride = R.bstride;
  return true;
}

// The tiling trades redundant work at a tile's rim against a full chip.  For each limit on a
// block's threads every grid takes the strips x rows with the least redundancy, and for each
// chunk length the launch is costed as waves of resident blocks: a plane takes a block set
// 2.05 ns per resident thread of an SM, at least kPlaneNs (both fitted on GB300 to 150 measured
// tilings of 256^3, 512^3, 60 x 96^3 and 600 x 32^3, which it orders as measured within 5%).
SweepPlan plan_sweep(std::vector<SweepGrid>& grids, std::vector<SweepGrid>& back) {
  constexpr double kThreadNs = 2.05, kPlaneNs = 300.0;
  struct Shape {
    int N[3], periodic, count;
    int S, TY, hx, hy, threads;
  };
  std::vector<Shape> shapes;
  for (const SweepGrid& G : grids) {
    bool found = false;
    for (Shape& q : shapes)
      if (q.periodic == G.periodic && std::equal(q.N, q.N + 3, G.N)) {
        ++q.count;
        found = true;
        break;
      }
    if (!found) shapes.push_back({{G.N[0], G.N[1], G.N[2]}, G.periodic, 1, 0, 0, 0, 0, 0});
  }
  const int sms = num_sms();
  double best = 1e30;
  std::vector<Shape> best_shapes;
  int best_zc = 32;
  SweepPlan plan;
  for (int limit : {128, 160, 192, 288, 320}) {
    int threads = 0;
    bool ok = true;
    for (Shape& q : shapes) {
      const int strips = q.N[0] / 4;
      double eff = 0;
      for (int S : {strips, 8, 16, 24, 32}) {
        if (S > strips || S < 1) continue;
        for (int TY : {q.N[1], 8, 12, 16, 20, 28, 32, 44}) {
          if (TY > q.N[1]) continue;
          // a tile as wide as the domain wraps around (or ends at its faces) by itself; one
          // as high as a periodic domain too
          const int hx = S == strips ? 0 : 1, hy = TY == q.N[1] && (q.periodic & 2) ? 0 : 2;
          const int th = tile_threads(S, TY, hx, hy);
          if (th > limit) continue;
          const double e = (double)strips * q.N[1] /
                           (2.0 * th * ceil_div(strips, S) * ceil_div(q.N[1], TY));
          if (e > eff) {
            eff = e;
            q.S = S;
            q.TY = TY;
            q.hx = hx;
            q.hy = hy;
            q.threads = th;
          }
        }
      }
      if (eff == 0) ok = false;
      threads = std::max(threads, q.threads);
    }
    if (!ok) continue;
    const int occ = std::min(std::max(65536 / (96 * threads), 1), 32);
    for (int zc : {4, 6, 8, 10, 12, 16, 20, 24, 28, 32, 37, 43, 52, 64, 86, 128}) {
      long long tiles = 0, planes = 0;
      for (const Shape& q : shapes) {
        const int z = std::min(zc, q.N[2]), nz = ceil_div(q.N[2], z);
        const long long t = (long long)q.count * ceil_div(q.N[0] / 4, q.S) * ceil_div(q.N[1], q.TY) * nz;
        tiles += t;
        planes += t * (ceil_div(q.N[2], nz) + 5);
      }
      const double per_tile = (double)planes / tiles;  // planes of an average tile
      const long long slots = (long long)sms * occ;
      const long long waves = tiles / slots, rest = tiles % slots;
      const int tail = (int)((rest + sms - 1) / sms);
      const double cost = per_tile * (waves * std::max(kPlaneNs, kThreadNs * threads * occ) +
                                      (rest ? std::max(kPlaneNs, kThreadNs * threads * tail) : 0.0));
      if (cost < best) {
        best = cost;
        best_shapes = shapes;
        best_zc = zc;
        plan.threads = threads;
      }
    }
  }
  plan.tiles = 0;
  for (size_t i = 0; i < grids.size(); ++i) {
    SweepGrid& G = grids[i];
    for (const Shape& q : best_shapes)
      if (q.periodic == G.periodic && std::equal(q.N, q.N + 3, G.N)) {
        G.S = q.S;
        G.TY = q.TY;
        G.hx = q.hx;
        G.hy = q.hy;
      }
    const int nz = ceil_div(G.N[2], std::min(best_zc, G.N[2]));
    G.ZC = ceil_div(G.N[2], nz);
    G.nt[0] = ceil_div(G.N[0] / 4, G.S);
    G.nt[1] = ceil_div(G.N[1], G.TY);
    G.nt[2] = ceil_div(G.N[2], G.ZC);
    G.tile_begin = plan.tiles;
    plan.tiles += G.nt[0] * G.nt[1] * G.nt[2];
    SweepGrid& B = back[i];
    const float* src = B.src;
    float* dst = B.dst;
    B = G;
    B.src = src;
    B.dst = dst;
  }
  return plan;
}

RestrictPlan plan_restrict(std::vector<RestrictGrid>& grids) {
  long long cols = 0;
  for (RestrictGrid& Q : grids) {
    Q.tiles_xy = ceil_div((Q.g.N[0] / 4) * (Q.g.N[1] / 2), kRestrictThreads);
    cols += (long long)Q.tiles_xy * Q.g.N[2];
  }
  int zc = kRestrictChunk;
  while (zc > 2 && cols / zc < 8ll * num_sms()) zc /= 2;
  RestrictPlan p;
  for (RestrictGrid& Q : grids) {
    Q.ZC = zc;
    Q.tile_begin = p.tiles;
    p.tiles += Q.tiles_xy * ceil_div(Q.g.N[2], zc);
  }
  return p;
}

cudaError_t launch_restrict_f32(const RestrictGrid* grids, int ngrids, const RestrictPlan& p, cudaStream_t s) {
  if (p.tiles <= 0) return cudaSuccess;
  launch_k(k_restrict_f32, (unsigned)p.tiles, kRestrictThreads, 0, s, grids, ngrids);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_sweep_f32(const SweepGrid* grids, int ngrids, const SweepPlan& p, int start,
                             cudaStream_t s) {
  if (p.tiles <= 0) return cudaSuccess;
  const auto k = start == SWEEP_ZERO      ? k_sweep_f32<SWEEP_ZERO>
                 : start == SWEEP_PROLONG ? k_sweep_f32<SWEEP_PROLONG>
                                          : k_sweep_f32<SWEEP_SOURCE>;
  // published pairs: 2 stages x 2 colours x 2 rows of 8 bytes; ring: kDepth planes of 2 rows of
  // phi and rhs, 16 bytes each, and of the two parents
  const size_t smem = (size_t)p.threads * (64 + (64 + (start == SWEEP_PROLONG ? 8 : 0)) * kDepth);
  cudaError_t e = opt_in_smem((const void*)k, smem);
  if (e != cudaSuccess) return e;
  launch_k(k, (unsigned)p.tiles, p.threads, smem, s, grids, ngrids);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_sweep_f32_fabs(const SweepGrid* grid, const SweepPlan& p, int phi_ghosts, cudaStream_t s) {
  // (rows start on 16 bytes, so the first valid cell is as aligned as the ghost cells before it)
  const auto k = phi_ghosts % 2 == 0 ? k_sweep_f32<SWEEP_SOURCE, 8, 4> : k_sweep_f32<SWEEP_SOURCE, 4, 4>;
  const size_t smem = (size_t)p.threads * (64 + 64 * kDepth);
  cudaError_t e = opt_in_smem((const void*)k, smem);
  if (e != cudaSuccess) return e;
  launch_k(k, (unsigned)p.tiles, p.threads, smem, s, grid, 1);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace gbmg
