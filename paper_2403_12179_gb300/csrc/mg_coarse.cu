// The coarse end of the V-cycle in one launch.
//
// Below a few thousand cells a level's stage kernels finish in a microsecond or two, so the
// cycle there is bound by launch latency (about 20 dependent launches per level).  This
// kernel runs the whole sub-cycle from level lc down to the bottom and back in one launch:
// each level is copied into shared memory as a single dense box (results of this multigrid are
// independent of the box decomposition), and every stage -- red and black half-sweeps, fused
// residual + restriction, exact bottom solve, prolongation -- is the same arithmetic, in the
// same order, as the per-stage kernels, so the result is bit-identical to the multi-launch path.
//
// One CTA a job (batches: the jobs fill the SMs), or a cluster of eight for a solve on its own, which
// then starts from a finer level: its larger levels lie in slabs of z-planes over the CTAs, a stage reads
// its own shared memory only -- the neighbours' planes are kept beside the slab, and whoever updates a
// cell of its first or last plane also writes it to the neighbour -- and ends with a cluster barrier;
// the smaller levels are the first CTA's.
//
// What bounds it is the chain of stages, each a barrier apart (1.1 us a stage in one CTA, about 2 us
// in slabs, against 3 to 4 us a launch), so a stage is kept short: a thread owns the same cells in
// every stage of a level and works out their neighbours' places once (periodic image, or the cell
// itself, negated, across a Dirichlet face: no ghost cells, no fill stage); the residuals of all fine
// cells are taken side by side before the 8-cell means; in FP64 half of the warps (every second four, one
// a scheduler) sum on the integer units (mg_isum.hpp), as one SM's FP64 pipe (1.68 lanes a clock) would
// hold each half-sweep of 8^3 cells for a microsecond.  Measured on GB300: FP64 from 8^3 33 -> 24 us (ncu,
// cold), the 64^3 FP64 solve 1.60 -> 1.46 ms, the 64^3 mixed one (FP32 from 16^3) 1.16 -> 0.91 ms against
// the form with ghost cells and fill stages; with the cluster 1.35 and 0.90 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "mg_isum_dev.cuh"
#include "mg_kernels.hpp"

namespace gbmg {

// Cells from which a level is split over the CTAs of a cluster (one CTA does the smaller ones in the
// time that the cluster's barriers take: FP64 8^3 in slabs the same), and the most cells of one CTA
// for which the cluster is the faster way: on GB300, 64^3 FP64 solve (16^3 in slabs of 512 cells) 1.46 -> 1.35
// ms, with 32^3 in slabs of 4096 too 1.83; 64^3 mixed (16^3 in slabs) 0.912 -> 0.899, with 32^3 0.955.
// Clusters of 4 instead of 8: 1.39 and 0.907 ms.
constexpr long long kSplitF64 = 1024, kSplitF32 = 4096, kMostF64 = 1024, kMostF32 = 2048;

namespace {

template <class T>
struct A;
template <>
struct A<double> {
  static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
  static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
  static __device__ __forceinline__ double neg(double a) {
    return __longlong_as_double(__double_as_longlong(a) ^ (long long)0x8000000000000000ull);
  }
};
template <>
struct A<float> {
  static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
  static __device__ __forceinline__ float neg(float a) {
    return __int_as_float(__float_as_int(a) ^ (int)0x80000000u);
  }
};

template <class T>
__device__ __forceinline__ T residual_of(T s, T phi, T rhs, T ih2) {
  return A<T>::fma(A<T>::neg(ih2), A<T>::fma(T(-6), phi, s), rhs);
}
__device__ __forceinline__ float flip_sign(float v, unsigned n) {  // -v if n is 1
  return __int_as_float(__float_as_int(v) ^ (int)(n << 31));
}
__device__ __forceinline__ double flip_sign(double v, unsigned n) { return flip(v, n); }

// Sum of six in order; FP64: on the integer units if `ints` (the same in all lanes of a warp).
__device__ __forceinline__ float sum_of(const float (&v)[6], bool, unsigned) {
  float s = A<float>::add(v[0], v[1]);
#pragma unroll
  for (int i = 2; i < 6; ++i) s = A<float>::add(s, v[i]);
  return s;
}
__device__ __forceinline__ double sum_of(const double (&v)[6], bool ints, unsigned mask) {
  return ints ? sum6_int(v, mask) : sum6_f64(v);
}
__device__ __forceinline__ float update_of(float s, float rhs, float h2) {
  constexpr float inv6 = 1.0f / 6.0f;
  return A<float>::mul(A<float>::fma(A<float>::neg(h2), rhs, s), inv6);
}
__device__ __forceinline__ double update_of(double s, double rhs, double h2) {
  return gs_update<true>(s, rhs, A<double>::neg(h2));
}

// Cluster: another CTA's shared memory (an address of this CTA's mapped to it), and the barrier that
// also makes the writes to it visible.
__device__ __forceinline__ uint32_t peer(const void* p, int rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_peer(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void ld_peer(uint32_t a, double& v) {
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void ld_peer(uint32_t a, float& v) {
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// Dense level in shared memory, x fastest; of a level in slabs this CTA's planes z0 .. z0 + np, phi
// with the neighbouring planes before and after.
template <class T>
struct Lev {
  T* phi;
  T* rhs;
  int n0, n1, n2;
  int lo;  // lo0 + lo1 + lo2 of the level domain (colour parity)
  int planes;       // planes of a slab; 0: whole in the first CTA
  int z0, np;       // this CTA's planes
  uint32_t before, after;  // where the CTAs before and after keep this CTA's first and last plane (0: none)
  T h2, ih2;
  __device__ __forceinline__ int cells() const { return n0 * n1 * np; }
};
template <class T>
__device__ Lev<T> lev_of(const CoarseLevel& c, T* arena, int rank, bool pz) {
  Lev<T> v;
  v.phi = arena + c.off_phi;
  v.rhs = arena + c.off_rhs;
  v.n0 = c.n[0];
  v.n1 = c.n[1];
  v.n2 = c.n[2];
  v.lo = c.lo[0] + c.lo[1] + c.lo[2];
  v.planes = c.planes;
  v.before = v.after = 0;
  v.h2 = (T)c.h2;
  v.ih2 = (T)c.ih2;
  if (!c.planes) {
    v.z0 = 0;
    v.np = rank ? 0 : v.n2;
    return v;
  }
  const int p = v.n0 * v.n1, last = (v.n2 - 1) / c.planes;
  v.z0 = rank * c.planes;
  v.np = max(0, min(c.planes, v.n2 - v.z0));
  if (v.np) {
    const int rb = rank > 0 ? rank - 1 : pz ? last : -1, ra = rank < last ? rank + 1 : pz ? 0 : -1;
    const int npb = rb == last ? v.n2 - last * c.planes : c.planes;  // planes of the CTA before
    if (rb >= 0) v.before = peer(v.phi + npb * p, rb);
    if (ra >= 0) v.after = peer(v.phi - p, ra);
  }
  return v;
}

// One cell: its place, its neighbours' (x-, x+, y-, y+, z-, z+), bit f of neg: neighbour f is read
// negated; its place in a neighbouring CTA's copy (0: none).  o < 0: no cell.
struct Cell {
  int o, nb[6];
  unsigned neg;
  uint32_t copy;
};
template <class T, bool CL>
__device__ __forceinline__ Cell cell_of(const Lev<T>& L, int3 per, int x, int y, int z) {
  const int p = L.n0 * L.n1;
  Cell c;
  c.o = z * p + y * L.n0 + x;
  c.neg = 0;
  c.copy = 0;
  bool e[6] = {x == 0, x == L.n0 - 1, y == 0, y == L.n1 - 1, z == 0, z == L.np - 1};
  if (CL && L.planes) {
    const uint32_t xy = (y * L.n0 + x) * sizeof(T);
    if (e[4] && L.before) c.copy = L.before + xy;
    if (e[5] && L.after) c.copy = L.after + xy;
    e[4] = e[4] && !L.before;  // (elsewhere the plane before is there, at negative places)
    e[5] = e[5] && !L.after;
  }
  const int step[3] = {1, L.n0, p}, wrap[3] = {L.n0 - 1, (L.n1 - 1) * L.n0, (L.n2 - 1) * p};
  const int pd[3] = {per.x, per.y, per.z};
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const int d = f >> 1, s = (f & 1) ? 1 : -1;
    c.nb[f] = !e[f] ? c.o + s * step[d] : pd[d] ? c.o - s * wrap[d] : c.o;
    if (e[f] && !pd[d]) c.neg |= 1u << f;
  }
  return c;
}
// The t-th cell of one colour.
template <class T, bool CL>
__device__ __forceinline__ Cell colour_cell(const Lev<T>& L, int3 per, int color, int t) {
  const int hx = (L.n0 + 1) >> 1;
  const int k = t % hx, r = t / hx, y = r % L.n1, z = r / L.n1;
  const int x = ((color + L.lo + y + L.z0 + z) & 1) + 2 * k;
  Cell c;
  if (z < L.np && x < L.n0) return cell_of<T, CL>(L, per, x, y, z);
  c = cell_of<T, CL>(L, per, 0, 0, 0);
  c.o = -1;
  return c;
}
template <class T>
__device__ __forceinline__ void nbr_vals(const Lev<T>& L, const Cell& c, T (&v)[6]) {
#pragma unroll
  for (int f = 0; f < 6; ++f) v[f] = flip_sign(L.phi[c.nb[f]], (c.neg >> f) & 1u);
}

// Cells a thread keeps of each colour.
template <class T>
constexpr int kKeep = sizeof(T) == 8 ? 1 : 2;

template <class T, bool CL>
struct Mine {
  Cell c[2][kKeep<T>];
  bool all;  // the level's cells are all kept; else they are worked out in every stage
  __device__ void init(const Lev<T>& L, int3 per) {
    const int half = ((L.n0 + 1) >> 1) * L.n1 * L.np;
    all = half <= kKeep<T> * (int)blockDim.x;
    if (!all) return;
#pragma unroll
    for (int q = 0; q < kKeep<T>; ++q)
      if (q * (int)blockDim.x < half) {
        c[0][q] = colour_cell<T, CL>(L, per, 0, threadIdx.x + q * blockDim.x);
        c[1][q] = colour_cell<T, CL>(L, per, 1, threadIdx.x + q * blockDim.x);
      } else {
        c[0][q].o = c[1][q].o = -1;
      }
  }
  // f(cell) for this thread's cells of one colour, in uniform control flow (cells with o < 0 too,
  // their neighbours readable)
  template <class F>
  __device__ __forceinline__ void each(const Lev<T>& L, int3 per, int color, F&& f) const {
    const int half = ((L.n0 + 1) >> 1) * L.n1 * L.np;
    if (all) {
#pragma unroll
      for (int q = 0; q < kKeep<T>; ++q)
        if ((int)(threadIdx.x & ~31u) + q * (int)blockDim.x < half) f(color ? c[1][q] : c[0][q]);
    } else {
      for (int t = threadIdx.x; (t & ~31) < half; t += blockDim.x) f(colour_cell<T, CL>(L, per, color, t));
    }
  }
};

// Barrier of a level's stages: of the cluster for a level in slabs.
template <class T, bool CL>
__device__ __forceinline__ void level_sync(const Lev<T>& L) {
  if (CL && L.planes) cluster_sync();
  else __syncthreads();
}

template <class T, bool CL>
__device__ void smooth(const Lev<T>& L, const Mine<T, CL>& M, const int3 per, int sweeps, bool ints) {
  for (int s = 0; s < sweeps; ++s)
    for (int color = 0; color < 2; ++color) {
      M.each(L, per, color, [&](const Cell& c) {
        T v[6];
        nbr_vals(L, c, v);
        const int o = c.o < 0 ? 0 : c.o;
        const T u = update_of(sum_of(v, ints, 0xffffffffu), L.rhs[o], L.h2);
        if (c.o >= 0) {
          L.phi[o] = u;
          if (CL && c.copy) st_peer(c.copy, u);
        }
      });
      level_sync<T, CL>(L);
    }
}

// rhs of C = mean of the 8 child residuals of F (x fastest); phi of C = 0.  res: F's residuals.
template <class T, bool CL>
__device__ void residual_restrict(const Lev<T>& F, const Mine<T, CL>& M, const Lev<T>& C, T* res, const int3 per,
                                  bool ints) {
  for (int color = 0; color < 2; ++color)
    M.each(F, per, color, [&](const Cell& c) {
      T v[6];
      nbr_vals(F, c, v);
      const int o = c.o < 0 ? 0 : c.o;
      const T r = residual_of(sum_of(v, ints, 0xffffffffu), F.phi[o], F.rhs[o], F.ih2);
      if (c.o >= 0) res[o] = r;
    });
  __syncthreads();
  const int pc = C.n0 * C.n1, nc = pc * (F.np >> 1);
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    const int X = i % C.n0, q = i / C.n0, Y = q % C.n1, Z = q / C.n1;
    const T* r = res + (2 * Z * F.n1 + 2 * Y) * F.n0 + 2 * X;
    const int p = F.n0 * F.n1;
    T acc = A<T>::add(r[0], r[1]);
    acc = A<T>::add(acc, r[F.n0]);
    acc = A<T>::add(acc, r[F.n0 + 1]);
    acc = A<T>::add(acc, r[p]);
    acc = A<T>::add(acc, r[p + 1]);
    acc = A<T>::add(acc, r[p + F.n0]);
    acc = A<T>::add(acc, r[p + F.n0 + 1]);
    acc = A<T>::mul(acc, (T)0.125);
    if (CL && F.planes) {
      const int Zd = (F.z0 >> 1) + Z, owner = C.planes ? Zd / C.planes : 0;
      st_peer(peer(C.rhs + (Zd - owner * C.planes) * pc + (i - Z * pc), owner), acc);
    } else {
      C.rhs[i] = acc;
    }
  }
  const int before = CL && C.planes ? pc : 0;  // the neighbours' planes too
  for (int i = threadIdx.x; i < C.cells() + 2 * before; i += blockDim.x) C.phi[i - before] = T(0);
  level_sync<T, CL>(F);
}

template <class T, bool CL>
__device__ void prolong_add(const Lev<T>& C, const Lev<T>& F) {
  const int nf = F.cells(), pf = F.n0 * F.n1;
  for (int i = threadIdx.x; i < nf; i += blockDim.x) {
    const int x = i % F.n0, q = i / F.n0, y = q % F.n1, z = q / F.n1;
    const int Z = (F.z0 + z) >> 1, xy = (y >> 1) * C.n0 + (x >> 1);
    T e;
    if (CL && F.planes) {
      const int owner = C.planes ? Z / C.planes : 0;
      ld_peer(peer(C.phi + (Z - owner * C.planes) * C.n0 * C.n1 + xy, owner), e);
    } else {
      e = C.phi[Z * C.n0 * C.n1 + xy];
    }
    const T u = A<T>::add(F.phi[i], e);
    F.phi[i] = u;
    if (CL && F.planes) {
      if (z == 0 && F.before) st_peer(F.before + i * (uint32_t)sizeof(T), u);
      if (z == F.np - 1 && F.after) st_peer(F.after + (i - z * pf) * (uint32_t)sizeof(T), u);
    }
  }
}

// Rows [i0, i1) of the exact bottom solve; phi(i, value) takes them.
template <class T, class F>
__device__ void bottom(const T* rhs, const double* __restrict__ Mt, int N, int i0, int i1, F&& phi) {
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    double s = 0.0;
#pragma unroll 16
    for (int j = 0; j < N; ++j) s = __dadd_rn(s, __dmul_rn(Mt[(long long)j * N + i], (double)rhs[j]));
    phi(i, (T)s);
  }
}
// Cells from which the bottom solve's rows are spread over the CTAs of a cluster: one SM's FP64 pipe
// takes 2 N^2 / 1.68 clocks (27 us for 210 cells).  Against stage launches and the bottom kernel: 88 x 88 x 56
// (bottom of 847 cells) 2.10 -> 2.00 ms, 88 x 56 x 56 (539) 1.69 -> 1.55, 72 x 72 x 40 (405) 1.43 -> 1.32.
constexpr int kBottomSpread = 64;

// 512 threads for FP64 (128 registers each), 1024 for FP32.  RANKS: CTAs of a job, a cluster.
// Every CTA of a cluster passes the same cluster barriers: one after the gather, those of the levels
// in slabs, two around a bottom solve that is spread, and one between the levels of the first CTA alone
// and those in slabs.
template <class T, int RANKS>
__global__ void __launch_bounds__(sizeof(T) == 8 ? 512 : 1024, 1) k_coarse_cycle(const CoarseJob* __restrict__ jobs) {
  constexpr bool CL = RANKS > 1;
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Lev<T> L[kMaxCoarseLevels];
  const CoarseJob& J = jobs[blockIdx.x / RANKS];
  const int rank = blockIdx.x % RANKS;
  T* arena = (T*)smem_raw;
  const int nl = J.nlev, ns = CL ? J.nslab : 0;
  const int3 per = make_int3(J.periodic[0], J.periodic[1], J.periodic[2]);
  if (threadIdx.x < nl) L[threadIdx.x] = lev_of(J.lev[threadIdx.x], arena, rank, J.periodic[2] != 0);
  T* const res = arena + J.off_res;
  const bool ints = sizeof(T) == 8 && ((threadIdx.x >> 7) & 1);
  __syncthreads();
  // gather phi (the current guess) and rhs of level lc
  T* const gphi = (T*)J.phi;
  const T* const grhs = (const T*)J.rhs;
  {
    const Lev<T>& F = L[0];
    const int pf = F.n0 * F.n1, first = F.z0 * pf, nc = F.cells();
    for (int i = threadIdx.x; i < nc; i += blockDim.x) {
      F.rhs[i] = grhs[J.off_rhs[first + i]];
      F.phi[i] = gphi[J.off_phi[first + i]];
    }
    if (CL && F.planes && nc) {  // the neighbours' planes
      const int zb = F.z0 > 0 ? F.z0 - 1 : F.n2 - 1, za = F.z0 + F.np < F.n2 ? F.z0 + F.np : 0;
      for (int i = threadIdx.x; i < pf; i += blockDim.x) {
        if (F.before) F.phi[i - pf] = gphi[J.off_phi[zb * pf + i]];
        if (F.after) F.phi[nc + i] = gphi[J.off_phi[za * pf + i]];
      }
    }
  }
  if (CL) cluster_sync();
  else __syncthreads();
  Mine<T, CL> M;
  for (int k = 0; k + 1 < nl; ++k) {
    if (CL && k >= ns && rank) break;
    M.init(L[k], per);
    smooth<T, CL>(L[k], M, per, J.nu1, ints);
    residual_restrict<T, CL>(L[k], M, L[k + 1], res, per, ints);
  }
  const Lev<T>& B = L[nl - 1];
  const bool spread = CL && J.N >= kBottomSpread;
  if (spread) {
    cluster_sync();
    if (rank)
      for (int i = threadIdx.x; i < J.N; i += blockDim.x) ld_peer(peer(B.rhs + i, 0), B.rhs[i]);
    __syncthreads();
    bottom(B.rhs, J.Mt, J.N, J.N * rank / RANKS, J.N * (rank + 1) / RANKS,
           [&](int i, T v) { st_peer(peer(B.phi + i, 0), v); });
    cluster_sync();
  }
  if (!CL || !rank) {
    if (!spread) bottom(B.rhs, J.Mt, J.N, 0, J.N, [&](int i, T v) { B.phi[i] = v; });
    __syncthreads();
    for (int k = nl - 2; k >= ns; --k) {
      if (k < nl - 2) M.init(L[k], per);
      prolong_add<T, CL>(L[k + 1], L[k]);
      __syncthreads();
      smooth<T, CL>(L[k], M, per, J.nu2, ints);
    }
  }
  if (CL) {
    cluster_sync();
    for (int k = ns - 1; k >= 0; --k) {
      if (k < nl - 2) M.init(L[k], per);
      prolong_add<T, CL>(L[k + 1], L[k]);
      cluster_sync();
      smooth<T, CL>(L[k], M, per, J.nu2, ints);
    }
  }
  // scatter phi of level lc back
  {
    const Lev<T>& F = L[0];
    const int nc = F.cells(), first = F.z0 * F.n0 * F.n1;
    for (int i = threadIdx.x; i < nc; i += blockDim.x) gphi[J.off_phi[first + i]] = F.phi[i];
  }
}

}  // namespace

size_t coarse_layout(int dt, CoarseJob& J, bool cluster, bool bounded) {
  // Cells from which a level is split over the CTAs: below, a cluster barrier a stage costs more than
  // the one CTA's work.
  const long long split = dt == DT_F64 ? kSplitF64 : kSplitF32;
  J.ranks = 1;
  J.nslab = 0;
  long long off = 0, res = 0;
  bool prefix = cluster;
  for (int k = 0; k < J.nlev; ++k) {
    CoarseLevel& V = J.lev[k];
    const long long p = (long long)V.n[0] * V.n[1];
    V.planes = V.pad_ = 0;
    if (prefix && k + 1 < J.nlev && p * V.n[2] >= split && V.n[2] >= 4) {
      V.planes = 2 * ((V.n[2] / 2 + kCoarseRanks - 1) / kCoarseRanks);
      J.ranks = kCoarseRanks;
      ++J.nslab;
    } else {
      prefix = false;
    }
    const long long mine = p * (V.planes ? V.planes : V.n[2]);
    if (bounded && mine > (dt == DT_F64 ? kMostF64 : kMostF32)) return 0;
    off += V.planes ? p : 0;
    V.off_phi = (int)off;
    off += mine + (V.planes ? p : 0);
    V.off_rhs = (int)off;
    off += mine;
    if (k + 1 < J.nlev) res = std::max(res, mine);
  }
  J.off_res = (int)off;
  return (size_t)(off + res) * (dt == DT_F64 ? 8 : 4);
}

cudaError_t coarse_opt_in(int dt, size_t smem, int ranks) {
  const void* k = dt == DT_F64 ? (ranks > 1 ? (const void*)k_coarse_cycle<double, kCoarseRanks> : (const void*)k_coarse_cycle<double, 1>)
                               : (ranks > 1 ? (const void*)k_coarse_cycle<float, kCoarseRanks> : (const void*)k_coarse_cycle<float, 1>);
  return opt_in_smem(k, smem);
}

cudaError_t launch_coarse_cycle(int dt, const CoarseJob* jobs, int njobs, size_t smem,
                                cudaStream_t s, int ranks) {
  if (njobs <= 0) return cudaSuccess;
  if (smem > kCoarseSmemMax || (ranks != 1 && ranks != kCoarseRanks)) return cudaErrorInvalidValue;
  cudaError_t e = coarse_opt_in(dt, smem, ranks);
  if (e != cudaSuccess) return e;
  const int th = dt == DT_F64 ? 512 : 1024;
  if (ranks > 1) {
    if (dt == DT_F64) launch_cluster_k(ranks, k_coarse_cycle<double, kCoarseRanks>, njobs * ranks, th, smem, s, jobs);
    else launch_cluster_k(ranks, k_coarse_cycle<float, kCoarseRanks>, njobs * ranks, th, smem, s, jobs);
  } else {
    if (dt == DT_F64) launch_k(k_coarse_cycle<double, 1>, njobs, th, smem, s, jobs);
    else launch_k(k_coarse_cycle<float, 1>, njobs, th, smem, s, jobs);
  }
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace gbmg
