// The coarse end of the V-cycle in one launch.
//
// Below a few thousand cells a level's stage kernels finish in a microsecond or two, so the
// cycle there is bound by launch latency (about 20 dependent launches per level).  This
// kernel runs the whole sub-cycle from level lc down to the bottom and back inside ONE CTA:
// each level is copied into shared memory as a single dense box (results of this multigrid are
// independent of the box decomposition), and every stage -- red and black half-sweeps, fused
// residual + restriction, exact bottom solve, prolongation -- is the same arithmetic, in the
// same order, as the per-stage kernels, so the result is bit-identical to the multi-launch path.
//
// What bounds it is the chain of stages, each a barrier apart, so a stage is kept short: a thread
// owns the same cells in every stage of a level and works out their neighbours' places once
// (periodic image, or the cell itself, negated, across a Dirichlet face: no ghost cells, no fill
// stage); the residuals of all fine cells are taken side by side before the 8-cell means; in FP64
// every second warp sums on the integer units (mg_isum.hpp), as one SM's FP64 pipe (1.68 lanes a
// clock) would hold each half-sweep of 8^3 cells for a microsecond.  Measured on GB300: FP64 from 8^3
// 33 -> 24 us (ncu, cold), the 64^3 FP64 solve 1.60 -> 1.49 ms, the 64^3 mixed one (FP32 from 16^3)
// 1.16 -> 1.01 ms against the form with ghost cells and fill stages.
#include <cuda_runtime.h>

#include <mutex>

#include "mg_isum_dev.cuh"
#include "mg_kernels.hpp"

namespace gbmg {

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

// Dense level in shared memory, x fastest.
template <class T>
struct Lev {
  T* phi;
  T* rhs;
  int n0, n1, n2;
  int lo;  // lo0 + lo1 + lo2 of the level domain (colour parity)
  T h2, ih2;
  __device__ __forceinline__ int cells() const { return n0 * n1 * n2; }
};

// One cell: its place, its neighbours' (x-, x+, y-, y+, z-, z+), bit f of neg: neighbour f is read
// negated.  o < 0: no cell.
struct Cell {
  int o, nb[6];
  unsigned neg;
};
template <class T>
__device__ __forceinline__ Cell cell_of(const Lev<T>& L, int3 per, int x, int y, int z) {
  const int p = L.n0 * L.n1;
  Cell c;
  c.o = z * p + y * L.n0 + x;
  c.neg = 0;
  const bool e[6] = {x == 0, x == L.n0 - 1, y == 0, y == L.n1 - 1, z == 0, z == L.n2 - 1};
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
template <class T>
__device__ __forceinline__ Cell colour_cell(const Lev<T>& L, int3 per, int color, int t) {
  const int hx = (L.n0 + 1) >> 1;
  const int k = t % hx, r = t / hx, y = r % L.n1, z = r / L.n1;
  const int x = ((color + L.lo + y + z) & 1) + 2 * k;
  Cell c;
  if (z < L.n2 && x < L.n0) return cell_of(L, per, x, y, z);
  c = cell_of(L, per, 0, 0, 0);
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

template <class T>
struct Mine {
  Cell c[2][kKeep<T>];
  bool all;  // the level's cells are all kept; else they are worked out in every stage
  __device__ void init(const Lev<T>& L, int3 per) {
    const int half = ((L.n0 + 1) >> 1) * L.n1 * L.n2;
    all = half <= kKeep<T> * (int)blockDim.x;
    if (!all) return;
#pragma unroll
    for (int q = 0; q < kKeep<T>; ++q)
      if (q * (int)blockDim.x < half) {
        c[0][q] = colour_cell(L, per, 0, threadIdx.x + q * blockDim.x);
        c[1][q] = colour_cell(L, per, 1, threadIdx.x + q * blockDim.x);
      } else {
        c[0][q].o = c[1][q].o = -1;
      }
  }
  // f(cell) for this thread's cells of one colour, in uniform control flow (cells with o < 0 too,
  // their neighbours readable)
  template <class F>
  __device__ __forceinline__ void each(const Lev<T>& L, int3 per, int color, F&& f) const {
    const int half = ((L.n0 + 1) >> 1) * L.n1 * L.n2;
    if (all) {
#pragma unroll
      for (int q = 0; q < kKeep<T>; ++q)
        if ((int)(threadIdx.x & ~31u) + q * (int)blockDim.x < half) f(color ? c[1][q] : c[0][q]);
    } else {
      for (int t = threadIdx.x; (t & ~31) < half; t += blockDim.x) f(colour_cell(L, per, color, t));
    }
  }
};

template <class T>
__device__ void smooth(const Lev<T>& L, const Mine<T>& M, const int3 per, int sweeps, bool ints) {
  for (int s = 0; s < sweeps; ++s)
    for (int color = 0; color < 2; ++color) {
      M.each(L, per, color, [&](const Cell& c) {
        T v[6];
        nbr_vals(L, c, v);
        const int o = c.o < 0 ? 0 : c.o;
        const T u = update_of(sum_of(v, ints, 0xffffffffu), L.rhs[o], L.h2);
        if (c.o >= 0) L.phi[o] = u;
      });
      __syncthreads();
    }
}

// rhs of C = mean of the 8 child residuals of F (x fastest); phi of C = 0.  res: F's residuals.
template <class T>
__device__ void residual_restrict(const Lev<T>& F, const Mine<T>& M, const Lev<T>& C, T* res, const int3 per,
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
  const int nc = C.cells();
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
    C.rhs[i] = A<T>::mul(acc, (T)0.125);
    C.phi[i] = T(0);
  }
}

template <class T>
__device__ void prolong_add(const Lev<T>& C, const Lev<T>& F) {
  const int nf = F.cells();
  for (int i = threadIdx.x; i < nf; i += blockDim.x) {
    const int x = i % F.n0, q = i / F.n0, y = q % F.n1, z = q / F.n1;
    F.phi[i] = A<T>::add(F.phi[i], C.phi[((z >> 1) * C.n1 + (y >> 1)) * C.n0 + (x >> 1)]);
  }
}

template <class T>
__device__ void bottom(const Lev<T>& B, const double* __restrict__ Mt, int N) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    double s = 0.0;
#pragma unroll 8
    for (int j = 0; j < N; ++j) s = __dadd_rn(s, __dmul_rn(Mt[(long long)j * N + i], (double)B.rhs[j]));
    B.phi[i] = (T)s;
  }
}

// 512 threads for FP64 (128 registers each), 1024 for FP32.
template <class T>
__global__ void __launch_bounds__(sizeof(T) == 8 ? 512 : 1024, 1) k_coarse_cycle(const CoarseJob* __restrict__ jobs) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Lev<T> L[kMaxCoarseLevels];
  const CoarseJob& J = jobs[blockIdx.x];
  T* arena = (T*)smem_raw;
  const int nl = J.nlev;
  const int3 per = make_int3(J.periodic[0], J.periodic[1], J.periodic[2]);
  if (threadIdx.x < nl) {
    const CoarseLevel& c = J.lev[threadIdx.x];
    Lev<T> v;
    v.phi = arena + c.off_phi;
    v.rhs = arena + c.off_rhs;
    v.n0 = c.n[0];
    v.n1 = c.n[1];
    v.n2 = c.n[2];
    v.lo = c.lo[0] + c.lo[1] + c.lo[2];
    v.h2 = (T)c.h2;
    v.ih2 = (T)c.ih2;
    L[threadIdx.x] = v;
  }
  T* const res = arena + J.off_res;
  const bool ints = sizeof(T) == 8 && ((threadIdx.x >> 5) & 1);
  // gather phi (the current guess) and rhs of level lc
  T* const gphi = (T*)J.phi;
  const T* const grhs = (const T*)J.rhs;
  {
    const int nc = J.lev[0].n[0] * J.lev[0].n[1] * J.lev[0].n[2];
    T* p = arena + J.lev[0].off_phi;
    T* r = arena + J.lev[0].off_rhs;
    for (int i = threadIdx.x; i < nc; i += blockDim.x) {
      r[i] = grhs[J.off_rhs[i]];
      p[i] = gphi[J.off_phi[i]];
    }
  }
  __syncthreads();
  Mine<T> M;
  for (int k = 0; k + 1 < nl; ++k) {
    M.init(L[k], per);
    smooth(L[k], M, per, J.nu1, ints);
    residual_restrict(L[k], M, L[k + 1], res, per, ints);
    __syncthreads();
  }
  bottom(L[nl - 1], J.Mt, J.N);
  __syncthreads();
  for (int k = nl - 2; k >= 0; --k) {
    if (k < nl - 2) M.init(L[k], per);
    prolong_add(L[k + 1], L[k]);
    __syncthreads();
    smooth(L[k], M, per, J.nu2, ints);
  }
  // scatter phi of level lc back
  {
    const Lev<T>& F = L[0];
    const int nc = F.cells();
    for (int i = threadIdx.x; i < nc; i += blockDim.x) gphi[J.off_phi[i]] = F.phi[i];
  }
}

}  // namespace

size_t coarse_smem_bytes(int dt, const int (*n)[3], int nlev) {
  size_t es = dt == DT_F64 ? 8 : 4, elems = 0;
  for (int k = 0; k < nlev; ++k)
    elems += 2 * (size_t)n[k][0] * n[k][1] * n[k][2];
  return (elems + (size_t)n[0][0] * n[0][1] * n[0][2]) * es;  // phi and rhs of each, residuals of one
}

cudaError_t coarse_opt_in(int dt, size_t smem) {
  return dt == DT_F64 ? opt_in_smem((const void*)k_coarse_cycle<double>, smem)
                      : opt_in_smem((const void*)k_coarse_cycle<float>, smem);
}

cudaError_t launch_coarse_cycle(int dt, const CoarseJob* jobs, int njobs, size_t smem,
                                cudaStream_t s) {
  if (njobs <= 0) return cudaSuccess;
  if (smem > kCoarseSmemMax) return cudaErrorInvalidValue;
  cudaError_t e = coarse_opt_in(dt, smem);
  if (e != cudaSuccess) return e;
  if (dt == DT_F64) launch_k(k_coarse_cycle<double>, njobs, 512, smem, s, jobs);
  else launch_k(k_coarse_cycle<float>, njobs, 1024, smem, s, jobs);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace gbmg
