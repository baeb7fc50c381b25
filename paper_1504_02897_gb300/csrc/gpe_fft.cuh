// The GPE's Fourier passes over the plan's n[0] x n[1] x n[2] grid, instantiated for FP32 and FP64
// by gpe_fft_f32.cu and gpe_fft_f64.cu.
//
// A multiplier in Fourier space (the kinetic phase, the gradient flow's solve) takes five passes
// in 3D instead of seven: x and y forward, then the last axis forward, multiplied and back in
// one pass (k_fft_pair), then y and x back.  What the steps do pointwise before or after rides on
// the x passes: |psi|^2 is written as the last pass stores psi, the gradient flow's right-hand side
// is formed as the first pass loads, and its change max |new - old| as the last one stores.
// Measured at 128^3 FP32: a time step without its DDI 105 -> 62 us; the grid (17 MB) stays in L2.
// Every pass applies the FP32 twiddles as head + tail: these transforms repeat on the same data.
#pragma once
#include "fft_core.cuh"

namespace ddi {
namespace {
using namespace fftcore;

struct GridDims3 {
  int n[3];
};

// v * k for a constant known in FP64: head + tail in FP32 (a rounded 1/N would scale the
// state by the same wrong factor every step)
template <typename T>
__device__ __forceinline__ T scale_const(T v, double k) {
  if constexpr (sizeof(T) == 4) {
    const float hi = (float)k;
    return fmaf(v, hi, v * (float)(k - (double)hi));
  } else {
    return v * (T)k;
  }
}

struct GpePolicy : PolicyBase {
  static constexpr bool kPrecise = true;
};

// rows along x, from src to data (they may be the same); RHO: also writes |v|^2 of what it stores
template <typename T, bool RHO>
struct GridX : GpePolicy {
  using C = cx_t<T>;
  using Ref = int;  // grids hold < 2^31 points
  const C* src;
  C* data;
  T* rho;
  GridDims3 d;
  __host__ __device__ long long nlines() const { return (long long)d.n[1] * d.n[2]; }
  static constexpr bool kStrided = false;
  __device__ Ref ref(long long L) const { return (int)L * d.n[0]; }
  __device__ C load(Ref r, int i) const { return chain_load(src + (r + i)); }
  __device__ void store(Ref r, int i, C v, Acc&) const {
    data[r + i] = v;
    if (RHO) rho[r + i] = v.x * v.x + v.y * v.y;
  }
};

// lines along y (axis 1) or z (axis 2), in place
template <typename T>
struct GridLines : GpePolicy {
  using C = cx_t<T>;
  using Ref = int;  // grids hold < 2^31 points
  C* data;
  GridDims3 d;
  int axis;
  __host__ __device__ long long nlines() const { return (long long)d.n[0] * (axis == 1 ? d.n[2] : d.n[1]); }
  __device__ Ref ref(long long L) const {
    if (axis == 2) return (int)L;
    const int q = (int)((unsigned)L / (unsigned)d.n[0]);
    return q * d.n[0] * d.n[1] + ((int)L - q * d.n[0]);
  }
  __device__ int at(Ref r, int i) const { return r + i * (axis == 1 ? d.n[0] : d.n[0] * d.n[1]); }
  __device__ C load(Ref r, int i) const { return chain_load(data + at(r, i)); }
  __device__ void store(Ref r, int i, C v, Acc&) const { data[at(r, i)] = v; }
};

// the last axis forward, times the kinetic phase e^{i f |mu|^2} / N_tot, and back.  tab: the
// per-axis tables of e - 1, combined as (1+A)(1+B)(1+C) - 1 = P + C + C P with P = A + B + A B
template <typename T>
struct KineticRef {
  int off;
  cx_t<T> P;  // the other axes' factor minus 1
};
template <typename T>
struct KineticPair : GridLines<T> {
  using C = cx_t<T>;
  using Ref = KineticRef<T>;
  using typename GridLines<T>::Acc;
  const C* tab;
  double inv_n;
  __device__ Ref ref(long long L) const {
    const int x = (int)(L % this->d.n[0]);
    const C A = tab[x];
    if (this->axis == 1) return Ref{GridLines<T>::ref(L), A};
    const C B = tab[this->d.n[0] + (int)(L / this->d.n[0])];
    return Ref{(int)L, cadd(cadd(A, B), cmul(A, B))};
  }
  __device__ C load(const Ref& r, int i) const { return GridLines<T>::load(r.off, i); }
  __device__ C apply(const Ref& r, int i, C v) const {
    const C Z = chain_load(tab + this->d.n[0] + (this->axis == 2 ? this->d.n[1] : 0) + i);
    const C E = cadd(cadd(r.P, Z), cmul(Z, r.P));
    const C o = cadd(v, cmul(v, E));
    return cmk<C>(scale_const(o.x, inv_n), scale_const(o.y, inv_n));
  }
  __device__ void store(const Ref& r, int i, C v, Acc& a) const { GridLines<T>::store(r.off, i, v, a); }
};

// ---- gradient flow: one sweep of the fixed point ---------------------------------------------------
// A sweep is skipped once an earlier one has converged: prev holds the last sweep's largest
// |change|^2 (FP64 bits; cleared before the first sweep, so the sweeps after a skipped one skip too)
struct GfSkip {
  const unsigned long long* prev;
  double tol2;
  __device__ bool done() const { return prev && __longlong_as_double((long long)*prev) <= tol2; }
};

// x forward of phi/dt + (alpha - W) cur
template <typename T>
struct GfRhsX : GpePolicy {
  using C = cx_t<T>;
  using Ref = int;  // grids hold < 2^31 points
  const C *phi, *cur;
  C* out;
  const T* W;
  T alpha, inv_dt;
  GridDims3 d;
  GfSkip sk;
  __host__ __device__ long long nlines() const { return (long long)d.n[1] * d.n[2]; }
  __device__ bool skip() const { return sk.done(); }
  static constexpr bool kStrided = false;
  __device__ Ref ref(long long L) const { return (int)L * d.n[0]; }
  __device__ C load(Ref r, int i) const {
    const T f = alpha - chain_load(W + (r + i));
    const C a = phi[r + i], c = cur[r + i];
    return cmk<C>(a.x * inv_dt + f * c.x, a.y * inv_dt + f * c.y);
  }
  __device__ void store(Ref r, int i, C v, Acc&) const { out[r + i] = v; }
};

template <typename T>
struct GfLines : GridLines<T> {
  GfSkip sk;
  __device__ bool skip() const { return sk.done(); }
};

// the last axis forward, divided by (1/dt + alpha + |mu|^2/2) and N_tot, and back (in the working
// precision: the fixed point's own tolerance is the plan's)
template <typename T>
struct GfSolveRef {
  int off;
  T m2;
};
template <typename T>
struct GfSolvePair : GridLines<T> {
  using C = cx_t<T>;
  using Ref = GfSolveRef<T>;
  using typename GridLines<T>::Acc;
  GfSkip sk;
  T ksx, ksy, ksl;  // 2 pi / len along x, y and the last axis
  int nl;           // points of the last axis
  T c0, sc;
  __device__ bool skip() const { return sk.done(); }
  __device__ static T mu2(int l, int n, T ks) {
    const T m = (T)(l < n / 2 ? l : l - n) * ks;
    return m * m;
  }
  __device__ Ref ref(long long L) const {
    const int x = (int)(L % this->d.n[0]);
    T m2 = mu2(x, this->d.n[0], ksx);
    if (this->axis == 2) m2 += mu2((int)(L / this->d.n[0]), this->d.n[1], ksy);
    return Ref{GridLines<T>::ref(L), m2};
  }
  __device__ C load(const Ref& r, int i) const { return GridLines<T>::load(r.off, i); }
  __device__ C apply(const Ref& r, int i, C v) const {
    const T m2 = r.m2 + mu2(i, nl, ksl);
    return cscale(v, sc / (c0 + (T)0.5 * m2));
  }
  __device__ void store(const Ref& r, int i, C v, Acc& a) const { GridLines<T>::store(r.off, i, v, a); }
};

// x inverse; the largest |stored - cur|^2 (in the working precision; a non-finite difference counts
// as infinite) goes to *change
template <typename T>
struct GfChangeX : GpePolicy {
  using C = cx_t<T>;
  using Ref = int;  // grids hold < 2^31 points
  struct Acc {
    T m;
  };
  C* data;
  const C* cur;
  unsigned long long* change;
  GridDims3 d;
  GfSkip sk;
  __host__ __device__ long long nlines() const { return (long long)d.n[1] * d.n[2]; }
  __device__ bool skip() const { return sk.done(); }
  static constexpr bool kStrided = false;
  __device__ Ref ref(long long L) const { return (int)L * d.n[0]; }
  __device__ C load(Ref r, int i) const { return chain_load(data + (r + i)); }
  __device__ void store(Ref r, int i, C v, Acc& a) const {
    data[r + i] = v;
    const C y = cur[r + i];
    const T dr = v.x - y.x, di = v.y - y.y;
    const T d2 = dr * dr + di * di;
    a.m = isfinite(d2) ? (d2 > a.m ? d2 : a.m) : (T)INFINITY;
  }
  // maxima of non-negative numbers: the order of their bits is theirs, and the result does not depend
  // on the order of the atomics
  __device__ void finish(const Acc& a) const {
    __shared__ unsigned long long top;
    if (threadIdx.x == 0) top = 0;
    __syncthreads();
    T m = a.m;
    for (int o = 16; o > 0; o >>= 1) {  // CTAs of contiguous lines are whole warps (launch_policy)
      const T q = __shfl_xor_sync(0xffffffffu, m, o);
      m = q > m ? q : m;
    }
    if (threadIdx.x % 32 == 0) atomicMax(&top, (unsigned long long)__double_as_longlong((double)m));
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(change, top);
  }
};

template <typename T, int DIR, typename P>
int grid_pass(const Plan& p, int axis, const P& pol, cudaStream_t s) {
  return dispatch_policy<T, DIR, 8, 1024>(p, p.n[axis], pol, s);
}
GridDims3 grid_dims(const Plan& p) { return GridDims3{{p.n[0], p.n[1], p.n[2]}}; }

}  // namespace

template <typename T>
int gpe_forward(Plan& p, const cx_t<T>* src, cx_t<T>* a, cudaStream_t s) {
  const GridDims3 d = grid_dims(p);
  DDI_TRY((grid_pass<T, -1>(p, 0, GridX<T, false>{{}, src, a, nullptr, d}, s)));
  for (int ax = 1; ax < p.dim; ++ax) DDI_TRY((grid_pass<T, -1>(p, ax, GridLines<T>{{}, a, d, ax}, s)));
  return DDI_OK;
}

template <typename T>
int gpe_kinetic(Plan& p, const cx_t<T>* src, cx_t<T>* a, const cx_t<T>* tab, T* rho, cudaStream_t s) {
  const GridDims3 d = grid_dims(p);
  const int last = p.dim - 1;
  DDI_TRY((grid_pass<T, -1>(p, 0, GridX<T, false>{{}, src, a, nullptr, d}, s)));
  if (last == 2) DDI_TRY((grid_pass<T, -1>(p, 1, GridLines<T>{{}, a, d, 1}, s)));
  DDI_TRY((grid_pass<T, 0>(p, last, KineticPair<T>{{{}, a, d, last}, tab, 1.0 / (double)p.grid_points()}, s)));
  if (last == 2) DDI_TRY((grid_pass<T, +1>(p, 1, GridLines<T>{{}, a, d, 1}, s)));
  if (rho) return grid_pass<T, +1>(p, 0, GridX<T, true>{{}, a, a, rho, d}, s);
  return grid_pass<T, +1>(p, 0, GridX<T, false>{{}, a, a, nullptr, d}, s);
}

template <typename T>
int gpe_gf_sweep(Plan& p, const GfSweep<T>& w, cudaStream_t s) {
  const GridDims3 d = grid_dims(p);
  const int last = p.dim - 1;
  const GfSkip sk{w.prev, w.tol2};
  DDI_TRY((grid_pass<T, -1>(p, 0,
                            GfRhsX<T>{{}, w.phi, w.cur, w.out, w.W, w.alpha, w.inv_dt, d, sk}, s)));
  if (last == 2) DDI_TRY((grid_pass<T, -1>(p, 1, GfLines<T>{{{}, w.out, d, 1}, sk}, s)));
  DDI_TRY((grid_pass<T, 0>(p, last,
                           GfSolvePair<T>{{{}, w.out, d, last},
                                          sk,
                                          (T)w.ks[0],
                                          (T)w.ks[1],
                                          (T)w.ks[last],
                                          p.n[last],
                                          (T)w.inv_dt_alpha,
                                          (T)(1.0 / (double)p.grid_points())},
                           s)));
  if (last == 2) DDI_TRY((grid_pass<T, +1>(p, 1, GfLines<T>{{{}, w.out, d, 1}, sk}, s)));
  return grid_pass<T, +1>(p, 0, GfChangeX<T>{{}, w.out, w.cur, w.change, d, sk}, s);
}

}  // namespace ddi
