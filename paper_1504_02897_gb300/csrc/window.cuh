// The window factor of the split algorithm (Eq. 3.9), e^{-|k|^2/k0^2} - 1, from per-axis tables.
//
// Joining the axes' factors a = e^{-k_x^2/k0^2} - 1, .. as (1 + a)(1 + b) - 1 = a + b (1 + a) needs no
// expm1 per mode, and its terms have one sign, so nothing cancels near k = 0.  But an FP32 table rounds
// each axis' factor, and those errors add up.  So FP32 plans hold the tables as head + tail pairs,
// the two axes of a line are joined in FP64, once per line, and a mode's factor is rounded only
// where it is formed: one FMA of the heads (their product exact) plus the tails' part.  Largest
// relative error over the modes |l| < 24 of a 256^3 split (box 48, k0 0.2) 7.4e-8, r.m.s. 8e-9; with
// tables rounded to FP32 and a + b + a b per mode 1.6e-7 and 2.9e-8, with expm1f(-|k|^2/k0^2) of the
// FP32 |k|^2 1.8e-7 and 7e-9.
#pragma once
#include <cmath>

#if defined(__CUDACC__)
#define DDI_HD __host__ __device__ __forceinline__
#else
#define DDI_HD inline
#endif

namespace ddi {
#if !defined(__CUDACC__)
using std::fma;
#endif

// a table entry e^{-k_d^2/k0^2} - 1: head and tail (FP64 plans: the number and 0)
template <typename T>
struct WindowEntry {
  T hi, lo;
};

template <typename T>
DDI_HD WindowEntry<T> window_entry(double v) {
  WindowEntry<T> e;
  e.hi = (T)v;
  e.lo = (T)(v - (double)e.hi);
  return e;
}

// the factor of two joined axes, a = (1 + x)(1 + y) - 1, and E = 1 + a, as head + tail
template <typename T>
struct WindowLine {
  WindowEntry<T> a, E;
};

template <typename T>
DDI_HD WindowLine<T> window_line(WindowEntry<T> x, WindowEntry<T> y) {
  const double u = (double)x.hi + (double)x.lo, v = (double)y.hi + (double)y.lo;
  const double a = fma(v, 1.0 + u, u);
  WindowLine<T> w;
  w.a = window_entry<T>(a);
  w.E = window_entry<T>(1.0 + a);
  return w;
}

// e^{-|k|^2/k0^2} - 1 of a line's mode with the last axis' factor z: a + z E
template <typename T>
DDI_HD T window_join(const WindowLine<T>& w, WindowEntry<T> z) {
  const T tail = fma(z.lo, w.E.hi, fma(z.hi, w.E.lo, w.a.lo));
  return fma(z.hi, w.E.hi, w.a.hi) + tail;
}

}  // namespace ddi
