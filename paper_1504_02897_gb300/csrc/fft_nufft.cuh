// Fine-grid FFTs of the NUFFT with the zero padding and the cropping built in, instantiated for
// FP32 and FP64 by fft_nufft_f32.cu and fft_nufft_f64.cu.
//
// The type-2 input occupies the n^d centred positions j' mod nf (j' = -n/2..n/2-1) of the
// 2n-oversampled grid and the type-1 output is read back at the same positions.  The density is
// real, so one half of the spectrum holds all of it, and one node of each (k, -k) pair is
// processed, the one with k_y >= 0 (the first half of the azimuth): its taps lie on about half of
// the fine y lines (the plan finds the shortest cyclic range holding all of them).  So in 3D y is
// transformed first and returned last, and every other pass works on the lines of that range only:
//   forward  y: the n_x n_z lines of the density (read straight from rho: pad and deconvolution
//               fused); only the y lines of the range are stored, in the first n_x cells of
//               their fine-grid rows;
//            x: the rows on those y lines, from n_x cells to the whole row, in place;
//            z: the columns on those y lines; elements outside the block read as zero.
//   inverse  z: the same columns; only the z in the block are stored;
//            x: the rows on those y lines, back to the first n_x cells of the row;
//            y: the n_x n_z lines; the y lines off the range are zero (no tap reaches them); the
//               y in the block are stored as Re(u) / psihat into phi (crop, deconvolution and real
//               part fused).
// (Transforming x first, as this file did, carries whole x rows of every y through two passes:
// 128^3 FP32 48 + 42 us for the x and y passes of the two directions against 36 + 31 us now.)
// The NUFFT passes run once per evaluation and use the twiddles' FP32 heads only (the
// path's error budget is 1e-6); the GPE's repeated transforms use heads and tails.
// Split plans (Eq. 3.9): the ball's taps lie in a band of y and x lines around k = 0, and the same
// passes run on those lines.  The smooth part I_1 runs them on the y lines 0..nf/2, the half
// spectrum of the real density, without the deconvolution, and its z passes are one: forward,
// symbol, inverse.
// Grid positions that are not read are never written in the same evaluation, so no
// zero-fill of the fine grid is needed.  Each CTA reads its own lines before it writes
// them and no other CTA of the pass touches them; the kernel before may still be writing them when
// the pass starts, so they are read coherently (chain_load, common.cuh).
#pragma once
#include "fft_core.cuh"
#include "window.cuh"

namespace ddi {
namespace {
using namespace fftcore;

struct Axis {
  int n;   // grid points
  int nf;  // fine points
  // grid index j (0..n-1) of fine position l in the block
  __host__ __device__ int grid_of(int l) const { return l < n / 2 ? l + n / 2 : l - (nf - n / 2); }
  // fine position of grid index j
  __host__ __device__ int fine_of(int j) const { return j < n / 2 ? j - n / 2 + nf : j - n / 2; }
};

template <typename T>
struct Geo {
  using C = cx_t<T>;
  Axis ax, ay, az;
  // deconvolution factors 1 / psihat, FP64 (x: [0, n0), y: [n0, n0 + n1), z: after), and for
  // FP32 plans the y factors (2D: x) as FP32 head + tail pairs (the FP64 value to ~2^-48)
  const double* dc;
  const float2* dcx2;
  C* fine;
  // the fine-grid y lines that hold node taps: ylo, ylo + 1, .. (mod nf_y), nyr of them; and
  // the x lines (xlo, .., nxr of them; every line except for split plans' ball)
  int ylo, nyr;
  int xlo, nxr;
  int* nonfinite;  // set when the pad pass reads a NaN / Inf
  int* counters;   // the work counters of the spread and the interpolation, cleared by the pad pass
  int sz;  // fine cells per plane
  // offsets into the fine grid (at most 1024^3 cells) and into rho / phi fit 32 bits
  __device__ int fidx(int lz, int ly, int lx) const { return lz * sz + ly * ax.nf + lx; }
  __host__ __device__ bool in_yr(int l) const {
    int d = l - ylo;
    if (d < 0) d += ay.nf;
    return d < nyr;
  }
  __host__ __device__ bool in_xr(int l) const {
    int d = l - xlo;
    if (d < 0) d += ax.nf;
    return d < nxr;
  }
  __host__ __device__ int yr_line(int i) const {
    const int l = ylo + i;
    return l >= ay.nf ? l - ay.nf : l;
  }
  __host__ __device__ int xr_line(int i) const {
    const int l = xlo + i;
    return l >= ax.nf ? l - ax.nf : l;
  }
};

// lines of the density and the potential: along y, one per (x, z) of the grid (3D), or rows (2D)
template <typename T>
struct YRef {
  int grid;        // offset of the line's first element in rho / phi
  int fine;        // the same in the fine grid (3D: row y of plane z, cell x)
  T hi, lo;        // the line's deconvolution factor (FP64 product of the other axes'): FP64 value, or FP32
                   // head + tail
};

template <typename T>
__device__ __forceinline__ YRef<T> line_ref(int grid, int fine, double f) {
  YRef<T> r;
  r.grid = grid;
  r.fine = fine;
  r.hi = (T)f;
  r.lo = sizeof(T) == 4 ? (T)(f - (double)r.hi) : (T)0;
  return r;
}

template <typename T>
__device__ __forceinline__ YRef<T> y_ref(const Geo<T>& g, long long L) {
  const int jz = (int)((unsigned)L / (unsigned)g.ax.n), jx = (int)L - jz * g.ax.n;
  return line_ref<T>(jz * g.ay.n * g.ax.n + jx, g.fidx(g.az.fine_of(jz), 0, jx),
                     g.dc[jx] * g.dc[g.ax.n + g.ay.n + jz]);
}

// v times the deconvolution factor of element j of line r (d: the FP64 factors along the line),
// rounded once: in FP64 directly; in FP32 the factor dx dy dz is formed as a head + tail pair (the
// exact product error of the heads by an FMA plus the cross terms), so only the final product is
// rounded
template <typename T>
__device__ __forceinline__ T deconv(const Geo<T>& g, const double* d, const YRef<T>& r, int j, T v) {
  if constexpr (sizeof(T) == 8) {
    return v * (d[j] * r.hi);
  } else {
    const float2 f = __ldg(g.dcx2 + j);
    const float ph = f.x * r.hi;
    const float pe = fmaf(f.x, r.hi, -ph) + fmaf(f.x, r.lo, f.y * r.hi);
    return fmaf(v, ph, v * pe);
  }
}

// an element of the density: its deconvolved value, with a NaN / Inf recorded (a policy's use(), after
// the loads: no load passes the atomic, and with each element loaded and recorded in turn the 256^3
// pads took 121 us each instead of 93)
template <typename T>
__device__ __forceinline__ cx_t<T> pad_value(const Geo<T>& g, const double* d, const YRef<T>& r, int j, T v) {
  if (!isfinite(v) && *(volatile int*)g.nonfinite == 0) atomicOr(g.nonfinite, 1);
  return cmk<cx_t<T>>(deconv<T>(g, d, r, j, v), (T)0);
}

template <typename T>
struct PadY : PolicyBase {
  using C = cx_t<T>;
  using Ref = YRef<T>;
  static constexpr bool kBlockIn = true;
  Geo<T> g;
  const T* rho;
  __host__ __device__ long long nlines() const { return (long long)g.ax.n * g.az.n; }
  __device__ Ref ref(long long L) const { return y_ref<T>(g, L); }
  __device__ void begin() const {
    if (blockIdx.x == 0 && threadIdx.x < 2) g.counters[threadIdx.x] = 0;
  }
  __device__ C load(const Ref& r, int i) const {
    return cmk<C>(chain_load(rho + (r.grid + g.ay.grid_of(i) * g.ax.n)), (T)0);
  }
  __device__ C use(const Ref& r, int i, C v) const {
    return pad_value<T>(g, g.dc + g.ax.n, r, g.ay.grid_of(i), v.x);
  }
  __device__ void store(const Ref& r, int i, C v, Acc&) const {
    if (g.in_yr(i)) g.fine[r.fine + i * g.ax.nf] = v;
  }
};

// inverse y with crop, deconvolution and real part; ACC adds the result to phi instead of
// storing it
template <typename T, bool ACC>
struct CropY : PolicyBase {
  using C = cx_t<T>;
  using Ref = YRef<T>;
  static constexpr bool kBlockOut = true;
  Geo<T> g;
  T* phi;
  __host__ __device__ long long nlines() const { return (long long)g.ax.n * g.az.n; }
  __device__ Ref ref(long long L) const { return y_ref<T>(g, L); }
  __device__ C load(const Ref& r, int i) const {
    if (!g.in_yr(i)) return cmk<C>((T)0, (T)0);
    return chain_load(g.fine + (r.fine + i * g.ax.nf));
  }
  __device__ void store(const Ref& r, int i, C v, Acc&) const {
    const int jy = g.ay.grid_of(i);
    const T val = deconv<T>(g, g.dc + g.ax.n, r, jy, v.x);
    T* at = phi + (r.grid + jy * g.ax.n);
    if (ACC)
      *at += val;
    else
      *at = val;
  }
};

// 2D: x first and last, as rows of the density and the potential; y in between, storing or reading
// only the y lines of the range.  (A pass's rounding noise is white along its own axis and follows
// the spectrum along the axes transformed before it, and the 2D symbol grows like |k|^2 / |k|: with
// y first the x noise of the rows near k_y = 0 met the symbol of a dipole tilted towards x, and the
// error of a 256^2 density grew from 2.3e-6 to 3.9e-6.)
template <typename T>
__device__ __forceinline__ YRef<T> x_ref(const Geo<T>& g, long long L) {
  return line_ref<T>((int)L * g.ax.n, g.ay.fine_of((int)L) * g.ax.nf, g.dc[g.ax.n + (int)L] * g.dc[g.ax.n + g.ay.n]);
}

template <typename T>
struct PadX2 : PolicyBase {
  using C = cx_t<T>;
  using Ref = YRef<T>;
  static constexpr bool kBlockIn = true, kStrided = false;
  Geo<T> g;
  const T* rho;
  __host__ __device__ long long nlines() const { return g.ay.n; }
  __device__ Ref ref(long long L) const { return x_ref<T>(g, L); }
  __device__ void begin() const {
    if (blockIdx.x == 0 && threadIdx.x < 2) g.counters[threadIdx.x] = 0;
  }
  __device__ C load(const Ref& r, int i) const { return cmk<C>(chain_load(rho + (r.grid + g.ax.grid_of(i))), (T)0); }
  __device__ C use(const Ref& r, int i, C v) const { return pad_value<T>(g, g.dc, r, g.ax.grid_of(i), v.x); }
  __device__ void store(const Ref& r, int i, C v, Acc&) const { g.fine[r.fine + i] = v; }
};

template <typename T, bool FWD>
struct ColY2 : PolicyBase {
  using C = cx_t<T>;
  using Ref = int;  // the column
  static constexpr bool kBlockIn = FWD, kBlockOut = !FWD;
  Geo<T> g;
  __host__ __device__ long long nlines() const { return g.ax.nf; }
  __device__ Ref ref(long long L) const { return (int)L; }
  __device__ C load(Ref r, int i) const {
    if (!FWD && !g.in_yr(i)) return cmk<C>((T)0, (T)0);
    return chain_load(g.fine + (i * g.ax.nf + r));
  }
  __device__ void store(Ref r, int i, C v, Acc&) const {
    if (!FWD || g.in_yr(i)) g.fine[i * g.ax.nf + r] = v;
  }
};

template <typename T>
struct CropX2 : PolicyBase {
  using C = cx_t<T>;
  using Ref = YRef<T>;
  static constexpr bool kBlockOut = true, kStrided = false;
  Geo<T> g;
  T* phi;
  __host__ __device__ long long nlines() const { return g.ay.n; }
  __device__ Ref ref(long long L) const { return x_ref<T>(g, L); }
  __device__ C load(const Ref& r, int i) const { return chain_load(g.fine + (r.fine + i)); }
  __device__ void store(const Ref& r, int i, C v, Acc&) const {
    const int jx = g.ax.grid_of(i);
    phi[r.grid + jx] = deconv<T>(g, g.dc, r, jx, v.x);
  }
};

// rows on the y lines of the range in the planes z of the block, between their first n_x cells
// (grid order) and the whole row
template <typename T, bool FWD>
struct RowX : PolicyBase {
  using C = cx_t<T>;
  using Ref = int;  // fine-grid offset of the row
  static constexpr bool kBlockIn = FWD, kBlockOut = !FWD;
  Geo<T> g;
  __host__ __device__ long long nlines() const { return (long long)g.nyr * g.az.n; }
  static constexpr bool kStrided = false;
  __device__ Ref ref(long long L) const {
    const int q = (int)((unsigned)L / (unsigned)g.nyr);
    return g.fidx(g.az.fine_of(q), g.yr_line((int)L - q * g.nyr), 0);
  }
  __device__ C load(Ref r, int i) const {
    if (FWD) return chain_load(g.fine + (r + g.ax.grid_of(i)));
    // x lines outside the taps' range were neither written by the spread nor transformed
    if (!g.in_xr(i)) return cmk<C>((T)0, (T)0);
    return chain_load(g.fine + (r + i));
  }
  __device__ void store(Ref r, int i, C v, Acc&) const {
    if (!FWD)
      g.fine[r + g.ax.grid_of(i)] = v;
    else if (g.in_xr(i))
      g.fine[r + i] = v;
  }
};

// z columns on the y and x lines of the ranges: forward (pruned input), inverse (pruned output)
template <typename T, bool FWD>
struct ColZ : PolicyBase {
  using C = cx_t<T>;
  using Ref = int;  // the column's (y, x) offset
  static constexpr bool kBlockIn = FWD, kBlockOut = !FWD;
  Geo<T> g;
  __host__ __device__ long long nlines() const { return (long long)g.nxr * g.nyr; }
  __device__ Ref ref(long long L) const {
    const int q = (int)((unsigned)L / (unsigned)g.nxr);
    return g.yr_line(q) * g.ax.nf + g.xr_line((int)L - q * g.nxr);
  }
  __device__ C load(Ref r, int i) const { return chain_load(g.fine + (i * g.sz + r)); }
  __device__ void store(Ref r, int i, C v, Acc&) const { g.fine[i * g.sz + r] = v; }
};

// The smooth symbol of the split algorithm (Eq. 3.9) at the fine grid's modes,
//   p(k) = (1 - e^{-|k|^2/k0^2}) / |k|^2 * (3 (n.k)(m.k) - (n.m) |k|^2),  p(0) = 0,
// times the inverse transform's 1 / (nf0 nf1 nf2).  Mode l of an axis with nf points is the
// wavenumber (2 pi / (nf h)) l~ with l~ = l for l < nf/2, else l - nf.  e^{-|k|^2/k0^2} - 1 comes
// from the plan's per-axis tables (window.cuh).
template <typename T>
struct SmoothSymbol {
  T dk[3];    // 2 pi / (nf_d h_d)
  T n[3], m[3];
  T nm;       // n.m
  T inv_k02;  // 1 / k0^2
  T scale;    // 1 / (nf0 nf1 nf2)
  const WindowEntry<T>* em1;  // [nf0 + nf1 + nf2]: e^{-k_d^2/k0^2} - 1
  __host__ __device__ T k_of(int a, int l, int nf) const { return dk[a] * (T)(l < nf / 2 ? l : l - nf); }
  // em: e^{-|k|^2/k0^2} - 1
  __device__ T operator()(T kx, T ky, T kz, T em) const {
    const T k2 = (kx * kx + ky * ky) + kz * kz;
    const T nk = (n[0] * kx + n[1] * ky) + n[2] * kz;
    const T mk = (m[0] * kx + m[1] * ky) + m[2] * kz;
    const T poly = (T)3 * (nk * mk) - nm * k2;
    const T f = k2 > (T)0 ? -em / k2 : inv_k02;
    return (f * poly) * scale;
  }
};

// Forward z, symbol, inverse z of the split algorithm's smooth part: the columns (y, x) of the
// half spectrum y = 0..nf/2.  The real part taken at the end makes a mode stand for itself and its
// conjugate partner: modes with 0 < y < nf/2 count twice.  The partner of a mode on the x or z
// Nyquist line is the one on the same line (-nf/2) with the other components negated, so such a
// mode takes the mean of the symbol at both signs of its Nyquist components (the whole complex
// transform sums the two modes).
template <typename T>
struct ZRef {
  int col;        // the column's (y, x) offset
  T kx, ky;       // the column's x and y wavenumbers
  WindowLine<T> em;  // e^{-(kx^2 + ky^2)/k0^2} - 1
  T w;            // 1 or 2
  int nyq;        // x is on its Nyquist line (and the column counts twice)
};

template <typename T>
struct SmoothZ : PolicyBase {
  using C = cx_t<T>;
  using Ref = ZRef<T>;
  static constexpr bool kBlockIn = true, kBlockOut = true;
  Geo<T> g;
  SmoothSymbol<T> sy;
  __host__ __device__ long long nlines() const { return (long long)g.ax.nf * g.nyr; }
  __device__ Ref ref(long long L) const {
    const int ly = (int)((unsigned)L / (unsigned)g.ax.nf), lx = (int)L - ly * g.ax.nf;
    const bool twice = ly > 0 && 2 * ly < g.ay.nf;
    return Ref{ly * g.ax.nf + lx, sy.k_of(0, lx, g.ax.nf), sy.k_of(1, ly, g.ay.nf),
               window_line(sy.em1[lx], sy.em1[g.ax.nf + ly]), (T)(twice ? 2 : 1), twice && 2 * lx == g.ax.nf};
  }
  __device__ C load(const Ref& r, int i) const { return chain_load(g.fine + (i * g.sz + r.col)); }
  __device__ C apply(const Ref& r, int i, C v) const {
    const T kz = sy.k_of(2, i, g.az.nf);
    const C z = __ldg(reinterpret_cast<const C*>(sy.em1) + g.ax.nf + g.ay.nf + i);
    const T em = window_join(r.em, WindowEntry<T>{z.x, z.y});
    T p = r.w * sy(r.kx, r.ky, kz, em);
    const bool nz = r.w > (T)1 && 2 * i == g.az.nf;
    if (r.nyq || nz) p = (T)0.5 * (p + r.w * sy(r.nyq ? -r.kx : r.kx, r.ky, nz ? -kz : kz, em));
    return cscale(v, p);
  }
  __device__ void store(const Ref& r, int i, C v, Acc&) const {
    g.fine[i * g.sz + r.col] = v;
  }
};

// unit: the split algorithm's smooth part (the half spectrum, no deconvolution)
template <typename T>
Geo<T> geo_of(Plan& p, bool unit = false) {
  Geo<T> g;
  g.ax = Axis{p.n[0], p.nf[0]};
  g.ay = Axis{p.n[1], p.nf[1]};
  g.az = Axis{p.n[2], p.nf[2]};
  g.ylo = unit ? 0 : p.yr[0];
  g.nyr = unit ? p.nf[1] / 2 + 1 : p.yr[1];
  g.xlo = unit ? 0 : p.xr[0];
  g.nxr = unit ? p.nf[0] : p.xr[1];
  g.nonfinite = p.d_nonfinite;
  g.sz = p.nf[0] * p.nf[1];
  g.counters = p.d_counter;
  g.dc = static_cast<const double*>(unit ? p.d_ones : p.d_deconv);
  g.dcx2 = static_cast<const float2*>(unit ? p.d_ones_x2 : p.d_deconv_x2);
  g.fine = static_cast<cx_t<T>*>(p.d_fine);
  return g;
}

// a policy with the twiddles applied as head + tail (FP32 tables hold both)
template <typename P>
struct Precise : P {
  static constexpr bool kPrecise = true;
};

// one pass of the NUFFT's fine-grid transforms, with precise twiddles when the plan asks
template <typename T, int DIR, int HI, typename P>
int pass(Plan& p, int n, const P& pol, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (p.precise_nufft) return dispatch_policy<T, DIR, 16, HI>(p, n, Precise<P>{pol}, s);
  }
  return dispatch_policy<T, DIR, 16, HI>(p, n, pol, s);
}

}  // namespace

template <typename T>
int nufft_forward_fft(Plan& p, const T* rho, cudaStream_t s) {
  const Geo<T> g = geo_of<T>(p);
  if (p.dim == 2) {
    DDI_TRY((pass<T, -1, 2048>(p, p.nf[0], PadX2<T>{{}, g, rho}, s)));
    p.mark("pad_fft_x", s);
    DDI_TRY((pass<T, -1, 2048>(p, p.nf[1], ColY2<T, true>{{}, g}, s)));
    p.mark("fft_y_fwd", s);
    return DDI_OK;
  }
  DDI_TRY((pass<T, -1, 1024>(p, p.nf[1], PadY<T>{{}, g, rho}, s)));
  p.mark("pad_fft_y", s);
  DDI_TRY((pass<T, -1, 1024>(p, p.nf[0], RowX<T, true>{{}, g}, s)));
  p.mark("fft_x_fwd", s);
  DDI_TRY((pass<T, -1, 1024>(p, p.nf[2], ColZ<T, true>{{}, g}, s)));
  p.mark("fft_z_fwd", s);
  return DDI_OK;
}

template <typename T>
int nufft_inverse_fft(Plan& p, T* phi, cudaStream_t s, bool acc) {
  const Geo<T> g = geo_of<T>(p);
  if (p.dim == 2) {
    DDI_TRY((pass<T, +1, 2048>(p, p.nf[1], ColY2<T, false>{{}, g}, s)));
    p.mark("fft_y_inv", s);
    DDI_TRY((pass<T, +1, 2048>(p, p.nf[0], CropX2<T>{{}, g, phi}, s)));
    p.mark("fft_x_inv_crop", s);
    return DDI_OK;
  }
  DDI_TRY((pass<T, +1, 1024>(p, p.nf[2], ColZ<T, false>{{}, g}, s)));
  p.mark("fft_z_inv", s);
  DDI_TRY((pass<T, +1, 1024>(p, p.nf[0], RowX<T, false>{{}, g}, s)));
  p.mark("fft_x_inv", s);
  if (acc)
    DDI_TRY((pass<T, +1, 1024>(p, p.nf[1], CropY<T, true>{{}, g, phi}, s)));
  else
    DDI_TRY((pass<T, +1, 1024>(p, p.nf[1], CropY<T, false>{{}, g, phi}, s)));
  p.mark(acc ? "fft_y_inv_crop_add" : "fft_y_inv_crop", s);
  return DDI_OK;
}

// I_1 of Eq. 3.9: rho zero-padded into the fine grid (the centred block, as for the NUFFT,
// which leaves the circular convolution unchanged), forward y, x, then forward z, p and inverse z
// in one pass, inverse x, y, crop and real part.  The 2x padding makes the circular
// convolution linear up to the kernel's tail beyond one box length.
template <typename T>
int split_smooth_part(Plan& p, const T* rho, T* phi, cudaStream_t s) {
  if (p.dim != 3 || !p.split() || !p.d_ones) {
    set_error("split_smooth_part: not a 3D split plan");
    return DDI_ERR_ARG;
  }
  const Geo<T> g = geo_of<T>(p, /*unit=*/true);
  SmoothSymbol<T> sy;
  for (int a = 0; a < 3; ++a) {
    sy.dk[a] = (T)((2.0 * M_PI) / ((double)p.nf[a] * p.h[a]));
    sy.n[a] = (T)p.desc.axis_n[a];
    sy.m[a] = (T)p.desc.axis_m[a];
  }
  const double* n = p.desc.axis_n;
  const double* m = p.desc.axis_m;
  sy.nm = (T)((n[0] * m[0] + n[1] * m[1]) + n[2] * m[2]);
  sy.inv_k02 = (T)(1.0 / (p.desc.split_k0 * p.desc.split_k0));
  sy.em1 = static_cast<const WindowEntry<T>*>(p.d_em1);
  sy.scale = (T)(1.0 / ((double)p.nf[0] * (double)p.nf[1] * (double)p.nf[2]));
  DDI_TRY((dispatch_policy<T, -1, 16, 1024>(p, p.nf[1], PadY<T>{{}, g, rho}, s)));
  p.mark("smooth_pad_fft_y", s);
  DDI_TRY((dispatch_policy<T, -1, 16, 1024>(p, p.nf[0], RowX<T, true>{{}, g}, s)));
  p.mark("smooth_fft_x_fwd", s);
  DDI_TRY((dispatch_policy<T, 0, 16, 1024>(p, p.nf[2], SmoothZ<T>{{}, g, sy}, s)));
  p.mark("smooth_fft_z_pair", s);
  DDI_TRY((dispatch_policy<T, +1, 16, 1024>(p, p.nf[0], RowX<T, false>{{}, g}, s)));
  p.mark("smooth_fft_x_inv", s);
  DDI_TRY((dispatch_policy<T, +1, 16, 1024>(p, p.nf[1], CropY<T, false>{{}, g, phi}, s)));
  p.mark("smooth_fft_y_inv_crop", s);
  return DDI_OK;
}

}  // namespace ddi
