// Stockham FFT core shared by the pruned and fused NUFFT passes (fft_nufft.cuh) and the GPE's
// passes (gpe_fft.cuh): in-register radix-16/12/8/4/2/3 DFTs, the Stockham stage loop over a
// padded shared-memory line, and CTA-level kernels that take LPB lines from and to global memory
// through a load/store policy, one transform a pass (k_fft_policy) or forward and inverse in one
// (k_fft_pair).
#pragma once
#include <cmath>

#include "common.cuh"

namespace ddi {
namespace fftcore {

// cos(2 pi k / 16), k = 0..15: exact mathematical constants rounded from 40 digits.
#define DDI_C1 0.9238795325112867561281831893967882868224
#define DDI_C2 0.7071067811865475244008443621048490392848
#define DDI_C3 0.3826834323650897717284599840303988667613
__host__ __device__ constexpr double cos16(int k) {
  return (k & 15) == 0   ? 1.0
         : (k & 15) == 1 ? DDI_C1
         : (k & 15) == 2 ? DDI_C2
         : (k & 15) == 3 ? DDI_C3
         : (k & 15) == 4 ? 0.0
         : (k & 15) == 5 ? -DDI_C3
         : (k & 15) == 6 ? -DDI_C2
         : (k & 15) == 7 ? -DDI_C1
         : (k & 15) == 8 ? -1.0
         : (k & 15) == 9 ? -DDI_C1
         : (k & 15) == 10 ? -DDI_C2
         : (k & 15) == 11 ? -DDI_C3
         : (k & 15) == 12 ? 0.0
         : (k & 15) == 13 ? DDI_C3
         : (k & 15) == 14 ? DDI_C2
                          : DDI_C1;
}
__host__ __device__ constexpr double sin16(int k) { return cos16(k + 12); }  // sin x = cos(x - pi/2)

// v * k for a constant k known in FP64.  In FP32 the constant is applied as head + tail
// (k_hi = fl(k), k_lo = fl(k - k_hi)): a single rounded constant would scale every butterfly
// that uses it by the same |w|^2 != 1 (e.g. 1 - 5.7e-8 for the pi/8 pair), a bias that
// accumulates over the stages and, in a time-splitting run, drains the mass step after
// step; with the tail only the unbiased rounding of each operation remains.
template <typename T>
__device__ __forceinline__ T mul_const(T v, double k) {
  if constexpr (sizeof(T) == 4) {
    const float hi = (float)k;
    const float lo = (float)(k - (double)hi);
    return fmaf(v, hi, v * lo);
  } else {
    return v * (T)k;
  }
}

template <int R, int DIR, typename C>
__device__ __forceinline__ C tw_const(C x, int k) {
  // x * exp(DIR * 2 pi i k / R) with the trivial factors special-cased
  if (k == 0) return x;
  if (4 * k == R) return DIR < 0 ? cmk<C>(x.y, -x.x) : cmk<C>(-x.y, x.x);
  const int idx = (k * (16 / R)) & 15;
  const double c = cos16(idx);
  const double s = DIR * sin16(idx);
  if constexpr (sizeof(C) == 8) {
    // x c + (i x) s, each product head + tail as mul_const's, both components at once
    const float ch = (float)c, cl = (float)(c - (double)ch), sh = (float)s, sl = (float)(s - (double)sh);
    const C y = make_float2(-x.y, x.x);
    const C p = __ffma2_rn(x, make_float2(ch, ch), __fmul2_rn(x, make_float2(cl, cl)));
    const C q = __ffma2_rn(y, make_float2(sh, sh), __fmul2_rn(y, make_float2(sl, sl)));
    return __fadd2_rn(p, q);
  } else {
    return cmk<C>(mul_const(x.x, c) - mul_const(x.y, s), mul_const(x.x, s) + mul_const(x.y, c));
  }
}

// In-register R-point DFT (natural order in and out), radix-2 decimation in time.
template <int R, int DIR, typename C>
struct Dft {
  __device__ __forceinline__ static void run(C* v) {
    C e[R / 2], o[R / 2];
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      e[k] = v[2 * k];
      o[k] = v[2 * k + 1];
    }
    Dft<R / 2, DIR, C>::run(e);
    Dft<R / 2, DIR, C>::run(o);
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      const C t = tw_const<R, DIR>(o[k], k);
      v[k] = cadd(e[k], t);
      v[k + R / 2] = csub(e[k], t);
    }
  }
};
template <int DIR, typename C>
struct Dft<1, DIR, C> {
  __device__ __forceinline__ static void run(C*) {}
};
template <int DIR, typename C>
struct Dft<3, DIR, C> {
  // X1,2 = a - (b + c)/2 +- i DIR (sqrt(3)/2) (b - c)
  __device__ __forceinline__ static void run(C* v) {
    using T = decltype(C::x);
    const double s3 = 0.8660254037844386467637231707529361834714;
    const C t1 = cadd(v[1], v[2]);
    const C d = csub(v[1], v[2]);
    const C t2 = cmk<C>(v[0].x - (T)0.5 * t1.x, v[0].y - (T)0.5 * t1.y);
    const C rot = cmk<C>(-(T)DIR * mul_const(d.y, s3), (T)DIR * mul_const(d.x, s3));
    v[0] = cadd(v[0], t1);
    v[1] = cadd(t2, rot);
    v[2] = csub(t2, rot);
  }
};

// 12 = 3 x 4 points by the prime-factor map (no twiddles between the factors): with
// n = (4 n1 + 3 n2) mod 12 and k = (4 k1 + 9 k2) mod 12, n k = 4 n1 k1 + 3 n2 k2 (mod 12)
template <int DIR, typename C>
struct Dft<12, DIR, C> {
  __device__ __forceinline__ static void run(C* v) {
    C a[4][3];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 3; ++n1) a[n2][n1] = v[(4 * n1 + 3 * n2) % 12];
      Dft<3, DIR, C>::run(a[n2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      C u[4];
#pragma unroll
      for (int n2 = 0; n2 < 4; ++n2) u[n2] = a[n2][k1];
      Dft<4, DIR, C>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[(4 * k1 + 9 * k2) % 12] = u[k2];
    }
  }
};

__device__ __forceinline__ int pidx(int i) { return i + (i >> 4); }
// pidx(i + r STEP) given pi = pidx(i): one constant offset where STEP is a multiple of 16 (the
// compiler cannot split the shift of a sum)
template <int STEP>
__device__ __forceinline__ int pidx_at(int i, int pi, int r) {
  return STEP % 16 == 0 ? pi + r * (STEP + STEP / 16) : pidx(i + r * STEP);
}

// Radix of the stage that follows sub-transform length NS: 16, then what is left (8, 4, 2 and 3).
// Lengths 3 * 2^a up to 192 take 12 first and 32 takes 8 and 4: two stages for 96 and 192 where 16, 2
// or 4 and 3 made three (96^3 gradient-flow sweep 51 -> 46 us).  384 and 512 stay with 16 first:
// 12 or 16, 8 and 4 took their passes from 76 to 96 and from 110 to 160 us.
__host__ __device__ constexpr int pow2_part(int n) { return n & (-n); }
__host__ __device__ constexpr int radix_for(int N, int NS) {
  const int left = N / NS;
  if (N <= 192 && left % 3 == 0) return 12;
  if (left == 32 && N == 32) return 8;
  return pow2_part(left) >= 16 ? 16 : (pow2_part(left) > 1 ? pow2_part(left) : 3);
}

template <int N>
struct Shape {
  static constexpr int RM = radix_for(N, 1);   // the first radix: elements per thread
  static constexpr int TPL = N / RM;           // threads per line
  static constexpr int LS = N + N / 16 + 1;    // padded line stride in shared memory
};

// shared-memory index of the first stage's output r of butterfly t, element t R0 + r
template <int R0>
__device__ __forceinline__ int first_out(int t, int r) {
  return R0 == 16 ? t * 17 + r : pidx(t * R0 + r);
}

// One Stockham stage of radix R with sub-transform length NS; each thread owns
// G = ceil(RM / R) butterflies of its line (the last ones masked when R does not divide RM).
// PRECISE: apply the twiddle table's tails (FP32), for transforms repeated many times on
// the same data (time splitting), where a rounded twiddle's |w| != 1 would accumulate.
// stage_compute reads the stage's inputs from the line, twiddles and transforms them.
template <typename C, int N, int R, int NS, int DIR, bool PRECISE>
__device__ __forceinline__ void stage_compute(const C* line, int t, const C* __restrict__ tw,
                                              C (&v)[(Shape<N>::RM + R - 1) / R][R]) {
  constexpr int RM = Shape<N>::RM;
  constexpr int TPL = Shape<N>::TPL;
  constexpr int G = (RM + R - 1) / R;
  constexpr int NB = N / R;  // butterflies per line
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int j = t + g * TPL;  // butterfly index in [0, N/R)
    if (RM % R == 0 || j < NB) {
      const int pj = pidx(j);
#pragma unroll
      for (int r = 0; r < R; ++r) v[g][r] = line[pidx_at<NB>(j, pj, r)];
      if (NS > 1) {
        const int jm = j % NS;
        constexpr int STRIDE = N / (NS * R);
#pragma unroll
        for (int r = 1; r < R; ++r) {
          const int ti = jm * r * STRIDE;
          C w = tw[ti];
          if (DIR > 0) w.y = -w.y;
          if constexpr (PRECISE && sizeof(w.x) == 4) {
            // head + tail twiddle (the table holds N heads, then N tails)
            C wl = tw[N + ti];
            if (DIR > 0) wl.y = -wl.y;
            const C x = v[g][r];
            v[g][r] = cmk<C>(fmaf(x.x, w.x, fmaf(-x.y, w.y, x.x * wl.x - x.y * wl.y)),
                             fmaf(x.x, w.y, fmaf(x.y, w.x, x.x * wl.y + x.y * wl.x)));
          } else {
            v[g][r] = cmul(v[g][r], w);
          }
        }
      }
      Dft<R, DIR, C>::run(v[g]);
    }
  }
}

// a middle stage: shared memory to shared memory (Stockham output order)
template <typename C, int N, int R, int NS, int DIR, bool PRECISE>
__device__ __forceinline__ void stage(C* line, int t, const C* __restrict__ tw) {
  constexpr int RM = Shape<N>::RM;
  constexpr int TPL = Shape<N>::TPL;
  constexpr int G = (RM + R - 1) / R;
  constexpr int NB = N / R;
  C v[G][R];
  stage_compute<C, N, R, NS, DIR, PRECISE>(line, t, tw, v);
  __syncthreads();
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int j = t + g * TPL;
    if (RM % R == 0 || j < NB) {
      const int jm = j % NS;
      const int idxD = (j - jm) * R + jm, pD = pidx(idxD);
#pragma unroll
      for (int r = 0; r < R; ++r) line[pidx_at<NS>(idxD, pD, r)] = v[g][r];
    }
  }
  __syncthreads();
}

// sub-transform length before the last stage
__host__ __device__ constexpr int last_ns(int N, int NS = 1) {
  return NS * radix_for(N, NS) >= N ? NS : last_ns(N, NS * radix_for(N, NS));
}

// the middle stages, from sub-transform length NS up to (not including) STOP
template <typename C, int N, int DIR, int NS, int STOP, bool PRECISE>
struct MidStages {
  __device__ __forceinline__ static void run(C* line, int t, const C* tw) {
    constexpr int R = radix_for(N, NS);
    stage<C, N, R, NS, DIR, PRECISE>(line, t, tw);
    MidStages<C, N, DIR, NS * R, STOP, PRECISE>::run(line, t, tw);
  }
};
template <typename C, int N, int DIR, int STOP, bool PRECISE>
struct MidStages<C, N, DIR, STOP, STOP, PRECISE> {
  __device__ __forceinline__ static void run(C*, int, const C*) {}
};

template <int N>
__host__ __device__ constexpr int lines_per_cta_base() {
  // powers of two, so that a CTA is whole warps and lines stay aligned
  return N <= 16 ? 128 : N <= 32 ? 64 : N <= 64 ? 32 : N <= 256 ? 16 : N <= 512 ? 8 : N <= 1024 ? 4 : 2;
}

// Generic batched-line FFT: a policy P supplies nlines(), ref(L) (the line's addresses,
// computed once per line by one thread), load(ref, i), use(ref, i, v) (what becomes of a loaded
// value, called after all of a thread's loads) / store(ref, i, v, acc) for element i of the line, skip() (the whole pass is not needed), an
// accumulator Acc with finish(acc), begin() (once per thread, before the lines), and the constants
//   kStrided   the lines' elements are strided in memory and neighbouring lines adjacent (else the
//              element index is fastest)
//   kPrecise   apply the twiddle tails (FP32)
//   kBlockIn   only the elements i < N/4 and i >= 3 N/4 are nonzero and loaded (the zero padding
//              of a twofold oversampled line): the first stage's other inputs are literal zeros,
//              so their loads and most of their butterfly drop out at compile time
//   kBlockOut  only those elements are stored (the crop)
// The first Stockham stage takes its inputs straight from global memory and the last one
// writes its outputs straight back (both are in natural element order there), so each
// element crosses shared memory once per middle stage plus once between the first stage
// and the next.  Threads are (line b, butterfly t) pairs: lines fastest when lines are
// strided in memory (a warp's accesses then cover adjacent lines), butterflies fastest
// when lines are contiguous.
struct PolicyBase {
  struct Acc {};
  static constexpr bool kPrecise = false, kBlockIn = false, kBlockOut = false, kStrided = true;
  __device__ bool skip() const { return false; }
  __device__ void begin() const {}
  template <typename Ref, typename C> __device__ C use(const Ref&, int, C v) const { return v; }
  __device__ void finish(const Acc&) const {}
};

__host__ __device__ constexpr bool outside_block(int r, int R) { return r >= R / 4 && r < R - R / 4; }

// first stage: butterfly t's inputs are elements t + r N/R0 (all loads issued before use)
template <int N, int R0, typename C, typename P, typename Ref>
__device__ __forceinline__ void load_first(const P& pol, const Ref& ref, bool live, int t, C (&v)[R0]) {
  static_assert(!P::kBlockIn || R0 % 4 == 0, "the block is whole quarters of the first stage");
#pragma unroll
  for (int r = 0; r < R0; ++r) {
    if (P::kBlockIn && outside_block(r, R0))
      v[r] = cmk<C>(0, 0);
    else
      v[r] = live ? pol.load(ref, t + r * (N / R0)) : cmk<C>(0, 0);
  }
#pragma unroll
  for (int r = 0; r < R0; ++r)
    if (!(P::kBlockIn && outside_block(r, R0)) && live) v[r] = pol.use(ref, t + r * (N / R0), v[r]);
}
// last stage: butterfly j's outputs are elements j + r NSL
template <int N, int RL, int NSL, typename C, typename P, typename Ref>
__device__ __forceinline__ void store_last(const P& pol, const Ref& ref, int j, const C (&v)[RL], typename P::Acc& acc) {
#pragma unroll
  for (int r = 0; r < RL; ++r) {
    if (P::kBlockOut && RL % 4 == 0 && outside_block(r, RL)) continue;
    const int i = j + r * NSL;
    if (P::kBlockOut && RL % 4 != 0 && i >= N / 4 && i < N - N / 4) continue;
    pol.store(ref, i, v[r], acc);
  }
}

template <typename T, int N, int LPB, int DIR, typename P>
__global__ void __launch_bounds__(LPB * Shape<N>::TPL)
    k_fft_policy(P pol, const cx_t<T>* __restrict__ tw) {
  using C = cx_t<T>;
  using Ref = typename P::Ref;
  constexpr bool PR = P::kPrecise;
  constexpr int LS = Shape<N>::LS;
  constexpr int TPL = Shape<N>::TPL;
  constexpr int RM = Shape<N>::RM;
  constexpr int R0 = radix_for(N, 1);
  constexpr int NSL = last_ns(N);      // the last stage's sub-transform length
  constexpr int RL = N / NSL;          // and its radix
  constexpr int GL = (RM + RL - 1) / RL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Ref refs[LPB];
  chain_release();
  chain_wait();
  if (pol.skip()) return;
  pol.begin();
  C* sm = reinterpret_cast<C*>(smem_raw);
  const long long L0 = (long long)blockIdx.x * LPB;
  const long long left = pol.nlines() - L0;
  const int nb = left < LPB ? (int)left : LPB;  // lines of this CTA
  if ((int)threadIdx.x < nb) refs[threadIdx.x] = pol.ref(L0 + threadIdx.x);
  __syncthreads();
  constexpr bool contig = !P::kStrided;
  const int b = contig ? (int)threadIdx.x / TPL : (int)threadIdx.x % LPB;
  const int t = contig ? (int)threadIdx.x % TPL : (int)threadIdx.x / LPB;
  const bool live = b < nb;
  C* line = sm + b * LS;
  typename P::Acc acc{};
  C v0[R0];
  load_first<N, R0>(pol, refs[b], live, t, v0);
  Dft<R0, DIR, C>::run(v0);
  if constexpr (R0 == N) {
    if (live) store_last<N, N, 1>(pol, refs[b], 0, v0, acc);
  } else {
#pragma unroll
    for (int r = 0; r < R0; ++r) line[first_out<R0>(t, r)] = v0[r];
    __syncthreads();
    MidStages<C, N, DIR, R0, NSL, PR>::run(line, t, tw);
    C v[GL][RL];
    stage_compute<C, N, RL, NSL, DIR, PR>(line, t, tw, v);
#pragma unroll
    for (int g = 0; g < GL; ++g) {
      const int j = t + g * TPL;
      if (live && (RM % RL == 0 || j < N / RL)) store_last<N, RL, NSL>(pol, refs[b], j, v[g], acc);
    }
  }
  pol.finish(acc);
}

// Forward transform, pol.apply(ref, i, v) on every mode, inverse transform of the same line in one
// pass: the line crosses global memory once each way instead of twice.  Where the last stage has
// the first stage's radix (N = 16^k), a thread's modes are the inverse's first inputs and stay in
// registers; otherwise they cross shared memory once.  FP32 passes without twiddle tails are held to
// 64 registers, so that a second 512-thread CTA loads while one transforms (256^3 split 1187 -> 1110
// us); with the tails that spills (128^3 steps 1345 -> 1429 us).
template <typename T, int N, int LPB, typename P>
constexpr int pair_ctas() {
  return sizeof(T) == 4 && !P::kPrecise && 1024 / (LPB * Shape<N>::TPL) > 1 ? 1024 / (LPB * Shape<N>::TPL) : 1;
}
template <typename T, int N, int LPB, typename P>
__global__ void __launch_bounds__(LPB * Shape<N>::TPL, pair_ctas<T, N, LPB, P>())
    k_fft_pair(P pol, const cx_t<T>* __restrict__ tw) {
  using C = cx_t<T>;
  using Ref = typename P::Ref;
  constexpr bool PR = P::kPrecise;
  constexpr int LS = Shape<N>::LS;
  constexpr int TPL = Shape<N>::TPL;
  constexpr int RM = Shape<N>::RM;
  constexpr int R0 = radix_for(N, 1);
  constexpr int NSL = last_ns(N);
  constexpr int RL = N / NSL;
  constexpr int GL = (RM + RL - 1) / RL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Ref refs[LPB];
  chain_release();
  chain_wait();
  if (pol.skip()) return;
  pol.begin();
  C* sm = reinterpret_cast<C*>(smem_raw);
  const long long L0 = (long long)blockIdx.x * LPB;
  const long long left = pol.nlines() - L0;
  const int nb = left < LPB ? (int)left : LPB;
  if ((int)threadIdx.x < nb) refs[threadIdx.x] = pol.ref(L0 + threadIdx.x);
  __syncthreads();
  constexpr bool contig = !P::kStrided;
  const int b = contig ? (int)threadIdx.x / TPL : (int)threadIdx.x % LPB;
  const int t = contig ? (int)threadIdx.x % TPL : (int)threadIdx.x / LPB;
  const bool live = b < nb;
  C* line = sm + b * LS;
  typename P::Acc acc{};
  C v0[R0];
  load_first<N, R0>(pol, refs[b], live, t, v0);
  Dft<R0, -1, C>::run(v0);
  if constexpr (R0 == N) {
    if (live) {
#pragma unroll
      for (int r = 0; r < R0; ++r) v0[r] = pol.apply(refs[b], r, v0[r]);
    }
    Dft<R0, 1, C>::run(v0);
    if (live) store_last<N, N, 1>(pol, refs[b], 0, v0, acc);
  } else {
#pragma unroll
    for (int r = 0; r < R0; ++r) line[first_out<R0>(t, r)] = v0[r];
    __syncthreads();
    MidStages<C, N, -1, R0, NSL, PR>::run(line, t, tw);
    {
      C v[GL][RL];
      stage_compute<C, N, RL, NSL, -1, PR>(line, t, tw, v);
      __syncthreads();  // every input of the stage has been read
#pragma unroll
      for (int g = 0; g < GL; ++g) {
        const int j = t + g * TPL;
        if (RM % RL == 0 || j < N / RL) {
#pragma unroll
          for (int r = 0; r < RL; ++r) {
            const C m = live ? pol.apply(refs[b], j + r * NSL, v[g][r]) : v[g][r];
            if constexpr (RL == R0)
              v0[r] = m;
            else
              line[pidx_at<NSL>(j, pidx(j), r)] = m;
          }
        }
      }
      if constexpr (RL != R0) {
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R0; ++r) v0[r] = line[pidx_at<N / R0>(t, pidx(t), r)];
        __syncthreads();
      }
    }
    Dft<R0, 1, C>::run(v0);
#pragma unroll
    for (int r = 0; r < R0; ++r) line[first_out<R0>(t, r)] = v0[r];
    __syncthreads();
    MidStages<C, N, 1, R0, NSL, PR>::run(line, t, tw);
    C v[GL][RL];
    stage_compute<C, N, RL, NSL, 1, PR>(line, t, tw, v);
#pragma unroll
    for (int g = 0; g < GL; ++g) {
      const int j = t + g * TPL;
      if (live && (RM % RL == 0 || j < N / RL)) store_last<N, RL, NSL>(pol, refs[b], j, v[g], acc);
    }
  }
  pol.finish(acc);
}

// Lines per CTA.  Strided lines: a power of two, so that the lines of a CTA are whole 128-byte
// pieces of memory at every element (10 lines of N = 384 made 80-byte pieces: 192^3 z passes 103
// -> 76 us; 8 of N = 512 64-byte ones: the 256^3 split's z pass 571 -> 530 us).  Contiguous
// lines: ~35 KB of shared memory per CTA in FP32.  FP64 takes half the lines.
template <typename T, int N, bool STRIDED>
constexpr int lines_per_cta() {
  constexpr int f32 = !STRIDED ? lines_per_cta_base<N>() : N <= 64 ? 32 : N <= 512 ? 16 : N <= 1024 ? 8 : 4;
  return sizeof(T) == 8 ? (f32 > 1 ? f32 / 2 : 1) : f32;
}

// DIR = 0: forward and inverse in one pass (k_fft_pair)
template <typename T, int N, int DIR, typename P>
int launch_policy(const Plan& p, const P& pol, cudaStream_t s) {
  constexpr int LPB = lines_per_cta<T, N, P::kStrided>();
  constexpr int threads = LPB * Shape<N>::TPL;
  static_assert(P::kStrided || threads % 32 == 0, "a CTA of contiguous lines is whole warps");
  const size_t smem = (size_t)LPB * Shape<N>::LS * sizeof(cx_t<T>);
  void (*kern)(P, const cx_t<T>*);
  if constexpr (DIR == 0)
    kern = k_fft_pair<T, N, LPB, P>;
  else
    kern = k_fft_policy<T, N, LPB, DIR, P>;
  DDI_TRY(prepare_kernel(reinterpret_cast<const void*>(kern), smem));
  if (!twiddles(p, N)) {
    set_error("missing twiddle table for FFT length %d", N);
    return DDI_ERR_ARG;
  }
  const long long blocks = (pol.nlines() + LPB - 1) / LPB;
  if (blocks <= 0) return DDI_OK;
  return launch_chain(p, kern, (unsigned)blocks, threads, smem, s, pol, static_cast<const cx_t<T>*>(twiddles(p, N)));
}

// FFT lengths built, 2^a and 3 * 2^a: LO and HI bound the lengths a policy is built for (fine-grid
// lines 16..2048, 3D 1024; grid lines 8..1024)
template <typename T, int DIR, int LO, int HI, typename P>
int dispatch_policy(const Plan& p, int n, const P& pol, cudaStream_t s) {
#define DDI_LEN(NN)                                                        \
  case NN:                                                                 \
    if constexpr (NN >= LO && NN <= HI) return launch_policy<T, NN, DIR>(p, pol, s); \
    break;
  switch (n) {
    DDI_LEN(8) DDI_LEN(12) DDI_LEN(16) DDI_LEN(24) DDI_LEN(32) DDI_LEN(48) DDI_LEN(64) DDI_LEN(96) DDI_LEN(128)
    DDI_LEN(192) DDI_LEN(256) DDI_LEN(384) DDI_LEN(512) DDI_LEN(768) DDI_LEN(1024) DDI_LEN(1536) DDI_LEN(2048)
    default: break;
  }
#undef DDI_LEN
  set_error("FFT length %d not supported (2^a or 3 * 2^a, %d..%d here)", n, LO, HI);
  return DDI_ERR_ARG;
}

}  // namespace fftcore
}  // namespace ddi
