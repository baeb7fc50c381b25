// Column spread and interpolation of 3D plans (Sec. 2.1, Eq. DDI-Trun1), FP32 and FP64, and the block
// spread of FP32 2D plans.
//
// A warp takes a unit: a range of groups of one column and a window of z-planes.  Lane (lx, ly)
// owns the cells (lx, ly) and (lx, ly + 4) of the column and keeps W planes of both in
// registers: plane p lives in register p mod W, so the window advances by writing its oldest
// plane and never moves a register.  For a run of one z class the lane sums
// g = sum c_q psi_x psi_y over the run's visits and then adds g psi_z to its W planes once.
// No shared-memory read-modify-write and no atomics: each cell belongs to one lane.  Planes that
// several units touch go to partial slots (contiguous per plane, in unit order) that
// k_reduce_col3 sums in order: results are deterministic.
//
// What bounds it.  FP64: this part issues a warp's FP64 instruction over 16 cycles of an SM, so
// the count of FP64 operations is the time.  A tile plane's read-modify-write costs 3 per tap and
// shares nothing between nodes; here the taps of a ring's nodes are summed before psi_z, so a
// visit costs 6 per lane (its 64 cells) and a run 4 W.  FP32: instruction issue.  The rows a visit
// needs do not change between evaluations, so the plan stores them laid out per group
// (columns.cuh) and the warp copies a group ahead with cp.async instead of gathering and
// zero-padding each row.  Its inner step takes two visits at once: four shared loads bring their
// u = c psi_x (real, imaginary) and psi_y (two cells) as pairs, four packed FMAs add them, and no
// value has to be duplicated into a pair.  Units are cut to equal work (plan.cu), because one
// warp that walks a sparse column's 256 planes alone outlasts the rest of the launch.
//
// Measured (spread + reduction): 128^3 FP32, 524288 nodes: 198 -> 101 us (4 CTAs per SM at up to
// 128 registers; 5 CTAs at 96 spill and take 118); 192^3 FP32 564 -> 277 us; 128^3 FP64 27.4 ->
// 2.6 ms (the FP64 operations above take 2.3 ms at this part's rate).
#include <algorithm>

#include "columns.cuh"

namespace ddi {
namespace {

constexpr int kColThreads3 = 128;  // 4 warps per CTA, each taking units on its own

// c + a b per component
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
template <typename C> __device__ __forceinline__ C both(decltype(C::x) v) { return cmk<C>(v, v); }
// the sum of a.x b.x + a.y b.y over a run, as a pair (FP32: packed) or a scalar chain (FP64: no
// addition to close it); dot_sum closes it
__device__ __forceinline__ float2 dot2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 dot2(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.y, b.y, fma(a.x, b.x, c.x)), 0.0);
}
__device__ __forceinline__ float dot_sum(float2 v) { return v.x + v.y; }
__device__ __forceinline__ double dot_sum(double2 v) { return v.x; }

// a += x with the rounding error of the sum carried in c (compensated summation, Kahan):
// y = x - c, t = a + y, c = (t - a) - y, a = t
__device__ __forceinline__ void kahan_add2(float2& a, float2& c, float2 x) {
  const float2 y = __fadd2_rn(x, make_float2(-c.x, -c.y));
  const float2 t = __fadd2_rn(a, y);
  c = __fadd2_rn(__fadd2_rn(t, make_float2(-a.x, -a.y)), make_float2(-y.x, -y.y));
  a = t;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// a group's image into the warp's shared memory, 16 bytes per lane and step
template <int BYTES>
__device__ __forceinline__ void copy_image(unsigned char* dst, const unsigned char* src, int lane) {
#pragma unroll
  for (int i = 0; i < (BYTES + 511) / 512; ++i) {
    const int o = (i * 32 + lane) * 16;
    if ((i + 1) * 512 <= BYTES || o < BYTES) cp_async16(dst + o, src + o);
  }
}

struct ColArgs3 {
  int nf[3];
  int ncx;
  const ColUnit* units;
  int nunits;
  int* counter;
  const unsigned char* image;  // [group][ColImage::BYTES]
  const int* nodes;            // [group][32] node of each visit, -1: none
  const void* c;               // [node]
  void* fine;
  void* partial;               // [slot][kColY * kColX]
  const int* dest;             // [unit][kColPlanes]: partial slot of each plane of its window, -1: the fine grid
};

// per-warp shared memory of the spread: two group images and u = c psi_x of each visit, rows of
// 32 visits per x cell, real parts, then imaginary parts
template <typename T, int W>
struct SpreadSmem {
  static constexpr int U = 2 * ColImage<T, W>::BYTES;
  static constexpr int BYTES = (U + 16 * ColImage<T, W>::RS + 127) / 128 * 128;
};

#define DDI_COL3_CASES(X) X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15)

template <typename T, int W, bool COMP>
__global__ void __launch_bounds__(kColThreads3, sizeof(T) == 4 ? 4 : 2) k_spread_col3(ColArgs3 a) {
  using C = cx_t<T>;
  using I = ColImage<T, W>;
  using S = SpreadSmem<T, W>;
  static_assert(W <= 16 && W % 2 == 0, "planes in register pairs 0..W/2-1 of the window");
  static_assert(!COMP || sizeof(T) == 4, "compensated sums are built for FP32");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  chain_release();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* sm = smem_raw + warp * S::BYTES;
  unsigned char* su = sm + S::U;
  const int lx = lane & 7, ly = lane >> 3;
  const int nfx = a.nf[0], nfz = a.nf[2];
  const long long plane = (long long)nfx * a.nf[1];
  const C* cg = static_cast<const C*>(a.c);
  // units are taken from a counter, the first one by position; the next unit's index, entry and
  // first group are requested while the current one is being worked on
  const int nwarps = gridDim.x * (blockDim.x >> 5);
  int un = warp * gridDim.x + blockIdx.x;
  int uw = 0;            // word (lane mod 8) of the next unit's entry
  int n0 = -1, n1 = -1;  // node of this lane in the next unit's first and second group
  int buf = 0;
  static_assert(sizeof(ColUnit) == 32, "eight words per unit");
  auto load_unit = [&]() { uw = __ldg(reinterpret_cast<const int*>(a.units + un) + (lane & 7)); };
  auto word = [&](int k) { return __shfl_sync(0xffffffffu, uw, k); };
  auto request_first = [&]() {  // the next unit's first image into the free buffer
    n0 = n1 = -1;
    const int lo = word(1), hi = word(2);
    if (un < a.nunits && lo < hi) {
      copy_image<I::BYTES>(sm + buf * I::BYTES, a.image + (size_t)lo * I::BYTES, lane);
      n0 = __ldg(a.nodes + (size_t)lo * 32 + lane);
      if (lo + 1 < hi) n1 = __ldg(a.nodes + (size_t)(lo + 1) * 32 + lane);
    }
    cp_async_commit();
  };
  if (un < a.nunits) load_unit();
  request_first();
  chain_wait();
  while (un < a.nunits) {
    const ColUnit U = {word(0), word(1), word(2), word(3), word(4), word(5), word(6), word(7)};
    int nx = 0;
    if (lane == 0) nx = atomicAdd(a.counter, 1);
    // where each plane of the window goes, one plane per lane
    static_assert(kColPlanes == 32, "a lane per plane of the window");
    const int mydest = __ldg(a.dest + (size_t)un * kColPlanes + lane);
    const int cx = U.col % a.ncx, cy = U.col / a.ncx;
    const long long cell = (long long)(cy * kColY + ly) * nfx + cx * kColX + lx;
    // planes 2 q and 2 q + 1 (mod W) of cells 0 and 1, real and imaginary parts; compensations
    C r0[W / 2], i0[W / 2], r1[W / 2], i1[W / 2];
    C cr0[COMP ? W / 2 : 1], ci0[COMP ? W / 2 : 1], cr1[COMP ? W / 2 : 1], ci1[COMP ? W / 2 : 1];
    const C zero = cmk<C>((T)0, (T)0);
#pragma unroll
    for (int q = 0; q < W / 2; ++q) {
      r0[q] = i0[q] = r1[q] = i1[q] = zero;
      if constexpr (COMP) cr0[q] = ci0[q] = cr1[q] = ci1[q] = zero;
    }
    if (U.lo == U.hi) {  // no visits: zeros
      for (int z = U.z0; z < U.z1; ++z) {
        C* dst = static_cast<C*>(a.fine) + (z >= nfz ? z - nfz : z) * plane + cell;
        __stcs(dst, zero);
        __stcs(dst + 4 * nfx, zero);
      }
      un = nwarps + __shfl_sync(0xffffffffu, nx, 0);
      if (un < a.nunits) load_unit();
      request_first();
      continue;
    }
    int zb = U.z0, zslot = U.z0 % W;
    // write plane zb (direct, or a partial slot when other units touch it), clear its registers
    auto flush = [&]() {
      C v0 = zero, v1 = zero;
      switch (zslot) {
#define DDI_TAKE3(R)                                                      \
  case R:                                                                 \
    if constexpr (R < W) {                                                \
      constexpr int Q = R / 2;                                            \
      if constexpr (COMP) {                                               \
        if constexpr (R % 2 == 0) {                                       \
          v0 = cmk<C>(r0[Q].x - cr0[Q].x, i0[Q].x - ci0[Q].x);            \
          v1 = cmk<C>(r1[Q].x - cr1[Q].x, i1[Q].x - ci1[Q].x);            \
          cr0[Q].x = ci0[Q].x = cr1[Q].x = ci1[Q].x = (T)0;               \
        } else {                                                          \
          v0 = cmk<C>(r0[Q].y - cr0[Q].y, i0[Q].y - ci0[Q].y);            \
          v1 = cmk<C>(r1[Q].y - cr1[Q].y, i1[Q].y - ci1[Q].y);            \
          cr0[Q].y = ci0[Q].y = cr1[Q].y = ci1[Q].y = (T)0;               \
        }                                                                 \
      } else if constexpr (R % 2 == 0) {                                  \
        v0 = cmk<C>(r0[Q].x, i0[Q].x);                                    \
        v1 = cmk<C>(r1[Q].x, i1[Q].x);                                    \
      } else {                                                            \
        v0 = cmk<C>(r0[Q].y, i0[Q].y);                                    \
        v1 = cmk<C>(r1[Q].y, i1[Q].y);                                    \
      }                                                                   \
      if constexpr (R % 2 == 0)                                           \
        r0[Q].x = i0[Q].x = r1[Q].x = i1[Q].x = (T)0;                     \
      else                                                                \
        r0[Q].y = i0[Q].y = r1[Q].y = i1[Q].y = (T)0;                     \
    }                                                                     \
    break;
        DDI_COL3_CASES(DDI_TAKE3)
#undef DDI_TAKE3
      }
      const int d = __shfl_sync(0xffffffffu, mydest, zb - U.z0);
      if (d >= 0) {
        C* dst = static_cast<C*>(a.partial) + (size_t)d * (kColX * kColY) + lane;
        dst[0] = v0;
        dst[32] = v1;
      } else {
        // streaming stores: the partial slots stay in L2 for the reduction
        C* dst = static_cast<C*>(a.fine) + (zb >= nfz ? zb - nfz : zb) * plane + cell;
        __stcs(dst, v0);
        __stcs(dst + 4 * nfx, v1);
      }
      ++zb;
      zslot = zslot + 1 == W ? 0 : zslot + 1;
    };
    // group images are copied one ahead, node values read one ahead, node indices two ahead
    int nnext = n1;
    C cnext = zero;
    if (n0 >= 0) cnext = chain_load(cg + n0);
    // after the last group: one more turn that only writes the planes left up to z1
    for (int gi = U.lo; gi <= U.hi; ++gi) {
      const bool end = gi == U.hi;
      if (gi + 1 == U.hi) {
        un = nwarps + __shfl_sync(0xffffffffu, nx, 0);
        if (un < a.nunits) load_unit();
      }
      const C c = cnext;
      cnext = zero;
      const unsigned char* im = sm + buf * I::BYTES;
      if (!end) {
        if (gi + 1 < U.hi) {
          copy_image<I::BYTES>(sm + (buf ^ 1) * I::BYTES, a.image + (size_t)(gi + 1) * I::BYTES, lane);
          if (nnext >= 0) cnext = chain_load(cg + nnext);
          nnext = gi + 2 < U.hi ? __ldg(a.nodes + (size_t)(gi + 2) * 32 + lane) : -1;
        }
        cp_async_commit();
        cp_async_wait<1>();
        __syncwarp();
        buf ^= 1;
      } else {
        request_first();
      }
      // u = c psi_x, lane = visit
      if (!end) {
#pragma unroll
        for (int ch = 0; ch < I::CH; ++ch) {
          T x[I::EPC];
          *reinterpret_cast<int4*>(x) = *reinterpret_cast<const int4*>(im + I::X + ch * 512 + lane * 16);
#pragma unroll
          for (int k = 0; k < I::EPC; ++k) {
            T* dst = reinterpret_cast<T*>(su + (ch * I::EPC + k) * I::RS) + lane;
            dst[0] = c.x * x[k];
            *reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(dst) + 8 * I::RS) = c.y * x[k];
          }
        }
      }
      __syncwarp();
      const int nruns = end ? 1 : *reinterpret_cast<const int*>(im + I::COUNTS + 4);
      for (int r = 0; r < nruns; ++r) {
        const int hd = end ? U.z1 << 12 : *reinterpret_cast<const int*>(im + I::HEAD + 4 * r);
        const int j0 = hd & 63, j1 = (hd >> 6) & 63, sr = hd >> 12;
        while (zb < sr) flush();
        if (end) break;
        // the run's sum of u psi_y, two visits at a time
        C a0r = zero, a0i = zero, a1r = zero, a1i = zero;
        const unsigned char* pu = su + lx * I::RS + j0 * (int)sizeof(T);
        const unsigned char* py = im + I::Y + ly * I::RS + j0 * (int)sizeof(T);
#pragma unroll 2
        for (int j = j0; j < j1; j += 2) {
          const C ur = *reinterpret_cast<const C*>(pu), ui = *reinterpret_cast<const C*>(pu + 8 * I::RS);
          const C y0 = *reinterpret_cast<const C*>(py), y1 = *reinterpret_cast<const C*>(py + 4 * I::RS);
          a0r = dot2(ur, y0, a0r);
          a0i = dot2(ui, y0, a0i);
          a1r = dot2(ur, y1, a1r);
          a1i = dot2(ui, y1, a1i);
          pu += sizeof(C);
          py += sizeof(C);
        }
        const C g0 = cmk<C>(dot_sum(a0r), dot_sum(a0i)), g1 = cmk<C>(dot_sum(a1r), dot_sum(a1i));
        const C* pz = reinterpret_cast<const C*>(im + I::Z + r * I::ZS);
#pragma unroll
        for (int q = 0; q < W / 2; ++q) {
          const C z = pz[q];
          if constexpr (COMP) {
            kahan_add2(r0[q], cr0[q], __fmul2_rn(both<C>(g0.x), z));
            kahan_add2(i0[q], ci0[q], __fmul2_rn(both<C>(g0.y), z));
            kahan_add2(r1[q], cr1[q], __fmul2_rn(both<C>(g1.x), z));
            kahan_add2(i1[q], ci1[q], __fmul2_rn(both<C>(g1.y), z));
          } else {
            r0[q] = fma2(both<C>(g0.x), z, r0[q]);
            i0[q] = fma2(both<C>(g0.y), z, i0[q]);
            r1[q] = fma2(both<C>(g1.x), z, r1[q]);
            i1[q] = fma2(both<C>(g1.y), z, i1[q]);
          }
        }
      }
      __syncwarp();  // the next group overwrites this image and u
    }
  }
  cp_async_wait<0>();
}

// 2D spread (FP32): a warp takes a unit, a range of groups of one 8 x 8 block, and sums
// c_q psi_x psi_y for its two cells per lane, four visits at a time: four 16-byte shared loads and
// eight packed FMAs, three issues a visit.  A block of several units goes to partial slots that
// k_reduce_col3 sums in unit order.
//
// The 2N x 2N polar rule puts about 1.3 nodes on every fine cell, so the blocks' visit lists are long
// and there is nothing to share between nodes (no rings of one k_z).  The kernels this replaces kept
// windows of rows whose runs were 1-3 visits (columns) or read and wrote each tap in shared memory
// (tiles).  Bound by issue and by reading the images (72 bytes a visit, 3.5 visits a node).  Spread +
// reduction, against the tiles: 128^2 39 -> 17 us, 512^2 90 -> 51 us, 1024^2 299 -> 135 us.
struct BlockArgs {
  int nfx, ncx;
  const ColUnit* units;  // col: block index; z0: -1 (the fine grid) or the partial slot
  int nunits;
  int* counter;
  const unsigned char* image;
  const int* nodes;
  const float2* c;
  float2* fine;
  float2* partial;
};

struct BlockSmem {
  static constexpr int U = 2 * BlockImage<float>::BYTES;
  static constexpr int BYTES = (U + 16 * BlockImage<float>::RS + 127) / 128 * 128;
};

__global__ void __launch_bounds__(kColThreads3, 8) k_spread_block(BlockArgs a) {
  using I = BlockImage<float>;
  using S = BlockSmem;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  chain_release();
  chain_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* sm = smem_raw + warp * S::BYTES;
  unsigned char* su = sm + S::U;
  const int lx = lane & 7, ly = lane >> 3;
  const int nwarps = gridDim.x * (blockDim.x >> 5);
  const float2 zero = make_float2(0.f, 0.f);
  for (int un = warp * gridDim.x + blockIdx.x; un < a.nunits;) {
    const ColUnit U = a.units[un];
    int nx = 0;
    if (lane == 0) nx = atomicAdd(a.counter, 1);
    float2 s0r = zero, s0i = zero, s1r = zero, s1i = zero;
    // group images are copied one ahead, node values read one ahead, node indices two ahead
    int buf = 0, nnext = -1;
    float2 cnext = zero;
    if (U.lo < U.hi) {
      copy_image<I::BYTES>(sm, a.image + (size_t)U.lo * I::BYTES, lane);
      const int n0 = __ldg(a.nodes + (size_t)U.lo * 32 + lane);
      if (U.lo + 1 < U.hi) nnext = __ldg(a.nodes + (size_t)(U.lo + 1) * 32 + lane);
      if (n0 >= 0) cnext = chain_load(a.c + n0);
    }
    cp_async_commit();
    for (int gi = U.lo; gi < U.hi; ++gi) {
      const float2 c = cnext;
      cnext = zero;
      if (gi + 1 < U.hi) {
        copy_image<I::BYTES>(sm + (buf ^ 1) * I::BYTES, a.image + (size_t)(gi + 1) * I::BYTES, lane);
        if (nnext >= 0) cnext = chain_load(a.c + nnext);
        nnext = gi + 2 < U.hi ? __ldg(a.nodes + (size_t)(gi + 2) * 32 + lane) : -1;
      }
      cp_async_commit();
      cp_async_wait<1>();
      __syncwarp();
      const unsigned char* im = sm + buf * I::BYTES;
      buf ^= 1;
      // u = c psi_x, lane = visit
#pragma unroll
      for (int ch = 0; ch < I::CH; ++ch) {
        const float4 x = *reinterpret_cast<const float4*>(im + I::X + ch * 512 + lane * 16);
        const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float* dst = reinterpret_cast<float*>(su + (ch * 4 + k) * I::RS) + lane;
          dst[0] = c.x * xs[k];
          *reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(dst) + 8 * I::RS) = c.y * xs[k];
        }
      }
      __syncwarp();
      // the group's sums, then added to the unit's: a cell takes some hundred terms of the size of its
      // total, and one running sum of them all lost 1.5 times the accuracy of the result
      float2 a0r = zero, a0i = zero, a1r = zero, a1i = zero;
      const float4* ur = reinterpret_cast<const float4*>(su + lx * I::RS);
      const float4* ui = reinterpret_cast<const float4*>(su + (8 + lx) * I::RS);
      const float4* y0 = reinterpret_cast<const float4*>(im + I::Y + ly * I::RS);
      const float4* y1 = reinterpret_cast<const float4*>(im + I::Y + (ly + 4) * I::RS);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 r = ur[j], i = ui[j], p = y0[j], q = y1[j];
        a0r = dot2(make_float2(r.x, r.y), make_float2(p.x, p.y), a0r);
        a0i = dot2(make_float2(i.x, i.y), make_float2(p.x, p.y), a0i);
        a1r = dot2(make_float2(r.x, r.y), make_float2(q.x, q.y), a1r);
        a1i = dot2(make_float2(i.x, i.y), make_float2(q.x, q.y), a1i);
        a0r = dot2(make_float2(r.z, r.w), make_float2(p.z, p.w), a0r);
        a0i = dot2(make_float2(i.z, i.w), make_float2(p.z, p.w), a0i);
        a1r = dot2(make_float2(r.z, r.w), make_float2(q.z, q.w), a1r);
        a1i = dot2(make_float2(i.z, i.w), make_float2(q.z, q.w), a1i);
      }
      s0r = __fadd2_rn(s0r, a0r);
      s0i = __fadd2_rn(s0i, a0i);
      s1r = __fadd2_rn(s1r, a1r);
      s1i = __fadd2_rn(s1i, a1i);
      __syncwarp();  // the next group overwrites this image and u
    }
    const float2 v0 = make_float2(dot_sum(s0r), dot_sum(s0i)), v1 = make_float2(dot_sum(s1r), dot_sum(s1i));
    if (U.z0 >= 0) {
      float2* dst = a.partial + (size_t)U.z0 * (kColX * kColY) + lane;
      dst[0] = v0;
      dst[32] = v1;
    } else {
      const int bx = U.col % a.ncx, by = U.col / a.ncx;
      float2* dst = a.fine + (long long)(by * kColY + ly) * a.nfx + bx * kColX + lx;
      dst[0] = v0;
      dst[4 * a.nfx] = v1;
    }
    un = nwarps + __shfl_sync(0xffffffffu, nx, 0);
  }
  cp_async_wait<0>();
}

// Planes of a column that several units touch: the entry's partial slots are contiguous (s0 ..
// s0 + ns - 1, in unit order).  The first `nlong` entries hold many slots (the dense columns
// around k = 0: hundreds): a CTA's 8 warps sum a contiguous eighth each, then warp 0 adds the
// eight sums in order.  The others take a warp each.  The order is fixed by the plan
// (deterministic); a lane sums two cells, eight loads in flight at a time.
template <typename T>
__global__ void __launch_bounds__(256)
    k_reduce_col3(const ColRed* __restrict__ red, int nred, int nlong, const cx_t<T>* partial,
                  cx_t<T>* __restrict__ fine, int nfx, int nfy, int ncx) {
  using C = cx_t<T>;
  __shared__ C sh[7][64];
  chain_release();
  chain_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool team = (int)blockIdx.x < nlong;
  const int e = team ? (int)blockIdx.x : nlong + ((int)blockIdx.x - nlong) * 8 + warp;
  if (e >= nred) return;
  const int4 r = __ldg(reinterpret_cast<const int4*>(red) + e);  // col, z, s0, ns
  const int k0 = team ? r.w * warp / 8 : 0, k1 = team ? r.w * (warp + 1) / 8 : r.w;
  C v0 = cmk<C>((T)0, (T)0), v1 = v0;  // cells 2 lane and 2 lane + 1 of the slot (row-major 8 x 8)
  const C* src = partial + (size_t)r.z * (kColX * kColY) + 2 * lane;
  auto load = [&](int k, C& p, C& q) {
    const C* at = src + (size_t)k * (kColX * kColY);
    if constexpr (sizeof(T) == 4) {
      const float4 f = __ldcs(reinterpret_cast<const float4*>(at));
      p = make_float2(f.x, f.y);
      q = make_float2(f.z, f.w);
    } else {
      p = __ldcs(at);
      q = __ldcs(at + 1);
    }
  };
  int k = k0;
  for (; k + 8 <= k1; k += 8) {
    C p[8], q[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) load(k + i, p[i], q[i]);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      v0 = cadd(v0, p[i]);
      v1 = cadd(v1, q[i]);
    }
  }
  for (; k < k1; ++k) {
    C p, q;
    load(k, p, q);
    v0 = cadd(v0, p);
    v1 = cadd(v1, q);
  }
  if (team) {
    if (warp > 0) {
      sh[warp - 1][2 * lane] = v0;
      sh[warp - 1][2 * lane + 1] = v1;
    }
    __syncthreads();
    if (warp > 0) return;
#pragma unroll
    for (int w = 0; w < 7; ++w) {
      v0 = cadd(v0, sh[w][2 * lane]);
      v1 = cadd(v1, sh[w][2 * lane + 1]);
    }
  }
  const int cx = r.x % ncx, cy = r.x / ncx, c0 = 2 * lane;
  C* dst = fine + (long long)r.y * nfx * nfy + (long long)(cy * kColY + c0 / 8) * nfx + cx * kColX + c0 % 8;
  if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(dst) = make_float4(v0.x, v0.y, v1.x, v1.y);
  } else {
    dst[0] = v0;
    dst[1] = v1;
  }
}

// ---- interpolation (type 2) ------------------------------------------------------------------------
// The spread's transpose over the same groups.  A warp holds W planes of its column in registers
// (lane (lx, ly): cells (lx, ly) and (lx, ly + 4); plane p in register p mod W), loading each plane
// of the unit's window once.  Per run of one z class every lane sums H = sum_z psi_z F for its
// two cells; the group's H blocks (one per run) go to shared memory, and then a lane per visit
// sums sum_y psi_y sum_x psi_x H over the 8 x 8 cells of its run's block: no reduction across
// lanes.  The visit's sum is its column's share of f_q; k_node_sum3 adds a node's shares in a
// fixed order (deterministic) and applies 2 h^d W_q.
//
// What bounds it: FP64 operations (4 W per run and lane, 144 per visit, against 2 per tap and 8/7
// idle lanes of a gather), in FP32 instruction issue; the gather kernel (k_interp) was bound by L1
// wavefronts, 64-byte pieces of unrelated rows.
struct InterpArgs3 {
  int nf[3];
  int ncx;
  int xlo, nx, ylo, ny;  // fine x and y lines that hold transformed values (cyclic ranges)
  const ColUnit* units;  // the units with visits come first
  int nunits;
  int* counter;
  const unsigned char* image;
  const void* fine;
  void* share;           // [group][32] each visit's sum
};

template <typename T, int W>
struct InterpSmem {
  static constexpr int HS = kColX * kColY * 2 * (int)sizeof(T) + 16;  // bytes between the runs' H blocks
  static constexpr int H = 2 * ColImage<T, W>::BYTES;
  static constexpr int BYTES = (H + kColRuns * HS + 127) / 128 * 128;
};

template <typename T, int W>
__global__ void __launch_bounds__(kColThreads3, sizeof(T) == 4 ? 4 : 2) k_interp_col3(InterpArgs3 a) {
  using C = cx_t<T>;
  using I = ColImage<T, W>;
  using S = InterpSmem<T, W>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  chain_release();
  chain_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* sm = smem_raw + warp * S::BYTES;
  unsigned char* sh = sm + S::H;
  const int lx = lane & 7, ly = lane >> 3;
  const int nfx = a.nf[0], nfy = a.nf[1], nfz = a.nf[2];
  const long long plane = (long long)nfx * nfy;
  const C zero = cmk<C>((T)0, (T)0);
  auto inside = [](int l, int lo, int n, int nf) {
    int d = l - lo;
    if (d < 0) d += nf;
    return d < n;
  };
  const int nwarps = gridDim.x * (blockDim.x >> 5);
  for (int un = warp * gridDim.x + blockIdx.x; un < a.nunits;) {
    const ColUnit U = a.units[un];
    int nx = 0;
    if (lane == 0) nx = atomicAdd(a.counter, 1);
    int buf = 0;
    copy_image<I::BYTES>(sm, a.image + (size_t)U.lo * I::BYTES, lane);
    cp_async_commit();
    const int x = (U.col % a.ncx) * kColX + lx, y = (U.col / a.ncx) * kColY + ly;
    // cells off the transformed lines hold no value of this evaluation: they count as zero (no
    // visit has a tap there)
    const bool inx = inside(x, a.xlo, a.nx, nfx);
    const bool ok0 = inx && inside(y, a.ylo, a.ny, nfy), ok1 = inx && inside(y + 4, a.ylo, a.ny, nfy);
    const C* col = static_cast<const C*>(a.fine) + (long long)y * nfx + x;
    auto load = [&](int z, C& v0, C& v1) {
      const C* at = col + (z >= nfz ? z - nfz : z) * plane;
      v0 = ok0 ? chain_load(at) : zero;
      v1 = ok1 ? chain_load(at + 4 * nfx) : zero;
    };
    C r0[W / 2], i0[W / 2], r1[W / 2], i1[W / 2];  // planes 2 q and 2 q + 1 (mod W)
    C p0 = zero, p1 = zero;                          // plane zl, requested ahead
    int zl = U.z0 - W, zslot = 0;                    // planes zl - W .. zl - 1 are in the window
    for (int gi = U.lo; gi < U.hi; ++gi) {
      if (gi + 1 < U.hi)
        copy_image<I::BYTES>(sm + (buf ^ 1) * I::BYTES, a.image + (size_t)(gi + 1) * I::BYTES, lane);
      cp_async_commit();
      cp_async_wait<1>();
      __syncwarp();
      const unsigned char* im = sm + buf * I::BYTES;
      buf ^= 1;
      const int nslots = *reinterpret_cast<const int*>(im + I::COUNTS);
      const int nruns = *reinterpret_cast<const int*>(im + I::COUNTS + 4);
      int myrun = 0;
      for (int r = 0; r < nruns; ++r) {
        const int hd = *reinterpret_cast<const int*>(im + I::HEAD + 4 * r);
        const int j0 = hd & 63, sr = hd >> 12;
        if (lane >= j0) myrun = r;
        if (sr + W - zl > 3) {
          // the unit's first run, or a gap: the whole window in one go (all loads in flight)
          const int rot = sr % W;
#pragma unroll
          for (int k = 0; k < W; ++k) {
            C v0, v1;
            load(sr + (k >= rot ? k - rot : k - rot + W), v0, v1);
            if (k % 2 == 0) {
              r0[k / 2].x = v0.x, i0[k / 2].x = v0.y, r1[k / 2].x = v1.x, i1[k / 2].x = v1.y;
            } else {
              r0[k / 2].y = v0.x, i0[k / 2].y = v0.y, r1[k / 2].y = v1.x, i1[k / 2].y = v1.y;
            }
          }
          zl = sr + W;
          zslot = rot;
          if (zl < U.z1) load(zl, p0, p1);
        }
        while (zl < sr + W) {
          switch (zslot) {
#define DDI_PUT3(R)                                                      \
  case R:                                                                \
    if constexpr (R < W) {                                               \
      constexpr int Q = R / 2;                                           \
      if constexpr (R % 2 == 0)                                          \
        r0[Q].x = p0.x, i0[Q].x = p0.y, r1[Q].x = p1.x, i1[Q].x = p1.y;  \
      else                                                               \
        r0[Q].y = p0.x, i0[Q].y = p0.y, r1[Q].y = p1.x, i1[Q].y = p1.y;  \
    }                                                                    \
    break;
            DDI_COL3_CASES(DDI_PUT3)
#undef DDI_PUT3
          }
          ++zl;
          zslot = zslot + 1 == W ? 0 : zslot + 1;
          if (zl < U.z1) load(zl, p0, p1);
        }
        C h0r = zero, h0i = zero, h1r = zero, h1i = zero;
        const C* pz = reinterpret_cast<const C*>(im + I::Z + r * I::ZS);
#pragma unroll
        for (int q = 0; q < W / 2; ++q) {
          const C z = pz[q];
          h0r = dot2(z, r0[q], h0r);
          h0i = dot2(z, i0[q], h0i);
          h1r = dot2(z, r1[q], h1r);
          h1i = dot2(z, i1[q], h1i);
        }
        C* h = reinterpret_cast<C*>(sh + r * S::HS) + lane;  // row-major 8 x 8 cells
        h[0] = cmk<C>(dot_sum(h0r), dot_sum(h0i));
        h[32] = cmk<C>(dot_sum(h1r), dot_sum(h1i));
      }
      __syncwarp();
      // lane = visit
      T wx[8];
#pragma unroll
      for (int ch = 0; ch < I::CH; ++ch)
        *reinterpret_cast<int4*>(wx + ch * I::EPC) = *reinterpret_cast<const int4*>(im + I::X + ch * 512 + lane * 16);
      const unsigned char* h = sh + myrun * S::HS;
      C f = zero;
#pragma unroll
      for (int yy = 0; yy < 8; ++yy) {
        const T wy = reinterpret_cast<const T*>(im + I::Y + yy * I::RS)[lane];
        C t = zero;
#pragma unroll
        for (int xx = 0; xx < 8; xx += 16 / (int)sizeof(C)) {
          C v[16 / sizeof(C)];
          *reinterpret_cast<int4*>(v) = *reinterpret_cast<const int4*>(h + (yy * 8 + xx) * (int)sizeof(C));
#pragma unroll
          for (int k = 0; k < (int)(16 / sizeof(C)); ++k) t = fma2(both<C>(wx[xx + k]), v[k], t);
        }
        f = fma2(both<C>(wy), t, f);
      }
      if (lane < nslots) static_cast<C*>(a.share)[(size_t)gi * 32 + lane] = f;
      __syncwarp();  // the next group overwrites this image and the H blocks
    }
    un = nwarps + __shfl_sync(0xffffffffu, nx, 0);
  }
  cp_async_wait<0>();
}

// c_q = 2 h^d W_q times the sum of the node's shares, in the order of its columns
template <typename T>
__global__ void __launch_bounds__(256)
    k_node_sum3(const int* __restrict__ off, const int* __restrict__ pos, const cx_t<T>* share,
                const T* __restrict__ scale, cx_t<T>* __restrict__ c, int count) {
  using C = cx_t<T>;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  chain_release();
  chain_wait();
  if (i >= count) return;
  const int b = off[i], e = off[i + 1];
  C sum = cmk<C>((T)0, (T)0);
  for (int k = b; k < e; k += 4) {
    C v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = k + q < e ? __ldcs(share + pos[k + q]) : cmk<C>((T)0, (T)0);
#pragma unroll
    for (int q = 0; q < 4; ++q) sum = cadd(sum, v[q]);
  }
  c[i] = cscale(sum, scale[i]);
}

// ---- group images (plan time) -----------------------------------------------------------------
// one warp per group; vis: (node or -1, (oy + 16) << 6 | (ox + 16)); runs: the head's entries;
// counts: (visits, runs)
template <typename T, int W>
__global__ void __launch_bounds__(128)
    k_col_image(const int2* __restrict__ vis, const int* __restrict__ runs, const int2* __restrict__ counts,
                const T* __restrict__ psi, unsigned char* __restrict__ image, int* __restrict__ nodes, int ngroups) {
  using I = ColImage<T, W>;
  const int g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (g >= ngroups) return;
  unsigned char* im = image + (size_t)g * I::BYTES;
  for (int i = lane; i < I::BYTES / 16; i += 32) reinterpret_cast<int4*>(im)[i] = make_int4(0, 0, 0, 0);
  __syncwarp();
  const int2 v = vis[(size_t)g * 32 + lane];
  nodes[(size_t)g * 32 + lane] = v.x;
  if (v.x >= 0) {
    const int ox = (v.y & 63) - 16, oy = ((v.y >> 6) & 63) - 16;
    const T* ps = psi + (size_t)v.x * 3 * W;
    for (int c = 0; c < 8; ++c) {
      if ((unsigned)(c - ox) < (unsigned)W)
        *reinterpret_cast<T*>(im + I::X + c / I::EPC * 512 + lane * 16 + c % I::EPC * (int)sizeof(T)) = ps[c - ox];
      if ((unsigned)(c - oy) < (unsigned)W)
        *reinterpret_cast<T*>(im + I::Y + c * I::RS + lane * (int)sizeof(T)) = ps[W + c - oy];
    }
  }
  const int2 n = counts[g];
  if (lane < n.y) {
    const int hd = runs[(size_t)g * kColRuns + lane];
    *reinterpret_cast<int*>(im + I::HEAD + 4 * lane) = hd;
    const int node = vis[(size_t)g * 32 + (hd & 63)].x, rot = (hd >> 12) % W;
    T* z = reinterpret_cast<T*>(im + I::Z + lane * I::ZS);
    for (int k = 0; k < W; ++k) z[rot + k < W ? rot + k : rot + k - W] = psi[(size_t)node * 3 * W + 2 * W + k];
  }
  if (lane == 0) *reinterpret_cast<int2*>(im + I::COUNTS) = n;
}

// the 2D images: vis as in k_col_image
template <int W>
__global__ void __launch_bounds__(128)
    k_block_image(const int2* __restrict__ vis, const float* __restrict__ psi, unsigned char* __restrict__ image,
                  int* __restrict__ nodes, int ngroups) {
  using I = BlockImage<float>;
  const int g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (g >= ngroups) return;
  unsigned char* im = image + (size_t)g * I::BYTES;
  const int2 v = vis[(size_t)g * 32 + lane];
  nodes[(size_t)g * 32 + lane] = v.x;
  const int ox = (v.y & 63) - 16, oy = ((v.y >> 6) & 63) - 16;
  const float* ps = psi + (size_t)(v.x < 0 ? 0 : v.x) * 3 * W;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const bool inx = v.x >= 0 && (unsigned)(c - ox) < (unsigned)W, iny = v.x >= 0 && (unsigned)(c - oy) < (unsigned)W;
    *reinterpret_cast<float*>(im + I::X + c / I::EPC * 512 + lane * 16 + c % I::EPC * 4) = inx ? ps[c - ox] : 0.f;
    *reinterpret_cast<float*>(im + I::Y + c * I::RS + lane * 4) = iny ? ps[W + c - oy] : 0.f;
  }
  if (lane < 8) *reinterpret_cast<int4*>(im + I::Y + lane * I::RS + 128) = make_int4(0, 0, 0, 0);  // row padding
}

enum class ColOp { ImageBytes, BuildImage, Configure, Spread, Interp };

struct ColBuild {
  const int2* vis;
  const int* runs;
  const int2* counts;
};

template <typename T, int W, bool COMP>
int col_op(Plan& p, cudaStream_t s, ColOp op, const ColBuild* b, size_t* out) {
  using I = ColImage<T, W>;
  if (op == ColOp::ImageBytes) {
    *out = I::BYTES;
    return DDI_OK;
  }
  if (op == ColOp::BuildImage) {
    if (p.ngroups == 0) return DDI_OK;
    k_col_image<T, W><<<(unsigned)((p.ngroups + 3) / 4), 128, 0, s>>>(b->vis, b->runs, b->counts,
                                                                      static_cast<const T*>(p.d_psi), p.d_cimage,
                                                                      p.d_cnodes, p.ngroups);
    DDI_LAUNCH_CHECK();
    return DDI_OK;
  }
  auto kern = k_spread_col3<T, W, COMP>;
  auto interp = k_interp_col3<T, W>;
  constexpr size_t smem = (size_t)SpreadSmem<T, W>::BYTES * (kColThreads3 / 32);
  constexpr size_t ismem = (size_t)InterpSmem<T, W>::BYTES * (kColThreads3 / 32);
  constexpr int wpc = kColThreads3 / 32;
  if (op == ColOp::Configure) {
    DDI_TRY(prepare_kernel(reinterpret_cast<const void*>(kern), smem));
    DDI_TRY(prepare_kernel(reinterpret_cast<const void*>(interp), ismem));
    int per_sm = 0, iper_sm = 0, sms = 0;
    DDI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kColThreads3, smem));
    DDI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&iper_sm, interp, kColThreads3, ismem));
    DDI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p.device));
    p.spread_smem = smem;
    p.spread_blocks = std::max(1, std::min(per_sm * sms, (p.ncunits + wpc - 1) / wpc));
    p.interp_blocks = std::max(1, std::min(iper_sm * sms, (p.ncvunits + wpc - 1) / wpc));
    return DDI_OK;
  }
  if (op == ColOp::Interp) {
    if (p.Mh == 0) return DDI_OK;
    InterpArgs3 a;
    for (int d = 0; d < 3; ++d) a.nf[d] = p.nf[d];
    a.ncx = p.nf[0] / kColX;
    a.xlo = p.xr[0], a.nx = p.xr[1], a.ylo = p.yr[0], a.ny = p.yr[1];
    a.units = p.d_cunits;
    a.nunits = p.ncvunits;
    a.counter = p.d_counter + 1;
    a.image = p.d_cimage;
    a.fine = p.d_fine;
    a.share = p.d_cshare;
    DDI_TRY(launch_chain(p, interp, p.interp_blocks, kColThreads3, ismem, s, a));
    p.mark("interp", s);
    DDI_TRY(launch_chain(p, k_node_sum3<T>, (unsigned)((p.Mh + 255) / 256), 256, 0, s, p.d_cnoff, p.d_cnpos,
                         static_cast<const cx_t<T>*>(p.d_cshare), static_cast<const T*>(p.d_scale),
                         static_cast<cx_t<T>*>(p.d_c), (int)p.Mh));
    p.mark("node_sum", s);
    return DDI_OK;
  }
  ColArgs3 a;
  for (int d = 0; d < 3; ++d) a.nf[d] = p.nf[d];
  a.ncx = p.nf[0] / kColX;
  a.units = p.d_cunits;
  a.nunits = p.ncunits;
  a.counter = p.d_counter;
  a.image = p.d_cimage;
  a.nodes = p.d_cnodes;
  a.c = p.d_c;
  a.fine = p.d_fine;
  a.partial = p.d_cpart;
  a.dest = p.d_cslots;
  DDI_TRY(launch_chain(p, kern, p.spread_blocks, kColThreads3, p.spread_smem, s, a));
  p.mark("spread", s);
  if (p.ncred > 0) {
    DDI_TRY(launch_chain(p, k_reduce_col3<T>, (unsigned)(p.ncred_long + (p.ncred - p.ncred_long + 7) / 8), 256, 0, s,
                         p.d_cred, p.ncred, p.ncred_long, static_cast<const cx_t<T>*>(p.d_cpart), static_cast<cx_t<T>*>(p.d_fine), p.nf[0], p.nf[1], a.ncx));
    p.mark("spread_reduce", s);
  }
  return DDI_OK;
}

template <int W>
int block_op(Plan& p, cudaStream_t s, ColOp op, const ColBuild* b, size_t* out) {
  using I = BlockImage<float>;
  constexpr int wpc = kColThreads3 / 32;
  constexpr size_t smem = (size_t)BlockSmem::BYTES * wpc;
  if (op == ColOp::ImageBytes) {
    *out = I::BYTES;
    return DDI_OK;
  }
  if (op == ColOp::BuildImage) {
    if (p.ngroups == 0) return DDI_OK;
    k_block_image<W><<<(unsigned)((p.ngroups + 3) / 4), 128, 0, s>>>(b->vis, static_cast<const float*>(p.d_psi),
                                                                     p.d_cimage, p.d_cnodes, p.ngroups);
    DDI_LAUNCH_CHECK();
    return DDI_OK;
  }
  if (op == ColOp::Configure) {
    DDI_TRY(prepare_kernel(reinterpret_cast<const void*>(k_spread_block), smem));
    int per_sm = 0, sms = 0;
    DDI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spread_block, kColThreads3, smem));
    DDI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p.device));
    p.spread_smem = smem;
    p.spread_blocks = std::max(1, std::min(per_sm * sms, (p.ncunits + wpc - 1) / wpc));
    return DDI_OK;
  }
  if (op != ColOp::Spread) {
    set_error("column interpolation: not built in 2D");
    return DDI_ERR_INTERNAL;
  }
  BlockArgs a;
  a.nfx = p.nf[0];
  a.ncx = p.nf[0] / kColX;
  a.units = p.d_cunits;
  a.nunits = p.ncunits;
  a.counter = p.d_counter;
  a.image = p.d_cimage;
  a.nodes = p.d_cnodes;
  a.c = static_cast<const float2*>(p.d_c);
  a.fine = static_cast<float2*>(p.d_fine);
  a.partial = static_cast<float2*>(p.d_cpart);
  DDI_TRY(launch_chain(p, k_spread_block, p.spread_blocks, kColThreads3, p.spread_smem, s, a));
  p.mark("spread", s);
  if (p.ncred > 0) {
    DDI_TRY(launch_chain(p, k_reduce_col3<float>, (unsigned)(p.ncred_long + (p.ncred - p.ncred_long + 7) / 8), 256, 0, s,
                         p.d_cred, p.ncred, p.ncred_long, static_cast<const float2*>(p.d_cpart), static_cast<float2*>(p.d_fine), p.nf[0], p.nf[1], a.ncx));
    p.mark("spread_reduce", s);
  }
  return DDI_OK;
}

int col_dispatch(Plan& p, cudaStream_t s, ColOp op, const ColBuild* b, size_t* out) {
  if (p.dim == 2) {
    if (p.w == 6) return block_op<6>(p, s, op, b, out);
    if (p.w == 8) return block_op<8>(p, s, op, b, out);
  } else if (p.prec == DDI_FP32) {
    switch (p.w) {
      case 6: return p.col_comp ? col_op<float, 6, true>(p, s, op, b, out) : col_op<float, 6, false>(p, s, op, b, out);
      case 8: return p.col_comp ? col_op<float, 8, true>(p, s, op, b, out) : col_op<float, 8, false>(p, s, op, b, out);
    }
  } else {
    switch (p.w) {
      case 10: return col_op<double, 10, false>(p, s, op, b, out);
      case 12: return col_op<double, 12, false>(p, s, op, b, out);
      case 14: return col_op<double, 14, false>(p, s, op, b, out);
      case 16: return col_op<double, 16, false>(p, s, op, b, out);
    }
  }
  set_error("column spread: kernel width %d not built", p.w);
  return DDI_ERR_ARG;
}

}  // namespace

size_t col_image_bytes(Plan& p) {
  size_t n = 0;
  return col_dispatch(p, nullptr, ColOp::ImageBytes, nullptr, &n) == DDI_OK ? n : 0;
}
int build_col_images(Plan& p, const int2* vis, const int* runs, const int2* counts, cudaStream_t s) {
  const ColBuild b{vis, runs, counts};
  return col_dispatch(p, s, ColOp::BuildImage, &b, nullptr);
}
int configure_spread_col(Plan& p) { return col_dispatch(p, nullptr, ColOp::Configure, nullptr, nullptr); }
int launch_interp_col(Plan& p, cudaStream_t s) { return col_dispatch(p, s, ColOp::Interp, nullptr, nullptr); }
int launch_spread_col(Plan& p, cudaStream_t s) { return col_dispatch(p, s, ColOp::Spread, nullptr, nullptr); }

}  // namespace ddi
