// NUFFT evaluation of the DDI quadrature sum (Sec. 2.1, Eq. DDI-Trun1).
//
//   Phi_j = Re sum_q W_q e^{i k_q.x_j} h^d sum_j' rho_j' e^{-i k_q.x_j'}
//
// With t_q = k_q h (per axis) and centred indices j' = j - n/2 the box centre cancels
// between the two transforms, so the path evaluates
//   f_q   = sum_j' rho_j' e^{-i t_q.j'}                         (type 2)
//   c_q   = 2 h^d W_q f_q       over one node of each (k, -k) pair
//   Phi_j = Re sum_q c_q e^{+i t_q.j'}                            (type 1)
// (the node set is closed under k -> -k with equal weights and rho is real, so the sum
// over the pair is twice the real part of one term).  Both transforms use a 2x
// oversampled grid and the exponential-of-semicircle kernel
//   psi(x) = exp(beta (sqrt(1 - (2x/w)^2) - 1)), |x| < w/2 (x in fine cells),
// with deconvolution by its Fourier transform psihat(2 pi j'/nf).  The nodes are fixed by
// the plan, so the per-axis kernel values psi_d(l - s_q) of every node are built once
// (k_taps, plan.cu: in FP64, rounded to the working precision) and read here.
//
// Launches (fft_nufft.cuh holds the FFT passes, columns.cu the column and block kernels):
//   forward FFT (3D: y with pad + deconvolution fused, x, z; 2D: x, y), pruned to the padded
//               block and to the lines that hold taps
//   interpolation: c_q = 2 h^d W_q f_q, f_q = sum over the w^d taps of psi F.  3D plans that spread
//               by columns interpolate by columns too where that is faster; the others gather:
//               k_interp (3D) and k_interp2 (2D), 8 (w <= 8) or 16 lanes per node, each footprint
//               row read as one contiguous segment
//   spread      by columns (3D) or blocks (2D), or by tiles: k_spread, owner-computes over work
//               units (tile, z-plane in 3D; tile in 2D): a warp takes a unit, streams the nodes
//               whose taps reach that plane (ranges built by the plan) and adds c psi_z psi_y psi_x
//               into its shared-memory plane with plain read-modify-writes (no other unit owns
//               those cells).  Every plane is written once; long units are split into partial
//               planes that k_reduce sums
//   inverse FFT (3D: z, x, y; 2D: y, x), pruned likewise; the last pass fused with crop,
//               deconvolution and real part
#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace ddi {
namespace {

struct GridDims {
  int n[3];
  int nf[3];
};

GridDims dims_of(const Plan& p) {
  GridDims g;
  for (int d = 0; d < 3; ++d) {
    g.n[d] = p.n[d];
    g.nf[d] = p.nf[d];
  }
  return g;
}

// i in [0, 2 nf) -> i mod nf
__device__ __forceinline__ int wrap1(int i, int nf) { return i >= nf ? i - nf : i; }

// kernel values of one axis of a node (w contiguous values), in 16- or 8-byte loads
template <typename T, int W>
__device__ __forceinline__ void load_taps(const T* __restrict__ src, T (&dst)[W]) {
  if constexpr (sizeof(T) == 4 && W % 4 == 0) {
#pragma unroll
    for (int k = 0; k < W / 4; ++k) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(src) + k);
      dst[4 * k] = v.x;
      dst[4 * k + 1] = v.y;
      dst[4 * k + 2] = v.z;
      dst[4 * k + 3] = v.w;
    }
  } else if constexpr (sizeof(T) == 4 && W % 2 == 0) {
#pragma unroll
    for (int k = 0; k < W / 2; ++k) {
      const float2 v = __ldg(reinterpret_cast<const float2*>(src) + k);
      dst[2 * k] = v.x;
      dst[2 * k + 1] = v.y;
    }
  } else if constexpr (sizeof(T) == 8 && W % 2 == 0) {
#pragma unroll
    for (int k = 0; k < W / 2; ++k) {
      const double2 v = __ldg(reinterpret_cast<const double2*>(src) + k);
      dst[2 * k] = v.x;
      dst[2 * k + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < W; ++k) dst[k] = __ldg(src + k);
  }
}

// ---- interpolation (type 2) -----------------------------------------------------------------
// XL lanes per node (one x tap each; 8 for w <= 8, else 16), 32 / XL nodes per warp: the
// lanes of a node read each footprint row of the fine grid as one contiguous segment,
// accumulate the psi_y (and psi_z) weighted sums in registers, and the node's value is
// the psi_x-weighted sum over its lanes (shuffle reduction).
// (at most 64 registers in FP32, so that 4 CTAs per SM keep enough loads in flight)
template <typename T, int W>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2)
    k_interp(const cx_t<T>* fine, const ushort4* __restrict__ l0, const T* __restrict__ psi,
             const T* __restrict__ scale, cx_t<T>* __restrict__ cout, long long count, GridDims g) {
  using C = cx_t<T>;
  constexpr int XL = W <= 8 ? 8 : 16;
  chain_release();
  chain_wait();
  const int lane = threadIdx.x & 31;
  const int rx = lane % XL;
  const long long i0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / XL;
  const bool valid = i0 < count;  // lanes past the end compute a copy of the last node
  const long long i = valid ? i0 : count - 1;
  const ushort4 s = l0[i];
  const T* ps = psi + i * 3 * W;
  T ky[W], kz[W];
  load_taps<T, W>(ps + W, ky);
  load_taps<T, W>(ps + 2 * W, kz);
  const bool on = rx < W;
  const T kx = on ? __ldg(ps + rx) : (T)0;
  const int xx = wrap1(s.x + (on ? rx : 0), g.nf[0]);
  int yoff[W];  // row offsets within a plane (a plane holds < 2^31 cells)
#pragma unroll
  for (int ay = 0; ay < W; ++ay) yoff[ay] = wrap1(s.y + ay, g.nf[1]) * g.nf[0];
  T ar = 0, ai = 0;
  const long long plane = (long long)g.nf[1] * g.nf[0];
#pragma unroll
  for (int az = 0; az < W; ++az) {
    const C* zp = fine + wrap1(s.z + az, g.nf[2]) * plane + xx;
    T zr = 0, zi = 0;
#pragma unroll
    for (int ay = 0; ay < W; ++ay) {
      const C v = chain_load(zp + yoff[ay]);
      zr += ky[ay] * v.x;
      zi += ky[ay] * v.y;
    }
    ar += kz[az] * zr;
    ai += kz[az] * zi;
  }
  ar *= kx;
  ai *= kx;
#pragma unroll
  for (int o = XL / 2; o > 0; o >>= 1) {
    ar += __shfl_xor_sync(0xffffffffu, ar, o);
    ai += __shfl_xor_sync(0xffffffffu, ai, o);
  }
  if (rx == 0 && valid) {
    const T sc = scale[i];
    cout[i] = cmk<C>(sc * ar, sc * ai);
  }
}

// 2D interpolation: as k_interp, but a lane group walks over nodes and requests the next node's taps
// and kernel values before it gathers for the current one.  With 64 taps a node the gather kernel was
// latency-bound: the node's data from memory, then its taps, once per thread (1024^2 143 -> 107 us).
template <typename T, int W>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2)
    k_interp2(const cx_t<T>* fine, const ushort4* __restrict__ l0, const T* __restrict__ psi,
              const T* __restrict__ scale, cx_t<T>* __restrict__ cout, int count, GridDims g) {
  using C = cx_t<T>;
  constexpr int XL = W <= 8 ? 8 : 16;
  chain_release();
  chain_wait();
  const int rx = threadIdx.x % XL;
  const bool on = rx < W;
  const int groups = (int)(gridDim.x * blockDim.x) / XL;
  const int first = (int)(blockIdx.x * blockDim.x + threadIdx.x) / XL;
  ushort4 sn;
  T kyn[W], kxn, scn;
  auto request = [&](int i) {
    const int q = i < count ? i : count - 1;  // lanes past the end work on a copy of the last node
    sn = __ldg(l0 + q);
    const T* ps = psi + (size_t)q * 3 * W;
    load_taps<T, W>(ps + W, kyn);
    kxn = on ? __ldg(ps + rx) : (T)0;
    scn = __ldg(scale + q);
  };
  request(first);
  // every lane of the block makes the same number of turns (the shuffles are of whole warps)
  const int turns = (count - (int)(blockIdx.x * (blockDim.x / XL)) + groups - 1) / groups;
  for (int k = 0; k < turns; ++k) {
    const int i = first + k * groups;
    const ushort4 s = sn;
    const T kx = kxn, sc = scn;
    T ky[W];
#pragma unroll
    for (int a = 0; a < W; ++a) ky[a] = kyn[a];
    const C* at = fine + wrap1(s.x + (on ? rx : 0), g.nf[0]);
    C v[W];
#pragma unroll
    for (int a = 0; a < W; ++a) v[a] = chain_load(at + wrap1(s.y + a, g.nf[1]) * g.nf[0]);
    if (k + 1 < turns) request(i + groups);
    T ar = 0, ai = 0;
#pragma unroll
    for (int a = 0; a < W; ++a) {
      ar += ky[a] * v[a].x;
      ai += ky[a] * v[a].y;
    }
    ar *= kx;
    ai *= kx;
#pragma unroll
    for (int o = XL / 2; o > 0; o >>= 1) {
      ar += __shfl_xor_sync(0xffffffffu, ar, o);
      ai += __shfl_xor_sync(0xffffffffu, ai, o);
    }
    if (rx == 0 && i < count) cout[i] = cmk<C>(sc * ar, sc * ai);
  }
}

// ---- spreading (type 1) ------------------------------------------------------------------------
struct SpreadArgs {
  GridDims g;
  int tile[3];
  int ntile[3];
  const SpreadUnit* units;  // (tile, plane, visit range, slot), largest first
  int nunits;
  int* counter;             // next unit to take (zeroed before the launch)
  const int4* visits;       // (node, ox, oy, oz): starts relative to the tile origin
  const void* c;            // [node] c_q
  const void* psi;          // [node][3][w]
  void* fine;
  void* partial;            // [slot][TY][TX]
};

// per-warp shared memory of k_spread: the plane buffer and a stage of 32 nodes
template <typename T>
struct alignas(16) NodeHead {
  cx_t<T> cz;     // c_q psi_z(plane) (3D), c_q (2D)
  int base;       // buffer index of the footprint's first cell
  unsigned mask;  // taps inside the tile: bit t (x tap t), bit 16 + t (y tap t)
};
template <typename T, int W>
struct alignas(16) WarpStage {
  static constexpr int XL = W <= 8 ? 8 : 16, RL = 32 / XL, MR = (W + RL - 1) / RL, PW = MR * RL;
  T px[32][W];
  T py[32][PW];  // psi_y regrouped per lane row: py[j][MR r + m] = psi_y(r + RL m), 0 past w
  NodeHead<T> hd[32];
};
static_assert(sizeof(WarpStage<float, 8>) == spread_stage_bytes(8, 4), "stage size");
static_assert(sizeof(WarpStage<float, 6>) == spread_stage_bytes(6, 4), "stage size");
static_assert(sizeof(WarpStage<double, 14>) == spread_stage_bytes(14, 8), "stage size");
static_assert(sizeof(WarpStage<double, 10>) == spread_stage_bytes(10, 8), "stage size");

// taps t in [0, w) of a footprint starting at o that land inside [0, T), as a bit mask
__device__ __forceinline__ unsigned tap_mask(int o, int T, int w) {
  const int lo = o < 0 ? -o : 0;
  const int hi = T - o < w ? T - o : w;
  if (hi <= lo) return 0u;
  return ((1u << hi) - 1u) & ~((1u << lo) - 1u);
}

// Spread, one warp per work unit.  A unit is a (tile, z-plane) in 3D and a whole tile in
// 2D: a plane of TY x TX fine cells that no other unit writes, so the warp accumulates it
// in its own shared-memory buffer with plain read-modify-writes and writes it once.
// Persistent: warps take units from a counter (largest first).  Lanes stage 32 nodes at a
// time (kernel values along x and y, c_q psi_z(plane), the footprint's first cell and the
// mask of its taps inside the tile), then the warp adds each node's w x w footprint
// c psi_y psi_x into the plane: lanes are (x, row) pairs, XL along x and 32/XL rows per
// instruction.  Long units are split into pieces that write partial planes (k_reduce).
template <typename T, int W, int DIM>
__global__ void __launch_bounds__(kSpreadThreads) k_spread(SpreadArgs a) {
  using C = cx_t<T>;
  using S = WarpStage<T, W>;
  constexpr int XL = S::XL, RL = S::RL, MR = S::MR;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  chain_release();
  chain_wait();
  const int TX = a.tile[0], TY = a.tile[1], TZ = a.tile[2];
  const int RS = spread_row_stride(TX);
  const int PSZ = TY * RS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t per_warp = spread_warp_bytes(PSZ * sizeof(C), sizeof(S));
  C* plane = reinterpret_cast<C*>(smem_raw + warp * per_warp);
  S* stage = reinterpret_cast<S*>(smem_raw + warp * per_warp + ((PSZ * sizeof(C) + 15) & ~(size_t)15));
  const int nfx = a.g.nf[0], nfy = a.g.nf[1], nfz = a.g.nf[2];
  // an axis held by a single tile wraps around inside it
  const bool wrx = a.ntile[0] == 1, wry = a.ntile[1] == 1, wrz = DIM == 3 && a.ntile[2] == 1;
  const bool wrap = wrx || wry;
  const int4* __restrict__ vis = a.visits;
  const C* cg = static_cast<const C*>(a.c);
  const T* __restrict__ psi = static_cast<const T*>(a.psi);
  const int rx = lane % XL, ry = lane / XL;
  const int rxc = rx < W ? rx : W - 1;
  // this lane's cell of the footprint per row iteration: required mask bits, buffer offset
  unsigned lbit[MR];
  int loff[MR];
#pragma unroll
  for (int m = 0; m < MR; ++m) {
    const int r = ry + RL * m;
    lbit[m] = (rx < W && r < W) ? ((1u << rx) | (1u << (16 + r))) : 0xFFFFFFFFu;
    loff[m] = r * RS + rx;
  }

  for (;;) {
    int u = 0;
    if (lane == 0) u = atomicAdd(a.counter, 1);
    u = __shfl_sync(0xffffffffu, u, 0);
    if (u >= a.nunits) break;
    const SpreadUnit U = a.units[u];
    for (int i = lane; i < PSZ; i += 32) plane[i] = cmk<C>((T)0, (T)0);
    __syncwarp();
    const int p = U.plane;
    for (int kb = U.lo; kb < U.hi; kb += 32) {
      const int cnt = min(32, U.hi - kb);
      if (lane < cnt) {
        const int4 e = vis[kb + lane];
        const size_t node = (size_t)e.x;
        const T* ps = psi + node * 3 * W;
        bool use = true;
        T pz = (T)1;
        if (DIM == 3) {
          int az = p - e.w;
          if (wrz) az = az < 0 ? az + nfz : (az >= nfz ? az - nfz : az);
          use = az >= 0 && az < W;
          pz = use ? ps[2 * W + az] : (T)0;
        }
        const C cq = cg[node];
        T tx[W], ty[W];
        load_taps<T, W>(ps, tx);
        load_taps<T, W>(ps + W, ty);
        const unsigned xm = wrx ? (1u << W) - 1u : tap_mask(e.y, TX, W);
        const unsigned ym = wry ? (1u << W) - 1u : tap_mask(e.z, TY, W);
        NodeHead<T> h;
        h.cz = cmk<C>(cq.x * pz, cq.y * pz);
        h.base = e.z * RS + e.y;
        h.mask = use ? (xm | (ym << 16)) : 0u;
        stage->hd[lane] = h;
#pragma unroll
        for (int q = 0; q < W; ++q) stage->px[lane][q] = tx[q];
#pragma unroll
        for (int r = 0; r < RL; ++r)
#pragma unroll
          for (int m = 0; m < MR; ++m) stage->py[lane][MR * r + m] = r + RL * m < W ? ty[r + RL * m] : (T)0;
      }
      __syncwarp();
      if (!wrap) {
        for (int j = 0; j < cnt; ++j) {
          const NodeHead<T> h = stage->hd[j];
          const T wx = stage->px[j][rxc];
          T wy[MR];
#pragma unroll
          for (int m = 0; m < MR; ++m) wy[m] = stage->py[j][MR * ry + m];
#pragma unroll
          for (int m = 0; m < MR; ++m) {
            if ((h.mask & lbit[m]) == lbit[m]) {
              const T w = wy[m] * wx;
              C* cell = plane + h.base + loff[m];
              C v = *cell;
              v.x += h.cz.x * w;
              v.y += h.cz.y * w;
              *cell = v;
            }
          }
          __syncwarp();  // the next node's cells may belong to other lanes
        }
      } else {
        for (int j = 0; j < cnt; ++j) {
          const NodeHead<T> h = stage->hd[j];
          if (h.mask == 0u) continue;  // this node misses plane p (uniform over the warp)
          const int4 e = vis[kb + j];
          const T wx = stage->px[j][rxc];
          int xx = e.y + rx;
          if (wrx && xx < 0) xx += nfx;
          const bool okx = rx < W && (unsigned)xx < (unsigned)TX;
#pragma unroll
          for (int m = 0; m < MR; ++m) {
            const int r = ry + RL * m;
            int yy = e.z + r;
            if (wry && yy < 0) yy += nfy;
            if (okx && r < W && (unsigned)yy < (unsigned)TY) {
              const T w = stage->py[j][MR * ry + m] * wx;
              C* cell = plane + yy * RS + xx;
              C v = *cell;
              v.x += h.cz.x * w;
              v.y += h.cz.y * w;
              *cell = v;
            }
          }
          __syncwarp();
        }
      }
      __syncwarp();
    }
    __syncwarp();
    // write the plane (or this unit's partial plane)
    const int tx = U.tile % a.ntile[0];
    const int ty = (U.tile / a.ntile[0]) % a.ntile[1];
    const int tz = U.tile / (a.ntile[0] * a.ntile[1]);
    if (U.slot < 0) {
      const int T0x = tile_origin(tx, TX, a.ntile[0], nfx);
      const int T0y = tile_origin(ty, TY, a.ntile[1], nfy);
      int gz = DIM == 3 ? tile_origin(tz, TZ, a.ntile[2], nfz) + p : 0;
      gz -= gz >= nfz ? nfz : 0;
      C* fine = static_cast<C*>(a.fine) + (long long)gz * nfy * nfx;
      for (int ly = 0; ly < TY; ++ly) {
        int gy = T0y + ly;
        gy -= gy >= nfy ? nfy : 0;
        for (int lx = lane; lx < TX; lx += 32) {
          int gx = T0x + lx;
          gx -= gx >= nfx ? nfx : 0;
          fine[(long long)gy * nfx + gx] = plane[ly * RS + lx];
        }
      }
    } else {
      C* part = static_cast<C*>(a.partial) + (long long)U.slot * TX * TY;
      for (int ly = 0; ly < TY; ++ly)
        for (int lx = lane; lx < TX; lx += 32) part[ly * TX + lx] = plane[ly * RS + lx];
    }
    __syncwarp();
  }
}

// Sums the partial planes of split units into the fine grid: one thread per (split unit,
// cell), blockIdx.y = split unit - split0, partials summed in slot order (deterministic).
template <typename T, int DIM>
__global__ void __launch_bounds__(256)
    k_reduce(const SplitUnit* __restrict__ split, const cx_t<T>* partial, cx_t<T>* __restrict__ fine,
             GridDims g, int TX, int TY, int TZ, int ntx, int nty, int ntz, int split0) {
  using C = cx_t<T>;
  const int ncell = TX * TY;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ncell) return;
  const SplitUnit st = split[split0 + blockIdx.y];
  const int tx = st.tile % ntx, ty = (st.tile / ntx) % nty, tz = st.tile / (ntx * nty);
  const C* src = partial + (long long)st.slot0 * ncell + i;
  T sr = 0, si = 0;
  int k = 0;
  for (; k + 4 <= st.nslots; k += 4) {
    C v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = chain_load(src + (long long)(k + q) * ncell);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      sr += v[q].x;
      si += v[q].y;
    }
  }
  for (; k < st.nslots; ++k) {
    const C v = chain_load(src + (long long)k * ncell);
    sr += v.x;
    si += v.y;
  }
  int gx = tile_origin(tx, TX, ntx, g.nf[0]) + i % TX;
  int gy = tile_origin(ty, TY, nty, g.nf[1]) + i / TX;
  int gz = (DIM == 3 ? tile_origin(tz, TZ, ntz, g.nf[2]) : 0) + (DIM == 3 ? st.plane : 0);
  gx -= gx >= g.nf[0] ? g.nf[0] : 0;
  gy -= gy >= g.nf[1] ? g.nf[1] : 0;
  gz -= gz >= g.nf[2] ? g.nf[2] : 0;
  fine[((long long)gz * g.nf[1] + gy) * g.nf[0] + gx] = cmk<C>(sr, si);
}

int spread_col(Plan& p, cudaStream_t s, bool configure) {
  return configure ? configure_spread_col(p) : launch_spread_col(p, s);
}

// ---- launch helpers ----------------------------------------------------------------------------
template <typename T, int W, int DIM>
int launch_interp(Plan& p, cudaStream_t s) {
  const long long cnt = p.Mh;
  constexpr int XL = W <= 8 ? 8 : 16;
  if (cnt == 0) return DDI_OK;
  if constexpr (DIM == 2) {
    // two waves of resident CTAs
    const long long need = (cnt * XL + 255) / 256, most = 152LL * (sizeof(T) == 4 ? 4 : 2) * 2;
    return launch_chain(p, k_interp2<T, W>, (unsigned)std::min(need, most), 256, 0, s,
                        static_cast<const cx_t<T>*>(p.d_fine), static_cast<const ushort4*>(p.d_l0),
                        static_cast<const T*>(p.d_psi), static_cast<const T*>(p.d_scale),
                        static_cast<cx_t<T>*>(p.d_c), (int)cnt, dims_of(p));
  } else {
    return launch_chain(p, k_interp<T, W>, (unsigned)((cnt * XL + 255) / 256), 256, 0, s,
                        static_cast<const cx_t<T>*>(p.d_fine), static_cast<const ushort4*>(p.d_l0),
                        static_cast<const T*>(p.d_psi), static_cast<const T*>(p.d_scale),
                        static_cast<cx_t<T>*>(p.d_c), cnt, dims_of(p));
  }
}

// launch geometry of the spread, fixed per plan (computed once so that applies make no
// host-side queries and can be recorded into a CUDA graph)
template <typename T, int W, int DIM>
int configure_spread(Plan& p, cudaStream_t) {
  const size_t plane_bytes = p.spread_plane_cells() * sizeof(cx_t<T>);
  const size_t smem = spread_warp_bytes(plane_bytes, sizeof(WarpStage<T, W>)) * (kSpreadThreads / 32);
  auto kern = k_spread<T, W, DIM>;
  {
    // the limit belongs to the kernel, shared by every plan (and thread): only raise it
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    cudaFuncAttributes fa;
    DDI_CUDA(cudaFuncGetAttributes(&fa, kern));
    if ((size_t)fa.maxDynamicSharedSizeBytes < smem)
      DDI_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  }
  int per_sm = 0;
  DDI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSpreadThreads, smem));
  int sms = 0;
  DDI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p.device));
  p.spread_smem = smem;
  p.spread_blocks = std::max(1, std::min(per_sm * sms, (p.nunits + kSpreadThreads / 32 - 1) / (kSpreadThreads / 32)));
  return DDI_OK;
}

template <typename T, int W, int DIM>
int launch_spread(Plan& p, cudaStream_t s) {
  SpreadArgs a;
  a.g = dims_of(p);
  for (int d = 0; d < 3; ++d) {
    a.tile[d] = p.tile[d];
    a.ntile[d] = p.ntile[d];
  }
  a.units = p.d_units;
  a.nunits = p.nunits;
  a.counter = p.d_counter;
  a.visits = p.d_visits;
  a.c = p.d_c;
  a.psi = p.d_psi;
  a.fine = p.d_fine;
  a.partial = p.d_partial;
  auto kern = k_spread<T, W, DIM>;
  const size_t smem = p.spread_smem;
  const int blocks = p.spread_blocks;
  DDI_TRY(launch_chain(p, kern, (unsigned)blocks, kSpreadThreads, smem, s, a));
  p.mark("spread", s);
  if (p.nsplit > 0) {
    for (int s0 = 0; s0 < p.nsplit; s0 += 65535) {
      const dim3 grid((unsigned)((p.tile[0] * p.tile[1] + 255) / 256), (unsigned)std::min(65535, p.nsplit - s0));
      k_reduce<T, DIM><<<grid, 256, 0, s>>>(p.d_split, static_cast<const cx_t<T>*>(p.d_partial),
                                            static_cast<cx_t<T>*>(p.d_fine), dims_of(p), p.tile[0], p.tile[1],
                                            p.tile[2], p.ntile[0], p.ntile[1], p.ntile[2], s0);
      DDI_LAUNCH_CHECK();
    }
    p.mark("spread_reduce", s);
  }
  return DDI_OK;
}

// kernel widths built per precision (the plan picks one of them from its tolerance)
#define DDI_WIDTH_SWITCH(FN)                                         \
  template <typename T, int DIM>                                    \
  int FN##_w(Plan& p, cudaStream_t s) {                             \
    if (sizeof(T) == 4) {                                           \
      switch (p.w) {                                                \
        case 6: return FN<T, 6, DIM>(p, s);                         \
        case 8: return FN<T, 8, DIM>(p, s);                         \
      }                                                             \
    } else {                                                        \
      switch (p.w) {                                                \
        case 10: return FN<T, 10, DIM>(p, s);                       \
        case 12: return FN<T, 12, DIM>(p, s);                       \
        case 14: return FN<T, 14, DIM>(p, s);                       \
        case 16: return FN<T, 16, DIM>(p, s);                       \
      }                                                             \
    }                                                               \
    set_error("kernel width %d not built for this precision", p.w); \
    return DDI_ERR_ARG;                                             \
  }

DDI_WIDTH_SWITCH(launch_interp)
DDI_WIDTH_SWITCH(launch_spread)
DDI_WIDTH_SWITCH(configure_spread)

}  // namespace

int configure_kernels(Plan& p) {
  if (p.spread_kind == DDI_SPREAD_COLUMNS) return spread_col(p, nullptr, /*configure=*/true);
  if (p.prec == DDI_FP64)
    return p.dim == 3 ? configure_spread_w<double, 3>(p, nullptr) : configure_spread_w<double, 2>(p, nullptr);
  return p.dim == 3 ? configure_spread_w<float, 3>(p, nullptr) : configure_spread_w<float, 2>(p, nullptr);
}

// Device time of what the plan's current work lists drive, the spread with its partial-plane
// reduction and, in plans that interpolate by columns, the interpolation with its node sums:
// the best of `reps` timed launches after one untimed one (the cost depends on the node set and
// the lists, not on the values).
int time_spread(Plan& p, cudaStream_t s, int reps, float* ms) {
  DDI_CUDA(cudaMemsetAsync(p.d_c, 0, p.cx_size() * (size_t)p.Mh, s));
  if (p.col_interp) DDI_CUDA(cudaMemsetAsync(p.d_fine, 0, p.cx_size() * (size_t)p.fine_points(), s));
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    set_error("time_spread: %s", cudaGetErrorString(cudaGetLastError()));
    return DDI_ERR_CUDA;
  }
  auto once = [&]() -> int {
    DDI_CUDA(cudaMemsetAsync(p.d_counter, 0, 2 * sizeof(int), s));
    if (p.col_interp) DDI_TRY(launch_interp_col(p, s));
    if (p.spread_kind == DDI_SPREAD_COLUMNS) return spread_col(p, s, false);
    if (p.prec == DDI_FP64) return p.dim == 3 ? launch_spread_w<double, 3>(p, s) : launch_spread_w<double, 2>(p, s);
    return p.dim == 3 ? launch_spread_w<float, 3>(p, s) : launch_spread_w<float, 2>(p, s);
  };
  int st = once();
  float best = 0.f;
  for (int r = 0; r < reps && st == DDI_OK; ++r) {
    cudaEventRecord(e0, s);
    st = once();
    cudaEventRecord(e1, s);
    float t = 0.f;
    if (st == DDI_OK && cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess) {
      if (r == 0 || t < best) best = t;
    } else if (st == DDI_OK) {
      set_error("time_spread: %s", cudaGetErrorString(cudaGetLastError()));
      st = DDI_ERR_CUDA;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *ms = best;
  return st;
}

template <typename T>
int run_type2(Plan& p, const T* rho, cudaStream_t s) {
  DDI_TRY(nufft_forward_fft<T>(p, rho, s));
  if (p.col_interp) return launch_interp_col(p, s);
  DDI_TRY((p.dim == 3 ? launch_interp_w<T, 3>(p, s) : launch_interp_w<T, 2>(p, s)));
  p.mark("interp", s);
  return DDI_OK;
}

template <typename T>
int run_type1(Plan& p, T* phi, cudaStream_t s, bool acc = false) {
  if (p.spread_kind == DDI_SPREAD_COLUMNS) {
    DDI_TRY(spread_col(p, s, false));
  } else {
    DDI_TRY((p.dim == 3 ? launch_spread_w<T, 3>(p, s) : launch_spread_w<T, 2>(p, s)));
  }
  return nufft_inverse_fft<T>(p, phi, s, acc);
}

template <typename T>
int run_type1_from_c(Plan& p, T* phi, cudaStream_t s) {
  DDI_CUDA(cudaMemsetAsync(p.d_counter, 0, sizeof(int), s));  // run_ddi: cleared by the forward transform
  return run_type1<T>(p, phi, s);
}

template <typename T>
int run_ddi(Plan& p, const T* rho, T* phi, cudaStream_t s) {
  DDI_TRY(run_type2<T>(p, rho, s));
  if (!p.split()) return run_type1<T>(p, phi, s);
  // split plans (Eq. 3.9): the ball's node values are in d_c, so the fine grid is free for
  // the smooth part I_1 until the spread; I_1 reads rho before it writes phi (which may
  // alias rho), and the ball's part I_2 is added to it
  DDI_TRY(split_smooth_part<T>(p, rho, phi, s));
  return run_type1<T>(p, phi, s, /*acc=*/true);
}

template int run_type2<float>(Plan&, const float*, cudaStream_t);
template int run_type2<double>(Plan&, const double*, cudaStream_t);
template int run_type1_from_c<float>(Plan&, float*, cudaStream_t);
template int run_type1_from_c<double>(Plan&, double*, cudaStream_t);
template int run_ddi<float>(Plan&, const float*, float*, cudaStream_t);
template int run_ddi<double>(Plan&, const double*, double*, cudaStream_t);

}  // namespace ddi
