// Shared device/host definitions of the DDI library: the plan object, complex helpers,
// error reporting.  Included by every .cu translation unit of the library.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <exception>
#include <new>
#include <string>
#include <vector>

#include "../../include/ddi.h"
#include "tables.h"

namespace ddi {

// ---- error reporting (thread-local message behind ddi_last_error) ----------------
void set_error(const char* fmt, ...);
const char* last_error();

#define DDI_CUDA(call)                                                                  \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) {                                                            \
      ::ddi::set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, \
                       __LINE__);                                                       \
      return DDI_ERR_CUDA;                                                              \
    }                                                                                   \
  } while (0)

#define DDI_LAUNCH_CHECK()                                                              \
  do {                                                                                  \
    cudaError_t e_ = cudaGetLastError();                                                \
    if (e_ != cudaSuccess) {                                                            \
      ::ddi::set_error("kernel launch failed: %s (%s:%d)", cudaGetErrorString(e_),      \
                       __FILE__, __LINE__);                                             \
      return DDI_ERR_CUDA;                                                              \
    }                                                                                   \
  } while (0)

// Runs f() (returning a status) so that no C++ exception crosses the C ABI: a failed host
// allocation becomes DDI_ERR_OOM, any other exception DDI_ERR_INTERNAL, with the message
// kept for ddi_last_error().
template <typename F>
int guarded(const char* where, F&& f) noexcept {
  try {
    return f();
  } catch (const std::bad_alloc&) {
    set_error("%s: host allocation failed", where);
    return DDI_ERR_OOM;
  } catch (const std::exception& e) {
    set_error("%s: %s", where, e.what());
    return DDI_ERR_INTERNAL;
  } catch (...) {
    set_error("%s: unknown exception", where);
    return DDI_ERR_INTERNAL;
  }
}

#define DDI_TRY(expr)          \
  do {                         \
    int s_ = (expr);           \
    if (s_ != DDI_OK) return s_; \
  } while (0)

// ---- complex types -------------------------------------------------------------
template <typename T> struct Cx;
template <> struct Cx<float> { using type = float2; };
template <> struct Cx<double> { using type = double2; };
template <typename T> using cx_t = typename Cx<T>::type;

template <typename C> __host__ __device__ __forceinline__ C cmk(decltype(C::x) a, decltype(C::x) b) {
  C r;
  r.x = a;
  r.y = b;
  return r;
}
// (FP32: both components in one packed instruction, rounded as the scalar operations)
template <typename C> __device__ __forceinline__ C cadd(C a, C b) {
  if constexpr (sizeof(C) == 8)
    return __fadd2_rn(a, b);
  else
    return cmk<C>(a.x + b.x, a.y + b.y);
}
template <typename C> __device__ __forceinline__ C csub(C a, C b) {
  if constexpr (sizeof(C) == 8)
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
  else
    return cmk<C>(a.x - b.x, a.y - b.y);
}
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return cmk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C cscale(C a, decltype(C::x) s) { return cmk<C>(a.x * s, a.y * s); }
template <typename C> __device__ __forceinline__ C cconj(C a) { return cmk<C>(a.x, -a.y); }

// ---- spread work list ------------------------------------------------------------
struct SpreadUnit {
  int tile;   // linear tile index (tz * ntiles_y + ty) * ntiles_x + tx
  int plane;  // owned z-plane of the tile in 3D; 0 in 2D (the unit is the whole tile)
  int lo, hi; // range of visit-list entries whose taps cover the plane
  int slot;   // -1: write the plane to the fine grid; >= 0: write to partial slot
};
struct SplitUnit {
  int tile, plane, slot0, nslots;
};

// ---- column spread work list -------------------------------------------------------------------
// 3D: a column is a kColX x kColY block of fine cells in x-y with all its z-planes.  A work unit
// takes a range of the column's visits, sorted by their first z tap, and a window of planes.
// 2D: a block is kColX x kColY cells; a unit takes a range of its visits.
constexpr int kColX = 8, kColY = 8;
constexpr int kColRuns = 8;     // 3D: most runs of one z class per group of 32 visits (columns.cuh)
constexpr int kColPlanes = 32;  // 3D: most planes of a unit's window
struct alignas(16) ColUnit {
  int col;       // column or block index cy * (nf_x / kColX) + cx
  int lo, hi;    // range of groups
  int z0, z1;    // 3D: planes [z0, z1) the unit writes (plane z mod nf_z; z1 may exceed nf_z);
                 // 2D: z0 = -1 (the unit writes the block) or its partial slot
  int plo, phi;  // 3D: leading / trailing planes that other units also touch: go to partial slots
  int slot0;     // 3D, plan time: its shared planes (leading, then trailing) count from slot0
};
struct alignas(16) ColRed {  // a plane of a column touched by several units: the sum of their partial slots
  int col, z;
  int s0, ns;    // partial slots [s0, s0 + ns), one per unit touching the plane, in unit order
};

// ---- spread tile geometry (host and device) -------------------------------------------------
constexpr int kSpreadThreads = 128;  // 4 warps per CTA, each taking work units on its own

// first fine cell of tile t along an axis: t T - T/2 (mod nf), i.e. the tile lattice is
// shifted by half a tile so that k = 0 lies inside a tile; unshifted with a single tile
__host__ __device__ inline int tile_origin(int t, int T, int ntile, int nf) {
  if (ntile == 1) return 0;
  const int o = t * T - T / 2;
  return o < 0 ? o + nf : o;
}
// start of a footprint relative to a tile origin: l0 - T0 wrapped into [-(w-1), nf-(w-1)),
// so that footprints reaching the tile from below through the periodic wrap are negative
__host__ __device__ inline int rel_start(int l0, int T0, int nf, int w) {
  int o = l0 - T0;
  if (o < 0) o += nf;
  if (o > nf - w) o -= nf;
  return o;
}
// Row stride (cells) of the spread's shared-memory plane.  A warp touches 4 rows of 8
// consecutive cells (8-byte cells: half the 128-byte bank window each); with a stride of
// 8 (mod 16) cells consecutive rows fall in opposite halves, so the 32 accesses take the
// minimum two wavefronts.  (16-byte cells fill the window with one 8-cell row segment.)
__host__ __device__ inline int spread_row_stride(int TX) { return TX + ((8 - TX % 16) + 16) % 16; }

// a processed node's symbol direction (x, y, z; 2D: cos, sin, 0) and weight without the
// symbol, FP64, from which its weight is rebuilt for other dipole axes
struct alignas(16) NodeDir {
  double x, y, z, w;
};

// ---- the plan ----------------------------------------------------------------------
struct Plan {
  ddi_plan_desc desc{};
  int dim = 3, prec = DDI_FP64;
  int n[3] = {1, 1, 1};
  int nf[3] = {1, 1, 1};
  double h[3] = {1, 1, 1};
  double dv = 1.0;  // h_1 h_2 h_3
  int w = 8;
  double beta = 0.0;
  int64_t M = 0, Mh = 0;
  int tile[3] = {1, 1, 1};
  int ntile[3] = {1, 1, 1};
  int chunk = 0;
  int device = 0;
  size_t bytes = 0;

  QuadTables quad;                   // host copy of the tables (export, tests)
  std::vector<int64_t> order;        // processing order -> original node index
  std::vector<ushort4> h_l0;         // host copy of d_l0 (spread lists are rebuilt from it)
  std::vector<int> h_zcls;           // z class of each processed node (equal first z tap and psi_z row)
  bool gpe_ready = false;            // GPE workspace allocated (plans of a batch have none)
  size_t spread_bytes = 0;           // device bytes of the spread lists and partial planes
  double tuned_ms = 0.0;             // spread time of the tile the autotuner chose (0: not tuned)

  // device arrays (element types depend on prec), nodes in processing order
  void* d_l0 = nullptr;       // ushort4 [Mh]: wrapped first tap (x, y, z)
  void* d_psi = nullptr;      // T [Mh][3][w]: kernel values along x, y, z at the w taps
  void* d_scale = nullptr;    // T [Mh]: 2 h^d W_q
  NodeDir* d_dirw = nullptr;  // [Mh]: direction and weight without the symbol (ddi_plan_set_axes)
  void* d_c = nullptr;        // cx [Mh]: node values c_q
  void* d_deconv = nullptr;   // double [n0 + n1 + n2]: 1/psihat per axis, index j (0..n-1)
  void* d_deconv_x2 = nullptr;  // float2 [n1] (2D: [n0]): the y (x) factors as FP32 head + tail (FP32 plans)
  void* d_ones = nullptr;     // double [n0 + n1 + n2] of ones: the pad and crop of a split plan's smooth part
  void* d_em1 = nullptr;      // WindowEntry<T> [nf0 + nf1 + nf2], split plans: e^{-k_d^2/k0^2} - 1 at the fine grid's
                              // modes (window.cuh)
  void* d_ones_x2 = nullptr;  // float2 [n1] of (1, 0)
  void* d_fine = nullptr;     // cx [nf0 nf1 nf2]
  void* d_partial = nullptr;  // cx [nslots * tile cells]
  int4* d_visits = nullptr;   // spread visit lists: (node, ox, oy, oz) relative to the tile
  SpreadUnit* d_units = nullptr;
  SplitUnit* d_split = nullptr;
  int* d_counter = nullptr;   // unit counters of the persistent spread and of the column interpolation
  int* d_nonfinite = nullptr; // set by the pad pass when rho holds NaN / Inf (cleared by checks)
  // column spread (spread_kind == DDI_SPREAD_COLUMNS)
  int spread_kind = DDI_SPREAD_TILES;
  unsigned char* d_cimage = nullptr;  // the groups' images (columns.cuh)
  int* d_cnodes = nullptr;    // [group][32] node of each visit, -1: none
  int ngroups = 0;            // groups of visits
  void* d_cshare = nullptr;   // 3D: [group][32] each visit's share of its node's value (interpolation)
  int* d_cnoff = nullptr;     // 3D: [Mh + 1] ranges of d_cnpos
  int* d_cnpos = nullptr;     // 3D: where a node's shares are in d_cshare
  int ncvunits = 0;           // 3D: units with visits (they come first)
  int interp_blocks = 1;
  bool col_interp = false;    // 3D: interpolate by columns too
  ColUnit* d_cunits = nullptr;
  ColRed* d_cred = nullptr;
  int* d_cslots = nullptr;    // 3D: [unit][kColPlanes], the partial slot of each plane of its window, -1 where it
                              // alone writes the plane
  void* d_cpart = nullptr;    // partial planes: [slot][kColY * kColX] complex
  int ncunits = 0, ncred = 0, ncslots = 0;
  int ncred_long = 0;         // the first reduce entries, each summed by a whole CTA
  bool col_comp = false;      // column spread: compensated (Kahan) plane accumulation
  long long visits = 0;       // total visit-list entries
  long long pairs = 0;        // total (node, plane) pairs of all units
  int npl = 1;                // owned planes per tile (z-planes in 3D; 1 in 2D)
  int nunits = 0;
  size_t spread_smem = 0;     // launch geometry of the spread (fixed per plan)
  int spread_blocks = 1;
  int nsplit = 0, nslots = 0;
  // split plans: half-widths of the band of fine-grid lines around k = 0 that hold every tap
  // of the ball's nodes (x and y; 0 = all lines); the ball's NUFFT passes skip the others
  int band[2] = {0, 0};
  // fine-grid y lines that hold node taps: yr[0], yr[0] + 1, .. (mod nf_y), yr[1] of them;
  // the NUFFT's z passes transform only these columns and its y passes only store / read them
  int yr[2] = {0, 1};
  // fine-grid x lines that hold node taps (every line, except for split plans' ball band)
  int xr[2] = {0, 1};
  bool precise_nufft = false;  // NUFFT passes apply FP32 twiddles as head + tail
  bool batch_item = false;     // built by ddi_batch_create
  int tw_n[8] = {};           // lengths of the twiddle tables below
  void* d_tw[8] = {};         // cx twiddle tables e^{-2 pi i k / n} (FP32: n heads, then n tails)
  // GPE workspace
  void* d_psi1 = nullptr;     // cx [N]
  void* d_rho = nullptr;      // T [N]
  void* d_phi = nullptr;      // T [N]
  void* d_work = nullptr;     // cx [N]
  void* d_work2 = nullptr;    // cx [N]
  void* d_kin = nullptr;      // cx [2][n0 + n1 + n2]: per-axis kinetic phase factors for two times
  double* d_red = nullptr;    // reduction partials
  double* h_red = nullptr;    // pinned host copy of reduction results
  void* d_io_in = nullptr;    // staging for ddi_apply_host
  void* d_io_out = nullptr;
  int red_blocks = 0;

  // per-launch CUDA events for ddi_apply_timed (recorded only while `timing` is set)
  bool timing = false;
  int nmarks = 0;
  const char* mark_names[64] = {};
  cudaEvent_t mark_ev[65] = {};
  bool ev_created = false;
  void mark(const char* name, cudaStream_t s) {
    if (!timing || nmarks >= 64) return;
    mark_names[nmarks] = name;
    cudaEventRecord(mark_ev[nmarks + 1], s);
    ++nmarks;
  }

  // the improved split algorithm (Eq. 3.9): the nodes are the small ball's, and the smooth
  // part is added by a padded FFT convolution
  bool split() const { return desc.split_k0 > 0.0; }
  int64_t grid_points() const { return (int64_t)n[0] * n[1] * n[2]; }
  // cells of one owned plane's shared-memory buffer (padded row stride)
  size_t spread_plane_cells() const { return (size_t)tile[1] * spread_row_stride(tile[0]); }
  int64_t fine_points() const { return (int64_t)nf[0] * nf[1] * nf[2]; }
  size_t real_size() const { return prec == DDI_FP64 ? 8 : 4; }
  size_t cx_size() const { return prec == DDI_FP64 ? 16 : 8; }
};

// ---- launches of the DDI's chain of kernels ------------------------------------------------------
// The kernels of an evaluation follow one another on one stream, each needing all of the one before.
// They are launched programmatically dependent: a kernel's CTAs may be placed, and do what needs only
// the plan's constants, while the last CTAs of the one before are still running; chain_wait() then
// holds them until that kernel has completed and its writes are visible.  Every such kernel calls
// chain_wait() in all its threads before it touches what an evaluation writes (or anything a
// caller's work on the stream may still use), so completion carries over along the chain.  Saves
// the launch gap of each of the 9-14 kernels: 24^3 49 -> 36 us, 96x64x48 138 -> 127 us, 128^3 293 -> 270
// us, 256^3 split 1154 -> 1128 us, four 128^3 steps 1479 -> 1349 us.  Not used inside batches, whose side streams fill the gaps, nor in FP64, whose
// kernels are long (128^3 6.73 against 6.75 ms; rotating 64^3 steps were slower with it, 2.95
// against 2.72 ms).
//
// Such a kernel is alive while the ones before it still write.  So what an evaluation or a caller writes
// (the fine grid, node values, shares, partial planes, densities, states, traps, phase tables) is read
// with coherent loads after chain_wait(): through chain_load() or a pointer that is not __restrict__.
// ld.global.nc, which __ldg and const __restrict__ parameters give, is defined only for data that
// nothing writes in the kernel's whole life: it is for the plan's constants (work lists, images, taps,
// factors, twiddles, and the node scales, which ddi_plan_set_axes writes by an ordinary launch).
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// (a plain load: chain_wait's memory clobber keeps it behind the wait.  As a volatile ld.global.ca,
// which the compiler cannot schedule, 192^3 took 869 us instead of 852)
template <typename V> __device__ __forceinline__ V chain_load(const V* p) { return *p; }

// Once per kernel and device: raises the kernel's dynamic shared memory limit to `smem` (the limit
// belongs to the kernel, shared by every plan and thread: only raised).
int prepare_kernel(const void* fn, size_t smem);

template <typename... P, typename... A>
int launch_chain(const Plan& p, void (*kern)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                 A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = p.batch_item || p.prec == DDI_FP64 ? 0 : 1;
  DDI_CUDA(cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...));
  return DDI_OK;
}

inline const void* twiddles(const Plan& p, int n) {
  for (int i = 0; i < 8; ++i)
    if (p.tw_n[i] == n) return p.d_tw[i];
  return nullptr;
}

// ---- FFT twiddle tables (fft.cu) -----------------------------------------------------------
int make_twiddles(Plan& p, int n);

// ---- the GPE's Fourier passes on the plan's grid (gpe_fft.cuh) ---------------------------------
// transforms are unnormalised, dir = -1: e^{-2 pi i jk/n}
template <typename T> int gpe_forward(Plan& p, const cx_t<T>* src, cx_t<T>* a, cudaStream_t s);  // a <- F src
// a <- F^{-1} e^{i f |mu|^2} F src (src may be a) for the per-axis tables tab of e^{i f mu_d^2} - 1 (x, y, z); rho,
// if not null, <- |a|^2
template <typename T>
int gpe_kinetic(Plan& p, const cx_t<T>* src, cx_t<T>* a, const cx_t<T>* tab, T* rho, cudaStream_t s);
// one sweep of the gradient flow's fixed point,
//   out <- F^{-1}[F(phi/dt + (alpha - W) cur) / (1/dt + alpha + |mu|^2/2)],
// and *change <- max |out - cur|^2 (FP64 bits, cleared by the caller); skipped when prev is not
// null and the FP64 number at *prev is <= tol2
template <typename T>
struct GfSweep {
  const cx_t<T>*phi, *cur;
  cx_t<T>* out;
  const T* W;
  T alpha, inv_dt;
  double inv_dt_alpha, ks[3];
  const unsigned long long* prev;
  double tol2;
  unsigned long long* change;
};
template <typename T> int gpe_gf_sweep(Plan& p, const GfSweep<T>& w, cudaStream_t s);

// ---- pruned / fused fine-grid FFTs of the NUFFT (fft_nufft.cuh) ----------------------
template <typename T> int nufft_forward_fft(Plan& p, const T* rho, cudaStream_t s);  // rho -> F (fine grid)
// U (fine grid) -> phi; acc: phi += the result instead of phi = the result
template <typename T> int nufft_inverse_fft(Plan& p, T* phi, cudaStream_t s, bool acc = false);
// split plans: phi = I_1 of Eq. 3.9 (zero-padded FFT convolution of rho with the smooth
// symbol p = (1 - q) Uhat on the fine grid); reads rho before it writes phi (they may alias)
template <typename T> int split_smooth_part(Plan& p, const T* rho, T* phi, cudaStream_t s);

// ---- NUFFT stages (nufft.cu) --------------------------------------------------------
template <typename T> int run_type2(Plan& p, const T* rho, cudaStream_t s);         // rho -> d_c
template <typename T> int run_type1_from_c(Plan& p, T* phi, cudaStream_t s);       // d_c -> phi
template <typename T> int run_ddi(Plan& p, const T* rho, T* phi, cudaStream_t s);
// bytes of the spread's per-warp node stage of 32 nodes: psi_x and psi_y rows (psi_y padded
// to the lanes' row groups) and a 16-byte (FP32) / 32-byte (FP64) header per node
__host__ __device__ constexpr int spread_rows_per_instr(int w) { return 32 / (w <= 8 ? 8 : 16); }
__host__ __device__ constexpr size_t spread_stage_bytes(int w, size_t real_bytes) {
  return 32 * (size_t)w * real_bytes +
         32 * (size_t)(((w + spread_rows_per_instr(w) - 1) / spread_rows_per_instr(w)) * spread_rows_per_instr(w)) *
             real_bytes +
         32 * (real_bytes == 4 ? 16 : 32);
}
// shared memory of one spread warp: its plane buffer and its node stage, 16-byte aligned
__host__ __device__ inline size_t spread_warp_bytes(size_t plane_bytes, size_t stage_bytes) {
  return ((plane_bytes + 15) & ~(size_t)15) + ((stage_bytes + 15) & ~(size_t)15);
}

// 3D column spread (columns.cu): bytes of a group's image, the images from device lists, the
// launch geometry, and the spread with its reduction
size_t col_image_bytes(Plan& p);
int build_col_images(Plan& p, const int2* vis, const int* runs, const int2* counts, cudaStream_t s);
int configure_spread_col(Plan& p);
int launch_spread_col(Plan& p, cudaStream_t s);
int launch_interp_col(Plan& p, cudaStream_t s);  // fine grid -> d_c
int configure_kernels(Plan& p);  // per-plan launch geometry (nufft.cu)
// reads and clears the plan's non-finite-input record after synchronising s:
// DDI_ERR_NONFINITE if it was set (plan.cu)
int take_nonfinite(Plan& p, cudaStream_t s);

// ---- plans (plan.cu) ------------------------------------------------------------------------
int create_plan(Plan& p, const ddi_plan_desc* desc, cudaStream_t stream, bool gpe = true, bool batch_item = false);
void set_tile(Plan& p, const int want[3]);         // tile rounded as for ddi_plan_desc.tile
int build_spread(Plan& p, cudaStream_t stream);     // spread lists for the current tile
int build_spread_col(Plan& p, cudaStream_t stream); // column (2D: block) spread lists for desc.chunk (plan.cu)
bool columns_apply(const Plan& p);                   // the column spread fits the plan (plan.cu)
int time_spread(Plan& p, cudaStream_t s, int reps, float* ms);  // what the lists drive, best of reps (nufft.cu)
int tune_spread_tile(Plan& p, cudaStream_t s);      // autotuner (batch.cu)
void destroy_plan(Plan& p);
void fill_info(const Plan& p, ddi_plan_info* info);
int set_axes(Plan& p, const double* axis_n, const double* axis_m, cudaStream_t s);  // (plan.cu)

}  // namespace ddi

struct ddi_plan_s {
  ddi::Plan p;
};
