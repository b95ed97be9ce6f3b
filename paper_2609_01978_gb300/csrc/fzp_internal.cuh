// fzp_internal.cuh -- shared declarations of libfzp (CUDA C++, sm_103a).
//
// Notation (Eq. 2 and Fig. 2):
//   aperture sample (j, i), i, j in [0, N), centred index di = i - c, c = (N-1)/2,
//   u_i = di * dx;  ROI sample (n, m), x_m = (m - msh) p, msh = -x0 / p
//   (msh = M/2 for the ROI centred on the focus).
//   Row kernel K[m, i] = exp(2 pi i theta(m, i)) with the phase in turns
//     theta(m, i) = di^2 kappa / 2 - (m - msh) di delta,
//     kappa = dx^2 / (lambda f),  delta = p dx / (lambda f)   (Eq. 2, Eq. 10).
//   The same matrix serves the column pass (the grids of both axes coincide):
//     U = Pre * chirp_out .* (K T K^T).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <utility>
#include <vector>

#include "../../include/fzp.h"

namespace fzp {

// --------------------------------------------------------------------------
// Host-side error handling (thread-local message, no exceptions across ABI)
// --------------------------------------------------------------------------
fzp_status set_error(fzp_status st, const char* fmt, ...);

#define FZP_CUDA_TRY(call)                                                              \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess)                                                              \
      return ::fzp::set_error(e_ == cudaErrorMemoryAllocation ? FZP_E_OOM : FZP_E_CUDA, \
                              "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_),   \
                              __FILE__, __LINE__);                                      \
  } while (0)

// Dynamic shared memory above 48 KiB is an attribute of a kernel on one
// device: set it on each device that launches the kernel, once.  `done` holds
// a bit per device ordinal (ordinals from 64 up set it at every call).
inline cudaError_t smem_attr_once(const void* kernel, int bytes, std::atomic<uint64_t>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? (1ull << dev) : 0ull;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

// --------------------------------------------------------------------------
// Mask geometry: exact binary FZP rule (paraxial radii, centre opaque)
//   open(s) = s <= s_R  and  zone(s) odd,   zone(s) = floor(fl(s * kappa)),
//   s = di^2 + dj^2 an exact integer.  zone(s) = #{m >= 1 : S_m <= s} with the
//   threshold table S_m = min{s : floor(fl(s kappa)) >= m} built on the host.
// --------------------------------------------------------------------------
struct MaskGeom {
  int64_t c;          // on-axis index
  int64_t sR;         // largest s inside the aperture disc
  uint64_t K64;       // floor(kappa * 2^64): fixed-point zone rate
  const int64_t* thr; // device: thr[m-1] = S_m, m = 1..nthr
  int64_t nthr;
  int levels;         // 0: binary amplitude (open on odd zones); L >= 2: phase level = zone mod L
  int centre_open;    // binary amplitude: 1 = open on even zones (positive-centred)
};

// zone(s) for 0 <= s <= sR (the zone rate kappa is kappa_L for phase plates).
// The 64x64->128 fixed-point product s K64 / 2^64 lies below s kappa by less
// than s / 2^64 < 2^-18 (s < 2^46), and fl(s kappa) differs from s kappa by
// less than 2^-29 (s kappa < 2^24); so outside a window of 2^-17 below and
// 2^-28 above an integer the product's integer part is floor(fl(s kappa)), and
// inside it the threshold table decides, bit for bit.
__device__ __forceinline__ int64_t zone_of(int64_t s, const MaskGeom& g) {
  const uint64_t hi = __umul64hi((uint64_t)s, g.K64);
  const uint64_t lo = (uint64_t)s * g.K64;
  int64_t z = (int64_t)hi;
  if (lo < (1ull << 36) || lo >= 0xFFFF800000000000ull) {
    if (z >= 1 && __ldg(g.thr + (z - 1)) > s) z -= 1;
    else if (z < g.nthr && __ldg(g.thr + z) <= s) z += 1;
  }
  return z;
}

__device__ __forceinline__ bool mask_open(int64_t dj, int64_t di, const MaskGeom& g) {
  const int64_t s = dj * dj + di * di;
  if (s > g.sR) return false;
  return ((zone_of(s, g) ^ g.centre_open) & 1) != 0;
}

// --------------------------------------------------------------------------
// Membrane deformation phase in turns, 2 w / lambda (phi / 2 pi, phi = (4 pi /
// lambda) w), as FP32 coefficients in sample units (di = i - c, dj = j - c):
//   amp2 sin(2 pi (di kx + dj ky)) (1 - tq (di^2 + dj^2)) + sum_k h2_k exp(-q_k d_k^2),
//   d_k = (di - pi_k) nx_k + (dj - pj_k) ny_k  ((pi_k, pj_k) on the k-th crease).
// kx, ky are split hi + lo with hi a multiple of 2^-14: for |di| < 2^20 and the
// configured wrinkle periods (>= 1 mm at sub-micron pitch) di * kxh is exact in
// FP32, so the integer turns drop exactly before the sine.
// --------------------------------------------------------------------------
struct DeformCoef {
  float kxh, kxl, kyh, kyl, amp2, tq;
  int n;
  float nx[3], ny[3], pi_[3], pj[3], q[3], h2[3];
  // steps along a row (di -> di + 1) for generators that walk columns:
  // the wrinkle phasor turns by e^{2 pi i kx}; a ridge's ratio g(di+1)/g(di)
  // is multiplied by rho_k = exp(-2 q_k nx_k^2)
  float zc, zs, rho[3], eta[3];  // eta = 1 - rho
  float z4;  // 4 sin^2(pi kx): the wrinkle's second difference per column
  // Columns evaluated one by one instead of walked: 1 by the FP32 rows, 2 by the dense
  // generators, too.  In FP32 a walk of 32 columns holds a ridge to 8e-7 of its height
  // down to a full width of 64 columns along the row, to 6e-6 at 16, and loses it
  // at 8 (0.03) and below; 16 columns: 2e-6 at 12, lost at 4 and below; a column by
  // itself: 1.5e-7 at any.  The wrinkle's second difference is ill-conditioned below
  // a period of 3 columns (3e-7 at 3, 5e-6 at 2.1).  The FP32 rows evaluate from 64
  // columns down (they did at any width before they walked), the dense forms,
  // whose values are kept to 2^-17, from 12.
  int direct;
};

// --------------------------------------------------------------------------
// Phase helpers.  Phases are carried in turns; the integer part is removed in
// FP64 before the (co)sine is evaluated.
// --------------------------------------------------------------------------
__device__ __forceinline__ double frac_turns(double t) { return t - rint(t); }

__device__ __forceinline__ float2 cis_turns_f(double t) {
  float s, c;
  sincospif((float)(2.0 * frac_turns(t)), &s, &c);
  return make_float2(c, s);
}

__device__ __forceinline__ double2 cis_turns_d(double t) {
  double s, c;
  sincospi(2.0 * frac_turns(t), &s, &c);
  return make_double2(c, s);
}

template <typename R> struct Cplx;
template <> struct Cplx<float> { using T = float2; };
template <> struct Cplx<double> { using T = double2; };

template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  C r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { C r; r.x = a.x + b.x; r.y = a.y + b.y; return r; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { C r; r.x = a.x - b.x; r.y = a.y - b.y; return r; }
// FP32: both parts in one instruction (the same two roundings).
template <> __device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 p, q, s;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n add.rn.f32x2 s, p, q;\n mov.b64 {%0, %1}, s;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
template <> __device__ __forceinline__ float2 csub(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 p, q, s;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n sub.rn.f32x2 s, p, q;\n mov.b64 {%0, %1}, s;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
// Pairs of FP32 values, both in one instruction.
__device__ __forceinline__ float2 pair2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 p, q, s;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n mul.rn.f32x2 s, p, q;\n mov.b64 {%0, %1}, s;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n .reg .b64 p, q, t, s;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n mov.b64 t, {%6, %7};\n"
      " fma.rn.f32x2 s, p, q, t;\n mov.b64 {%0, %1}, s;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}

template <typename R> __device__ __forceinline__ typename Cplx<R>::T cis_turns(double t);
template <> __device__ __forceinline__ float2 cis_turns<float>(double t) { return cis_turns_f(t); }
template <> __device__ __forceinline__ double2 cis_turns<double>(double t) { return cis_turns_d(t); }

// e^{sign 2 pi i r / L} for an exact integer r (0 <= r < L, L a power of two).
template <typename R> __device__ __forceinline__ typename Cplx<R>::T twiddle(int64_t r, int64_t L, float sign);
template <> __device__ __forceinline__ float2 twiddle<float>(int64_t r, int64_t L, float sign) {
  float s, c;
  sincospif(sign * 2.0f * (float)r / (float)L, &s, &c);
  return make_float2(c, s);
}
template <> __device__ __forceinline__ double2 twiddle<double>(int64_t r, int64_t L, float sign) {
  double s, c;
  sincospi((double)sign * 2.0 * (double)r / (double)L, &s, &c);
  return make_double2(c, s);
}

// --------------------------------------------------------------------------
// Plan
// --------------------------------------------------------------------------
// Decimated rows (k_dec): grid points that a column's value is spread over.
constexpr int DTAPS = 6;

struct Bluestein {
  int64_t L = 0;     // convolution length, power of two >= N + M - 1
  int64_t L1 = 1;    // four-step split L = L1 * L2 (L1 = 1: single pass)
  int64_t L2 = 0;
  void* d_pre = nullptr;  // N entries: e^{2 pi i pre(i)} (complex64 or complex128)
  void* d_H = nullptr;    // L entries: FFT_L of the convolution chirp, stored [k1][k2]
  void* d_Z = nullptr;    // workspace [rows][L1][L2]
  void* d_G = nullptr;    // workspace [rows][L1][M]
  void* d_tab = nullptr;  // table block: chirp v (L) | twiddles (L2/2) | post (M)
  void* d_tw = nullptr;   // into d_tab
  void* d_post = nullptr; // into d_tab
  void* d_twL = nullptr;  // into d_tab: e^{-2 pi i t / L}, t < 4096
  int64_t rows = 0;       // rows per batch of the workspace
  // partitioned convolution (FP32): blocks of S columns, 4096-point spectra of
  // the chirp pieces in d_H as [nseg][4096]; d_Z, d_G unused
  int seg = 0;
  int S = 0;
  int64_t nseg = 0;
  int dec = 0;            // decimated rows: columns to a grid point (then S counts those); 0: none
  float2 T[2][DTAPS][4];  // their weights (decimation_weights), each twice
  int64_t col0 = 0;       // first input column (the axis when `half`)
  bool half = false;      // columns from the axis on, outputs x and -x added
  int64_t L_full = 0;     // power of two >= N + M - 1 (what the plan reports)
};

// One signed-mask pass of a phase plate in the dense form: the mask is +1 on
// the levels in `pos`, -1 on those in `neg` (bit q for level q), 0 elsewhere,
// and the pass's field enters the ROI accumulator times (wr + i wi).
struct MaskPass {
  uint64_t pos = 0, neg = 0;
  double wr = 1.0, wi = 0.0;
  int cx = -1;  // membrane deformation (complex T e^{i phi}): 0 -> mask T cos(phi), 1 -> T sin(phi)
};

struct Dense {
  void* d_A = nullptr;     // kernel matrix, split-BF16, pre-swizzled tiles
  int64_t kblocks = 0;     // ceil(N / 32)
  int ntiles = 0;          // 2M / 128 row tiles of the kernel matrix
  int promote_kblocks = 0; // K blocks per TMEM accumulation chunk
  int group_kblocks = 0;   // K blocks per work-list chunk (promotions of one unit)
  int npairs = 0;          // kernel tile pairs, padded to a multiple of the cluster size
  int cluster = 1;         // CTAs per cluster sharing each mask tile
  int num_sms = 0;
  int max_ctas = 0;        // CTAs that can be resident at once (whole clusters)
  int* d_sched = nullptr;  // work list of a row-pass launch (3 nchunks + 1 ints)
  // SMs that hold no whole cluster: a concurrent single-CTA launch takes a
  // band of stripes there (single plans of cluster launches only)
  int extra_ctas = 0;
  int* d_sched2 = nullptr;
  cudaStream_t s2 = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
};

// A form on interpolation nodes (nodes.cu): n nodes across the ROI, of which ns
// are evaluated (the positive half of them for an even field).
struct NodeSet {
  int n = 0, ns = 0;       // n = 0: the plan does not use nodes
  int Mo = 0;              // outputs per side of the interpolation (even: M / 2 + 1)
  bool even = false;       // flat plate, ROI centred on the focus
  int64_t kblocks = 0;     // ceil(columns / 32)
  double half = 0, h = 0;  // ROI half width and node pitch, in ROI pitches
  double band = 0;         // 2 R p / (lambda f): the field's band, cycles per pitch
  double delta = 0, msh = 0;  // the nodes as a grid: x_k = (k - msh) h p, delta = h p dx / (lambda f)
  double dist = 0;         // distance of the output chirp (f, or the SA-CZT's z_F)
  double* d_W = nullptr;   // interpolation [ns][Mo] (owned by the plan, also in a batch)
  double* d_Wy = nullptr;  // [n][M], behind d_W: along y when the rows are not symmetric
  bool yfull = false;      // the call being run takes all n nodes along y
  bool tri = false;        // its field (not on nodes) is its own transpose: column pass on and above the diagonal
  int64_t zero_acc = 0;    // accumulator elements that the next row pass is to zero first
  int slices = 1;          // images of C1 in the chunk being run, and their distance
  int64_t slice_elems = 0;
  double2* d_chirp = nullptr;  // [M] output chirp of the ROI samples, behind d_W
  double2* d_X = nullptr;  // [ns][M] rows interpolated
};

// What a row of the column pass stands for (flat plates: distances from the axis).
enum RowKind { ROWS_PLAIN = 0, ROWS_FOLDED = 1, ROWS_MIRRORED = 2 };

// SA-CZT (Sec. 3.6, Fig. 5): padded grid and its buffers.
struct SaCzt {
  int64_t P = 0;           // padded grid side, a power of two >= 1.5 N
  int logP = 0;
  int exact = 0;           // 1: exact zone radii of Eq. 3; 0: paraxial radii
  double zF = 0;           // distance of the Fresnel part
  double kmax = 0, d = 0;  // quadratic fit of k_z: c k_max + d K^2 / k_max, c = k0 / k_max
  void* d_G = nullptr;     // P x P complex64
  void* d_T = nullptr;     // P x P complex64 (transposed layout)
  void* d_tw = nullptr;    // P / 2 twiddles e^{-2 pi i t / P}, complex64
  void* d_K = nullptr;     // M x P complex64: Fresnel chirp and zoom kernel
  void* d_RT = nullptr;    // M x P complex64: row pass, transposed
  int64_t* d_xthr = nullptr;  // exact radii: first s of every zone m = 1 .. nx
  int64_t nx = 0;
  // whole apertures on nodes: the zoom kernel's transform E, its operand
  // images and the work list of the contraction
  void* d_E = nullptr;     // [nodes][E stride] complex64
  void* d_EA = nullptr;
  void* d_ZA = nullptr;    // images of K itself over the padded columns (a part of the rows)
  int* d_esched = nullptr;
  int64_t estride = 0;     // P / 2 + 32: the frequencies 0 .. P / 2 and padding
};

struct Plan {
  // problem
  double D, f, lambda, dx, R, p, x0;
  double msh = 0;  // ROI shift in pitches: x_m = (m - msh) p (M/2 when centred)
  int64_t N, c;
  int M;
  int form, precision, stripe_rows;
  int promote_req = 0, row_batch_req = 0, cluster_req = 0;  // tuning knobs as requested (0: default)
  int conv_req = 0;  // Bluestein row convolution as requested (fzp_params.conv)
  bool owns_buffers = true;  // false: tables and workspace belong to a batch
  // derived
  double kappa, delta, dx2, R2;
  int64_t total_zones;
  int levels = 0;               // 0: binary amplitude FZP; L >= 2: L-level phase FZP
  std::vector<MaskPass> passes; // dense form, L >= 4: the signed-mask passes summing to T
  int pass_index = -1;          // pass being run (-1: the plate's single pass)
  double kappa_mask = 0;        // zone rate of the mask rule: kappa, or kappa_L = fl(kappa L/2)
  MaskGeom mg;
  int64_t* d_thr = nullptr;
  bool has_deform = false;
  fzp_deform deform{};
  // workspace shared by both forms
  float* d_C1 = nullptr;       // row intermediate [2M][chunk_rows] (FP32 forms)
  double* d_C1d = nullptr;     // row intermediate [2M][chunk_rows] (FP64 form)
  int64_t chunk_rows = 0;
  bool c1_images = true;        // false: no memory for more than one image of C1
  int64_t c1_rows = 0;          // rows of C1: 2M rounded up to 512
  double2* d_Uacc = nullptr;   // FP64 ROI accumulator M*M
  int* d_err = nullptr;        // device error word (bounded waits)
  double* d_metrics = nullptr; // device scratch for the metric extractor
  size_t device_bytes = 0;
  Bluestein bs;
  SaCzt sa;
  Dense dn;
  NodeSet nd;
  bool fold = false;            // flat plate: the rows at distances +-d from the axis run once
  int64_t c1_stride = 0;        // row length of C1 in the chunk being run
  // tracing: kernel launches issued, and CUDA events around the dominant
  // kernel (recorded on the launching stream when profiling is enabled)
  int64_t launches = 0;
  bool profiling = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_events;
  size_t prof_used = 0;
  const char* dominant = "";
};

// Elements of a plan's row intermediate: C1 of one chunk; a small membrane on
// nodes takes eight images of its two masks' rows where the memory is there (they
// make its sums reproducible; c1_images).
inline size_t c1_elems(const Plan& P) {
  const size_t all = (size_t)((2 * (int64_t)P.M + 511) / 512 * 512) * (size_t)P.chunk_rows;
  if (P.c1_images && P.form == FZP_FORM_DENSE && P.nd.n > 0 && P.has_deform && P.N <= 8192)
    return all > 2048u * (size_t)P.chunk_rows ? all : 2048u * (size_t)P.chunk_rows;
  return all;
}

// Columns to a grid point of the FP32 form's decimated rows (host), 0: none.
int bluestein_decimation(const Plan& P);

// Rows of the partitioned row pass that are in flight at once.
int64_t bluestein_wave(const Plan& P);

// FP32 deformation coefficients of a plan with a deformation (host).
DeformCoef deform_coef(const Plan& P);

// Bracket one launch of the dominant kernel with events (no-op unless profiling).
void prof_begin(Plan& P, cudaStream_t s);
void prof_end(Plan& P, cudaStream_t s);

// Launchers implemented in the .cu files.  All enqueue on `stream`.
// Form layouts: sizes in bytes of the form's tables and transform workspace.
struct FormSizes {
  size_t pre = 0, H = 0, tab = 0, Z = 0, G = 0;  // Bluestein
  size_t A = 0, sched = 0;                       // dense
  size_t X = 0;                                  // dense on nodes
};
// FP64 row passes of a flat plate whose ROI is centred on the focus: only the
// samples x >= 0 (and x = (M / 2) p, the mirror image of the first) are
// evaluated, M / 2 + 1 per axis, unless the row range is not symmetric.
inline bool bluestein_even(const Plan& P) {
  return P.form == FZP_FORM_BLUESTEIN && P.precision == FZP_PREC_FP64 && !P.has_deform && P.msh == (double)(P.M / 2);
}
fzp_status bluestein_layout(Plan& P, FormSizes* out);
fzp_status bluestein_fill_tables(Plan& P, cudaStream_t s);  // buffers already assigned
fzp_status bluestein_build_tables(Plan& P);                 // layout + allocate + fill
fzp_status bluestein_rows(Plan& P, int64_t j0, int64_t rows, bool octant, cudaStream_t stream);
fzp_status dense_layout(Plan& P, FormSizes* out);
fzp_status dense_fill_tables(Plan& P, cudaStream_t s);
fzp_status dense_build_tables(Plan& P);
fzp_status dense_rows(Plan& P, int64_t j0, int64_t rows, cudaStream_t stream);
// The SA-CZT zoom on the tensor cores: kernel images of `ncols` columns with
// the chirp-kernel phase di^2 kappa / 2 - (m - msh) di delta turns (di = i - c),
// then row passes over a real FP32 matrix [rows][stride] loaded as the B operand.
fzp_status dense_zoom_build(Plan& P, int64_t ncols, int64_t c, double kappa, double delta);
fzp_status dense_zoom_rows(Plan& P, const float* src, int64_t rows, int64_t stride, cudaStream_t stream);
fzp_status column_pass(Plan& P, int64_t j0, int64_t rows, RowKind kind, cudaStream_t stream);
bool column_pass_tc_applies(const Plan& P);
// Aperture rows [a, b) (clipped to the disc's) into the ROI accumulator (zeroed
// first), chunk by chunk: row pass and column pass of every mask pass.  *sym:
// the field is the accumulator plus its transpose.
fzp_status propagate_rows(Plan& P, int64_t a, int64_t b, bool* sym, cudaStream_t stream);
// The accumulator to the caller's field (interpolation, output chirp, prefactor).
fzp_status finish_field(Plan& P, void* d_field, int accumulate, bool sym, cudaStream_t stream);
// Form (b) on nodes (nodes.cu).
void nodes_choose(Plan& P);
bool nodes_two_masks(const Plan& P);  // both real masks of a complex transmission in one row pass
fzp_status nodes_layout(Plan& P, FormSizes* out);
fzp_status nodes_upload(Plan& P);
fzp_status nodes_fill(Plan& P, cudaStream_t s);
fzp_status nodes_rows(Plan& P, int64_t j0, int64_t rows, bool octant, cudaStream_t s);
fzp_status nodes_epilogue(Plan& P, void* d_field, int accumulate, bool sym, cudaStream_t s);
fzp_status nodes_mask(Plan& P, int64_t j0, int64_t rows, uint8_t* out, cudaStream_t s);
// Contraction of a real FP32 matrix [rows][stride] (lower: a symmetric one, its
// lower triangle) of kblocks x 32 columns with node columns: row pass into the
// rows part * 2 ns .. of C1.  Images from a table, or of the SA-CZT's zoom kernel.
fzp_status nodes_table_images(Plan& P, const void* E, int64_t ncols, int64_t stride, int64_t kblocks, void* A);
fzp_status nodes_loaded_rows(Plan& P, const float* src, int64_t rows, int64_t stride, int64_t kblocks, const void* A,
                             int* sched, int part, bool lower, cudaStream_t s);
fzp_status nodes_zoom_images(Plan& P, int64_t ncols, int64_t kblocks, void* A);
// The column pass of that contraction: both parts, kernel columns from E, or of
// the zoom kernel of the distance z (lz = lambda z) over `rows` padded rows.
fzp_status column_pass_zoom(Plan& P, int64_t rows, double lz, cudaStream_t s);
fzp_status column_pass_table(Plan& P, const void* E, int64_t rows, int64_t estride, cudaStream_t s);
fzp_status column_pass_tc(Plan& P, int64_t j0, int64_t rows, cudaStream_t stream);
// The same with the pass's field weighted by (wr + i wi).
fzp_status column_pass_tc_w(Plan& P, int64_t j0, int64_t rows, double wr, double wi, cudaStream_t stream);
fzp_status epilogue(Plan& P, void* d_field, int accumulate, cudaStream_t stream);
// The epilogue with the Fresnel part's distance z in the output chirp and the
// amplitude dx^2 / (lambda z) (the phase e^{ikf} keeps the focal length).
fzp_status epilogue_z(Plan& P, void* d_field, int accumulate, double z, cudaStream_t stream);
fzp_status saczt_layout(Plan& P);                      // P, fit, z_F (host)
fzp_status saczt_build(Plan& P);                       // allocate and fill its tables
fzp_status saczt_propagate(Plan& P, int64_t j0, int64_t j1, cudaStream_t stream);  // into d_Uacc
bool saczt_folds(const Plan& P, int64_t j0, int64_t j1);  // the range is the whole aperture and the plan has nodes
fzp_status saczt_mask(Plan& P, int64_t j0, int64_t rows, uint8_t* out, cudaStream_t stream);
fzp_status intensity(Plan& P, const void* d_field, void* d_I, cudaStream_t stream);
fzp_status metrics(Plan& P, const void* d_field, cudaStream_t stream, fzp_metrics_t* out);
fzp_status bluestein_mask(Plan& P, int64_t j0, int64_t rows, uint8_t* out, cudaStream_t stream);
fzp_status dense_mask(Plan& P, int64_t j0, int64_t rows, uint8_t* out, cudaStream_t stream);

// Launch that may overlap the end of the stream's previous kernel (tc_ptx.cuh:
// the kernel waits for it itself).  The surrogate's chain of nine launches is
// bound by the gaps between them: gradients of a batch of 256, 130 -> 111 us.
// (The node form's chain got slower, 78 -> 84 us on the 2 mm plate: its blocks
// take the place of the running kernel's.)
template <typename... P, typename... A>
cudaError_t launch_after(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

// Row index into the C1 layout: kernel row tile t = m / 64 holds the real parts
// of m = 64t..64t+63 in rows [0,64) and the imaginary parts in rows [64,128).
__host__ __device__ __forceinline__ int c1_row_re(int m) { return (m >> 6) * 128 + (m & 63); }
__host__ __device__ __forceinline__ int c1_row_im(int m) { return (m >> 6) * 128 + 64 + (m & 63); }

}  // namespace fzp

// The opaque handle of the C ABI is the plan itself.
struct fzp_plan_s : public fzp::Plan {};

namespace fzp {
// Host part of fzp_plan (validation, grids, zone-rule limits; no CUDA call):
// fills P and returns the disc limit s_R and the last zone step.
fzp_status plan_host(const fzp_params* params, Plan& P, int64_t* sR, int64_t* zmax);
fzp_status autotune(const fzp_params* in, fzp_params* chosen, fzp_plan_t* keep);
}
