// bluestein.cu -- form (a): row chirp-z transform by Bluestein's identity
// (Sec. 2.6; Eq. 9-10; Fig. 2 Stage 3; Fig. 18 Stage 3 "row Bluestein at fixed
// length nfft"), with FFTs written here.
//
// For aperture row j the row transform is
//   C[j, m] = sum_i x_i K[m, i],  x_i = T[j, i] e^{i phi[j, i]},
//   K[m, i] = exp(2 pi i theta(m, i)),  theta = di^2 kappa/2 - (m - msh) di delta
// (msh = -x0/p: M/2 for the ROI centred on the focus).
// With m i = (m^2 + i^2 - (m - i)^2) / 2 (Bluestein):
//   theta(m, i) = pre(i) + post(m) + delta (m - i)^2 / 2,
//   pre(i)  = di^2 kappa/2 - delta i^2/2 + delta msh i,
//   post(m) = -delta m^2/2 + delta m c - delta msh c,
// so C[j, .] = e^{2 pi i post} .* (y * h)[0..M) with y_i = x_i e^{2 pi i pre(i)} and
// the chirp h_k = e^{i pi delta k^2}, k in (-N, M): one linear convolution of
// length >= N + M - 1, done as FFT_L, pointwise product with FFT_L(h), IFFT_L.
//
// Large L is split four-step (Bailey, ref. [24] of the paper), L = L1 * L2,
// n = L2 n1 + n2, k = k1 + L1 k2:
//   pass F1 (L1 > 1): for each column n2 an L1-point FFT over n1, times e^{-2 pi i n2 k1 / L}
//   pass F2         : for each row k1 an L2-point FFT over n2 -> Y[k1 + L1 k2],
//                     times H, L2-point inverse FFT; only m < M outputs kept,
//                     times e^{+2 pi i k1 m / L}
//   pass F3 (L1 > 1): sum over k1, times e^{2 pi i post(m)} / L -> row intermediate.
// The mask and the input chirp are generated inside F1 (or F2 when L1 = 1):
// the aperture is never stored.
//
// FP32 default (fzp_params.conv): the same convolution partitioned into
// 4096-point blocks, each row on chip from its mask to its M outputs (k_seg,
// below), its columns first spread over a coarse grid where the outputs' band is
// that narrow (k_dec); the four-step passes above remain the FP64 path and the
// single-convolution FP32 option.
#include <algorithm>
#include <cmath>

#include "fzp_internal.cuh"
#include "membrane.cuh"
#include "zone_phase.cuh"

namespace fzp {
namespace {

template <typename R> struct Traits;
template <> struct Traits<float> { static constexpr int L2MAX = 4096; };  // radix-16 pass kernel
template <> struct Traits<double> { static constexpr int L2MAX = 4096; };

__host__ __device__ inline int ilog2(int64_t v) { int r = 0; while ((1ll << r) < v) ++r; return r; }

__device__ __forceinline__ int brev(int v, int bits) { return (int)(__brev((unsigned)v) >> (32 - bits)); }

template <typename C> __device__ __forceinline__ C conjc(C a) { a.y = -a.y; return a; }

// Batched in-place radix-2 DIT: `batch` transforms of length n = 2^logn, column
// c at x + c * colstride; input in bit-reversed order, output natural; forward sign.
// tw[t] = e^{-2 pi i t / twN}.
template <typename C>
__device__ void dit(C* x, int logn, int batch, const C* __restrict__ tw, int twN, int colstride) {
  const int n = 1 << logn, nb = (n >> 1) * batch;
  for (int s = 1; s <= logn; ++s) {
    const int half = 1 << (s - 1);
    const int stride = twN >> s;
    for (int t = threadIdx.x; t < nb; t += blockDim.x) {
      const int col = t >> (logn - 1), b = t & ((n >> 1) - 1);
      const int k = b & (half - 1);
      const int i0 = col * colstride + ((b >> (s - 1)) << s) + k, i1 = i0 + half;
      const C w = tw[k * stride];
      const C a = x[i0], v = cmul(x[i1], w);
      x[i0] = cadd(a, v);
      x[i1] = csub(a, v);
    }
    __syncthreads();
  }
}

// The same transform with two radix-2 stages per pass (radix 2^2): each work
// item takes the four elements k, k + h, k + 2h, k + 3h of a group of 4h
// (h = 2^(s-1)), applies stage s to the pairs (0,1), (2,3) and stage s + 1 to
// (0,2), (1,3) in registers; a single radix-2 stage finishes odd lengths.
// tws[t] = e^{-2 pi i t / n} for t < n / 2, in shared memory.
template <typename C>
__device__ void dit22(C* x, int logn, int batch, const C* tws, int colstride) {
  const int n = 1 << logn;
  int s = 1;
  for (; s + 1 <= logn; s += 2) {
    const int h = 1 << (s - 1);
    const int items = (n >> 2) * batch;
    for (int t = threadIdx.x; t < items; t += blockDim.x) {
      const int col = t >> (logn - 2), g = t & ((n >> 2) - 1);
      const int k = g & (h - 1);
      const int i0 = col * colstride + ((g >> (s - 1)) << (s + 1)) + k;
      const C w1 = tws[k << (logn - s)];
      const C w2 = tws[k << (logn - s - 1)], w3 = tws[(k + h) << (logn - s - 1)];
      C a0 = x[i0], a1 = x[i0 + h], a2 = x[i0 + 2 * h], a3 = x[i0 + 3 * h];
      const C v1 = cmul(a1, w1), v3 = cmul(a3, w1);
      const C b0 = cadd(a0, v1), b1 = csub(a0, v1), b2 = cadd(a2, v3), b3 = csub(a2, v3);
      const C u2 = cmul(b2, w2), u3 = cmul(b3, w3);
      x[i0] = cadd(b0, u2);
      x[i0 + 2 * h] = csub(b0, u2);
      x[i0 + h] = cadd(b1, u3);
      x[i0 + 3 * h] = csub(b1, u3);
    }
    __syncthreads();
  }
  if (s == logn) {  // one radix-2 stage left
    const int h = 1 << (s - 1);
    const int items = (n >> 1) * batch;
    for (int t = threadIdx.x; t < items; t += blockDim.x) {
      const int col = t >> (logn - 1), b = t & ((n >> 1) - 1);
      const int k = b & (h - 1);
      const int i0 = col * colstride + ((b >> (s - 1)) << s) + k;
      const C w = tws[k << (logn - s)];
      const C a0 = x[i0], v = cmul(x[i0 + h], w);
      x[i0] = cadd(a0, v);
      x[i0 + h] = csub(a0, v);
    }
    __syncthreads();
  }
}

// In-place radix-2 DIF, natural input, bit-reversed output, inverse sign (no 1/n).
template <typename C>
__device__ void dif_inverse(C* x, int logn, const C* __restrict__ tw, int twN) {
  const int n = 1 << logn, nb = n >> 1;
  for (int s = logn; s >= 1; --s) {
    const int half = 1 << (s - 1);
    const int stride = twN >> s;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
      const int k = b & (half - 1);
      const int i0 = ((b >> (s - 1)) << s) + k, i1 = i0 + half;
      const C w = conjc(tw[k * stride]);
      const C a = x[i0], v = x[i1];
      x[i0] = cadd(a, v);
      x[i1] = cmul(csub(a, v), w);
    }
    __syncthreads();
  }
}

struct RowArgs {
  MaskGeom mg;
  int64_t N, L, L1, L2;
  int logL1, logL2, M;
  int64_t j0;        // first aperture row of this launch
  int64_t rows;      // rows in this launch
  int B, logB;       // columns per F1 block (a power of two)
  int has_deform;
  fzp_deform def;
  double dx, R, inv_lambda;
  // the deformation phase in turns, 2 w / lambda, as FP32 coefficients:
  //   amp2 sin(2 pi (di kx + dj ky)) (1 - tq (di^2 + dj^2)) + sum_k h2_k exp(-q_k d_k^2),
  //   d_k = (di - pi_k) nx_k + (dj - pj_k) ny_k  (sample units; (pi_k, pj_k) on the crease)
  DeformCoef df;
  const void* pre;   // N
  const void* H;     // [L1][L2]
  void* Z;           // [rows][L1][L2]
  void* G;           // [rows][L1][M]
  const void* post;  // M, includes 1/L
  const void* tw;    // twN entries: e^{-2 pi i t / twN}
  const void* twL;   // 4096 entries: e^{-2 pi i t / L}
  int twN;
  void* C1;          // [2M][c1_stride]
  int64_t c1_stride; // row length of C1
  int64_t c1_j0;     // aperture row of C1 column 0
  const void* vin;   // input sequence for the table-building mode (length L)
  int S;             // partitioned convolution: columns per block
  int64_t nseg;      // partitioned convolution: blocks per row (spectra in H)
  int64_t col0;      // first column of the transforms' input (the axis when `half`)
  PhaseRule ph;      // partitioned convolution: the zone phase of the mask walk
  int half;          // even output grid: columns from the axis on, outputs x and -x added
  int octant;        // columns up to the row's distance from the axis only, the last one halved
  // decimated rows: chirp turns per squared column (units of 2^-64; Kc2: the next 32
  // bits) and per column (2^-64), the second difference (2^-32), the sums' weights
  // on the grid points
  uint64_t Kc, Kl;
  uint32_t Kc2, cc2;
  float2 T[2][DTAPS][4];  // (each weight twice)
};

// Aperture transmission of sample (j, i): T e^{i phi}, optional deformation.
template <typename R>
__device__ __forceinline__ typename Cplx<R>::T aperture(const RowArgs& a, int64_t j, int64_t i) {
  typename Cplx<R>::T v;
  v.x = 0; v.y = 0;
  if (i >= a.N) return v;
  const int64_t dj = j - a.mg.c, di = i - a.mg.c, s = dj * dj + di * di;
  if (s > a.mg.sR) return v;
  const int64_t z = zone_of(s, a.mg);
  if (a.mg.levels >= 2) {
    // L-level phase plate: e^{-2 pi i q / L}, q = zone mod L (Fig. 18 Stage 3)
    // fewer than 2^24 zone steps (a plan limit): a 32-bit remainder
    const int q = (int)((uint32_t)z % (uint32_t)a.mg.levels);
    if (sizeof(R) == 4) {
      // FP32 form: -q / L turns lies in (-1, 0], so FP32 carries it to within
      // an ulp without the FP64 reduction
      float sn, cs;
      sincospif(-2.0f * (float)q / (float)a.mg.levels, &sn, &cs);
      v.x = cs;
      v.y = sn;
    } else {
      v = cis_turns<R>(-(double)q / (double)a.mg.levels);
    }
    if (!a.has_deform) return v;
  } else {
    if (((z ^ a.mg.centre_open) & 1) == 0) return v;  // binary amplitude: odd zones open (even: positive-centred)
    v.x = 1;
    if (!a.has_deform) return v;
  }
  if (sizeof(R) == 4) {
    // FP32 form: the phase is at most about a turn, so FP32 coefficients
    // (relative error ~1e-7 of it) are far inside the form's tolerance
    const float fi = (float)di, fj = (float)dj;
    // turns of the wrinkle: |di| < 2^20 and kxh a multiple of 2^-14 with few
    // significant bits, so di kxh is exact and its integer part drops exactly
    const float th = fi * a.df.kxh + fj * a.df.kyh;
    const float tt = (th - rintf(th)) + (fi * a.df.kxl + fj * a.df.kyl);
    float wz = a.df.amp2 * sinpif(2.0f * (tt - rintf(tt))) * (1.0f - a.df.tq * (fi * fi + fj * fj));
    for (int k = 0; k < a.df.n; ++k) {
      const float d = (fi - a.df.pi_[k]) * a.df.nx[k] + (fj - a.df.pj[k]) * a.df.ny[k];
      wz += a.df.h2[k] * __expf(-a.df.q[k] * d * d);
    }
    // wz - rint(wz) is exact in FP32, so the reduction adds nothing to wz's
    // own rounding (the FP64 reduction of the same FP32 value gave the same)
    float sn, cs;
    sincospif(2.0f * (wz - rintf(wz)), &sn, &cs);
    typename Cplx<R>::T e;
    e.x = cs;
    e.y = sn;
    return cmul(v, e);
  }
  const double u = (double)(i - a.mg.c) * a.dx, w = (double)(j - a.mg.c) * a.dx;
  const fzp_deform& d = a.def;
  const double tt = (u * cos(d.theta) + w * sin(d.theta)) / d.period;  // turns
  const double r2 = (u * u + w * w) / (a.R * a.R);
  double wz = d.amp * sinpi(2.0 * frac_turns(tt)) * (1.0 - d.taper * r2);
  for (int k = 0; k < d.n_ridges; ++k) {
    const double dist = (u - d.ridge_px[k]) * (-sin(d.ridge_alpha[k])) + (w - d.ridge_py[k]) * cos(d.ridge_alpha[k]);
    const double sg = d.ridge_width[k] / (2.0 * sqrt(2.0 * log(2.0)));
    wz += d.ridge_h[k] * exp(-dist * dist / (2.0 * sg * sg));
  }
  return cmul(v, cis_turns<R>(2.0 * wz * a.inv_lambda));  // phi / (2 pi) = 2 w / lambda
}

// Input n of a row's convolution: the transmission of column col0 + n times the
// chirp; with the columns from the axis on, the axis itself (which the two
// added outputs both count) at half weight.
template <typename R>
__device__ __forceinline__ typename Cplx<R>::T row_input(const RowArgs& a, int64_t j, int64_t n,
                                                         const typename Cplx<R>::T* pre) {
  typename Cplx<R>::T x = aperture<R>(a, j, n + a.col0);
  if (x.x != 0 || x.y != 0) x = cmul(x, pre[n]);
  if (a.half && n == 0) {
    x.x *= (R)0.5;
    x.y *= (R)0.5;
  }
  return x;
}

// e^{sign 2 pi i t / L} for 0 <= t < L = L1 * L2 from two tables:
// t = th * 4096 + tl, W_L^t = W_{L1}^{th} W_L^{tl}, W_{L1}^{th} = tw[th * (twN / L1)].
template <typename R>
__device__ __forceinline__ typename Cplx<R>::T twiddle_L(const RowArgs& a, int64_t t, bool conj) {
  using C = typename Cplx<R>::T;
  if (a.L <= 4096) {
    C w = reinterpret_cast<const C*>(a.twL)[t];
    if (conj) w.y = -w.y;
    return w;
  }
  const int64_t th = t >> 12, tl = t & 4095;
  C w1 = reinterpret_cast<const C*>(a.tw)[th * (a.twN / a.L1)];
  C w2 = reinterpret_cast<const C*>(a.twL)[tl];
  C w = cmul(w1, w2);
  if (conj) w.y = -w.y;
  return w;
}

// mode 0: generate y = aperture * pre; mode 1: read the table input `vin`.
template <typename R>
__global__ void __launch_bounds__(256) k_f1(RowArgs a, int mode) {
  using C = typename Cplx<R>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sm = reinterpret_cast<C*>(smem_raw);
  const int B = a.B;
  const int64_t r = blockIdx.y;
  const int64_t j = a.j0 + r;
  const int64_t n2_0 = (int64_t)blockIdx.x * B;
  const int L1 = (int)a.L1;
  const C* pre = reinterpret_cast<const C*>(a.pre);
  const C* vin = reinterpret_cast<const C*>(a.vin);
  C* tws = sm + (L1 + 1) * B;  // L1 / 2 twiddles of the column FFT
  for (int t = threadIdx.x; t < (L1 >> 1); t += blockDim.x)
    tws[t] = reinterpret_cast<const C*>(a.tw)[t * (a.twN / L1)];
  // load, bit-reversed within each column
  for (int t = threadIdx.x; t < L1 * B; t += blockDim.x) {
    const int n1 = t >> a.logB, b = t & (B - 1);
    const int64_t n = (int64_t)n1 * a.L2 + n2_0 + b;
    C x;
    if (mode == 0) x = row_input<R>(a, j, n, pre);
    else x = vin[n];
    sm[b * (L1 + 1) + brev(n1, a.logL1)] = x;  // odd column stride: no bank conflicts across columns
  }
  __syncthreads();
  dit22(sm, a.logL1, B, tws, L1 + 1);
  C* Z = reinterpret_cast<C*>(a.Z) + r * a.L;
  for (int t = threadIdx.x; t < L1 * B; t += blockDim.x) {
    const int k1 = t >> a.logB, b = t & (B - 1);
    const int64_t n2 = n2_0 + b;
    const C w = twiddle_L<R>(a, n2 * k1, false);
    Z[(int64_t)k1 * a.L2 + n2] = cmul(sm[b * (L1 + 1) + k1], w);
  }
}

// mode 0: full row transform; mode 1: forward FFT only, result -> Z as [k1][k2].
template <typename R>
__global__ void __launch_bounds__(512) k_f2(RowArgs a, int mode) {
  using C = typename Cplx<R>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sm = reinterpret_cast<C*>(smem_raw);
  const int64_t k1 = blockIdx.x;
  const int64_t r = blockIdx.y;
  const int64_t j = a.j0 + r;
  const int L2 = (int)a.L2;
  const C* tw = reinterpret_cast<const C*>(a.tw);
  const C* pre = reinterpret_cast<const C*>(a.pre);
  if (a.L1 == 1) {
    const C* vin = reinterpret_cast<const C*>(a.vin);
    for (int n = threadIdx.x; n < L2; n += blockDim.x) {
      C x;
      if (mode == 0) x = row_input<R>(a, j, n, pre);
      else x = vin[n];
      sm[brev(n, a.logL2)] = x;
    }
  } else {
    const C* Z = reinterpret_cast<const C*>(a.Z) + r * a.L + k1 * a.L2;
    for (int n = threadIdx.x; n < L2; n += blockDim.x) sm[brev(n, a.logL2)] = Z[n];
  }
  __syncthreads();
  dit(sm, a.logL2, 1, tw, a.twN, (int)a.L2);
  if (mode == 1) {
    C* out = reinterpret_cast<C*>(a.Z) + r * a.L + k1 * a.L2;
    for (int k = threadIdx.x; k < L2; k += blockDim.x) out[k] = sm[k];
    return;
  }
  const C* H = reinterpret_cast<const C*>(a.H) + k1 * a.L2;
  for (int k = threadIdx.x; k < L2; k += blockDim.x) sm[k] = cmul(sm[k], H[k]);
  __syncthreads();
  dif_inverse(sm, a.logL2, tw, a.twN);
  if (a.L1 == 1) {
    // finalize directly: C = post(m) * z[m]  (post includes 1/L)
    const C* post = reinterpret_cast<const C*>(a.post);
    R* C1 = reinterpret_cast<R*>(a.C1);
    const int64_t jl = j - a.c1_j0;
    const int hm = (a.M - 1) / 2;
    for (int m = threadIdx.x; m < (a.half ? hm + 1 : a.M); m += blockDim.x) {
      const int mp = a.half ? hm + m : m;
      C v = cmul(sm[brev(mp, a.logL2)], post[mp]);
      if (a.half) v = cadd(v, cmul(sm[brev(hm - m, a.logL2)], post[hm - m]));
      C1[(int64_t)c1_row_re(m) * a.c1_stride + jl] = v.x;
      C1[(int64_t)c1_row_im(m) * a.c1_stride + jl] = v.y;
    }
    return;
  }
  C* G = reinterpret_cast<C*>(a.G) + (r * a.L1 + k1) * a.M;
  for (int m = threadIdx.x; m < a.M; m += blockDim.x) {
    G[m] = cmul(sm[brev(m, a.logL2)], twiddle_L<R>(a, (k1 * m) & (a.L - 1), true));
  }
}

// ---------------------------------------------------------------- FP32 pass F2, radix 16
constexpr int RL = 4096;  // inner FFT length of the FP32 four-step split

__device__ __forceinline__ void dft4(float2& a0, float2& a1, float2& a2, float2& a3, bool inv) {
  const float2 s02 = make_float2(a0.x + a2.x, a0.y + a2.y), d02 = make_float2(a0.x - a2.x, a0.y - a2.y);
  const float2 s13 = make_float2(a1.x + a3.x, a1.y + a3.y), d13 = make_float2(a1.x - a3.x, a1.y - a3.y);
  const float2 t = inv ? make_float2(-d13.y, d13.x) : make_float2(d13.y, -d13.x);  // (+/-i) d13
  a0 = make_float2(s02.x + s13.x, s02.y + s13.y);
  a2 = make_float2(s02.x - s13.x, s02.y - s13.y);
  a1 = make_float2(d02.x + t.x, d02.y + t.y);
  a3 = make_float2(d02.x - t.x, d02.y - t.y);
}

// ---------------------------------------------------------------- FP32 pass F2, radix 8
// L2 = 4096 = 8^4 points, 512 threads x 8 values in registers, Stockham
// order (pass s, Ns = 8^s: x_r = in[j + 512 r] times W_{8 Ns}^{r k}, k = j mod
// Ns, 8-point DFT, y_q -> out[(j / Ns) 8 Ns + q Ns + k]).  After the forward
// passes thread j holds Y[j + 512 q], the layout the inverse's first pass
// reads, so the product with H needs no exchange; the inverse's last pass
// (Ns = 512) evaluates only the outputs q < ceil(M / 512) it keeps.  Shared
// memory (padded one element per 8 against bank conflicts) carries the three
// exchanges of each transform.  Twiddles: W^k, W^{2k}, W^{4k} from the table,
// the other four by products.
constexpr int R8T = 512;
__device__ __forceinline__ int pidx8(int i) { return i + (i >> 3); }

__device__ __forceinline__ void dft8(float2 (&v)[8], bool inv) {
  // radix 2 x 4: two 4-point DFTs on the even and odd inputs, then W_8^q
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4(e0, e1, e2, e3, inv);
  dft4(o0, o1, o2, o3, inv);
  const float h = 0.70710678118654752f;
  // o_q times W_8^{q} (forward e^{-2 pi i q / 8}; inverse conjugate)
  const float sg = inv ? 1.0f : -1.0f;
  float2 t1 = make_float2(h * (o1.x - sg * o1.y), h * (o1.y + sg * o1.x));  // W^1
  float2 t2 = make_float2(-sg * o2.y, sg * o2.x);                           // W^2 = -+i
  float2 t3 = make_float2(h * (-o3.x - sg * o3.y), h * (-o3.y + sg * o3.x)); // W^3
  v[0] = make_float2(e0.x + o0.x, e0.y + o0.y);
  v[4] = make_float2(e0.x - o0.x, e0.y - o0.y);
  v[1] = make_float2(e1.x + t1.x, e1.y + t1.y);
  v[5] = make_float2(e1.x - t1.x, e1.y - t1.y);
  v[2] = make_float2(e2.x + t2.x, e2.y + t2.y);
  v[6] = make_float2(e2.x - t2.x, e2.y - t2.y);
  v[3] = make_float2(e3.x + t3.x, e3.y + t3.y);
  v[7] = make_float2(e3.x - t3.x, e3.y - t3.y);
}

// v[r] *= W_{8 Ns}^{r k} (forward) or its conjugate; tw[t] = e^{-2 pi i t / 4096}.
__device__ __forceinline__ void twiddle8(float2 (&v)[8], int k, int step, const float2* __restrict__ tw, bool inv) {
  if (k == 0) return;
  float2 w1 = __ldg(tw + k * step), w2 = __ldg(tw + 2 * k * step), w4 = __ldg(tw + 4 * k * step);
  if (inv) { w1.y = -w1.y; w2.y = -w2.y; w4.y = -w4.y; }
  const float2 w3 = cmul(w1, w2), w5 = cmul(w1, w4), w6 = cmul(w2, w4), w7 = cmul(w3, w4);
  v[1] = cmul(v[1], w1); v[2] = cmul(v[2], w2); v[3] = cmul(v[3], w3); v[4] = cmul(v[4], w4);
  v[5] = cmul(v[5], w5); v[6] = cmul(v[6], w6); v[7] = cmul(v[7], w7);
}

// One Stockham pass with the exchange that feeds the next: twiddle, DFT,
// scatter to shared memory, gather the next pass's inputs.
__device__ __forceinline__ void r8_pass(float2 (&v)[8], float2* sm, int Ns, const float2* __restrict__ tw, bool inv) {
  const int j = threadIdx.x;
  const int k = j & (Ns - 1);
  twiddle8(v, k, 512 / Ns, tw, inv);
  dft8(v, inv);
  const int base = (j / Ns) * 8 * Ns + k;
#pragma unroll
  for (int q = 0; q < 8; ++q) sm[pidx8(base + q * Ns)] = v[q];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = sm[pidx8(j + R8T * q)];
  __syncthreads();
}

// mode 0: row transform; mode 1: forward FFT only, natural order -> Z row (table build).
__global__ void __launch_bounds__(R8T, 2) k_f2_r8(RowArgs a, int mode) {
  __shared__ float2 sm[RL + RL / 8];
  const int j = threadIdx.x;
  const int64_t k1 = blockIdx.x, r = blockIdx.y, row = a.j0 + r;
  const float2* tw = reinterpret_cast<const float2*>(a.tw);
  float2 v[8];
  if (a.L1 == 1) {
    const float2* pre = reinterpret_cast<const float2*>(a.pre);
    const float2* vin = reinterpret_cast<const float2*>(a.vin);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int n = j + R8T * q;
      if (mode == 0) {
        float2 x = aperture<float>(a, row, n);
        if (x.x != 0.f || x.y != 0.f) x = cmul(x, pre[n]);
        v[q] = x;
      } else {
        v[q] = vin[n];
      }
    }
  } else {
    const float2* Z = reinterpret_cast<const float2*>(a.Z) + r * a.L + k1 * RL;
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = Z[j + R8T * q];
  }
  // forward: passes Ns = 1, 8, 64 with exchanges, then Ns = 512 in registers
  r8_pass(v, sm, 1, tw, false);
  r8_pass(v, sm, 8, tw, false);
  r8_pass(v, sm, 64, tw, false);
  twiddle8(v, j, 1, tw, false);
  dft8(v, false);  // thread j now holds Y[j + 512 q] in v[q]
  if (mode == 1) {
    float2* out = reinterpret_cast<float2*>(a.Z) + r * a.L + k1 * RL;
#pragma unroll
    for (int q = 0; q < 8; ++q) out[q * R8T + j] = v[q];
    return;
  }
  const float2* H = reinterpret_cast<const float2*>(a.H) + k1 * RL;
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = cmul(v[q], __ldg(H + q * R8T + j));
  // inverse: passes Ns = 1, 8, 64, then the kept outputs of Ns = 512
  r8_pass(v, sm, 1, tw, true);
  r8_pass(v, sm, 8, tw, true);
  r8_pass(v, sm, 64, tw, true);
  twiddle8(v, j, 1, tw, true);
  // outputs m = q * 512 + j < M: y_q = sum_r v_r W_8^{-r q} (inverse sign)
  const int nq = (a.M + R8T - 1) / R8T;
  float2 y[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    y[q] = make_float2(0.f, 0.f);
    if (q < nq) {
#pragma unroll
      for (int rr = 0; rr < 8; ++rr) {
        float sn, cs;
        // W_8^{-r q} = e^{+2 pi i r q / 8}: exact for r q mod 8 in {0, 2, 4, 6}; 1/sqrt(2) otherwise
        const int t = (rr * q) & 7;
        const float h = 0.70710678118654752f;
        const float ct[8] = {1.f, h, 0.f, -h, -1.f, -h, 0.f, h};
        const float st[8] = {0.f, h, 1.f, h, 0.f, -h, -1.f, -h};
        cs = ct[t];
        sn = st[t];
        y[q].x += v[rr].x * cs - v[rr].y * sn;
        y[q].y += v[rr].x * sn + v[rr].y * cs;
      }
    }
  }
  if (a.L1 == 1) {
    const float2* post = reinterpret_cast<const float2*>(a.post);
    float* C1 = reinterpret_cast<float*>(a.C1);
    const int64_t jl = row - a.c1_j0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int m = q * R8T + j;
      if (q < nq && m < a.M) {
        const float2 z = cmul(y[q], post[m]);
        C1[(int64_t)c1_row_re(m) * a.c1_stride + jl] = z.x;
        C1[(int64_t)c1_row_im(m) * a.c1_stride + jl] = z.y;
      }
    }
    return;
  }
  float2* G = reinterpret_cast<float2*>(a.G) + (r * a.L1 + k1) * a.M;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int m = q * R8T + j;
    if (q < nq && m < a.M) G[m] = cmul(y[q], twiddle_L<float>(a, (k1 * m) & (a.L - 1), true));
  }
}

// Sum over k1; tile of 32 rows x 32 outputs; writes C1 coalesced along rows.
template <typename R>
__global__ void __launch_bounds__(256) k_f3(RowArgs a) {
  using C = typename Cplx<R>::T;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 8 warps
  const int m0 = blockIdx.x * 32;
  const int64_t r0 = (int64_t)blockIdx.y * 32;
  const int hm = (a.M - 1) / 2, nout = a.half ? hm + 1 : a.M;
  __shared__ C tile[32][33];
  const C* G = reinterpret_cast<const C*>(a.G);
  const C* post = reinterpret_cast<const C*>(a.post);
  auto out = [&](int64_t r, int m) {
    C acc;
    acc.x = 0; acc.y = 0;
    for (int64_t k1 = 0; k1 < a.L1; ++k1) acc = cadd(acc, G[(r * a.L1 + k1) * a.M + m]);
    return cmul(acc, post[m]);
  };
  for (int rr = ty; rr < 32; rr += 8) {
    const int64_t r = r0 + rr;
    const int m = m0 + tx;
    if (r >= a.rows || m >= nout) continue;
    tile[rr][tx] = a.half ? cadd(out(r, hm + m), out(r, hm - m)) : out(r, m);
  }
  __syncthreads();
  R* C1 = reinterpret_cast<R*>(a.C1);
  for (int mm = ty; mm < 32; mm += 8) {
    const int64_t r = r0 + tx;
    const int m = m0 + mm;
    if (r >= a.rows || m >= nout) continue;
    const int64_t jl = a.j0 + r - a.c1_j0;
    const C v = tile[tx][mm];
    C1[(int64_t)c1_row_re(m) * a.c1_stride + jl] = v.x;
    C1[(int64_t)c1_row_im(m) * a.c1_stride + jl] = v.y;
  }
}

// ---------------------------------------------------------------------------
// Partitioned convolution (FP32).  The row's convolution (y * h)[m], m < M, is
// a sum over blocks of S input columns, i in [i_s, i_s + S), i_s = s S.  With
// P = 4096 >= S + M - 1 a block's share is one P-point circular convolution of
// the zero-padded block with the chirp piece
//   g_s[q] = h_{q - i_s} (q < M),  g_s[q] = h_{q - P - i_s} (P - S < q < P),
// read at q = m < M: the two ranges hold every lag m - i the block needs and
// do not overlap.  The transform is linear, so a row needs one inverse
// transform of sum_s FFT_P(y_s) .* G_s, G_s = FFT_P(g_s) precomputed per block
// (the same for every row); blocks that miss the row's disc chord are skipped.
// A row's working set (the block, the spectrum sum, the transposes) stays in
// registers and shared memory.
//
// The P-point FFT: 256 threads, thread t holding elements t + 256 r, r < 16;
// P = 16 * 16 * 16 as three in-register 16-point DFTs with two shared-memory
// transposes (index t = a + 16 b + 256 r, frequency k = k0 + 16 c + 256 d):
//   pass A: over r -> k0, times e^{-2 pi i t k0 / P}
//   pass B: thread (a, k0) over b -> c, times e^{-2 pi i a c / 256}
//   pass C: thread (k0, c) over a -> d; thread t = k0 + 16 c then holds
//           X[t + 256 d], the same distribution as its input.
// ---------------------------------------------------------------------------
constexpr int SP = 4096;          // partition transform length
constexpr int STH = 256;          // threads per block
constexpr int SB0 = 256 * 17;     // transpose buffer A->B: [t][k0], row pitch 17
constexpr int SB1 = 16 * 273;     // transpose buffer B->C: [k0][c][a], pitches 273 and 17
constexpr int SBUF = SB1 > SB0 ? SB1 : SB0;
constexpr int NO_LEVEL = 64;      // level byte of a column outside the disc: phasor 0
constexpr size_t SEG_SMEM = sizeof(float2) * (2 * SBUF + 15 * 256 + 256 + NO_LEVEL + 2) + SP;
// row kernels: binary plate (chunk bits), phase plate (chunk zone steps),
// deformed binary plate (chunk bits and the membrane phasor, walked or, with
// DeformCoef::direct, by column), general transmission (a deformed phase plate)
enum { SEG_FLAT = 0, SEG_LEVELS = 1, SEG_MEMBRANE = 2, SEG_GENERAL = 3, SEG_DIRECT = 4 };
constexpr bool seg_membrane(int mode) { return mode == SEG_MEMBRANE || mode == SEG_DIRECT; }

// A membrane's phase (turns, 2 w / lambda) on the 16 columns from di0, CLOSED
// where the plate is (bits: open columns), to shared memory at a pitch of one.
constexpr float CLOSED = 1e30f;
template <typename Walk>
__device__ __forceinline__ void membrane_chunk(Walk walk, uint32_t bits, float* o) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float w = walk.next();
    o[k] = ((bits >> k) & 1u) ? w : CLOSED;
  }
}

// v e^{-2 pi i K / 16}
template <int K, typename C>
__device__ __forceinline__ C w16mul(C v) {
  using R = decltype(C::x);
  constexpr R C1 = (R)0.92387953251128675613, S1 = (R)0.38268343236508977173, R2 = (R)0.70710678118654752440;
  C r;
  if constexpr (K == 0) {
    r = v;
  } else if constexpr (K == 4) {
    r.x = v.y;
    r.y = -v.x;
  } else if constexpr (K == 2) {
    r.x = R2 * (v.x + v.y);
    r.y = R2 * (v.y - v.x);
  } else if constexpr (K == 6) {
    r.x = R2 * (v.y - v.x);
    r.y = -R2 * (v.x + v.y);
  } else {
    constexpr R wr = K == 1 ? C1 : (K == 3 ? S1 : -C1);  // K = 1, 3, 9
    constexpr R wi = K == 1 ? -S1 : (K == 3 ? -C1 : S1);
    r.x = v.x * wr - v.y * wi;
    r.y = v.x * wi + v.y * wr;
  }
  return r;
}

// Forward 4-point DFT in place.
template <typename C>
__device__ __forceinline__ void dft4(C& a0, C& a1, C& a2, C& a3) {
  const C t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = csub(a1, a3);
  a0 = cadd(t0, t2);
  a2 = csub(t0, t2);
  a1.x = t1.x + t3.y;
  a1.y = t1.y - t3.x;
  a3.x = t1.x - t3.y;
  a3.y = t1.y + t3.x;
}

// x[k] <- sum_n x[n] e^{-2 pi i n k / 16}: n = q + 4 n1, k = p + 4 k1; 4-point
// DFTs over n1, twiddles e^{-2 pi i q p / 16}, 4-point DFTs over q.
template <typename C>
__device__ __forceinline__ void dft16(C (&x)[16]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) dft4(x[q], x[q + 4], x[q + 8], x[q + 12]);  // (q, p) at q + 4 p
  x[5] = w16mul<1>(x[5]);
  x[9] = w16mul<2>(x[9]);
  x[13] = w16mul<3>(x[13]);
  x[6] = w16mul<2>(x[6]);
  x[10] = w16mul<4>(x[10]);
  x[14] = w16mul<6>(x[14]);
  x[7] = w16mul<3>(x[7]);
  x[11] = w16mul<6>(x[11]);
  x[15] = w16mul<9>(x[15]);
#pragma unroll
  for (int p = 0; p < 4; ++p) dft4(x[4 * p], x[4 * p + 1], x[4 * p + 2], x[4 * p + 3]);  // (p, k1) at 4 p + k1
  C y[16];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) y[p + 4 * k1] = x[4 * p + k1];
#pragma unroll
  for (int k = 0; k < 16; ++k) x[k] = y[k];
}

// The outputs k = 0 and 1 of the same, in x[0] and x[1].
template <typename C>
__device__ __forceinline__ void dft16_two(C (&x)[16]) {
  C e[4], o[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const C s02 = cadd(x[q], x[q + 8]), d02 = csub(x[q], x[q + 8]), s13 = cadd(x[q + 4], x[q + 12]),
            d13 = csub(x[q + 4], x[q + 12]);
    e[q] = cadd(s02, s13);
    o[q].x = d02.x + d13.y;
    o[q].y = d02.y - d13.x;
  }
  x[0] = cadd(cadd(e[0], e[1]), cadd(e[2], e[3]));
  x[1] = cadd(cadd(o[0], w16mul<1>(o[1])), cadd(w16mul<2>(o[2]), w16mul<3>(o[3])));
}

// Forward P-point DFT of the block distributed as v[r] = x[t + 256 r];
// on return v[d] = X[t + 256 d].  Two barriers; b0 and b1 alternate, so
// back-to-back calls need no further barrier.  twA[(k0 - 1) 256 + t] =
// e^{-2 pi i t k0 / P}, twB[c 16 + a] = e^{-2 pi i a c / 256}.
// TWO: only v[0] and v[1] are wanted.
template <bool TWO = false, typename C>
__device__ __forceinline__ void fft_p(C (&v)[16], C* b0, C* b1, const C* twA, const C* twB) {
  const int t = threadIdx.x;
  dft16(v);
#pragma unroll
  for (int k0 = 1; k0 < 16; ++k0) v[k0] = cmul(v[k0], twA[(k0 - 1) * 256 + t]);
#pragma unroll
  for (int k0 = 0; k0 < 16; ++k0) b0[t * 17 + k0] = v[k0];
  __syncthreads();
  {
    const int a = t & 15, k0 = t >> 4;
#pragma unroll
    for (int b = 0; b < 16; ++b) v[b] = b0[(a + 16 * b) * 17 + k0];
    dft16(v);
#pragma unroll
    for (int c = 1; c < 16; ++c) v[c] = cmul(v[c], twB[c * 16 + a]);
#pragma unroll
    for (int c = 0; c < 16; ++c) b1[k0 * 273 + c * 17 + a] = v[c];
  }
  __syncthreads();
  {
    const int k0 = t & 15, c = t >> 4;
#pragma unroll
    for (int a = 0; a < 16; ++a) v[a] = b1[k0 * 273 + c * 17 + a];
    if (TWO) dft16_two(v);
    else dft16(v);
  }
}

__device__ __forceinline__ void seg_twiddles(float2* twA, float2* twB) {
  for (int e = threadIdx.x; e < 15 * 256; e += blockDim.x) {
    const int k0 = e / 256 + 1, th = e % 256;
    float sn, cs;
    sincospif(-(float)(th * k0) / 2048.0f, &sn, &cs);  // exact argument: th k0 < 2^12
    twA[e] = make_float2(cs, sn);
  }
  {
    const int c = threadIdx.x >> 4, a = threadIdx.x & 15;
    float sn, cs;
    sincospif(-(float)(a * c) / 128.0f, &sn, &cs);
    twB[threadIdx.x] = make_float2(cs, sn);
  }
  __syncthreads();
}

// Largest b with b^2 <= t, 0 <= t < 2^46, from the FP32 root (every thread of a
// row takes it, and FP64 has two lanes per SM).
__device__ __forceinline__ int64_t isqrt_row(int64_t t) {
  int64_t b = (int64_t)sqrtf((float)t);
  while (b > 0 && b * b > t) --b;
  while ((b + 1) * (b + 1) <= t) ++b;
  return b;
}

// Open bits of the 16 columns [x, x + 16) of a row (bit p: column x + p) of
// the binary plate, dj2 = dj^2.  Between the chunk's two ends the zone index
// steps through the boundaries m in (zn, zf] (zn, zf: the zones at the ends
// nearer to and farther from the axis, squared radius clamped into the
// disc); boundary m sits at distance a_m = ceil(sqrt(S_m - dj^2)) from the
// axis: at column c + a_m right of the axis (the zone reaches m there), at
// c - a_m + 1 left of it (the zone drops below m there).  With the chunk at
// distance d >= 128 from the axis, a_m = d + k, k in [1, 15] the smallest k
// with k (k + 2d) >= S_m - dj^2 - d^2 (below 30 d + 225: 32-bit); the
// estimate (S_m - dj^2 - d^2) / (2d) exceeds k by k^2 / (2d) < 1, and with
// FP32 rounding it lies within [k - 1, k + 2]: one step up and two down make
// k exact.  Chunks nearer the axis take the zone rule column by column.
// Columns outside the disc chord come out arbitrary (their input is zero).
__device__ __forceinline__ uint32_t chunk_bits(int64_t x, int64_t dj2, const MaskGeom& g) {
  const int64_t dr = x - g.c, dl = g.c - (x + 15);
  if (dr < 128 && dl < 128) {
    uint32_t bits = 0;
    for (int p = 0; p < 16; ++p) {
      const int64_t di = x + p - g.c, sq = dj2 + di * di;
      if (sq <= g.sR && ((zone_of(sq, g) ^ g.centre_open) & 1) != 0) bits |= 1u << p;
    }
    return bits;
  }
  const bool right = dr >= 128;
  const int64_t d = right ? dr : dl;
  const int64_t sn = dj2 + d * d, sf = dj2 + (d + 15) * (d + 15);
  const int64_t zn = zone_of(min(sn, g.sR), g), zf = zone_of(min(sf, g.sR), g);
  uint32_t bits = ((((right ? zn : zf) ^ g.centre_open) & 1) != 0) ? 0xFFFFu : 0u;  // parity at p = 0
  const float inv2d = 0.5f / (float)d;
  const int32_t td = (int32_t)(2 * d);
  for (int64_t m = zn + 1; m <= zf; ++m) {
    const int32_t D = (int32_t)(__ldg(g.thr + (m - 1)) - sn);
    int32_t k = __float2int_ru((float)D * inv2d);
    k += (k * (k + td) < D) ? 1 : 0;
    k -= (k > 0 && (k - 1) * (k - 1 + td) >= D) ? 1 : 0;
    k -= (k > 0 && (k - 1) * (k - 1 + td) >= D) ? 1 : 0;
    bits ^= (0xFFFFu << (right ? k : 16 - k)) & 0xFFFFu;
  }
  return bits;
}

// The zone rule on four columns, a level byte each.
__device__ __noinline__ uint32_t exact_levels4(int64_t di0, int64_t dj2, const MaskGeom& g) {
  uint32_t v = 0u;
  for (int z = 0; z < 4; ++z) {
    const int64_t di = di0 + z;
    v |= ((uint32_t)zone_of(min(dj2 + di * di, g.sR), g) % (uint32_t)g.levels) << (8 * z);
  }
  return v;
}

// Levels of the 16 columns from di0 of a row of the phase plate, a byte each in
// the four words of `lv`: the phase's integer part over L, or, where a phase
// comes within E of a step, the zone rule column by column.
__device__ __forceinline__ void chunk_levels(int64_t di0, int64_t dj2, const MaskGeom& g, const PhaseRule& r,
                                             uint32_t (&lv)[4]) {
  Walk16 w = walk16(di0, dj2, r);
  const uint32_t L = (uint32_t)g.levels, el = r.E * L;
  uint32_t near = 0xFFFFFFFFu;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    uint32_t v = 0u;
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const uint64_t p = (uint64_t)w.f * L;
      near = min(near, (uint32_t)p + el);
      v |= (uint32_t)(p >> 32) << (8 * z);
      w.f += w.d;
      w.d += w.c2;
    }
    lv[k] = v;
  }
  if (near < 2u * el) {
#pragma unroll
    for (int k = 0; k < 4; ++k) lv[k] = exact_levels4(di0 + 4 * k, dj2, g);
  }
}

// The inner pass of the single convolution in FP64 (L2 = 4096; what k_f2 does for
// the other lengths): the 4096-point transforms above, in registers, resident
// CTAs over the (row, k1) pairs.  FP64 has two lanes per SM here (GB300: 1.25
// TFLOP/s), so operations are what counts: radix 16 takes 3.6 per point and
// stage instead of radix 2's 4, the inverse's last pass forms only the outputs
// that are kept, and a flat plate's columns from the axis on fit half the
// length.  4 mm plate (N = 5,057, L 8192 -> 4096), ROI 256^2: 6.2 -> 1.6 ms for
// the row transforms (375,000 FP64 operations a row, 2,529 rows: 1.6 ms at 0.58
// T/s, the pipe's rate), 22.2 -> 2.1 ms for a propagation with its metrics.
constexpr size_t D16_SMEM = sizeof(double2) * (2 * SBUF + 15 * 256 + 256);
__global__ void __launch_bounds__(STH, 1) k_f2_d16(RowArgs a, int mode) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* b0 = reinterpret_cast<double2*>(smem_raw);
  double2* b1 = b0 + SBUF;
  double2* twA = b1 + SBUF;
  double2* twB = twA + 15 * 256;
  const int t = threadIdx.x;
  const double2* tw = reinterpret_cast<const double2*>(a.tw);  // e^{-2 pi i t / 4096}
  for (int e = t; e < 15 * 256; e += STH) twA[e] = tw[(e / 256 + 1) * (e % 256)];
  twB[t] = tw[16 * (t >> 4) * (t & 15)];
  __syncthreads();
  const double2* pre = reinterpret_cast<const double2*>(a.pre);
  const double2* vin = reinterpret_cast<const double2*>(a.vin);
  const double2* post = reinterpret_cast<const double2*>(a.post);
  for (int64_t w = blockIdx.x; w < a.rows * a.L1; w += gridDim.x) {
    const int64_t r = w / a.L1, k1 = w % a.L1, j = a.j0 + r;
    double2 v[16];
    double2* Z = reinterpret_cast<double2*>(a.Z) + r * a.L + k1 * SP;
    if (a.L1 == 1) {
#pragma unroll
      for (int q = 0; q < 16; ++q) v[q] = mode == 0 ? row_input<double>(a, j, t + 256 * q, pre) : vin[t + 256 * q];
    } else {
#pragma unroll
      for (int q = 0; q < 16; ++q) v[q] = Z[t + 256 * q];
    }
    fft_p(v, b0, b1, twA, twB);
    if (mode == 1) {
#pragma unroll
      for (int d = 0; d < 16; ++d) Z[t + 256 * d] = v[d];
      continue;
    }
    const double2* H = reinterpret_cast<const double2*>(a.H) + k1 * SP + t;
#pragma unroll
    for (int d = 0; d < 16; ++d) {
      v[d] = cmul(v[d], H[256 * d]);
      v[d].y = -v[d].y;  // the inverse transform as conj(FFT(conj(.)))
    }
    if (a.M <= 512) fft_p<true>(v, b0, b1, twA, twB);
    else fft_p(v, b0, b1, twA, twB);
    const int64_t jl = j - a.c1_j0;
    double* C1 = reinterpret_cast<double*>(a.C1);
    if (a.L1 == 1 && a.half) {
      // outputs x and -x meet in the buffer that the last pass does not read
#pragma unroll
      for (int d = 0; d < 5; ++d) {
        const int m = t + 256 * d;
        if (m < a.M) b0[m] = cmul(make_double2(v[d].x, -v[d].y), post[m]);
      }
      __syncthreads();
      const int hm = (a.M - 1) / 2;
      for (int m = t; m <= hm; m += STH) {
        const double2 y = cadd(b0[hm + m], b0[hm - m]);
        C1[(int64_t)c1_row_re(m) * a.c1_stride + jl] = y.x;
        C1[(int64_t)c1_row_im(m) * a.c1_stride + jl] = y.y;
      }
      __syncthreads();
      continue;
    }
#pragma unroll
    for (int d = 0; d < 5; ++d) {
      const int m = t + 256 * d;
      if (m >= a.M) continue;
      const double2 y = make_double2(v[d].x, -v[d].y);
      if (a.L1 == 1) {
        const double2 z = cmul(y, post[m]);
        C1[(int64_t)c1_row_re(m) * a.c1_stride + jl] = z.x;
        C1[(int64_t)c1_row_im(m) * a.c1_stride + jl] = z.y;
      } else {
        reinterpret_cast<double2*>(a.G)[(r * a.L1 + k1) * a.M + m] =
            cmul(y, twiddle_L<double>(a, (k1 * m) & (a.L - 1), true));
      }
    }
    __syncthreads();  // the next row's first pass writes b0
  }
}

// G_s = FFT_P(g_s) for every block s (one CTA per block, grid-strided); blocks
// every S input columns, W of them long.
__global__ void __launch_bounds__(STH) k_seg_tables(int64_t nseg, int64_t col0, int S, int W, int M, double delta, float2* G) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* b0 = reinterpret_cast<float2*>(smem_raw);
  float2* b1 = b0 + SBUF;
  float2* twA = b1 + SBUF;
  float2* twB = twA + 15 * 256;
  seg_twiddles(twA, twB);
  const int t = threadIdx.x;
  for (int64_t s = blockIdx.x; s < nseg; s += gridDim.x) {
    const int64_t is = col0 + s * (int64_t)S;
    float2 v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int q = t + 256 * r;
      v[r] = make_float2(0.0f, 0.0f);
      int64_t k = 0;
      bool have = false;
      if (q < M) { k = q - is; have = true; }
      else if (q > SP - W) { k = (int64_t)q - SP - is; have = true; }
      if (have) {
        const double kk = (double)k;  // |k| < 2^24: k^2 exact in FP64
        v[r] = cis_turns<float>(0.5 * delta * kk * kk);
      }
    }
    fft_p(v, b0, b1, twA, twB);
    float2* out = G + s * SP + t;
#pragma unroll
    for (int d = 0; d < 16; ++d) out[256 * d] = v[d];
  }
}

// Row pass of the partitioned convolution: rows j0 + r, r = blockIdx.x,
// blockIdx.x + gridDim.x, ... (interleaved, so every CTA gets rows from the
// whole range of chord lengths); writes C1 like k_f3.  The transmission of a
// block's samples, by chunks of 16 columns whose zone phase is walked (the exact
// rule where it comes near a zone's end): SEG_FLAT, binary amplitude plate, open
// bits; SEG_LEVELS, phase plate, a level byte per column and the level's phasor
// from a table; SEG_MEMBRANE and SEG_DIRECT, deformed binary plate, open bits and
// the membrane's phase; SEG_GENERAL, deformed phase plate, the transmission
// function per sample.  A block's input chirp loads are issued together before the
// transmission is evaluated, and the spectra G_s before the last FFT pass,
// so each waits one memory latency.
//
// Flat plates (FOLD; rows j >= c: each stands for itself and its mirror image):
// `half`, for an output grid symmetric about the axis, transforms the columns
// from the axis on and adds the outputs at x and -x (the axis column, counted
// twice, at half weight); `octant`, for the whole aperture, stops at the
// diagonal |di| = dj with half weight there (the field is this one plus its
// transpose).  Half the blocks each, a quarter both, and half the rows; with the
// outputs on nodes (nodes.cu: 128 instead of 512) the column pass shrinks too.
// Whole propagation, ROI 512^2, with the masks from the walked zone phase: D = 5
// cm (N = 63,213) 17.1 -> 1.86 ms, L = 16 on N = 50,001 15.7 -> 1.38 ms; such
// plates now take k_dec, this kernel the grids too small for it, deformed phase
// plates and ROIs without nodes.
template <int MODE>
__global__ void __launch_bounds__(STH, 2) k_seg(RowArgs a) {
  constexpr bool FOLD = MODE == SEG_FLAT || MODE == SEG_LEVELS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* b0 = reinterpret_cast<float2*>(smem_raw);
  float2* b1 = b0 + SBUF;
  float2* twA = b1 + SBUF;
  float2* twB = twA + 15 * 256;
  float2* phs = twB + 256;                              // SEG_LEVELS: e^{-2 pi i q / L}, q < L <= 64; 0 at NO_LEVEL
  uint32_t* mk = reinterpret_cast<uint32_t*>(phs + NO_LEVEL + 2);  // SEG_FLAT: open bits per chunk of 16 columns
  uint8_t* lev = reinterpret_cast<uint8_t*>(mk);        // SEG_LEVELS: level per column
  const uint32_t nlev = (uint32_t)max(a.mg.levels, 1);
  if (MODE == SEG_LEVELS && threadIdx.x <= NO_LEVEL) {
    float sn, cs;
    sincospif(-2.0f * (float)threadIdx.x / (float)nlev, &sn, &cs);
    phs[threadIdx.x] = threadIdx.x == NO_LEVEL ? make_float2(0.0f, 0.0f) : make_float2(cs, sn);
  }
  seg_twiddles(twA, twB);
  const int t = threadIdx.x;
  const float2* pre = reinterpret_cast<const float2*>(a.pre);
  const float2* Gs = reinterpret_cast<const float2*>(a.H);
  const float2* post = reinterpret_cast<const float2*>(a.post);
  float* C1 = reinterpret_cast<float*>(a.C1);
  const int S = a.S, RS = a.S / 256;
  const float scale = (float)a.L / (float)SP;  // post carries 1/L; the inverse below is unnormalised
  for (int64_t r = blockIdx.x; r < a.rows; r += gridDim.x) {
    const int64_t j = a.j0 + r;
    const int64_t dj = j - a.mg.c;
    const int64_t rem = a.mg.sR - dj * dj;
    float2 acc[16];
#pragma unroll
    for (int d = 0; d < 16; ++d) acc[d] = make_float2(0.0f, 0.0f);
    CxRow cxr;
    if (seg_membrane(MODE)) cx_row_init(a.df, dj, cxr);
    if (rem >= 0) {
      int64_t bmax = isqrt_row(rem);
      if (FOLD && a.octant) bmax = min(bmax, dj);
      // the row's disc chord, within the grid (a given N may cut the disc)
      const int64_t lo = FOLD && a.half ? a.mg.c : max(a.mg.c - bmax, (int64_t)0), hi = min(a.mg.c + bmax, a.N - 1);
      const int64_t col0 = FOLD ? a.col0 : 0, s1 = (hi - col0) / S;
      for (int64_t s = (lo - col0) / S; s <= s1; ++s) {
        const int64_t is = col0 + s * (int64_t)S;
        float2 v[16];
        // the block's chord [olo, ohi] in block offsets; thread t makes the 16
        // columns from offset 16 t (element (t, q) is offset t + 256 q)
        const int olo = (int)max(lo - is, (int64_t)0), ohi = (int)min(hi - is, (int64_t)(S - 1)), xo = 16 * t;
        const bool meets = t < S / 16 && xo + 15 >= olo && xo <= ohi;
        const uint32_t inside = meets ? (0xFFFFu >> (15 - min(ohi - xo, 15) + max(olo - xo, 0))) << max(olo - xo, 0) : 0u;
        if (MODE == SEG_FLAT || MODE == SEG_LEVELS) {
          // loads clamped into the grid, every element's value decided by its bit or level
          const int lim = (int)min(a.N - 1 - is, (int64_t)(SP - 1));
          const float2* pb = pre + is;
#pragma unroll
          for (int q = 0; q < 16; ++q) v[q] = __ldg(pb + min(t + 256 * q, lim));
        }
        if (MODE == SEG_FLAT) {
          uint32_t w = 0u;
          if (meets && !walk_bits16(walk16(is + xo - a.mg.c, dj * dj, a.ph), a.ph, w)) w = chunk_bits(is + xo, dj * dj, a.mg);
          mk[t] = w & inside;
          __syncthreads();
#pragma unroll
          for (int q = 0; q < 16; ++q)
            if (((mk[16 * q + (t >> 4)] >> (t & 15)) & 1u) == 0) v[q] = make_float2(0.0f, 0.0f);
        } else if (seg_membrane(MODE)) {
          uint32_t w = 0u;
          if (meets && !walk_bits16(walk16(is + xo - a.mg.c, dj * dj, a.ph), a.ph, w)) w = chunk_bits(is + xo, dj * dj, a.mg);
          w &= inside;
          // phases by chunk through the first transpose buffer (its last readers
          // are two barriers back; pitch 17 a chunk), the chirp's turns added and
          // one hardware sine and cosine of the sum reduced to [-1/2, 1/2] turns
          // (absolute error below 4e-7 each) by element
          float* wz = reinterpret_cast<float*>(b0);
          float* o = wz + 17 * t;
          const float* pt = reinterpret_cast<const float*>(a.pre) + is;
          const int lim = (int)min(a.N - 1 - is, (int64_t)(SP - 1));
          float tc[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) tc[q] = __ldg(pt + min(t + 256 * q, lim));
          if (w != 0u) {
            const int32_t di0 = (int32_t)(is + xo - a.mg.c);
            if (MODE == SEG_DIRECT) {
              membrane_chunk(MembraneDirect(a.df, cxr, di0), w, o);
            } else {
              switch (a.df.n) {
                case 0: membrane_chunk(MembraneWalk<0>(a.df, cxr, di0), w, o); break;
                case 1: membrane_chunk(MembraneWalk<1>(a.df, cxr, di0), w, o); break;
                case 2: membrane_chunk(MembraneWalk<2>(a.df, cxr, di0), w, o); break;
                default: membrane_chunk(MembraneWalk<3>(a.df, cxr, di0), w, o); break;
              }
            }
          } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) o[k] = CLOSED;
          }
          __syncthreads();
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            constexpr float TWO_PI = 6.28318530717958648f;
            const float wv = wz[t + 256 * q + ((t + 256 * q) >> 4)];
            float x = wv + tc[q];
            x -= rintf(x);
            x *= TWO_PI;
            const bool open = wv < 0.5f * CLOSED;
            v[q] = make_float2(open ? __cosf(x) : 0.0f, open ? __sinf(x) : 0.0f);
          }
          __syncthreads();  // pass A writes this buffer
        } else if (MODE == SEG_LEVELS) {
          uint32_t lv[4] = {0x40404040u, 0x40404040u, 0x40404040u, 0x40404040u};
          if (meets) {
            chunk_levels(is + xo - a.mg.c, dj * dj, a.mg, a.ph, lv);
            if (inside != 0xFFFFu) {
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                uint32_t m = 0u;
#pragma unroll
                for (int z = 0; z < 4; ++z) m |= ((inside >> (4 * k + z)) & 1u) ? 0xFFu << (8 * z) : 0u;
                lv[k] = (lv[k] & m) | (0x40404040u & ~m);
              }
            }
          }
          *reinterpret_cast<uint4*>(lev + 16 * t) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
          __syncthreads();
#pragma unroll
          for (int q = 0; q < 16; ++q) v[q] = cmul(v[q], phs[lev[t + 256 * q]]);
        } else {
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int64_t i = is + t + 256 * q;
            v[q] = (q < RS && i >= lo && i <= hi) ? __ldg(pre + i) : make_float2(0.0f, 0.0f);
          }
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int64_t i = is + t + 256 * q;
            if (q < RS && i >= lo && i <= hi) v[q] = cmul(aperture<float>(a, j, i), v[q]);
          }
        }
        if (FOLD) {
          // half weight of the axis column and of the diagonal's columns (few blocks hold one)
          const int64_t oa = a.half ? a.mg.c - is : -1, od = a.octant ? a.mg.c + dj - is : -1,
                        oe = a.octant && !a.half && dj > 0 ? a.mg.c - dj - is : -1;
          const bool ha = oa >= 0 && oa < S, hd = od >= 0 && od < S, he = oe >= 0 && oe < S;
          if (ha || hd || he) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const int o = t + 256 * q;
              float w = ha && o == (int)oa ? 0.5f : 1.0f;
              if (hd && o == (int)od) w *= 0.5f;
              if (he && o == (int)oe) w *= 0.5f;
              v[q].x *= w;
              v[q].y *= w;
            }
          }
        }
        // forward FFT (passes A and B), spectrum loads, pass C, product-sum
        dft16(v);
#pragma unroll
        for (int k0 = 1; k0 < 16; ++k0) v[k0] = cmul(v[k0], twA[(k0 - 1) * 256 + t]);
#pragma unroll
        for (int k0 = 0; k0 < 16; ++k0) b0[t * 17 + k0] = v[k0];
        __syncthreads();
        {
          const int aa = t & 15, k0 = t >> 4;
#pragma unroll
          for (int b = 0; b < 16; ++b) v[b] = b0[(aa + 16 * b) * 17 + k0];
          dft16(v);
#pragma unroll
          for (int c = 1; c < 16; ++c) v[c] = cmul(v[c], twB[c * 16 + aa]);
#pragma unroll
          for (int c = 0; c < 16; ++c) b1[k0 * 273 + c * 17 + aa] = v[c];
        }
        __syncthreads();
        float2 g[16];
        const float2* G = Gs + s * SP + t;
#pragma unroll
        for (int d = 0; d < 16; ++d) g[d] = __ldg(G + 256 * d);
        {
          const int k0 = t & 15, c = t >> 4;
#pragma unroll
          for (int aa = 0; aa < 16; ++aa) v[aa] = b1[k0 * 273 + c * 17 + aa];
          dft16(v);
        }
#pragma unroll
        for (int d = 0; d < 16; ++d) {
          acc[d].x = fmaf(v[d].x, g[d].x, fmaf(-v[d].y, g[d].y, acc[d].x));
          acc[d].y = fmaf(v[d].x, g[d].y, fmaf(v[d].y, g[d].x, acc[d].y));
        }
      }
    }
    // inverse transform as conj(FFT(conj(.))), outputs m = t + 256 d < M
#pragma unroll
    for (int d = 0; d < 16; ++d) acc[d].y = -acc[d].y;
    fft_p(acc, b0, b1, twA, twB);
    const int64_t jl = j - a.c1_j0;
    if (FOLD && a.half) {
      // outputs x and -x meet in the transpose buffer that the transform's last
      // pass does not read (M <= 256 nodes: one output per thread)
      if (t < a.M) b0[t] = cmul(make_float2(acc[0].x * scale, -acc[0].y * scale), post[t]);
      __syncthreads();
      const int hm = a.M / 2;
      if (t < hm) {
        const float2 y = cadd(b0[hm + t], b0[hm - 1 - t]);
        C1[(int64_t)c1_row_re(t) * a.c1_stride + jl] = y.x;
        C1[(int64_t)c1_row_im(t) * a.c1_stride + jl] = y.y;
      }
      __syncthreads();
      continue;
    }
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const int m = t + 256 * d;
      if (m < a.M) {
        const float2 y = cmul(make_float2(acc[d].x * scale, -acc[d].y * scale), post[m]);
        C1[(int64_t)c1_row_re(m) * a.c1_stride + jl] = y.x;
        C1[(int64_t)c1_row_im(m) * a.c1_stride + jl] = y.y;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Decimated rows.  The outputs' band is narrow: between a row's columns the
// phases of the nodes' exponentials e^{-2 pi i delta (m - m_c) x} differ by at most
// u = pi delta (n - 1), so over a chunk of D = 16 or 32 columns each of them is a
// polynomial, and interpolating it from DTAPS = 6 points of a grid of pitch D is
// off by at most 0.0049 (D u)^6 (the outermost node, a quarter outside the ROI).
// Transposed: a column's value times the input chirp is spread over the six grid
// points, and the row goes on as N / D + 5 points through the convolution above:
// two rows to a 4096-point transform (offsets 0 and 2048: with S + 5 + n < 2050
// neither meets the other's outputs) instead of N / 3840 transforms a row.
//
// A lane takes one chunk of two neighbouring rows, all in registers: the chirp by
// a 64-bit fixed-point phase walked in 32 bits (as the zone phase), the value, and
// four running sums (c0 += z, c1 += c0, ...) per 16 columns, which are their
// binomial moments; the weights T (decimation_weights) take them to the grid
// points; lanes exchange the overlaps by shuffles.  No table is read per column.
// Whole propagations, k_seg -> k_dec: D = 5 cm 1.86 -> 0.80 ms, L = 16 1.38 -> 0.80,
// four membranes on N <= 34,567 13.2 -> 5.1 ms (9 transforms a row to a half).
// What bounds it: the issue slots (60 % busy at two CTAs of 128 registers a
// thread per SM); of a membrane's 45 instructions per column the walk in pairs,
// the mask's walk and the running sums take two thirds.
// ---------------------------------------------------------------------------
constexpr int DROW = SP / 2;                    // offset of the second row
constexpr int DGRP = DROW / 32;                 // warp groups of chunks a row
constexpr size_t DEC_SMEM = sizeof(float2) * (2 * SBUF + 15 * 256 + 256 + 2 * DGRP * (DTAPS - 1));

struct DecRow {
  int64_t dj;
  int32_t lo, hi;  // the row's chord (lo > hi: empty)
};

__device__ __forceinline__ float2 cis_rad(float x) { return make_float2(__cosf(x), __sinf(x)); }

// Bits of the 16 columns from x that lie in the row's chord.
__device__ __forceinline__ uint32_t chord_bits(const DecRow& r, int32_t x) {
  const int a = max(r.lo - x, 0), b = min(r.hi - x, 15);
  return a <= b ? (0xFFFFu >> (15 - b + a)) << a : 0u;
}

__device__ __forceinline__ uint32_t open_bits(const RowArgs& a, const DecRow& r, int32_t x) {
  const uint32_t in = chord_bits(r, x);
  uint32_t w = 0u;
  if (in != 0u && !walk_bits16(walk16((int64_t)x - a.mg.c, r.dj * r.dj, a.ph), a.ph, w)) w = chunk_bits(x, r.dj * r.dj, a.mg);
  return w & in;
}

// The running sums of 16 columns; add(z): the next column's value joins c[0] first.
__device__ __forceinline__ void sums_step(float2 (&c)[4]) {
#pragma unroll
  for (int q = 1; q < 4; ++q) c[q] = cadd(c[q], c[q - 1]);
}

// c += w times the sums of a single value z at column k of the 16.
__device__ __forceinline__ void sums_at(float2 (&c)[4], int k, float2 z, float w) {
  const float m = (float)(16 - k);
  const float b[4] = {w, w * m, w * m * (m + 1.0f) * 0.5f, w * m * (m + 1.0f) * (m + 2.0f) * (1.0f / 6.0f)};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c[q].x = fmaf(b[q], z.x, c[q].x);
    c[q].y = fmaf(b[q], z.y, c[q].y);
  }
}

__device__ __forceinline__ void sums_out(const RowArgs& a, int sub, const float2 (&c)[4], float2 (&tap)[DTAPS]) {
#pragma unroll
  for (int q = 0; q < DTAPS; ++q)
#pragma unroll
    for (int e = 0; e < 4; ++e) tap[q] = fma2(a.T[sub][q][e], c[e], tap[q]);
}

// The chirp's 32-bit phase and its first difference at column di0.  Without Kc2 the
// phase would be short by up to di0^2 2^-64 turns: 3.5e-6 at the rim of N = 16e6.
// (Its product with the lower half of di0^2 stays below a unit of f.)
struct Chirp16 {
  uint32_t f, d;
};
__device__ __forceinline__ Chirp16 chirp16(const RowArgs& a, int64_t di0) {
  Chirp16 p;
  const uint64_t d2 = (uint64_t)(di0 * di0);
  p.f = (uint32_t)((a.Kc * d2 + a.Kl * (uint64_t)di0) >> 32) + __umulhi(a.Kc2, (uint32_t)(d2 >> 32));
  p.d = (uint32_t)((a.Kc * (uint64_t)(2 * di0 + 1) + a.Kl + 0x80000000ull) >> 32);
  return p;
}

// Folded plates: half weight of the axis column and of the diagonal's columns, as
// a correction of the sums.  value(k): the chunk's column k.
template <typename F>
__device__ __forceinline__ void fold_weights(const RowArgs& a, const DecRow& r, int32_t x, float2 (&c)[4], F value) {
  const int32_t dj = (int32_t)r.dj, cc = (int32_t)a.mg.c;
  const int ka = a.half ? cc - x : -1, kd = a.octant ? cc + dj - x : -1, ke = a.octant && !a.half && dj > 0 ? cc - dj - x : -1;
  if ((unsigned)ka < 16u) sums_at(c, ka, value(ka), -0.5f);
  if ((unsigned)kd < 16u) sums_at(c, kd, value(kd), ka == kd ? -0.25f : -0.5f);
  if ((unsigned)ke < 16u) sums_at(c, ke, value(ke), -0.5f);
}

constexpr float RAD32 = 6.28318530717958648f / 4294967296.0f;  // 2^-32 turns in radians

// Binary plate: both rows share the chirp's sine and cosine.
template <int D>
__device__ __forceinline__ void dec_flat(const RowArgs& a, const DecRow (&row)[2], int32_t x0, float2 (&tap)[2][DTAPS]) {
#pragma unroll 1
  for (int sub = 0; sub < D / 16; ++sub) {
    const int32_t x = x0 + 16 * sub;
    const Chirp16 p0 = chirp16(a, (int64_t)x - a.mg.c);
    const uint32_t w0 = open_bits(a, row[0], x), w1 = open_bits(a, row[1], x);
    float2 c[2][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) c[0][e] = c[1][e] = make_float2(0.0f, 0.0f);
    uint32_t f = p0.f, d = p0.d;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float2 z = cis_rad((float)(int32_t)f * RAD32);
      if ((w0 >> k) & 1u) c[0][0] = cadd(c[0][0], z);
      if ((w1 >> k) & 1u) c[1][0] = cadd(c[1][0], z);
      sums_step(c[0]);
      sums_step(c[1]);
      f += d;
      d += a.cc2;
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const uint32_t w = e ? w1 : w0;
      fold_weights(a, row[e], x, c[e], [&](int k) {
        const float2 z = cis_rad((float)(int32_t)(p0.f + (uint32_t)k * p0.d + (uint32_t)(k * (k - 1) / 2) * a.cc2) * RAD32);
        return ((w >> k) & 1u) ? z : make_float2(0.0f, 0.0f);
      });
      sums_out(a, sub, c[e], tap[e]);
    }
  }
}

// Phase plate: the level's turns taken off the chirp's.
template <int D>
__device__ __forceinline__ void dec_levels(const RowArgs& a, const DecRow& row, int32_t x0, float2 (&tap)[DTAPS]) {
  const uint32_t turn = (uint32_t)((0x100000000ull + (uint32_t)a.mg.levels / 2) / (uint32_t)a.mg.levels);
#pragma unroll 1
  for (int sub = 0; sub < D / 16; ++sub) {
    const int32_t x = x0 + 16 * sub;
    const uint32_t in = chord_bits(row, x);
    if (in == 0u) continue;
    uint32_t lv[4];
    chunk_levels((int64_t)x - a.mg.c, row.dj * row.dj, a.mg, a.ph, lv);
    const Chirp16 p0 = chirp16(a, (int64_t)x - a.mg.c);
    float2 c[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) c[e] = make_float2(0.0f, 0.0f);
    uint32_t f = p0.f, d = p0.d;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const uint32_t q = (lv[k >> 2] >> (8 * (k & 3))) & 0xFFu;
      const float2 z = cis_rad((float)(int32_t)(f - q * turn) * RAD32);
      if ((in >> k) & 1u) c[0] = cadd(c[0], z);
      sums_step(c);
      f += d;
      d += a.cc2;
    }
    fold_weights(a, row, x, c, [&](int k) {
      const uint32_t w = k < 8 ? (k < 4 ? lv[0] : lv[1]) : (k < 12 ? lv[2] : lv[3]);
      const uint32_t q = (w >> (8 * (k & 3))) & 0xFFu;
      const float2 z = cis_rad((float)(int32_t)(p0.f + (uint32_t)k * p0.d + (uint32_t)(k * (k - 1) / 2) * a.cc2 - q * turn) * RAD32);
      return ((in >> k) & 1u) ? z : make_float2(0.0f, 0.0f);
    });
    sums_out(a, sub, c, tap);
  }
}

// Deformed binary plate: both rows' membrane phases walked along the chunk in
// pairs, one hardware sine and cosine of the sum with the chirp's reduced to
// [-1/2, 1/2] turns (absolute error below 4e-7 each).
template <int D, typename Walk2>
__device__ __forceinline__ void dec_membrane_n(const RowArgs& a, const DecRow (&row)[2], Walk2 walk, int32_t x0,
                                               float2 (&tap)[2][DTAPS]) {
#pragma unroll 1
  for (int sub = 0; sub < D / 16; ++sub) {
    const int32_t x = x0 + 16 * sub;
    const uint32_t w0 = open_bits(a, row[0], x), w1 = open_bits(a, row[1], x);
    const Chirp16 p0 = chirp16(a, (int64_t)x - a.mg.c);
    float2 c[2][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) c[0][e] = c[1][e] = make_float2(0.0f, 0.0f);
    uint32_t f = p0.f, d = p0.d;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float2 t = reduced_rad(fma2(pair2((float)(int32_t)f), pair2(1.0f / 4294967296.0f), walk.next()));
      if ((w0 >> k) & 1u) c[0][0] = cadd(c[0][0], cis_rad(t.x));
      if ((w1 >> k) & 1u) c[1][0] = cadd(c[1][0], cis_rad(t.y));
      sums_step(c[0]);
      sums_step(c[1]);
      f += d;
      d += a.cc2;
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) sums_out(a, sub, c[e], tap[e]);
  }
}
template <int NR>
__device__ __forceinline__ MembraneWalk2<NR> walk_rows(const DeformCoef& d, const CxRow (&cx)[2], int32_t di0) {
  return MembraneWalk2<NR>(MembraneWalk<NR>(d, cx[0], di0), MembraneWalk<NR>(d, cx[1], di0));
}
template <int D, bool DIRECT>
__device__ __forceinline__ void dec_membrane(const RowArgs& a, const DecRow (&row)[2], const CxRow (&cx)[2], int32_t x0,
                                             float2 (&tap)[2][DTAPS]) {
  const int32_t di0 = (int32_t)(x0 - a.mg.c);
  if (DIRECT) {
    dec_membrane_n<D>(a, row, MembraneDirect2(MembraneDirect(a.df, cx[0], di0), MembraneDirect(a.df, cx[1], di0)), x0, tap);
    return;
  }
  switch (a.df.n) {
    case 0: dec_membrane_n<D>(a, row, walk_rows<0>(a.df, cx, di0), x0, tap); break;
    case 1: dec_membrane_n<D>(a, row, walk_rows<1>(a.df, cx, di0), x0, tap); break;
    case 2: dec_membrane_n<D>(a, row, walk_rows<2>(a.df, cx, di0), x0, tap); break;
    default: dec_membrane_n<D>(a, row, walk_rows<3>(a.df, cx, di0), x0, tap); break;
  }
}

// Row pass: rows j0 + 2 p and j0 + 2 p + 1, p = blockIdx.x, blockIdx.x + gridDim.x,
// ...; warps take groups of 32 chunks.  Output as k_seg.
template <int MODE, int D>
__global__ void __launch_bounds__(STH, 2) k_dec(RowArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* b0 = reinterpret_cast<float2*>(smem_raw);
  float2* b1 = b0 + SBUF;
  float2* twA = b1 + SBUF;
  float2* twB = twA + 15 * 256;
  float2* over = twB + 256;  // [row][group][5]: a group's share of the next group's points
  seg_twiddles(twA, twB);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const float2* pre = reinterpret_cast<const float2*>(a.pre);
  const float2* Gs = reinterpret_cast<const float2*>(a.H);
  const float2* post = reinterpret_cast<const float2*>(a.post);
  float* C1 = reinterpret_cast<float*>(a.C1);
  const int S = a.S, W = S + DTAPS - 1;
  const int32_t base = (int32_t)a.col0;
  for (int64_t p = blockIdx.x; 2 * p < a.rows; p += gridDim.x) {
    DecRow row[2];
    CxRow cx[2];
    int32_t lo = INT32_MAX, hi = -1;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      row[e].dj = a.j0 + 2 * p + e - a.mg.c;
      row[e].lo = 0;
      row[e].hi = -1;
      const int64_t rem = a.mg.sR - row[e].dj * row[e].dj;
      if (rem >= 0 && 2 * p + e < a.rows) {
        int64_t bmax = isqrt_row(rem);
        if (!seg_membrane(MODE) && a.octant) bmax = min(bmax, row[e].dj);
        // the row's disc chord, within the grid (a given N may cut the disc)
        row[e].lo = (int32_t)(!seg_membrane(MODE) && a.half ? a.mg.c : max(a.mg.c - bmax, (int64_t)0));
        row[e].hi = (int32_t)min(a.mg.c + bmax, a.N - 1);
        lo = min(lo, row[e].lo);
        hi = max(hi, row[e].hi);
      }
      if (seg_membrane(MODE)) cx_row_init(a.df, row[e].dj, cx[e]);
    }
    float2 acc[16];
#pragma unroll
    for (int d = 0; d < 16; ++d) acc[d] = make_float2(0.0f, 0.0f);
    if (hi >= lo) {
      const int ch0 = (lo - base) / D, ch1 = (hi - base) / D;
      const int s0 = ch0 / S, s1 = ch1 / S;
      for (int s = s0; s <= s1; ++s) {
        const int g0 = max(ch0 - s * S, 0) >> 5, g1 = min(ch1 - s * S, S - 1) >> 5;
        for (int g = g0 + warp; g <= g1; g += STH / 32) {
          const int32_t x0 = base + D * (s * S + 32 * g + lane);
          float2 tap[2][DTAPS];
#pragma unroll
          for (int q = 0; q < DTAPS; ++q) tap[0][q] = tap[1][q] = make_float2(0.0f, 0.0f);
          if (MODE == SEG_FLAT) {
            dec_flat<D>(a, row, x0, tap);
          } else if (MODE == SEG_LEVELS) {
#pragma unroll
            for (int e = 0; e < 2; ++e) dec_levels<D>(a, row[e], x0, tap[e]);
          } else {
            dec_membrane<D, MODE == SEG_DIRECT>(a, row, cx, x0, tap);
          }
          __syncwarp();
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            // chunk ch's tap q belongs to point ch + q
            float2 in = tap[e][0], out = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int q = 1; q < DTAPS; ++q) {
              const int src = (lane - q) & 31;
              const float2 v = make_float2(__shfl_sync(0xFFFFFFFFu, tap[e][q].x, src), __shfl_sync(0xFFFFFFFFu, tap[e][q].y, src));
              if (lane >= q) in = cadd(in, v);
              else out = cadd(out, v);
            }
            b0[e * DROW + 32 * g + lane] = in;
            if (lane < DTAPS - 1) over[(e * DGRP + g) * (DTAPS - 1) + lane] = out;
          }
        }
        __syncthreads();
        float2 v[16];
        {
          const float2* pb = pre + (int64_t)s * S;
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int e = t + 256 * r, g = e >> 5;
            const float2 y = __ldg(pb + min(e, W - 1));
#pragma unroll
            for (int z = 0; z < 2; ++z) {
              float2 x = make_float2(0.0f, 0.0f);
              if (g >= g0 && g <= g1) x = b0[z * DROW + e];
              if (lane < DTAPS - 1 && g > g0 && g <= g1 + 1) x = cadd(x, over[(z * DGRP + g - 1) * (DTAPS - 1) + lane]);
              v[r + 8 * z] = cmul(x, y);
            }
          }
        }
        // the spectrum sum waits in the second buffer while the columns are made
#pragma unroll
        for (int d = 0; d < 16; ++d) acc[d] = s > s0 ? b1[t + 256 * d] : make_float2(0.0f, 0.0f);
        __syncthreads();  // pass A writes the points' buffer
        dft16(v);
#pragma unroll
        for (int k0 = 1; k0 < 16; ++k0) v[k0] = cmul(v[k0], twA[(k0 - 1) * 256 + t]);
#pragma unroll
        for (int k0 = 0; k0 < 16; ++k0) b0[t * 17 + k0] = v[k0];
        __syncthreads();
        {
          const int aa = t & 15, k0 = t >> 4;
#pragma unroll
          for (int b = 0; b < 16; ++b) v[b] = b0[(aa + 16 * b) * 17 + k0];
          dft16(v);
#pragma unroll
          for (int c = 1; c < 16; ++c) v[c] = cmul(v[c], twB[c * 16 + aa]);
#pragma unroll
          for (int c = 0; c < 16; ++c) b1[k0 * 273 + c * 17 + aa] = v[c];
        }
        __syncthreads();
        float2 g[16];
        const float2* G = Gs + (int64_t)s * SP + t;
#pragma unroll
        for (int d = 0; d < 16; ++d) g[d] = __ldg(G + 256 * d);
        {
          const int k0 = t & 15, c = t >> 4;
#pragma unroll
          for (int aa = 0; aa < 16; ++aa) v[aa] = b1[k0 * 273 + c * 17 + aa];
          dft16(v);
        }
#pragma unroll
        for (int d = 0; d < 16; ++d) {
          acc[d].x = fmaf(v[d].x, g[d].x, fmaf(-v[d].y, g[d].y, acc[d].x));
          acc[d].y = fmaf(v[d].x, g[d].y, fmaf(v[d].y, g[d].x, acc[d].y));
        }
        if (s < s1) {
          __syncthreads();
#pragma unroll
          for (int d = 0; d < 16; ++d) b1[t + 256 * d] = acc[d];
        }
      }
    }
    // inverse transform as conj(FFT(conj(.))): outputs m = t of the first row at
    // point t, of the second at DROW + t (n <= 256)
#pragma unroll
    for (int d = 0; d < 16; ++d) acc[d].y = -acc[d].y;
    fft_p(acc, b0, b1, twA, twB);
    const int64_t jl = a.j0 + 2 * p - a.c1_j0;
    float2 y[2];
    if (t < a.M) {
      const float2 w = post[t];
      y[0] = cmul(make_float2(acc[0].x, -acc[0].y), w);
      y[1] = cmul(make_float2(acc[DROW / 256].x, -acc[DROW / 256].y), w);
    }
    if (!seg_membrane(MODE) && a.half) {
      // outputs x and -x meet in the transpose buffer that the transform's last pass does not read
      if (t < a.M) {
        b0[t] = y[0];
        b0[256 + t] = y[1];
      }
      __syncthreads();
      const int hm = a.M / 2;
      if (t < hm) {
        y[0] = cadd(b0[hm + t], b0[hm - 1 - t]);
        y[1] = cadd(b0[256 + hm + t], b0[256 + hm - 1 - t]);
      }
    }
    if (t < (!seg_membrane(MODE) && a.half ? a.M / 2 : a.M)) {
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if (2 * p + e < a.rows) {
          C1[(int64_t)c1_row_re(t) * a.c1_stride + jl + e] = y[e].x;
          C1[(int64_t)c1_row_im(t) * a.c1_stride + jl + e] = y[e].y;
        }
    }
    __syncthreads();
  }
}

// Its tables: the convolution's input chirp on the grid points i, at D (i - i0)
// columns from the axis, and the outputs' (times 1 / 4096).
__global__ void k_dec_tables(int64_t npts, int n, double delta, double mc, double i0, float2* pre, float2* post) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < max(npts, (int64_t)n); t += stride) {
    const double x = (double)t;
    if (t < npts) pre[t] = cis_turns<float>(x * (delta * mc - 0.5 * delta * x));
    if (t < n) {
      float2 z = cis_turns<float>(delta * ((x - mc) * i0 - 0.5 * x * x));
      z.x *= 1.0f / SP;
      z.y *= 1.0f / SP;
      post[t] = z;
    }
  }
}

// Tables: pre(i), post(m)/L, convolution chirp v (length L), twiddles.
template <typename R>
__global__ void k_tables(int64_t N, int M, double msh, int64_t L, int64_t c, double kappa, double delta, int turns, void* pre,
                         void* post,
                         void* v, void* tw, int twN, void* twL) {
  using C = typename Cplx<R>::T;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < L; t += stride) {
    if (t < N) {
      const double di = (double)(t - c), ti = (double)t;
      const double ph = di * di * (0.5 * kappa) - (0.5 * delta) * (ti * ti) + delta * msh * ti;
      if (turns) reinterpret_cast<R*>(pre)[t] = (R)frac_turns(ph);  // the membrane walk adds its phase to them
      else reinterpret_cast<C*>(pre)[t] = cis_turns<R>(ph);
    }
    if (t < M) {
      const double tm = (double)t;
      const double ph = -(0.5 * delta) * tm * tm + delta * tm * (double)c - delta * msh * (double)c;
      C z = cis_turns<R>(ph);
      z.x /= (R)L; z.y /= (R)L;
      reinterpret_cast<C*>(post)[t] = z;
    }
    // chirp h_k = e^{i pi delta k^2}: index k for k < M, index L - k for 0 < k < N
    C h;
    h.x = 0; h.y = 0;
    int64_t k = -1;
    if (t < M) k = t;
    else if (t > L - N) k = L - t;
    if (k >= 0) {
      const double kk = (double)k;
      h = cis_turns<R>(0.5 * delta * kk * kk);
    }
    reinterpret_cast<C*>(v)[t] = h;
    if (t < twN) reinterpret_cast<C*>(tw)[t] = twiddle<R>(t, twN, -1.0f);
    if (t < 4096) reinterpret_cast<C*>(twL)[t] = twiddle<R>(t, L, -1.0f);
  }
}

template <typename R>
static size_t f1_smem(const RowArgs& a) {
  return sizeof(typename Cplx<R>::T) * (size_t)((a.L1 + 1) * a.B + a.L1 / 2);
}

}  // namespace

// D u <= 0.17 keeps the interpolation's error below 1.2e-7 (3e-8 at the ROI's
// edge); a deformed phase plate has its general per-sample transmission.
int bluestein_decimation(const Plan& P) {
  if (P.nd.n == 0 || (P.has_deform && P.levels >= 2)) return 0;
  const double u = M_PI * P.nd.delta * (P.nd.n - 1);
  return 32 * u <= 0.17 ? 32 : 16 * u <= 0.17 ? 16 : 0;
}

int64_t bluestein_wave(const Plan& P) {
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) cudaGetLastError();
  return (P.bs.dec ? 4 : 2) * (int64_t)sms;  // two CTAs to an SM, two decimated rows to a transform
}

DeformCoef deform_coef(const Plan& P) {
  DeformCoef c{};
  const fzp_deform& d = P.deform;
  const double k2 = 2.0 / P.lambda;  // metres -> turns of phase (phi / 2 pi = 2 w / lambda)
  const double kx = std::cos(d.theta) * P.dx / d.period, ky = std::sin(d.theta) * P.dx / d.period;
  c.kxh = (float)(std::rint(kx * 16384.0) / 16384.0);
  c.kyh = (float)(std::rint(ky * 16384.0) / 16384.0);
  c.kxl = (float)(kx - (double)c.kxh);
  c.kyl = (float)(ky - (double)c.kyh);
  c.amp2 = (float)(d.amp * k2);
  c.tq = (float)(d.taper * P.dx * P.dx / (P.R * P.R));
  c.zc = (float)std::cos(2.0 * M_PI * kx);
  c.zs = (float)std::sin(2.0 * M_PI * kx);
  c.z4 = (float)(4.0 * std::sin(M_PI * kx) * std::sin(M_PI * kx));
  c.n = d.n_ridges;
  for (int k = 0; k < d.n_ridges && k < 3; ++k) {
    const double nx = -std::sin(d.ridge_alpha[k]), ny = std::cos(d.ridge_alpha[k]);
    const double sg = d.ridge_width[k] / (2.0 * std::sqrt(2.0 * std::log(2.0)));
    c.nx[k] = (float)nx;
    c.ny[k] = (float)ny;
    c.pi_[k] = (float)(d.ridge_px[k] / P.dx);
    c.pj[k] = (float)(d.ridge_py[k] / P.dx);
    c.q[k] = (float)(P.dx * P.dx / (2.0 * sg * sg));
    c.h2[k] = (float)(d.ridge_h[k] * k2);
    c.rho[k] = (float)std::exp(-2.0 * (P.dx * P.dx / (2.0 * sg * sg)) * nx * nx);
    c.eta[k] = (float)-std::expm1(-2.0 * (P.dx * P.dx / (2.0 * sg * sg)) * nx * nx);
    const double across = std::fabs(nx) * P.dx;  // the full width along a row is width / across columns
    if (12.0 * across > d.ridge_width[k]) c.direct = 2;
    else if (64.0 * across > d.ridge_width[k]) c.direct = std::max(c.direct, 1);
  }
  if (c.z4 > 3.0f) c.direct = 2;
  return c;
}

namespace {

// The weights that take 16 columns' running sums to the grid points: the
// Lagrange polynomials of the six points on the columns of the chunk's part
// `sub`, fitted by least squares in the sums' own weights 1, m, m (m + 1) / 2,
// m (m + 1) (m + 2) / 6, m = 16 - k (a cubic follows a node's exponential over
// half of 16 columns to below 1e-8).
static void decimation_weights(int D, float2 (*T)[DTAPS][4]) {
  double B[16][4], Q[16][4], R[4][4] = {};
  for (int k = 0; k < 16; ++k) {
    const double m = 16 - k;
    B[k][0] = 1; B[k][1] = m; B[k][2] = m * (m + 1) / 2; B[k][3] = m * (m + 1) * (m + 2) / 6;
  }
  for (int e = 0; e < 4; ++e) {  // modified Gram-Schmidt
    for (int k = 0; k < 16; ++k) Q[k][e] = B[k][e];
    for (int f = 0; f < e; ++f) {
      for (int k = 0; k < 16; ++k) R[f][e] += Q[k][f] * Q[k][e];
      for (int k = 0; k < 16; ++k) Q[k][e] -= R[f][e] * Q[k][f];
    }
    for (int k = 0; k < 16; ++k) R[e][e] += Q[k][e] * Q[k][e];
    R[e][e] = std::sqrt(R[e][e]);
    for (int k = 0; k < 16; ++k) Q[k][e] /= R[e][e];
  }
  for (int sub = 0; sub < D / 16; ++sub)
    for (int q = 0; q < DTAPS; ++q) {
      double y[4] = {};
      for (int k = 0; k < 16; ++k) {
        const double xi = (16 * sub + k + 0.5) / D;  // from the point half a column before the chunk
        double w = 1;
        for (int p = 0; p < DTAPS; ++p)
          if (p != q) w *= (xi - (p - 2)) / (q - p);
        for (int e = 0; e < 4; ++e) y[e] += Q[k][e] * w;
      }
      for (int e = 3; e >= 0; --e) {
        for (int f = e + 1; f < 4; ++f) y[e] -= R[e][f] * y[f];
        y[e] /= R[e][e];
        T[sub][q][e] = make_float2((float)y[e], (float)y[e]);
      }
    }
}

// x turns in units of 2^-64, mod 1; *below: the next 32 bits
static uint64_t turns64(double x, uint32_t* below = nullptr) {
  x -= std::floor(x);
  const double t = std::ldexp(x, 64);
  const uint64_t k = t >= 18446744073709551616.0 ? 0 : (uint64_t)t;
  if (below) *below = (uint32_t)std::ldexp(t - std::floor(t), 32);
  return k;
}

static void (*dec_kernel(int mode, int D))(RowArgs) {
  switch (mode) {
    case SEG_FLAT: return D == 32 ? k_dec<SEG_FLAT, 32> : k_dec<SEG_FLAT, 16>;
    case SEG_LEVELS: return D == 32 ? k_dec<SEG_LEVELS, 32> : k_dec<SEG_LEVELS, 16>;
    case SEG_DIRECT: return D == 32 ? k_dec<SEG_DIRECT, 32> : k_dec<SEG_DIRECT, 16>;
    default: return D == 32 ? k_dec<SEG_MEMBRANE, 32> : k_dec<SEG_MEMBRANE, 16>;
  }
}

static RowArgs make_args(const Plan& P) {
  const Bluestein& b = P.bs;
  RowArgs a{};
  a.mg = P.mg;
  a.N = P.N; a.L = b.L; a.L1 = b.L1; a.L2 = b.L2; a.logL1 = ilog2(b.L1); a.logL2 = ilog2(b.L2); a.M = P.M;
  // F1 columns per block: a power of two, at most 16, F1 tile <= 64 KiB
  {
    const int64_t csz = P.precision == FZP_PREC_FP64 ? 16 : 8;
    int64_t B = 16;
    while (B > 1 && (B * (b.L1 + 1) + b.L1 / 2) * csz > 65536) B >>= 1;
    a.B = (int)std::min<int64_t>(B, b.L2);
    a.logB = ilog2(a.B);
  }
  a.has_deform = P.has_deform ? 1 : 0;
  a.def = P.deform;
  a.dx = P.dx; a.R = P.R; a.inv_lambda = 1.0 / P.lambda;
  if (P.has_deform) a.df = deform_coef(P);
  a.pre = b.d_pre; a.H = b.d_H; a.Z = b.d_Z; a.G = b.d_G; a.post = b.d_post; a.tw = b.d_tw;
  a.twN = (int)b.L2;
  a.twL = b.d_twL;
  a.c1_stride = P.chunk_rows;
  a.C1 = P.precision == FZP_PREC_FP64 ? (void*)P.d_C1d : (void*)P.d_C1;
  a.vin = b.d_tab;
  if (b.seg) a.ph = phase_rule(P, nullptr);
  a.S = b.S;
  a.nseg = b.nseg;
  a.col0 = b.col0;
  a.half = b.half ? 1 : 0;
  if (P.nd.n > 0) a.M = P.nd.n;
  else if (b.half) a.M = P.M + 1;
  if (b.dec) {
    const double mc = 0.5 * (P.nd.n - 1);
    a.Kc = turns64(0.5 * P.kappa, &a.Kc2);
    a.Kl = turns64(-P.nd.delta * (mc - P.nd.msh - (P.nd.even ? P.nd.n / 2 : 0)));
    a.cc2 = (uint32_t)((2 * a.Kc + 0x80000000ull) >> 32);
    std::copy(&b.T[0][0][0], &b.T[0][0][0] + 2 * DTAPS * 4, &a.T[0][0][0]);
  }
  return a;
}

template <typename R>
fzp_status layout_t(Plan& P, FormSizes* out) {
  using C = typename Cplx<R>::T;
  Bluestein& b = P.bs;
  b.seg = (sizeof(R) == 4 && P.conv_req != 1) ? 1 : 0;
  // columns from the axis on: flat plates whose outputs are symmetric about it
  // (nodes, or in FP64 the ROI's samples and x = +(M / 2) p besides)
  b.half = b.seg ? P.nd.even : sizeof(R) == 8 && bluestein_even(P);
  b.col0 = b.half ? P.c : 0;
  b.L = 1;
  while (b.L < P.N + P.M - 1) b.L <<= 1;
  b.L_full = b.L;
  if (!b.seg && b.half)
    for (b.L = 1; b.L < P.c + 1 + P.M;) b.L <<= 1;
  b.L2 = b.L < Traits<R>::L2MAX ? b.L : Traits<R>::L2MAX;
  b.L1 = b.L / b.L2;
  if (P.M > b.L2) return set_error(FZP_E_UNSUPPORTED, "M larger than the inner FFT length");
  // the F1 twiddles are read from the L2-entry table with stride L2 / L1 (a plan
  // that runs half the length is held to the same limit as fzp_plan_query)
  const int64_t L2_full = std::min<int64_t>(b.L_full, Traits<R>::L2MAX);
  if (b.L1 > b.L2 || b.L_full > L2_full * L2_full)
    return set_error(FZP_E_UNSUPPORTED, "FFT length %lld above %lld", (long long)b.L_full, (long long)L2_full * L2_full);
  if (b.seg) {
    // partitioned convolution: S + M - 1 <= 4096, S a multiple of 256 (at most 15 x 256)
    const int M = P.nd.n > 0 ? P.nd.n : P.M;  // outputs per row: the nodes, or the ROI samples
    b.S = 256 * std::min(15, (4097 - M) / 256);
    b.nseg = (P.N - b.col0 + b.S - 1) / b.S;
    b.dec = bluestein_decimation(P);
    if (b.dec) {
      decimation_weights(b.dec, b.T);
      // two rows to a transform: S + 5 + n < 2050, S a multiple of 32
      const int64_t chunks = (P.N - b.col0 + b.dec - 1) / b.dec, most = (DROW - M - DTAPS + 1) / 32 * 32;
      b.nseg = (chunks + most - 1) / most;
      b.S = (int)(((chunks + b.nseg - 1) / b.nseg + 31) / 32 * 32);
    }
    b.rows = P.chunk_rows;
    // decimated: a value per grid point, which on grids of up to 35 columns are
    // more than the columns (a block is at least 32 + 5 points)
    out->pre = sizeof(C) * (size_t)(b.dec ? b.nseg * b.S + DTAPS - 1 : P.N);
    out->H = sizeof(C) * (size_t)SP * (size_t)b.nseg;
    out->tab = sizeof(C) * (b.L + (int)b.L2 + std::max(P.M, M) + 4096);
    out->Z = 0;
    out->G = 0;
    out->X = (size_t)P.nd.ns * P.M * sizeof(double2);
    static std::atomic<uint64_t> attr_segt{0}, attr_seg[5];
    const void* kern[5] = {(const void*)k_seg<SEG_FLAT>, (const void*)k_seg<SEG_LEVELS>, (const void*)k_seg<SEG_MEMBRANE>,
                           (const void*)k_seg<SEG_GENERAL>, (const void*)k_seg<SEG_DIRECT>};
    for (int q = 0; q < 5; ++q) FZP_CUDA_TRY(smem_attr_once(kern[q], (int)SEG_SMEM, attr_seg[q]));
    static std::atomic<uint64_t> attr_dec[8];
    const int modes[4] = {SEG_FLAT, SEG_LEVELS, SEG_MEMBRANE, SEG_DIRECT};
    for (int q = 0; q < 8; ++q)
      FZP_CUDA_TRY(smem_attr_once((const void*)dec_kernel(modes[q / 2], q % 2 ? 32 : 16), (int)DEC_SMEM, attr_dec[q]));
    FZP_CUDA_TRY(smem_attr_once((const void*)k_seg_tables, (int)SEG_SMEM, attr_segt));
    return FZP_OK;
  }
  // rows per pass: requested, else a transform workspace of about 1 GiB
  const int64_t zbytes = (int64_t)sizeof(C) * b.L_full;  // (of the length that the plan reports)
  int64_t rows = P.row_batch_req > 0 ? P.row_batch_req : (1ll << 30) / zbytes;
  if (b.L_full <= Traits<R>::L2MAX) rows = P.row_batch_req > 0 ? P.row_batch_req : P.chunk_rows;
  b.rows = std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(rows, P.chunk_rows), 65535));
  const int twN = (int)b.L2, Mo = P.M + (b.half ? 1 : 0);
  out->pre = sizeof(C) * P.N;
  out->H = sizeof(C) * b.L;
  out->tab = sizeof(C) * (b.L + twN + Mo + 4096);
  out->Z = sizeof(C) * b.L * (b.L1 > 1 ? b.rows : 1);  // row 0 also serves the table build
  out->G = b.L1 > 1 ? sizeof(C) * b.L1 * Mo * b.rows : 0;
  // 64 KiB covers every FP32 case; FP64 at L1 = 4096 needs ~96 KiB
  static std::atomic<uint64_t> attr_f1{0}, attr_f2{0};
  FZP_CUDA_TRY(smem_attr_once((const void*)k_f1<R>, 200 * 1024, attr_f1));
  FZP_CUDA_TRY(smem_attr_once((const void*)k_f2<R>, (int)(sizeof(C) * Traits<R>::L2MAX), attr_f2));
  static std::atomic<uint64_t> attr_d16{0};
  FZP_CUDA_TRY(smem_attr_once((const void*)k_f2_d16, (int)D16_SMEM, attr_d16));
  return FZP_OK;
}

template <typename R>
fzp_status fill_tables_t(Plan& P, cudaStream_t s) {
  using C = typename Cplx<R>::T;
  Bluestein& b = P.bs;
  const int twN = (int)b.L2;
  b.d_tw = reinterpret_cast<C*>(b.d_tab) + b.L;
  b.d_post = reinterpret_cast<C*>(b.d_tw) + twN;
  // the outputs: the ROI's samples, or the nodes (all n of them)
  const bool nodes = P.nd.n > 0, half = b.half && !nodes;
  const int M = nodes ? P.nd.n : P.M + (half ? 1 : 0);
  const double delta = nodes ? P.nd.delta : P.delta;
  const double msh = nodes ? P.nd.msh + (P.nd.even ? P.nd.n / 2 : 0) : P.msh;
  b.d_twL = reinterpret_cast<C*>(b.d_post) + M;
  if (b.dec) {
    const double mc = 0.5 * (M - 1), i0 = 2.0 + (0.5 + (double)(P.c - b.col0)) / b.dec, dd = delta * b.dec;
    k_dec_tables<<<64, 256, 0, s>>>(b.nseg * b.S + DTAPS - 1, M, dd, mc, i0, reinterpret_cast<float2*>(b.d_pre),
                                    reinterpret_cast<float2*>(b.d_post));
    FZP_CUDA_TRY(cudaGetLastError());
    const unsigned g = (unsigned)std::min<int64_t>(b.nseg, 1024);
    k_seg_tables<<<g, STH, SEG_SMEM, s>>>(b.nseg, 0, b.S, b.S + DTAPS - 1, M, dd, reinterpret_cast<float2*>(b.d_H));
    FZP_CUDA_TRY(cudaGetLastError());
    P.launches += 2;
    return FZP_OK;
  }
  k_tables<R><<<1024, 256, 0, s>>>(half ? P.c + 1 : P.N, M, msh, b.L, half ? 0 : P.c, P.kappa, delta, b.seg && P.has_deform && P.levels < 2 ? 1 : 0, b.d_pre, b.d_post, b.d_tab, b.d_tw, twN,
                                   b.d_twL);
  FZP_CUDA_TRY(cudaGetLastError());
  if (b.seg) {
    const unsigned g = (unsigned)std::min<int64_t>(b.nseg, 1024);
    k_seg_tables<<<g, STH, SEG_SMEM, s>>>(b.nseg, b.col0, b.S, b.S, M, delta, reinterpret_cast<float2*>(b.d_H));
    FZP_CUDA_TRY(cudaGetLastError());
    P.launches += 2;
    return FZP_OK;
  }
  // H = FFT_L(v) in the [k1][k2] order: F1 (table mode) + F2 (forward only) into Z row 0, then copy.
  RowArgs a = make_args(P);
  a.j0 = 0;
  a.rows = 1;
  if (b.L1 > 1) k_f1<R><<<dim3((unsigned)(b.L2 / a.B), 1), 256, f1_smem<R>(a), s>>>(a, 1);
  if (sizeof(R) == 4 && b.L2 == RL) k_f2_r8<<<dim3((unsigned)b.L1, 1), R8T, 0, s>>>(a, 1);
  else if (sizeof(R) == 8 && b.L2 == SP) k_f2_d16<<<(unsigned)b.L1, STH, D16_SMEM, s>>>(a, 1);
  else k_f2<R><<<dim3((unsigned)b.L1, 1), 512, sizeof(C) * b.L2, s>>>(a, 1);
  FZP_CUDA_TRY(cudaGetLastError());
  FZP_CUDA_TRY(cudaMemcpyAsync(b.d_H, b.d_Z, sizeof(C) * b.L, cudaMemcpyDeviceToDevice, s));
  P.launches += b.L1 > 1 ? 3 : 2;
  return FZP_OK;
}

template <typename R>
fzp_status build_tables_t(Plan& P) {
  Bluestein& b = P.bs;
  FormSizes z;
  fzp_status st = layout_t<R>(P, &z);
  if (st != FZP_OK) return st;
  FZP_CUDA_TRY(cudaMalloc(&b.d_pre, z.pre));
  FZP_CUDA_TRY(cudaMalloc(&b.d_H, z.H));
  FZP_CUDA_TRY(cudaMalloc(&b.d_tab, z.tab));
  if (z.Z) FZP_CUDA_TRY(cudaMalloc(&b.d_Z, z.Z));
  if (z.G) FZP_CUDA_TRY(cudaMalloc(&b.d_G, z.G));
  P.device_bytes += z.pre + z.H + z.tab + z.Z + z.G;
  if (P.nd.n > 0) {
    FZP_CUDA_TRY(cudaMalloc(&P.nd.d_X, z.X));
    P.device_bytes += z.X;
    // the tables are built while the host factors the interpolation
    st = fill_tables_t<R>(P, 0);
    return st == FZP_OK ? nodes_upload(P) : st;
  }
  return fill_tables_t<R>(P, 0);
}

template <typename R>
fzp_status rows_t(Plan& P, int64_t j0, int64_t rows, bool octant, cudaStream_t s) {
  using C = typename Cplx<R>::T;
  const Bluestein& b = P.bs;
  RowArgs a = make_args(P);
  a.c1_j0 = j0;
  int sms = 0, dev = 0;
  FZP_CUDA_TRY(cudaGetDevice(&dev));
  FZP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (b.seg) {
    // resident CTAs only: each takes every gridDim.x-th row of the range
    int ctas_per_sm = 0;
    const int mode = P.has_deform ? (P.levels >= 2 ? SEG_GENERAL : a.df.direct ? SEG_DIRECT : SEG_MEMBRANE)
                                  : (P.levels >= 2 ? SEG_LEVELS : SEG_FLAT);
    a.octant = octant ? 1 : 0;
    void (*kern)(RowArgs) = mode == SEG_FLAT       ? k_seg<SEG_FLAT>
                            : mode == SEG_LEVELS   ? k_seg<SEG_LEVELS>
                            : mode == SEG_MEMBRANE ? k_seg<SEG_MEMBRANE>
                            : mode == SEG_DIRECT   ? k_seg<SEG_DIRECT>
                                                   : k_seg<SEG_GENERAL>;
    const size_t smem = b.dec ? DEC_SMEM : SEG_SMEM;
    if (b.dec) kern = dec_kernel(mode, b.dec);
    FZP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas_per_sm, kern, STH, smem));
    if (ctas_per_sm < 1) ctas_per_sm = 1;
    a.j0 = j0;
    a.rows = rows;
    const int64_t grid = std::min<int64_t>(b.dec ? (rows + 1) / 2 : rows, (int64_t)ctas_per_sm * sms);
    prof_begin(P, s);
    kern<<<(unsigned)grid, STH, smem, s>>>(a);
    prof_end(P, s);
    P.launches += 1;
    FZP_CUDA_TRY(cudaGetLastError());
    return FZP_OK;
  }
  for (int64_t r0 = 0; r0 < rows; r0 += b.rows) {
    const int64_t rb = std::min<int64_t>(b.rows, rows - r0);
    a.j0 = j0 + r0;
    a.rows = rb;
    const unsigned d16_grid = (unsigned)std::min<int64_t>(rb * b.L1, sms);
    if (b.L1 > 1) {
      k_f1<R><<<dim3((unsigned)(b.L2 / a.B), (unsigned)rb), 256, f1_smem<R>(a), s>>>(a, 0);
      prof_begin(P, s);
      if (sizeof(R) == 4 && b.L2 == RL) k_f2_r8<<<dim3((unsigned)b.L1, (unsigned)rb), R8T, 0, s>>>(a, 0);
      else if (sizeof(R) == 8 && b.L2 == SP) k_f2_d16<<<d16_grid, STH, D16_SMEM, s>>>(a, 0);
      else k_f2<R><<<dim3((unsigned)b.L1, (unsigned)rb), 512, sizeof(C) * b.L2, s>>>(a, 0);
      prof_end(P, s);
      k_f3<R><<<dim3((unsigned)((a.M + 31) / 32), (unsigned)((rb + 31) / 32)), 256, 0, s>>>(a);
      P.launches += 3;
    } else {
      prof_begin(P, s);
      if (sizeof(R) == 4 && b.L2 == RL) k_f2_r8<<<dim3(1, (unsigned)rb), R8T, 0, s>>>(a, 0);
      else if (sizeof(R) == 8 && b.L2 == SP) k_f2_d16<<<d16_grid, STH, D16_SMEM, s>>>(a, 0);
      else k_f2<R><<<dim3(1, (unsigned)rb), 512, sizeof(C) * b.L2, s>>>(a, 0);
      prof_end(P, s);
      P.launches += 1;
    }
  }
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

__global__ void k_mask(MaskGeom mg, int64_t N, int64_t j0, int64_t rows, uint8_t* out) {
  const int64_t total = rows * N;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t / N, i = t % N;
    const int64_t dj = j0 + r - mg.c, di = i - mg.c, sq = dj * dj + di * di;
    if (mg.levels >= 2) out[t] = sq > mg.sR ? 0 : (uint8_t)(1 + zone_of(sq, mg) % mg.levels);
    else out[t] = mask_open(dj, di, mg) ? 1 : 0;
  }
}

// The same through the walked zone phase and its exact rule, as the partitioned row
// pass makes its masks: a thread per 16 columns from col0, mirrored to the columns
// left of the axis where the row pass runs the others only.
__global__ void k_mask_walk(MaskGeom mg, PhaseRule ph, int64_t N, int64_t j0, int64_t rows, int64_t col0, uint8_t* out) {
  const int64_t chunks = (N - col0 + 15) / 16, total = rows * chunks;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t / chunks, x = col0 + 16 * (t % chunks), dj = j0 + r - mg.c, dj2 = dj * dj, di0 = x - mg.c;
    uint32_t lv[4] = {0u, 0u, 0u, 0u}, w = 0u;
    // (a chunk that misses the disc is closed, as in the row pass)
    const int64_t near = di0 > 0 ? di0 : di0 + 15 < 0 ? di0 + 15 : 0;
    const bool meets = dj2 + near * near <= mg.sR;
    if (meets) {
      if (mg.levels >= 2) chunk_levels(di0, dj2, mg, ph, lv);
      else if (!walk_bits16(walk16(di0, dj2, ph), ph, w)) w = chunk_bits(x, dj2, mg);
    }
    for (int k = 0; k < 16 && x + k < N; ++k) {
      const int64_t di = di0 + k;
      uint8_t v = 0;
      if (meets && dj2 + di * di <= mg.sR) v = mg.levels >= 2 ? (uint8_t)(1 + ((lv[k >> 2] >> (8 * (k & 3))) & 0xFFu)) : (uint8_t)((w >> k) & 1u);
      out[r * N + x + k] = v;
      if (col0 > 0 && mg.c - di >= 0) out[r * N + mg.c - di] = v;
    }
  }
}

}  // namespace

fzp_status bluestein_mask(Plan& P, int64_t j0, int64_t rows, uint8_t* out, cudaStream_t s) {
  // a deformed phase plate's row pass takes the zone rule per sample
  if (P.bs.seg && !(P.has_deform && P.levels >= 2))
    k_mask_walk<<<1024, 256, 0, s>>>(P.mg, phase_rule(P, nullptr), P.N, j0, rows, P.bs.col0, out);
  else
    k_mask<<<1024, 256, 0, s>>>(P.mg, P.N, j0, rows, out);
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status bluestein_build_tables(Plan& P) {
  return P.precision == FZP_PREC_FP64 ? build_tables_t<double>(P) : build_tables_t<float>(P);
}

fzp_status bluestein_layout(Plan& P, FormSizes* out) {
  return P.precision == FZP_PREC_FP64 ? layout_t<double>(P, out) : layout_t<float>(P, out);
}

fzp_status bluestein_fill_tables(Plan& P, cudaStream_t s) {
  return P.precision == FZP_PREC_FP64 ? fill_tables_t<double>(P, s) : fill_tables_t<float>(P, s);
}

fzp_status bluestein_rows(Plan& P, int64_t j0, int64_t rows, bool octant, cudaStream_t stream) {
  P.dominant = P.precision == FZP_PREC_FP64 ? "bluestein_f2<double>"
               : P.bs.dec                       ? "k_dec (partitioned convolution, decimated rows)"
               : P.bs.seg                       ? "k_seg (partitioned convolution)"
                                                : "bluestein_f2<float>";
  return P.precision == FZP_PREC_FP64 ? rows_t<double>(P, j0, rows, false, stream) : rows_t<float>(P, j0, rows, octant, stream);
}

}  // namespace fzp
