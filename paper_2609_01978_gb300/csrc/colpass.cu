// colpass.cu -- column pass, cross-stripe FP64 accumulation and output
// epilogue (Fig. 2 Stage 3 "column czt * dx_in^2/(lambda0 f)"; Fig. 18 Stage 4
// "output chirp and Fresnel prefactor").
//
//   Uacc[n, m] += sum_{j in rows} K[n, j] C[j, m]            (column pass)
//   U[n, m]     = Pre e^{i pi (x_m^2 + y_n^2)/(lambda f)} Uacc[n, m],
//   Pre         = e^{i k f} dx^2 / (i lambda f)              (Eq. 2)
//
// K[n, j] = exp(2 pi i (A_j - n B_j)) with A_j = dj^2 kappa/2 + msh dj delta and
// B_j = dj delta (turns, dj = j - c).  A_j and B_j are reduced in FP64 once per
// row j; for the FP32 path B_j is split as hi + lo with hi a multiple of 2^-14
// so that n * hi is exact in FP32 for n < 1024.
#include <algorithm>
#include <cmath>

#include "fzp_internal.cuh"
#include "sums.cuh"
#include "tc_ptx.cuh"

namespace fzp {
namespace {

constexpr int TN = 64, TM = 64, TJ = 16, PJ = 128;  // output tiles of 64 (48: NA = 3 outputs per thread and side)

constexpr int CZ = 4;        // blocks of a cluster along the rows
constexpr int BLOCKS = 288;  // two per SM as far as clusters of four fit into the GPCs (of 304 in eights a second wave ran)
// Clusters: where the tile of sums fits in static shared memory.
template <typename R, int NA> constexpr bool col_clusters = sizeof(R) == 4 || NA < 4;

struct ColArgs {
  int64_t c, j0, rows, c1_stride;
  int64_t jc;     // rows per block of the grid's z
  int kind;       // RowKind: the row's kernel K(dj), K(dj) + K(-dj) or K(-dj)
  int slices;       // images of C1 to be summed, slice_off values apart
  int64_t slice_off;
  int64_t sin_off;  // > 0: C1 holds the rows of Re T and, sin_off values on, of Im T
  const float2* E;
  int64_t estride;
  int M, ny;      // outputs per row (m) and of the column pass (n)
  double kappa, delta;
  double msh;     // ROI (or node) shift in pitches: y_n = (n - msh) p
  double wr, wi;  // weight of this pass's field (1, 0 for a single-pass plate)
  int tri;        // > 0: the field is its own transpose; blockIdx.x counts the tiles m >= n of tri x tri
};

template <typename R> struct RowPhase;
template <> struct RowPhase<float> { float fa, hi, lo; };
template <> struct RowPhase<double> { double a, b; };

__device__ __forceinline__ void row_phase(const ColArgs& g, double dj, RowPhase<float>& rp) {
  const double A = dj * dj * (0.5 * g.kappa) + g.msh * dj * g.delta;
  const double fb = frac_turns(dj * g.delta);
  const double hi = rint(fb * 16384.0) / 16384.0;
  rp.fa = (float)frac_turns(A);
  rp.hi = (float)hi;
  rp.lo = (float)(fb - hi);
}
__device__ __forceinline__ void row_phase(const ColArgs& g, double dj, RowPhase<double>& rp) {
  rp.a = frac_turns(dj * dj * (0.5 * g.kappa) + g.msh * dj * g.delta);
  rp.b = frac_turns(dj * g.delta);
}

__device__ __forceinline__ float2 kern(const RowPhase<float>& rp, int n) {
  const float x = (float)n * rp.hi;
  const float t = rp.fa - (x - floorf(x)) - (float)n * rp.lo;
  float s, c;
  sincospif(2.0f * t, &s, &c);
  return make_float2(c, s);
}
__device__ __forceinline__ double2 kern(const RowPhase<double>& rp, int n) {
  return cis_turns_d(rp.a - (double)n * rp.b);
}

// FP32, a row and its mirror image: K(dj) + K(-dj) = e^{i pi kappa dj^2} 2 cos(2 pi
// (n - msh) dj delta), one cosine instead of two sines and cosines.  The first
// part of a row's phases is the cosine's (msh dj delta, and B split as above),
// the second the exponential and the factor (the axis row: 1).
__device__ __forceinline__ void row_pair(const ColArgs& g, double dj, bool second, RowPhase<float>& rp) {
  if (second) {
    const float2 e = cis_turns_f(dj * dj * (0.5 * g.kappa));
    rp.fa = e.x;
    rp.hi = e.y;
    rp.lo = dj == 0.0 ? 1.0f : 2.0f;
    return;
  }
  row_phase(g, dj, rp);
  rp.fa = (float)frac_turns(g.msh * dj * g.delta);
}
__device__ __forceinline__ void row_pair(const ColArgs&, double, bool, RowPhase<double>&) {}
__device__ __forceinline__ float2 kern_pair(const RowPhase<float>& rp, const RowPhase<float>& e, int n) {
  const float x = (float)n * rp.hi;
  const float c = e.lo * cospif(2.0f * (rp.fa - (x - floorf(x)) - (float)n * rp.lo));
  return make_float2(c * e.fa, c * e.hi);
}
__device__ __forceinline__ double2 kern_pair(const RowPhase<double>&, const RowPhase<double>&, int) { return make_double2(0.0, 0.0); }

// Factors of a row's kernel values in an output tile from n0: q < 8: e^{-2 pi i
// (n0 + 8 q) B}; q < 16: e^{-2 pi i (q - 8) B}; 16, 17: e^{2 pi i A} at dj and, of
// a folded row, at -dj (where B changes sign: the conjugate product).
__device__ __forceinline__ double2 factor(int q, int n0, const RowPhase<double>& r0, const RowPhase<double>& r1, bool folded) {
  if (q == 17 && !folded) return make_double2(0.0, 0.0);
  return cis_turns_d(q < 8 ? -(double)(n0 + 8 * q) * r0.b : q < 16 ? -(double)(q - 8) * r0.b : q == 16 ? r0.a : r1.a);
}
__device__ __forceinline__ float2 factor(int, int, const RowPhase<float>&, const RowPhase<float>&, bool) {
  return make_float2(0.f, 0.f);  // (FP32 evaluates its sines)
}

__device__ __forceinline__ float2 peer_load(uint32_t addr, float2) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ double2 peer_load(uint32_t addr, double2) {
  double2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr) : "memory");
  return v;
}

// grid (M/TM, M/TN, ceil(rows/jc)); 256 threads; each thread 4 n x 4 m outputs.
// TAB: the kernel's columns from a table E [n][estride] instead of their phase.
// The blocks' sums meet in Uacc: in clusters of CZ along the rows, block k adds up
// its part of the tile over the cluster through distributed shared memory first
// (sum4: with what the FP32 additions round off, as if in FP64).
// Without that, 304 blocks put FP64 atomics on the same 8,192 values.  The next
// tile of C1 loads during the products.  18,965 rows, 64 x 64 nodes: 56 us without
// clusters and prefetch and with two sine pairs per folded kernel value, 49 with
// clusters of eight and prefetch, 33 with clusters of four and one cosine (issue
// slots 28 -> 35 % busy; the waits left are loads and the barriers of 16-row tiles),
// 35 with sum4 in place of FP32 additions.
// FP64, 2,529 rows, 129 x 129 outputs, bound by the FP64 pipe: 0.46 ms, with the
// tiles on and above the diagonal only a propagation takes 0.09 ms less.
// Large grids (FP32 outputs that are ROI samples) run it at 80 registers, three blocks
// to an SM (MINB) instead of two of 111: a membrane of 8,001 rows on 1024^2 2,678 us before
// the prefetch, 3,077 with it, 2,654 at 80 registers, 2,470 with balanced waves.
template <typename R, bool TAB = false, int NA = 4, int MINB = 1>
__global__ void __launch_bounds__(256, MINB) k_colpass(ColArgs g, const R* __restrict__ C1, double2* __restrict__ Uacc) {
  using C = typename Cplx<R>::T;
  constexpr int TN = 16 * NA, TM = 16 * NA;
  constexpr int TILE = TJ * (TN + 1), POOL = col_clusters<R, NA> && TN * TM > 2 * TILE ? TN * TM : 2 * TILE;
  __shared__ __align__(16) C pool[POOL];
  C(*sK)[TN + 1] = reinterpret_cast<C(*)[TN + 1]>(pool);
  C(*sC)[TM + 1] = reinterpret_cast<C(*)[TM + 1]>(pool + TILE);
  // phases of 128 rows at a time (they are FP64, at two operations per clock and
  // SM): of dj (mirrored rows: -dj) and, folded, of -dj
  __shared__ RowPhase<R> sP[2][PJ];
  // FP64: e^{-2 pi i n B} as products of 8 + 8 phasors per row (an FP64 sine per
  // element took as long as the products), and the rows' e^{2 pi i A}, A at dj and -dj
  constexpr bool FACT = sizeof(R) == 8 && !TAB, PAIR = sizeof(R) == 4 && !TAB;
  __shared__ C sF[FACT ? TJ : 1][18];
  int bx = blockIdx.x, by = blockIdx.y;
  if (g.tri) {
    for (; bx >= g.tri - by; ++by) bx -= g.tri - by;
    bx += by;
  }
  const int m0 = bx * TM, n0 = by * TN;
  const int64_t jb = (int64_t)blockIdx.z * g.jc;
  const int64_t je = jb + g.jc < g.rows ? jb + g.jc : g.rows;
  const int tid = threadIdx.x;
  const int tn = tid >> 4, tm = tid & 15;  // 16 x 16 threads, 4 x 4 outputs each
  // outputs of this warp's rows and of the tile's columns (uniform per warp)
  const int na = min(NA, max(0, (g.ny - n0 - (tn & ~1) + 15) / 16)), nb = min(NA, (g.M - m0 + 15) / 16);
  C acc[NA][NA];
#pragma unroll
  for (int a = 0; a < NA; ++a)
#pragma unroll
    for (int b = 0; b < NA; ++b) { acc[a][b].x = 0; acc[a][b].y = 0; }
  constexpr int CQ = TJ * TM / 256;
  C next[CQ];
  auto load_c = [&](int64_t j) {
#pragma unroll
    for (int q = 0; q < CQ; ++q) {
      const int t = tid + 256 * q, jj = t % TJ, m = m0 + t / TJ;
      C v;
      v.x = 0; v.y = 0;
      if (j + jj < je && m < g.M) {
        const int64_t re = (int64_t)c1_row_re(m) * g.c1_stride + j + jj, im = (int64_t)c1_row_im(m) * g.c1_stride + j + jj;
#pragma unroll 1
        for (int sl = 0; sl < g.slices; ++sl) {
          const R* S = C1 + sl * g.slice_off;
          v.x += S[re];
          v.y += S[im];
          if (g.sin_off > 0) {  // K (Re T + i Im T)
            v.x -= S[g.sin_off + im];
            v.y += S[g.sin_off + re];
          }
        }
      }
      next[q] = v;
    }
  };
  load_c(jb);
  for (int64_t j = jb; j < je; j += TJ) {
    const int pj = (int)(j - jb) & (PJ - 1);
    if (!TAB && pj == 0) {
      const int r = tid & (PJ - 1);
      if (j + r < je && (tid < PJ || g.kind == ROWS_FOLDED)) {
        const double dj = (double)(g.j0 + j + r - g.c);
        RowPhase<R> rp;
        if (PAIR && g.kind == ROWS_FOLDED) row_pair(g, dj, tid >= PJ, rp);
        else row_phase(g, (tid >= PJ) != (g.kind == ROWS_MIRRORED) ? -dj : dj, rp);
        sP[tid / PJ][r] = rp;
      }
    }
    // C tile: TJ rows x TM columns (j contiguous in C1), loaded during the last tile's products
#pragma unroll
    for (int q = 0; q < CQ; ++q) {
      const int t = tid + 256 * q;
      sC[t % TJ][t / TJ] = next[q];
    }
    __syncthreads();
    if (FACT) {
      for (int t = tid; t < TJ * 18; t += 256) {
        const int jj = t / 18, q = t % 18;
        const RowPhase<R> r0 = sP[0][pj + jj], r1 = sP[1][pj + jj];
        if (j + jj < je) sF[jj][q] = factor(q, n0, r0, r1, g.kind == ROWS_FOLDED && g.j0 + j + jj != g.c);
      }
      __syncthreads();
    }
    for (int t = tid; t < TJ * TN; t += 256) {
      const int jj = TAB ? t % TJ : t / TN, nn = TAB ? t / TJ : t % TN;
      C k;
      k.x = 0; k.y = 0;
      if (TAB && j + jj < je) {
        const float2 e = __ldg(g.E + (int64_t)(n0 + nn) * g.estride + j + jj);
        k.x = e.x;
        k.y = e.y;
      } else if (FACT && j + jj < je) {
        C e = cmul(sF[jj][nn >> 3], sF[jj][8 + (nn & 7)]);
        k = cmul(sF[jj][16], e);
        e.y = -e.y;
        k = cadd(k, cmul(sF[jj][17], e));
      } else if (PAIR && g.kind == ROWS_FOLDED && j + jj < je) {
        k = kern_pair(sP[0][pj + jj], sP[1][pj + jj], n0 + nn);
      } else if (j + jj < je) {
        k = kern(sP[0][pj + jj], n0 + nn);
      }
      sK[jj][nn] = k;
    }
    __syncthreads();
    load_c(j + TJ);
    if (na == 0) {
    } else if (na < NA || nb < NA) {  // an edge tile: the outputs it has
#pragma unroll 1
      for (int jj = 0; jj < TJ; ++jj)
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
          for (int b = 0; b < NA; ++b)
            if (a < na && b < nb) {
              const C kv = sK[jj][tn + 16 * a], cv = sC[jj][tm + 16 * b];
              acc[a][b].x = fma(kv.x, cv.x, fma(-kv.y, cv.y, acc[a][b].x));
              acc[a][b].y = fma(kv.x, cv.y, fma(kv.y, cv.x, acc[a][b].y));
            }
    } else
#pragma unroll 4
    for (int jj = 0; jj < TJ; ++jj) {
      C kv[NA], cv[NA];
#pragma unroll
      for (int a = 0; a < NA; ++a) kv[a] = sK[jj][tn + 16 * a];
#pragma unroll
      for (int b = 0; b < NA; ++b) cv[b] = sC[jj][tm + 16 * b];
#pragma unroll
      for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int b = 0; b < NA; ++b) {
          acc[a][b].x = fma(kv[a].x, cv[b].x, fma(-kv[a].y, cv[b].y, acc[a][b].x));
          acc[a][b].y = fma(kv[a].x, cv[b].y, fma(kv[a].y, cv[b].x, acc[a][b].y));
        }
    }
    __syncthreads();
  }
  auto add = [&](int n, int m, double ux, double uy) {
    if (n >= g.ny || m >= g.M) return;
    if (g.wi != 0.0 || g.wr != 1.0) {
      const double t = g.wr * ux - g.wi * uy;
      uy = g.wr * uy + g.wi * ux;
      ux = t;
    }
    atomicAdd(&Uacc[(int64_t)n * g.M + m].x, ux);
    atomicAdd(&Uacc[(int64_t)n * g.M + m].y, uy);
  };
  uint32_t cz = 1, rank = 0;
  if (col_clusters<R, NA>) asm("mov.u32 %0, %%cluster_nctarank;\n mov.u32 %1, %%cluster_ctarank;" : "=r"(cz), "=r"(rank));
  if (cz == CZ) {
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
      for (int b = 0; b < NA; ++b) pool[(tn + 16 * a) * TM + tm + 16 * b] = acc[a][b];
    tc::cluster_sync();
    uint32_t peer[CZ];
#pragma unroll
    for (int q = 0; q < CZ; ++q) peer[q] = tc::mapa(tc::smem_u32(pool), q);
    constexpr int PART = TN * TM / CZ;
    for (int e = (int)rank * PART + tid; e < ((int)rank + 1) * PART; e += 256) {
      R x[CZ], y[CZ];
#pragma unroll
      for (int q = 0; q < CZ; ++q) {
        const C v = peer_load(peer[q] + (uint32_t)(e * sizeof(C)), C{});
        x[q] = v.x;
        y[q] = v.y;
      }
      add(n0 + e / TM, m0 + e % TM, sum4(x), sum4(y));
    }
    tc::cluster_sync();  // the peers may still be reading this block's tile
    return;
  }
#pragma unroll
  for (int a = 0; a < NA; ++a)
#pragma unroll
    for (int b = 0; b < NA; ++b) add(n0 + tn + 16 * a, m0 + tm + 16 * b, (double)acc[a][b].x, (double)acc[a][b].y);
}

template <typename R, bool TAB = false, int NA = 4, int MINB = 1>
fzp_status run_colpass(const ColArgs& g, unsigned tx, unsigned ty, const R* C1, double2* Uacc, cudaStream_t s) {
  unsigned tz = (unsigned)((g.rows + g.jc - 1) / g.jc);
  const bool clusters = col_clusters<R, NA> && tz >= CZ;
  if (clusters) tz = (tz + CZ - 1) / CZ * CZ;  // (blocks past the last row add zeros)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tx, ty, tz);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = CZ;
  cfg.attrs = attr;
  cfg.numAttrs = clusters ? 1 : 0;
  FZP_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_colpass<R, TAB, NA, MINB>, g, C1, Uacc));
  return FZP_OK;
}

__global__ void k_epilogue(int M, double msh, double p, double lf, double f_over_lambda, double amp,
                           int evenx, int eveny, int tri, const double2* __restrict__ Uacc, double2* __restrict__ out,
                           int accumulate) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= M * M) return;
  const int n = t / M, m = t % M;
  const double xm = (double)m - msh, yn = (double)n - msh;
  // e^{ikf} (1/i) e^{i pi (x^2 + y^2)/(lambda f)}: turns f/lambda - 1/4 + (x^2 + y^2)/(2 lambda f)
  const double ph = frac_turns(f_over_lambda) - 0.25 + (xm * xm + yn * yn) * (p * p) / (2.0 * lf);
  double2 w = cis_turns_d(ph);
  w.x *= amp;
  w.y *= amp;
  // even: the accumulator holds the samples x >= 0, |m - M/2| of them from the axis
  const int h = M / 2;
  int un = eveny ? abs(n - h) : n, um = evenx ? abs(m - h) : m;
  if (tri > 0 && un / tri > um / tri) {  // the accumulator's tiles of `tri` below the diagonal are not filled
    const int x = un;
    un = um;
    um = x;
  }
  const double2 u = Uacc[(int64_t)un * (evenx ? h + 1 : M) + um];
  double2 v = make_double2(w.x * u.x - w.y * u.y, w.x * u.y + w.y * u.x);
  if (accumulate) {
    v.x += out[t].x;
    v.y += out[t].y;
  }
  out[t] = v;
}

__global__ void k_intensity(int64_t count, const double2* __restrict__ U, double* __restrict__ I) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < count) I[t] = U[t].x * U[t].x + U[t].y * U[t].y;
}

}  // namespace

fzp_status column_pass(Plan& P, int64_t j0, int64_t rows, RowKind kind, cudaStream_t s) {
  const bool nodes = P.nd.n > 0;
  ColArgs g{};
  g.c = P.form == FZP_FORM_DENSE && P.fold ? 0 : P.c;
  g.j0 = j0;
  g.rows = rows;
  g.c1_stride = P.c1_stride;
  g.kind = kind;
  // FP64 on the samples x >= 0: a grid from the axis on
  const bool even = !nodes && bluestein_even(P);
  g.M = nodes ? P.nd.ns : even ? P.M / 2 + 1 : P.M;
  g.ny = nodes ? (P.nd.yfull ? P.nd.n : P.nd.ns) : P.nd.yfull ? P.M : g.M;
  g.kappa = P.kappa;
  g.delta = nodes ? P.nd.delta : P.delta;
  g.msh = !nodes ? (even && !P.nd.yfull ? 0.0 : P.msh) : P.nd.yfull ? 0.5 * (P.nd.n - 1) : P.nd.msh;
  g.wr = 1.0;
  if (P.pass_index >= 0) {
    g.wr = P.passes[P.pass_index].wr;
    g.wi = P.passes[P.pass_index].wi;
  }
  g.slices = P.nd.slices;
  g.slice_off = P.nd.slice_elems;
  if (nodes_two_masks(P)) g.sin_off = 128 * P.c1_stride;
  // rows per block: 2048, fewer where that leaves the GPU idle (few output tiles)
  // FP64 on M / 2 + 1 outputs: tiles of 48 (129 = 3 x 43: nine equal tiles, where
  // tiles of 64 are four full ones and five slivers that share SMs with them)
  const int T = even ? 48 : TM;
  const int tx = (g.M + T - 1) / T, ty = (g.ny + T - 1) / T;
  // a symmetric field: the tiles on and above the diagonal (k_epilogue mirrors)
  const bool tri = P.nd.tri && tx == ty;
  g.tri = tri ? tx : 0;
  const int64_t tiles = tri ? (int64_t)tx * (tx + 1) / 2 : (int64_t)tx * ty;
  // As many blocks a tile as are resident at once (8 x 8 tiles: four; with the quotient
  // not rounded down five, which clusters made eight: 8,001 rows in BF16 877 -> 1,045 us).
  // More tiles than half of the blocks: unevenly long blocks, unless the second of a tile
  // had too few rows to be worth its sums (101 rows of 16 x 16 tiles: 50 us in one block
  // a tile, 63 in two).
  const int64_t fit = BLOCKS / tiles, share = fit > 1 ? (rows + fit - 1) / fit : rows * tiles / BLOCKS;
  g.jc = std::min<int64_t>(2048, std::max<int64_t>(2 * TJ, (share + TJ - 1) / TJ * TJ));
  if (fit <= 1 && rows > g.jc && rows < g.jc + 64 && rows <= 2048) g.jc = rows;
  // several waves: three blocks to an SM, as many a tile as leave the last wave fullest
  const int64_t least = (rows + 2047) / 2048;
  const bool many = !nodes && P.precision != FZP_PREC_FP64 && tiles * least > BLOCKS;
  if (many) {
    int64_t best = INT64_MAX;
    for (int64_t z = least; z <= least + 8; ++z) {
      const int64_t jc = ((rows + z - 1) / z + TJ - 1) / TJ * TJ, run = z < CZ ? z : (z + CZ - 1) / CZ * CZ;
      const int64_t t = (tiles * run + BLOCKS * 3 / 2 - 1) / (BLOCKS * 3 / 2) * jc;
      if (t < best) {
        best = t;
        g.jc = jc;
      }
    }
  }
  P.launches += 1;
  const unsigned gx = (unsigned)(tri ? tiles : tx), gy = (unsigned)(tri ? 1 : ty);
  return even                           ? run_colpass<double, false, 3>(g, gx, gy, P.d_C1d, P.d_Uacc, s)
         : P.precision == FZP_PREC_FP64 ? run_colpass<double>(g, gx, gy, P.d_C1d, P.d_Uacc, s)
         : many                         ? run_colpass<float, false, 4, 3>(g, gx, gy, P.d_C1, P.d_Uacc, s)
                                        : run_colpass<float>(g, gx, gy, P.d_C1, P.d_Uacc, s);
}

fzp_status column_pass_table(Plan& P, const void* E, int64_t rows, int64_t estride, cudaStream_t s) {
  ColArgs g{};
  g.rows = rows;
  g.c1_stride = P.c1_stride;
  g.M = P.nd.ns;
  g.wr = 1.0;
  g.slices = 1;
  g.sin_off = 2 * P.nd.ns * P.c1_stride;
  g.E = reinterpret_cast<const float2*>(E);
  g.estride = estride;
  g.ny = g.M;
  const int t = g.M / TM;
  g.jc = std::min<int64_t>(2048, std::max<int64_t>(2 * TJ, (rows * t * t / BLOCKS + TJ - 1) / TJ * TJ));
  P.launches += 1;
  return run_colpass<float, true>(g, t, t, P.d_C1, P.d_Uacc, s);
}

fzp_status column_pass_zoom(Plan& P, int64_t rows, double lz, cudaStream_t s) {
  const NodeSet& z = P.nd;
  ColArgs g{};
  g.c = rows / 2;
  g.rows = rows;
  g.c1_stride = P.c1_stride;
  g.M = z.ns;
  g.kappa = P.dx2 / lz;
  g.delta = z.h * P.p * P.dx / lz;
  g.msh = z.yfull ? 0.5 * (z.n - 1) : z.msh;
  g.wr = 1.0;
  g.slices = 1;
  g.sin_off = 2 * z.ns * P.c1_stride;
  g.ny = z.yfull ? z.n : z.ns;
  const int tx = g.M / TM, ty = g.ny / TN;
  g.jc = std::min<int64_t>(2048, std::max<int64_t>(2 * TJ, (rows * tx * ty / BLOCKS + TJ - 1) / TJ * TJ));
  P.launches += 1;
  return run_colpass<float>(g, tx, ty, P.d_C1, P.d_Uacc, s);
}

fzp_status epilogue(Plan& P, void* d_field, int accumulate, cudaStream_t s) {
  const double lf = P.lambda * P.f;
  const int count = P.M * P.M;
  const bool even = bluestein_even(P);
  k_epilogue<<<(count + 255) / 256, 256, 0, s>>>(P.M, P.msh, P.p, lf, P.f / P.lambda, P.dx2 / lf, even ? 1 : 0,
                                                 even && !P.nd.yfull ? 1 : 0, P.nd.tri ? (even ? 48 : TM) : 0, P.d_Uacc,
                                                 reinterpret_cast<double2*>(d_field), accumulate);
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status epilogue_z(Plan& P, void* d_field, int accumulate, double z, cudaStream_t s) {
  const double lz = P.lambda * z;
  const int count = P.M * P.M;
  k_epilogue<<<(count + 255) / 256, 256, 0, s>>>(P.M, P.msh, P.p, lz, P.f / P.lambda, P.dx2 / lz, 0, 0, 0, P.d_Uacc,
                                                 reinterpret_cast<double2*>(d_field), accumulate);
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status intensity(Plan& P, const void* d_field, void* d_I, cudaStream_t s) {
  const int64_t count = (int64_t)P.M * P.M;
  k_intensity<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(count, reinterpret_cast<const double2*>(d_field),
                                                               reinterpret_cast<double*>(d_I));
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

}  // namespace fzp
