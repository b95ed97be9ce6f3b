// nodes.cu -- form (b) on interpolation nodes: the dense contraction evaluated
// at as many focal-plane points as the aperture can distinguish.
//
// The field on the ROI is band limited: Eq. 2 without its output chirp is a
// Fourier sum over the aperture disc, so along x it has about
//   d = M p 2R / (lambda f)
// degrees of freedom on the ROI's M samples (64 of 512 at the usual pitch
// lambda f/# / 8).  The contraction U = K T K^T therefore runs on n uniform
// nodes x_k across the ROI (and a margin of a quarter of it), n = 64, 128 or
// 256 with d at most 0.56 n, 0.62 n, 0.66 n, and the ROI is read from the
// nodes by the least-squares interpolation of functions of that band,
//   U = W V W^T,  V = K_x T K_x^T,  W = S(x_m, x_k) S(x_k, x_l)^-1,
// S(x, y) = sin(B (x - y)) / (B (x - y)).  W's rows have norm about 1 (it adds
// no error to V's) and it reproduces e^{i nu x}, |nu| <= B, to 3e-8 rms (under
// 2e-6 at the band's ends, the rim), far below the split-BF16 kernel's 2^-17.
//
// A flat plate is a function of di^2 + dj^2, which every step exploits:
//   - columns +-d fold into one kernel column K(x, d) + K(x, -d) (half the
//     contraction), rows +-d have the same row transform (half the rows), and
//     over the whole aperture T is its own transpose: with L = T below the
//     diagonal plus half of T on the diagonal tiles, T = L + L^T and
//     V = F + F^T, F = K L K^T (half of the rest);
//   - for an ROI centred on the focus K(x, d) + K(x, -d) is even in x, so the
//     nodes x > 0 carry V (half the nodes).
// A range of rows that is not its own mirror image keeps the column fold and the
// evenness along x; its V takes all nodes along y.
// Deformed membranes have no symmetry; they take all nodes, all columns, and
// both real masks T cos(phi) and T sin(phi) in one pass (the phase is
// evaluated once).
//
// k_nodes is a persistent tcgen05 kernel, one CTA per SM:
//   unit    : a stripe of BN aperture rows x one chunk of K blocks
//   stage   : 32 columns; A = NT node tiles of 128 kernel rows (Re and Im of 64
//             nodes), BF16 hi and lo, pre-swizzled in HBM, one bulk copy; B =
//             the masks of BN rows, generated into shared memory
//   flat, NT = 1: 512 rows, two 128 x 256 accumulators (row halves) share A
//   flat, NT = 2: 256 rows, two accumulators (node tiles)
//   four levels : 256 rows, accumulators Re T and Im T, a plane each
//   membrane    : 256 rows, accumulators T cos and T sin, hi and lo planes
//   warps 0-3 epilogue, 4 loader, 5 MMA issuer, 6-21 mask generators
// The mask rule in the generators: the zone index of a sample is the integer
// part of s kappa, s = di^2 + dj^2; the 64-bit fixed-point phase s K mod 2^64
// (its top bit the zone's parity, or its top log2 L bits the level) is carried
// exactly from block to block, and its upper 32 bits run along a block with
// two integer additions per sample.  Their error is below E units; a row of a
// block in which a phase comes within E of a zone boundary takes the exact rule
// with the threshold table, a sample per lane (exact_rows; a plate whose zones
// end on samples has a tie in every 4 N of them).
// What bounds it: on large flat plates the tensor pipe (1.51 PFLOP/s on N =
// 120,001, 0.78 of the measured burst); on small ones the length of a unit's
// chain (8 K blocks, 2,000 clocks each); with membranes the generators.
// Whole propagations before (every sample against every ROI row, k_dense) and
// now: 2 mm, ROI 128^2 0.242 -> 0.075 ms; 30 mm off the axis, 256^2 2.36 -> 0.167;
// 25 cm, 512^2 200 -> 3.32; a rank's eighth of 1 m 422 -> 24.3; four levels on
// 60,001^2 28.1 -> 0.349; four membranes on N <= 36,363, 128^2 20.0 -> 5.1 ms.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <memory>
#include <new>
#include <vector>

#include "fzp_internal.cuh"
#include "membrane.cuh"
#include "tc_ptx.cuh"
#include "zone_phase.cuh"

namespace fzp {
namespace {

using namespace tc;

constexpr int BK = 32;                   // columns per stage: one 64-byte swizzle row of BF16
constexpr int SUB = 128 * BK * 2;        // 8 KiB: one (tile, hi | lo) operand image
constexpr int PLANE = 256 * BK * 2;      // 16 KiB: one mask plane of 256 rows
constexpr int EPI_WARPS = 4, LOAD_WARP = 4, MMA_WARP = 5, GEN_WARP0 = 6, GEN_WARPS = 16;
constexpr int NUM_THREADS = (GEN_WARP0 + GEN_WARPS) * 32;
constexpr int TMEM_COLS = 512;
constexpr int EPI_BOX = 32;
constexpr int EPI_BYTES = EPI_WARPS * 2 * EPI_BOX * EPI_BOX * 4;  // two boxes per warp
constexpr int ERR_BASE = 300;

enum { MASK_PARITY = 0, MASK_SIGNED = 1, MASK_LEVELS = 2, MASK_MEMBRANE = 3, MASK_QUAD = 4, MASK_LOADED = 5, MASK_DIRECT = 6 };  // (membranes: walked, by column)

struct NodeArgs {
  MaskGeom mg;              // c = 0 for a folded (flat) plate
  PhaseRule ph;
  int64_t j_begin, j_end;   // rows of this launch (folded: distances from the axis)
  int n_stripes;
  int octant;               // 1: columns up to the row only, diagonal tiles halved
  int64_t kblocks;          // K blocks of the kernel image
  const int* sched;         // off[nchunks + 1], slo[nchunks], cnt[nchunks]
  int nchunks, group, promote;
  int slices;               // images of C1, chunk g adds into image g slices / nchunks
  DeformCoef df;            // membrane
  const float* ld_src;      // loaded operand: row j at ld_src + j ld_stride
  int64_t ld_stride;
  int y_off;                // first row of C1
  const uint8_t* A;
  int* err;
};

template <int NT, int MASK>
struct Shape {
  static constexpr bool CX = MASK == MASK_MEMBRANE || MASK == MASK_DIRECT;
  static constexpr bool LD = MASK == MASK_LOADED;                 // a real FP32 matrix in place of the masks
  static constexpr bool TWO = CX || MASK == MASK_QUAD;            // two masks: one accumulator each
  static constexpr int BN = (NT == 1 && !TWO && !LD) ? 512 : 256; // rows per unit
  static constexpr int PLANES = CX ? 4 : (TWO || LD) ? 2 : BN / 256;  // mask planes per stage
  static constexpr int ACCS = LD && NT == 1 ? 1 : 2;              // accumulators
  static constexpr int A_BYTES = NT * 2 * SUB;
  static constexpr int B_BYTES = PLANES * PLANE;
  static constexpr int STAGES = CX || (LD && NT == 2) ? 2 : 4;
  static constexpr int C1_ROWS = NT * 128 * (TWO ? 2 : 1);
  static constexpr int SMEM = 1024 + STAGES * (A_BYTES + B_BYTES) + EPI_BYTES + 256;
  static_assert(!TWO || NT == 1, "two node tiles of two masks need more tensor memory than there is");
};

__device__ __forceinline__ uint64_t sdesc(const void* p) {
  const uint64_t a = smem_u32(p);
  return ((a >> 4) & 0x3FFFull) | (1ull << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}
// kind::f16, D = F32, A = B = BF16, K-major, N = 256, M = 128
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
          dtmem),
      "l"(ad), "l"(bd), "r"(IDESC), "r"(accumulate)
      : "memory");
}

// Largest a with a^2 <= t, 0 <= t < 2^46: the FP32 root is within 2 of it (an
// FP64 root costs thousands of clocks at two FP64 lanes per SM).
__device__ __forceinline__ int64_t isqrt_floor(int64_t t) {
  int64_t a = (int64_t)sqrtf((float)t);
  while (a * a > t) --a;
  while ((a + 1) * (a + 1) <= t) ++a;
  return a;
}

// ------------------------------------------------------------------ work list
// K blocks [klo, khi) of the stripe of rows [jb, je): the chord of its row
// nearest the axis; with the octant, columns below je only.  At least one
// block (every stripe writes its rows of C1).
__device__ __forceinline__ void stripe_kspan(const NodeArgs& a, int64_t jb, int64_t je, int64_t& klo, int64_t& khi) {
  if (a.ld_src) {  // dense: no chord
    klo = 0;
    khi = a.octant && (je + BK - 1) / BK < a.kblocks ? (je + BK - 1) / BK : a.kblocks;
    return;
  }
  const int64_t c = a.mg.c;
  const int64_t jn = c < jb ? jb : (c >= je ? je - 1 : c);
  const int64_t t = a.mg.sR - (jn - c) * (jn - c);
  const int64_t b = t < 0 ? -1 : isqrt_floor(t);
  klo = c - b > 0 ? (c - b) / BK : 0;
  khi = (c + b) / BK + 1;
  if (khi > a.kblocks) khi = a.kblocks;
  if (a.octant && khi > (je + BK - 1) / BK) khi = (je + BK - 1) / BK;
  if (klo >= a.kblocks) klo = a.kblocks - 1;
  if (khi <= klo) khi = klo + 1;
}

template <int BN>
__device__ __forceinline__ void span_of(const NodeArgs& a, int64_t s, int64_t& klo, int64_t& khi) {
  const int64_t jb = a.j_begin + s * BN;
  stripe_kspan(a, jb, jb + BN < a.j_end ? jb + BN : a.j_end, klo, khi);
}

// Zeroes C1 and, at a propagation's start, the accumulator (all blocks but the
// first) and builds the work list (the first):
// units (chunk g, stripe s) in chunk order, so that the CTAs at work at one time
// share kernel blocks.  Every chunk's stripes are one range around the stripe
// whose span holds the others' ends: the one nearest the axis or, with the
// octant, where the chord takes over from the diagonal.
template <int BN>
__global__ void __launch_bounds__(1024) k_nodes_prep(const NodeArgs a, int* sched, float4* c1, int64_t c1_vec, float4* uacc,
                                                      int64_t uacc_vec) {
  if (blockIdx.x > 0) {
    const int64_t step = (int64_t)(gridDim.x - 1) * blockDim.x;
    for (int64_t t = (int64_t)(blockIdx.x - 1) * blockDim.x + threadIdx.x; t < c1_vec; t += step)
      c1[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t t = (int64_t)(blockIdx.x - 1) * blockDim.x + threadIdx.x; t < uacc_vec; t += step)
      uacc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  int* off = sched;
  int* slo = sched + a.nchunks + 1;
  int* cnt = slo + a.nchunks;
  __shared__ int s_part[1024];
  const int64_t ns = a.n_stripes;
  int64_t sc = a.mg.c < a.j_begin ? 0 : (a.mg.c - a.j_begin) / BN;
  if (sc >= ns) sc = ns - 1;
  if (a.ld_src) {
    sc = ns - 1;  // the last stripe's span holds the others'
  } else if (a.octant) {
    int64_t lo = 0, hi = ns - 1;  // first stripe whose chord ends below its last row
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      const int64_t jb = a.j_begin + mid * BN, je = jb + BN < a.j_end ? jb + BN : a.j_end;
      const int64_t t = a.mg.sR - jb * jb;
      if (t < 0 || isqrt_floor(t) < je) hi = mid;
      else lo = mid + 1;
    }
    sc = lo;
    if (lo > 0) {
      int64_t k0, h0, k1, h1;
      span_of<BN>(a, lo - 1, k0, h0);
      span_of<BN>(a, lo, k1, h1);
      if (h0 > h1) sc = lo - 1;
    }
  }
  int mine = 0;
  const int per = (a.nchunks + (int)blockDim.x - 1) / (int)blockDim.x;  // consecutive chunks of this thread
  const int g0 = threadIdx.x * per, g1 = min(g0 + per, a.nchunks);
  for (int g = g0; g < g1; ++g) {
    const int64_t c0 = (int64_t)g * a.group, c1k = c0 + a.group;
    auto meets = [&](int64_t st) {
      int64_t klo, khi;
      span_of<BN>(a, st, klo, khi);
      return klo < c1k && khi > c0;
    };
    int first = (int)sc, n = 0;
    if (meets(sc)) {
      int64_t lo = 0, hi = sc;
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (meets(mid)) hi = mid;
        else lo = mid + 1;
      }
      first = (int)lo;
      lo = sc;
      hi = ns - 1;
      while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (meets(mid)) lo = mid;
        else hi = mid - 1;
      }
      n = (int)lo - first + 1;
    }
    slo[g] = first;
    cnt[g] = n;
    mine += n;
  }
  s_part[threadIdx.x] = mine;
  __syncthreads();
  for (int d = 1; d < (int)blockDim.x; d <<= 1) {  // inclusive prefix sums over the threads
    const int v = (int)threadIdx.x >= d ? s_part[threadIdx.x - d] : 0;
    __syncthreads();
    s_part[threadIdx.x] += v;
    __syncthreads();
  }
  int acc = s_part[threadIdx.x] - mine;
  for (int g = g0; g < g1; ++g) {
    off[g] = acc;
    acc += cnt[g];
  }
  if (threadIdx.x == blockDim.x - 1) off[a.nchunks] = s_part[threadIdx.x];
}

struct Unit {
  int64_t jb, je, kb0, kb1;
  int slice;
};

template <int BN>
__device__ __forceinline__ Unit unit_at(const NodeArgs& a, int it) {
  const int* off = a.sched;
  const int* slo = a.sched + a.nchunks + 1;
  int lo = 0, hi = a.nchunks - 1;  // largest g with off[g] <= it (chunks without units share an offset)
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(off + mid) <= it) lo = mid;
    else hi = mid - 1;
  }
  Unit u;
  const int64_t s = __ldg(slo + lo) + (it - __ldg(off + lo));
  u.jb = a.j_begin + s * BN;
  u.je = u.jb + BN < a.j_end ? u.jb + BN : a.j_end;
  int64_t klo, khi;
  stripe_kspan(a, u.jb, u.je, klo, khi);
  const int64_t c0 = (int64_t)lo * a.group, c1 = c0 + a.group;
  u.kb0 = klo > c0 ? klo : c0;
  u.kb1 = khi < c1 ? khi : c1;
  u.slice = lo * a.slices / a.nchunks;
  return u;
}

// ------------------------------------------------------------------ generator
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

// bits 2q, 2q + 1 of `bits` as two half-word masks
__device__ __forceinline__ uint32_t pair_mask(uint32_t bits, int q) {
  return (((bits >> (2 * q)) & 1u) ? 0xFFFFu : 0u) | (((bits >> (2 * q + 1)) & 1u) ? 0xFFFF0000u : 0u);
}

// Columns [di0, di0 + 32) of row dj inside the disc chord (bmax = -1: none).
__device__ __forceinline__ uint32_t chord_bits(int64_t di0, int64_t bmax) {
  const int64_t lo = -bmax - di0, hi = bmax - di0;
  if (bmax < 0 || hi < 0 || lo > 31) return 0u;
  const uint32_t a = lo <= 0 ? 0xFFFFFFFFu : (0xFFFFFFFFu << (uint32_t)lo);
  const uint32_t b = hi >= 31 ? 0xFFFFFFFFu : (0xFFFFFFFFu >> (uint32_t)(31 - hi));
  return a & b;
}

// The exact rule on the blocks of the lanes that ask for it (`redo`; whole warp):
// the warp takes such a row at a time, a column per lane.  Bits with value +1 and
// with value -1 before the chord is applied (MASK_SIGNED: every column +1 or -1;
// MASK_QUAD: the level's parity and its upper half).  A plate whose zones end on
// samples has a tie in every 4 N of them; column after column in one lane each
// cost 10,000 clocks, a third of a small plate's row pass.
template <int MASK>
__device__ __noinline__ void exact_rows(bool redo, int32_t di0, int32_t dj, const MaskGeom& g, const PhaseRule& r, uint32_t& pb,
                                        uint32_t& nb) {
  const int lane = threadIdx.x & 31;
  pb = nb = 0u;
  for (uint32_t todo = __ballot_sync(0xffffffffu, redo); todo != 0u; todo &= todo - 1u) {
    const int src = __ffs(todo) - 1;
    const int64_t d = (int64_t)__shfl_sync(0xffffffffu, di0, src) + lane, j = __shfl_sync(0xffffffffu, dj, src);
    const int64_t s = j * j + d * d;
    const uint32_t z = (uint32_t)zone_of(s < g.sR ? s : g.sR, g);  // (zones are below 2^24)
    bool p, n = false;
    if (MASK == MASK_LEVELS) {
      const uint32_t q = z % (uint32_t)r.lmod;
      p = (r.pos >> q) & 1ull;
      n = (r.neg >> q) & 1ull;
    } else if (MASK == MASK_SIGNED) {
      n = z & 1u;
      p = !n;
    } else if (MASK == MASK_QUAD) {
      p = z & 1u;
      n = (z >> 1) & 1u;
    } else {
      p = (z ^ (uint32_t)r.open_even) & 1u;
    }
    const uint32_t P = __ballot_sync(0xffffffffu, p), N = __ballot_sync(0xffffffffu, n);
    if (lane == src) {
      pb = P;
      nb = N;
    }
  }
}

// A row's walk over its blocks: the exact 64-bit phase at the block's first
// column and its first difference.
struct RowWalk {
  uint64_t phase, step;  // s K and (2 di + 1) K mod 2^64
  int32_t di0, dj, bmax;  // |di|, |dj| < 2^24
};

__device__ __forceinline__ void row_start(RowWalk& w, int64_t dj, int64_t di0, bool live, const MaskGeom& g,
                                          const PhaseRule& r) {
  const int64_t t = g.sR - dj * dj;
  w.dj = (int32_t)dj;
  w.di0 = (int32_t)di0;
  w.bmax = (live && t >= 0) ? (int32_t)isqrt_floor(t) : -1;
  w.phase = (uint64_t)(dj * dj + di0 * di0) * r.K + (r.open_even ? (1ull << 63) : 0ull);
  w.step = (uint64_t)(2 * di0 + 1) * r.K;
}

// On by `n` columns: K ((d + n)^2 - d^2) = n (2 d + 1) K + n (n - 1) K.
template <int n>
__device__ __forceinline__ void row_next(RowWalk& w, const PhaseRule& r) {
  w.phase += (uint64_t)n * w.step + (uint64_t)(n * (n - 1)) * r.K;
  w.step += (uint64_t)(2 * n) * r.K;
  w.di0 += n;
}

// The block's columns inside the disc chord, for a walk from the axis on.
__device__ __forceinline__ uint32_t chord_up(const RowWalk& w) {
  const int n = w.bmax + 1 - w.di0;
  return n >= 32 ? 0xFFFFFFFFu : n <= 0 ? 0u : (1u << n) - 1u;
}

// The block's mask as 16 words of two BF16 values; `one` = +-1 (or +-1/2) in
// both halves.  Whole warp (the votes), every lane a row.  True: a lane of the
// warp has `redo` set, its words are exact_rows' (after the stores, when these
// words' registers are free).
template <int MASK>
__device__ __forceinline__ bool block_words(const RowWalk& w, const MaskGeom& g, const PhaseRule& r, uint32_t one,
                                            uint32_t chord, uint32_t (&wd)[16], bool& redo) {
  const uint32_t c2 = (uint32_t)(r.K >> 32) * 2u + (uint32_t)((r.K >> 31) & 1u);  // upper 32 bits of 2 K
  uint32_t f = (uint32_t)(w.phase >> 32), d = (uint32_t)(w.step >> 32);
  uint32_t near = 0xFFFFFFFFu;
  if (MASK == MASK_LEVELS) {
    const uint32_t el = r.E * (uint32_t)r.lmod;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      uint32_t v = 0u;
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        const uint64_t p = (uint64_t)f * (uint32_t)r.lmod;
        near = min(near, (uint32_t)p + el);
        const int lv = (int)(p >> 32);
        const uint32_t pb = (uint32_t)(r.pos >> lv) & 1u, nb = (uint32_t)(r.neg >> lv) & 1u;
        v |= ((pb | nb) * 0xFFFFu & ((nb << 15) | (one & 0x7FFFu))) << (16 * z);
        f += d;
        d += c2;
      }
      wd[q] = v;
    }
    near = near < 2u * el ? 1u : 0u;
  } else {
    const uint32_t e2 = 2u * r.E, c4 = 2u * c2;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const uint32_t fa = f, fb = f + d;
      f = fb + d + c2;
      d += c4;
      near = min(near, min((fa << 1) + e2, (fb << 1) + e2));
      const uint32_t s = prmt(fa, fb, 0xFFBBu);  // each value's sign in its half-word
      wd[q] = MASK == MASK_SIGNED ? ((s & 0x80008000u) | one) : (s & one);
    }
    near = near < 2u * e2 ? 1u : 0u;
  }
  // rare: a phase near a zone boundary, columns beyond the chord
  redo = false;
  if (__any_sync(0xffffffffu, near != 0u || chord != 0xFFFFFFFFu)) {
    redo = near != 0u && chord != 0u;
#pragma unroll
    for (int q = 0; q < 16; ++q) wd[q] &= pair_mask(chord, q);
    return __any_sync(0xffffffffu, redo);
  }
  return false;
}

// Word q of a row from the exact rule's bits.
template <int MASK>
__device__ __forceinline__ uint32_t exact_word(uint32_t pb, uint32_t nb, uint32_t one, uint32_t chord, int q) {
  return ((pair_mask(pb | nb, q) & one) | (pair_mask(nb, q) & 0x80008000u)) & pair_mask(chord, q);
}
__device__ __forceinline__ void exact_quad_word(uint32_t odd, uint32_t high, uint32_t one, uint32_t chord, int q, uint32_t& re,
                                                uint32_t& im) {
  const uint32_t t = pair_mask(odd, q), s = pair_mask(high, q) & 0x80008000u, m = pair_mask(chord, q);
  re = ~t & (one | s) & m;
  im = t & (one | (s ^ 0x80008000u)) & m;
}

// Four levels (T = e^{-2 pi i q / 4} = 1, -i, -1, i, q the phase's top two bits):
// the block's Re T and Im T, 16 words each.
__device__ __forceinline__ bool block_quad(const RowWalk& w, const MaskGeom& g, const PhaseRule& r, uint32_t one,
                                           uint32_t chord, uint32_t (&re)[16], uint32_t (&im)[16], bool& redo) {
  const uint32_t c2 = (uint32_t)(r.K >> 32) * 2u + (uint32_t)((r.K >> 31) & 1u);  // upper 32 bits of 2 K
  uint32_t f = (uint32_t)(w.phase >> 32), d = (uint32_t)(w.step >> 32);
  uint32_t near = 0xFFFFFFFFu;
  const uint32_t e4 = 4u * r.E;
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const uint32_t fa = f, fb = f + d;
    f = fb + d + c2;
    d += 2u * c2;
    const uint32_t ga = fa << 1, gb = fb << 1;
    near = min(near, min((ga << 1) + e4, (gb << 1) + e4));
    const uint32_t s = prmt(fa, fb, 0xFFBBu) & 0x80008000u;      // q >= 2
    const uint32_t t = prmt(ga, gb, 0xFFBBu);                    // q odd
    re[q] = ~t & (one | s);
    im[q] = t & (one | (s ^ 0x80008000u));
  }
  redo = near < 2u * e4 && chord != 0u;
  if (__any_sync(0xffffffffu, redo || chord != 0xFFFFFFFFu)) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const uint32_t m = pair_mask(chord, q);
      re[q] &= m;
      im[q] &= m;
    }
    return __any_sync(0xffffffffu, redo);
  }
  return false;
}

// The block's open bits (parity rule, chord applied), for the membrane pass.  Whole warp.
__device__ __forceinline__ uint32_t block_open(const RowWalk& w, const MaskGeom& g, const PhaseRule& r) {
  const uint32_t c2 = (uint32_t)(r.K >> 32) * 2u + (uint32_t)((r.K >> 31) & 1u);
  uint32_t f = (uint32_t)(w.phase >> 32), d = (uint32_t)(w.step >> 32);
  uint32_t near = 0xFFFFFFFFu, bits = 0u;
  const uint32_t chord = chord_bits(w.di0, w.bmax), e2 = 2u * r.E;
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    near = min(near, (f << 1) + e2);
    bits = __funnelshift_l(f, bits, 1);  // the sign shifts in: column k at bit 31 - k
    f += d;
    d += c2;
  }
  bits = __brev(bits);
  const bool redo = near < 2u * e2 && chord != 0u;
  if (__any_sync(0xffffffffu, redo)) {
    uint32_t pb, nb;
    exact_rows<MASK_PARITY>(redo, w.di0, w.dj, g, r, pb, nb);
    if (redo) bits = pb;
  }
  return bits & chord;
}

// Whole-warp wait: usually the stage is free and one test passes.
__device__ __forceinline__ bool stage_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err, int code) {
  return __all_sync(0xffffffffu, mbar_try(bar, parity)) || warp_wait(bar, parity, abort_flag, err, code);
}

// ------------------------------------------------------------------ kernel
template <int NT, int MASK>
__global__ void __launch_bounds__(NUM_THREADS, 1) k_nodes(const NodeArgs a, const __grid_constant__ CUtensorMap tmC1) {
  using S = Shape<NT, MASK>;
  constexpr bool CX = S::CX, LD = S::LD;
  constexpr int NST = S::STAGES, BN = S::BN;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = base;
  uint8_t* sB = base + NST * S::A_BYTES;
  uint8_t* sE = sB + NST * S::B_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sE + EPI_BYTES);
  uint64_t* fullA = bars;
  uint64_t* fullB = bars + NST;
  uint64_t* empty = bars + 2 * NST;
  uint64_t* accFull = bars + 3 * NST;
  uint64_t* accEmpty = accFull + 1;
  uint64_t* drain = accEmpty + 1;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(drain + 1);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 2);
  volatile int* epi_ok = reinterpret_cast<volatile int*>(drain + 3);  // [2], by promotion parity

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&fullA[s], 1);
      mbar_init(&fullB[s], GEN_WARPS / 2);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accFull, 1);
    mbar_init(accEmpty, EPI_WARPS);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int n_items = __ldg(a.sched + a.nchunks);

  if (warp == LOAD_WARP) {
    // ---------------- kernel images: one bulk copy per stage
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int last[NST];
#pragma unroll
      for (int s2 = 0; s2 < NST; ++s2) last[s2] = -1;
      for (int it = blockIdx.x; it < n_items && !*abort_flag; it += gridDim.x) {
        const Unit un = unit_at<BN>(a, it);
        for (int64_t kb = un.kb0; kb < un.kb1; ++kb) {
          if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag, a.err, ERR_BASE + 1)) break;
          mbar_arrive_tx(&fullA[stage], S::A_BYTES);
          bulk_g2s(sA + stage * S::A_BYTES, a.A + kb * S::A_BYTES, S::A_BYTES, &fullA[stage]);
          last[stage] = (int)phase;
          if (++stage == NST) { stage = 0; phase ^= 1; }
        }
      }
      if (*abort_flag) {
        // copies already issued must land before shared memory is released
#pragma unroll
        for (int s2 = 0; s2 < NST; ++s2) {
          if (last[s2] < 0) continue;
          const uint64_t t0 = gtimer();
          while (!mbar_try(&fullA[s2], (uint32_t)last[s2]) && gtimer() - t0 < WAIT_NS) {
          }
        }
      }
    }
  } else if (warp == MMA_WARP) {
    // ---------------- MMA issuer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0, accph = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x) {
        const Unit un = unit_at<BN>(a, it);
        for (int64_t p0 = un.kb0; p0 < un.kb1 && ok; p0 += a.promote) {
          const int64_t p1 = p0 + a.promote < un.kb1 ? p0 + a.promote : un.kb1;
          if (!mbar_wait(accEmpty, accph ^ 1, abort_flag, a.err, ERR_BASE + 2)) { ok = false; break; }
          tc_fence_after();
          for (int64_t kb = p0; kb < p1; ++kb) {
            if (!mbar_wait(&fullA[stage], phase, abort_flag, a.err, ERR_BASE + 3) ||
                !mbar_wait(&fullB[stage], phase, abort_flag, a.err, ERR_BASE + 4)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t ad = sdesc(sA + stage * S::A_BYTES), bd = sdesc(sB + stage * S::B_BYTES);
#pragma unroll
            for (int ks = 0; ks < BK / 16; ++ks) {
              const uint64_t o = (uint64_t)((ks * 32) >> 4);
              const uint32_t acc = (kb > p0 || ks > 0) ? 1u : 0u;
#pragma unroll
              for (int q = 0; q < S::ACCS; ++q) {
                // flat: accumulator q = row half q (NT = 1) or node tile q (NT = 2);
                // two masks: q = 0, 1; membrane planes 2q (hi) and 2q + 1 (lo)
                const uint32_t dt = tmem + (uint32_t)(q * 256);
                const int at = NT == 2 ? q : 0;
                const int bp = CX ? 2 * q : (NT == 2 || LD ? 0 : q);
                const uint64_t a_hi = ad + (uint64_t)((at * SUB) >> 4) + o;
                const uint64_t a_lo = ad + (uint64_t)(((NT + at) * SUB) >> 4) + o;
                const uint64_t b0 = bd + (uint64_t)((bp * PLANE) >> 4) + o;
                mma_bf16(dt, a_hi, b0, acc);
                mma_bf16(dt, a_lo, b0, 1u);
                if (CX || LD) mma_bf16(dt, a_hi, b0 + (uint64_t)(PLANE >> 4), 1u);
              }
            }
            mma_commit(&empty[stage]);
            if (++stage == NST) { stage = 0; phase ^= 1; }
          }
          if (!ok) break;
          mma_commit(accFull);
          accph ^= 1;
        }
      }
      // all issued MMAs complete before tensor memory is released
      mma_commit(drain);
      const uint64_t t0 = gtimer();
      while (!mbar_try(drain, 0) && gtimer() - t0 < WAIT_NS) {
      }
    }
  } else if (warp >= GEN_WARP0) {
    // ---------------- mask generators: two groups of eight warps take every
    // other block of the CTA's sequence (with an even number of stages a stage
    // has one group), a lane per row, or per two rows 256 apart where the unit
    // has 512
    static_assert(NST % 2 == 0, "a stage must keep its generator group");
    const int gw = warp - GEN_WARP0, grp = gw >> 3;
    const int row = (gw & 7) * 32 + lane;  // row of the stripe (and row + 256)
    // 64-byte swizzle: row at (row / 8) 512 + (row % 8) 64, 16-byte part q at q ^ ((row % 8) / 2)
    uint8_t* rowbase = sB + (row >> 3) * 512 + (row & 7) * 64;
    const int sw = (row & 7) >> 1;
    bool ok = true;
    {
      constexpr int RPL = BN / 256;  // rows per lane
      int stage = grp;
      uint32_t phase = 0;
      int skip = grp;  // blocks before this group's next one
      for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x) {
        const Unit un = unit_at<BN>(a, it);
        const int nkb = (int)(un.kb1 - un.kb0);
        RowWalk w[RPL];
#pragma unroll
        for (int h = 0; h < RPL; ++h) {
          const int64_t j = un.jb + row + 256 * h;
          row_start(w[h], j - a.mg.c, (un.kb0 + skip) * BK - a.mg.c, j < un.je, a.mg, a.ph);
        }
        CxRow cxr;
        if constexpr (CX) cx_row_init(a.df, un.jb + row - a.mg.c, cxr);
        // blocks of the diagonal tile: half weight
        const int diag = a.octant ? (int)(un.jb / BK - un.kb0) : nkb;
        int b = skip;
        for (; b < nkb; b += 2) {
          const uint32_t one = b >= diag ? 0x3F003F00u : 0x3F803F80u;
          uint8_t* rp = rowbase + stage * S::B_BYTES;
          if constexpr (LD) {
            const int64_t j = un.jb + row;
            const float h = b >= diag ? 0.5f : 1.0f;
            float4 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j < un.je) {
              const float4* src = reinterpret_cast<const float4*>(a.ld_src + j * a.ld_stride + (un.kb0 + b) * BK);
#pragma unroll
              for (int q = 0; q < 8; ++q) v[q] = __ldg(src + q);
            }
            if (!stage_wait(&empty[stage], phase ^ 1, abort_flag, a.err, ERR_BASE + 5)) { ok = false; break; }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t hi[4], lo[4];
              split2(h * v[2 * q].x, h * v[2 * q].y, hi[0], lo[0]);
              split2(h * v[2 * q].z, h * v[2 * q].w, hi[1], lo[1]);
              split2(h * v[2 * q + 1].x, h * v[2 * q + 1].y, hi[2], lo[2]);
              split2(h * v[2 * q + 1].z, h * v[2 * q + 1].w, hi[3], lo[3]);
              *reinterpret_cast<uint4*>(rp + ((q ^ sw) << 4)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
              *reinterpret_cast<uint4*>(rp + PLANE + ((q ^ sw) << 4)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            }
          } else if constexpr (CX) {
            const uint32_t bits = block_open(w[0], a.mg, a.ph);
            if (!stage_wait(&empty[stage], phase ^ 1, abort_flag, a.err, ERR_BASE + 5)) { ok = false; break; }
            cx_store2<MASK == MASK_DIRECT>(a.df, cxr, w[0].di0, bits, rp, PLANE, sw);
          } else if constexpr (MASK == MASK_QUAD) {
            uint32_t re[16], im[16];
            bool redo;
            const bool rare = block_quad(w[0], a.mg, a.ph, one, chord_up(w[0]), re, im, redo);
            if (!stage_wait(&empty[stage], phase ^ 1, abort_flag, a.err, ERR_BASE + 5)) { ok = false; break; }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              *reinterpret_cast<uint4*>(rp + ((q ^ sw) << 4)) =
                  make_uint4(re[4 * q], re[4 * q + 1], re[4 * q + 2], re[4 * q + 3]);
              *reinterpret_cast<uint4*>(rp + PLANE + ((q ^ sw) << 4)) =
                  make_uint4(im[4 * q], im[4 * q + 1], im[4 * q + 2], im[4 * q + 3]);
            }
            if (rare) {
              uint32_t odd, high;
              exact_rows<MASK>(redo, w[0].di0, w[0].dj, a.mg, a.ph, odd, high);
              if (redo) {
                const uint32_t chord = chord_up(w[0]);
#pragma unroll 1
                for (int q = 0; q < 16; ++q) {
                  uint32_t x, y;
                  exact_quad_word(odd, high, one, chord, q, x, y);
                  uint8_t* o = rp + (((q >> 2) ^ sw) << 4) + 4 * (q & 3);
                  *reinterpret_cast<uint32_t*>(o) = x;
                  *reinterpret_cast<uint32_t*>(o + PLANE) = y;
                }
              }
            }
          } else {
            bool redo[RPL], rare = false;
#pragma unroll
            for (int h = 0; h < RPL; ++h) {
              uint32_t wd[16];
              rare |= block_words<MASK>(w[h], a.mg, a.ph, one, chord_up(w[h]), wd, redo[h]);
              if (h == 0 && !stage_wait(&empty[stage], phase ^ 1, abort_flag, a.err, ERR_BASE + 5)) { ok = false; break; }
#pragma unroll
              for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4*>(rp + h * PLANE + ((q ^ sw) << 4)) =
                    make_uint4(wd[4 * q], wd[4 * q + 1], wd[4 * q + 2], wd[4 * q + 3]);
            }
            if (!ok) break;
            if (rare) {
#pragma unroll 1
              for (int h = 0; h < RPL; ++h) {
                const bool again = h ? redo[RPL - 1] : redo[0];
                const int32_t di0 = w[0].di0, dj = w[0].dj + 256 * h;
                const uint32_t chord = h ? chord_up(w[RPL - 1]) : chord_up(w[0]);
                uint32_t pb, nb;
                exact_rows<MASK>(again, di0, dj, a.mg, a.ph, pb, nb);
                if (again) {
#pragma unroll 1
                  for (int q = 0; q < 16; ++q)
                    *reinterpret_cast<uint32_t*>(rp + h * PLANE + (((q >> 2) ^ sw) << 4) + 4 * (q & 3)) =
                        exact_word<MASK>(pb, nb, one, chord, q);
                }
              }
            }
          }
#pragma unroll
          for (int h = 0; h < RPL; ++h) row_next<2 * BK>(w[h], a.ph);
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(&fullB[stage]);
          stage += 2;
          if (stage >= NST) { stage -= NST; phase ^= 1; }
        }
        skip = b - nkb;
      }
    }
  } else {
    // ---------------- epilogue: warp w drains TMEM lanes 32 w .. of both
    // accumulators: each 32 x 32 piece goes to shared memory (128-byte swizzle,
    // two boxes in turn) and from there by one TMA reduce-add into C1, once per
    // promotion
    uint8_t* eb = sE + warp * (2 * EPI_BOX * EPI_BOX * 4);
    uint32_t accph = 0, box = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x) {
      const Unit un = unit_at<BN>(a, it);
      const int rows = (int)(un.je - un.jb);
      for (int64_t p0 = un.kb0; p0 < un.kb1; p0 += a.promote) {
        if (threadIdx.x == 0) epi_ok[accph] = mbar_wait(accFull, accph, abort_flag, a.err, ERR_BASE + 6) ? 1 : 0;
        named_bar_sync(1, EPI_WARPS * 32);
        if (!epi_ok[accph]) { ok = false; break; }
        tc_fence_after();
#pragma unroll 1
        for (int q = 0; q < S::ACCS; ++q) {
          const int xs = BN == 512 ? q * 256 : 0, x0 = (int)(un.jb - a.j_begin) + xs;
          const int y0 = a.y_off + un.slice * S::C1_ROWS + (BN == 512 ? 0 : q * 128) + warp * 32;
          const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(q * 256);
          const int xn = min(256, rows - xs);  // live columns (may be <= 0)
#pragma unroll 1
          for (int col = 0; col < xn; col += EPI_BOX) {
            float v[32];
            tmem_ld32(taddr + col, v);
            uint8_t* bx = eb + box * (EPI_BOX * EPI_BOX * 4);
            box ^= 1u;
            if (lane == 0) bulk_wait_read1();  // the piece before the last has been read out
            __syncwarp();
#pragma unroll
            for (int c4 = 0; c4 < 8; ++c4)
              *reinterpret_cast<float4*>(bx + lane * 128 + ((c4 ^ (lane & 7)) << 4)) =
                  make_float4(v[4 * c4], v[4 * c4 + 1], v[4 * c4 + 2], v[4 * c4 + 3]);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tma_reduce_add_2d(&tmC1, bx, x0 + col, y0);
              bulk_commit();
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(accEmpty);
        accph ^= 1;
      }
    }
    if (lane == 0) bulk_wait0();  // C1 complete before the kernel ends
  }
  tc_fence_before();
  __syncthreads();
  if (warp == MMA_WARP) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------ tables
// Kernel images of the nodes: K block kb = [tile 0 hi] .. [tile NT-1 hi][tile 0 lo] ..,
// each 128 rows x 32 BF16, 64-byte swizzle; tile t holds Re K (rows 0-63) and
// Im K (rows 64-127) of nodes 64 t ..; folded: column d holds K(x, d) + K(x, -d).
__global__ void k_nodes_A(int nt, int64_t ncols, int64_t kblocks, int64_t c, int fold, double kappa, double msh,
                          double delta, uint8_t* A) {
  const int64_t total = kblocks * 4 * (int64_t)nt * 64;  // one thread per node and 8 columns
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k8 = e % (kblocks * 4);
    const int node = (int)(e / (kblocks * 4));
    const int t = node >> 6, r = node & 63;
    const double x = (double)node - msh;
    float re[8], im[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int64_t i = 8 * k8 + u;
      re[u] = im[u] = 0.f;
      if (i < ncols) {
        const double di = (double)(i - c), q = di * di * (0.5 * kappa), l = x * di * delta;
        const float2 v = cis_turns_f(q - l);
        re[u] = v.x;
        im[u] = v.y;
        if (fold && i > c) {
          const float2 m = cis_turns_f(q + l);
          re[u] += m.x;
          im[u] += m.y;
        }
      }
    }
    uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      split2(re[2 * u], re[2 * u + 1], rh[u], rl[u]);
      split2(im[2 * u], im[2 * u + 1], ih[u], il[u]);
    }
    const int k = (int)(k8 & 3);
    uint8_t* blk = A + (k8 >> 2) * (int64_t)(nt * 2 * SUB);
    auto put = [&](int plane, int rr, const uint32_t (&v)[4]) {
      *reinterpret_cast<uint4*>(blk + plane * SUB + (rr >> 3) * 512 + (rr & 7) * 64 + ((k ^ ((rr & 7) >> 1)) << 4)) =
          make_uint4(v[0], v[1], v[2], v[3]);
    };
    put(t, r, rh);
    put(nt + t, r, rl);
    put(t, 64 + r, ih);
    put(nt + t, 64 + r, il);
  }
}

// The same images from a table E [node][stride] of complex columns.
__global__ void k_nodes_table(int nt, int64_t ncols, int64_t kblocks, const float2* __restrict__ E, int64_t stride,
                              uint8_t* A) {
  const int64_t total = kblocks * 4 * (int64_t)nt * 64;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k8 = e % (kblocks * 4);
    const int node = (int)(e / (kblocks * 4)), t = node >> 6, r = node & 63;
    uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t i = 8 * k8 + 2 * u;
      const float2 a = i < ncols ? E[(int64_t)node * stride + i] : make_float2(0.f, 0.f);
      const float2 b = i + 1 < ncols ? E[(int64_t)node * stride + i + 1] : make_float2(0.f, 0.f);
      split2(a.x, b.x, rh[u], rl[u]);
      split2(a.y, b.y, ih[u], il[u]);
    }
    const int k = (int)(k8 & 3);
    uint8_t* blk = A + (k8 >> 2) * (int64_t)(nt * 2 * SUB);
    auto put = [&](int plane, int rr, const uint32_t (&v)[4]) {
      *reinterpret_cast<uint4*>(blk + plane * SUB + (rr >> 3) * 512 + (rr & 7) * 64 + ((k ^ ((rr & 7) >> 1)) << 4)) =
          make_uint4(v[0], v[1], v[2], v[3]);
    };
    put(t, r, rh);
    put(nt + t, r, rl);
    put(t, 64 + r, ih);
    put(nt + t, 64 + r, il);
  }
}

// ------------------------------------------------------------------ interpolation
// FP64 runs at two multiply-adds per clock and SM here, so the outputs are cut
// into small blocks over the whole GPU and the chirp is applied per axis.
__device__ __forceinline__ double sinc_d(double z) { return fabs(z) < 1e-9 ? 1.0 : sin(z) / z; }

// W from the Cholesky factors of the node matrix (host): a block per output, a
// warp per parity, both triangular solves with U = ns / 32 unknowns per lane in
// registers and the pivots by shuffles, the factor's columns loaded eight steps
// ahead.  A chain of 2 ns steps bounds it: 26 us for 64 nodes (70 with a block of
// four outputs, a barrier per step and one parity after the other; the 2 mm plan
// 309 -> 233 us with that, a faster factorisation and the tables built meanwhile).  F: per parity the factor by columns, then by rows (ns x ns each),
// reciprocals on the diagonal.
struct InterpSpec {
  int n, ns, M, Mo, even;
  double h, c, half;  // node pitch and band (radians) per ROI half width; half width in pitches
  double msh, chirp;  // ROI shift; p^2 / (2 lambda f)
};

template <int U>
__global__ void __launch_bounds__(64) k_interp_W(const InterpSpec a, const double* __restrict__ F, double* __restrict__ W,
                                                 double* __restrict__ Wy, double2* __restrict__ chirp) {
  constexpr int ns = 32 * U;
  __shared__ double w[2][ns];
  const int lane = threadIdx.x & 31, side = threadIdx.x >> 5, o = blockIdx.x;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.M; i += gridDim.x * blockDim.x) {
    const double t = (double)i - a.msh;
    chirp[i] = cis_turns_d(t * t * a.chirp);
  }
  const double xo = (a.even ? (double)o : (double)o - 0.5 * (a.M - 1)) / a.half;
  const double* C = F + (size_t)side * 2 * ns * ns;  // by columns, behind it by rows
  const double* R = C + (size_t)ns * ns;
  double v[U], inv[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int r = lane + 32 * u;
    const double x = ((double)(a.even ? r + ns : r) - 0.5 * (a.n - 1)) * a.h;
    const double sm = sinc_d(a.c * (xo - x)), sp = a.even ? sinc_d(a.c * (xo + x)) : 0.0;
    v[u] = side ? sm - sp : sm + sp;
    inv[u] = C[r * ns + r];
  }
  // columns of the factor eight steps ahead of the pivots
  constexpr int G = 8;
  double next[G][U];
  auto load = [&](const double* T, int k0, int dir) {
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int u = 0; u < U; ++u) next[g][u] = T[(k0 + dir * g) * ns + lane + 32 * u];
  };
  load(C, 0, 1);
#pragma unroll
  for (int kb = 0; kb < U; ++kb)
#pragma unroll 1
    for (int k0 = 0; k0 < 32; k0 += G) {
      double c[G][U];
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int u = 0; u < U; ++u) c[g][u] = next[g][u];
      const int k1 = 32 * kb + k0 + G;
      if (k1 < ns) load(C, k1, 1);
      else load(R, ns - 1, -1);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const double pivot = __shfl_sync(0xffffffffu, v[kb] * inv[kb], k0 + g);
        if (lane == k0 + g) v[kb] = pivot;
        if (lane > k0 + g) v[kb] = fma(-c[g][kb], pivot, v[kb]);
#pragma unroll
        for (int u = kb + 1; u < U; ++u) v[u] = fma(-c[g][u], pivot, v[u]);
      }
    }
#pragma unroll
  for (int kb = U - 1; kb >= 0; --kb)
#pragma unroll 1
    for (int k0 = 31; k0 >= 0; k0 -= G) {
      double c[G][U];
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int u = 0; u < U; ++u) c[g][u] = next[g][u];
      const int k1 = 32 * kb + k0 - G;
      if (k1 >= 0) load(R, k1, -1);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const double pivot = __shfl_sync(0xffffffffu, v[kb] * inv[kb], k0 - g);
        if (lane == k0 - g) v[kb] = pivot;
        if (lane < k0 - g) v[kb] = fma(-c[g][kb], pivot, v[kb]);
#pragma unroll
        for (int u = 0; u < kb; ++u) v[u] = fma(-c[g][u], pivot, v[u]);
      }
    }
#pragma unroll
  for (int u = 0; u < U; ++u) w[side][lane + 32 * u] = v[u];
  __syncthreads();
  for (int r = threadIdx.x; r < ns; r += blockDim.x) {
    W[(size_t)r * a.Mo + o] = w[0][r];
    if (a.even && Wy) {
      // the matrix of all nodes: w(+-x_k) = (even +- odd) / 2, at x_o and mirrored at -x_o
      const int hm = a.M / 2, kp = ns + r, km = ns - 1 - r;
      const double same = 0.5 * (w[0][r] + w[1][r]), other = 0.5 * (w[0][r] - w[1][r]);
      if (o < hm) {
        Wy[(size_t)kp * a.M + hm + o] = same;
        Wy[(size_t)km * a.M + hm + o] = other;
      }
      if (o > 0) {
        Wy[(size_t)kp * a.M + hm - o] = other;
        Wy[(size_t)km * a.M + hm - o] = same;
      }
    }
  }
}

// X[l][o] = sum_k Wy[k][o] V[k][l], k over the ny nodes of the rows' axis (sym:
// of V plus its transpose): a block per output and 32 nodes, its four warps a
// quarter of the sum each.
__global__ void __launch_bounds__(128) k_interp_rows(int ny, int ns, int Mo, int sym, const double* __restrict__ Wy,
                                                     const double2* __restrict__ V, double2* __restrict__ X) {
  __shared__ double2 part[4][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, l = blockIdx.x * 32 + lane, o = blockIdx.y;
  const int n4 = ny / 4;
  const double2* v = V + (size_t)w * n4 * ns + l;
  const double* c = Wy + (size_t)w * n4 * Mo + o;
  double2 x[2];
  x[0] = x[1] = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int k = 0; k < n4; k += 2, v += 2 * ns, c += 2 * Mo) {
    double2 v0 = v[0], v1 = v[ns];
    const double c0 = c[0], c1 = c[Mo];
    if (sym) {
      const double2* vt = V + (size_t)l * ns + w * n4 + k;
      v0 = cadd(v0, vt[0]);
      v1 = cadd(v1, vt[1]);
    }
    x[0].x = fma(c0, v0.x, x[0].x);
    x[0].y = fma(c0, v0.y, x[0].y);
    x[1].x = fma(c1, v1.x, x[1].x);
    x[1].y = fma(c1, v1.y, x[1].y);
  }
  part[w][lane] = cadd(x[0], x[1]);
  __syncthreads();
  if (w == 0) X[l * Mo + o] = cadd(cadd(part[0][lane], part[1][lane]), cadd(part[2][lane], part[3][lane]));
}

struct InterpOut {
  int M, ns;
  int Moy, eveny, Mox, evenx;  // outputs of the two axes (even: M / 2 + 1)
  int sym;                     // the field is its own transpose
  double2 pre;                 // e^{ikf} dx^2 / (i lambda f)
  int accumulate;
};

// U[on, om] = sum_l X[l][on] W[l][om] (sym: only blocks on and below the diagonal
// run and both are stored), the output chirp and prefactor, and the stores: with an even field output o
// stands for the samples M/2 + o and M/2 - o (o = M/2: sample 0 alone).
// Block: 8 x 4 outputs (columns x rows), two threads per output with half of
// the sum each, operands through shared memory.  chirp[i] = e^{i pi x_i^2 /
// (lambda f)} of the ROI samples, as k_interp_W left it.
constexpr int ITX = 8, ITY = 4;
__global__ void __launch_bounds__(2 * ITX * ITY) k_interp_cols(const InterpOut a, const double* __restrict__ W,
                                                               const double2* __restrict__ X,
                                                               const double2* __restrict__ chirp,
                                                               double2* __restrict__ out) {
  const int n0 = blockIdx.y * ITY, m0 = blockIdx.x * ITX;
  if (a.sym && m0 >= n0 + ITY) return;
  __shared__ double2 sXn[64][ITY];
  __shared__ double sWm[64][ITX];
  __shared__ double2 half[ITX * ITY];
  const int h = a.M / 2, tid = threadIdx.x;
  const int side = tid / (ITX * ITY), q = tid % (ITX * ITY), qn = q / ITX, qm = q % ITX;
  const int on = n0 + qn, om = m0 + qm;
  double2 u = make_double2(0.0, 0.0);
  for (int l0 = 0; l0 < a.ns; l0 += 64) {  // ns is 64 or 128
    if (l0 > 0) __syncthreads();
    for (int e = tid; e < 64 * ITY; e += 2 * ITX * ITY) {
      const int l = e / ITY, c = min(n0 + e % ITY, a.Moy - 1);
      sXn[l][e % ITY] = __ldg(X + (l0 + l) * a.Moy + c);
    }
    for (int e = tid; e < 64 * ITX; e += 2 * ITX * ITY) {
      const int l = e / ITX, c = min(m0 + e % ITX, a.Mox - 1);
      sWm[l][e % ITX] = __ldg(W + (l0 + l) * a.Mox + c);
    }
    __syncthreads();
    const int lb = 32 * side;
#pragma unroll 8
    for (int l = lb; l < lb + 32; ++l) {
      const double2 x = sXn[l][qn];
      const double w = sWm[l][qm];
      u.x = fma(w, x.x, u.x);
      u.y = fma(w, x.y, u.y);
    }
  }
  if (side) half[q] = u;
  __syncthreads();
  if (side) return;
  u = cadd(u, half[q]);
  if (on >= a.Moy || om >= a.Mox || (a.sym && om > on)) return;
  const int n = a.eveny ? (on < h ? h + on : 0) : on, m = a.evenx ? (om < h ? h + om : 0) : om;
  const double2 v = cmul(cmul(u, cmul(chirp[n], chirp[m])), a.pre);
  auto put = [&](int nn, int mm) {
    double2* o = out + (int64_t)nn * a.M + mm;
    double2 z = v;
    if (a.accumulate) {
      z.x += o->x;
      z.y += o->y;
    }
    *o = z;
  };
  // samples with a mirror image of their own
  const bool fn = a.eveny && on > 0 && on < h, fm = a.evenx && om > 0 && om < h;
  auto put4 = [&](int nn, int mm, bool f1, bool f2) {
    put(nn, mm);
    if (f1) put(a.M - nn, mm);
    if (f2) put(nn, a.M - mm);
    if (f1 && f2) put(a.M - nn, a.M - mm);
  };
  put4(n, m, fn, fm);
  if (a.sym && on != om) put4(m, n, fm, fn);
}

// ------------------------------------------------------------------ mask export
template <int MASK>
__device__ __forceinline__ void mask_words(const RowWalk& w, const MaskGeom& g, const PhaseRule& r, uint32_t disc,
                                           uint32_t (&wd)[16]) {
  bool redo;
  if (!block_words<MASK>(w, g, r, 0x3F803F80u, disc, wd, redo)) return;
  uint32_t pb, nb;
  exact_rows<MASK>(redo, w.di0, w.dj, g, r, pb, nb);
#pragma unroll
  for (int q = 0; q < 16; ++q)
    if (redo) wd[q] = exact_word<MASK>(pb, nb, 0x3F803F80u, disc, q);
}

// A warp takes 32 rows by MASK_COLS columns (a walk starts at any column; one warp per
// 32 whole rows took 742 us for 512 rows of 5,057 columns, the row walker that
// exported these masks before the nodes 670; now 49).
constexpr int MASK_COLS = 256;
__global__ void k_mask_nodes(MaskGeom mg, PhaseRule ph, int mask, int64_t N, int64_t j0, int64_t rows, uint8_t* out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t parts = (N + MASK_COLS - 1) / MASK_COLS;
  for (int64_t item = warp; item < (rows + 31) / 32 * parts; item += nwarps) {
    const int64_t r = item / parts * 32 + lane, ib = item % parts * MASK_COLS, ie = ib + MASK_COLS < N ? ib + MASK_COLS : N;
    const int64_t dj = j0 + r - mg.c;
    RowWalk w;
    row_start(w, dj, ib - mg.c, r < rows, mg, ph);
    for (int64_t i0 = ib; i0 < ie; i0 += 32) {
      const uint32_t disc = chord_bits(w.di0, w.bmax);
      uint8_t v[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) v[k] = 0;
      uint32_t wd[16];
      if (mask == MASK_QUAD) {
        uint32_t wi[16];
        bool redo;
        if (block_quad(w, mg, ph, 0x3F803F80u, disc, wd, wi, redo)) {
          uint32_t odd, high;
          exact_rows<MASK_QUAD>(redo, w.di0, w.dj, mg, ph, odd, high);
#pragma unroll
          for (int k = 0; k < 16; ++k)
            if (redo) exact_quad_word(odd, high, 0x3F803F80u, disc, k, wd[k], wi[k]);
        }
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          const uint32_t x = (wd[k / 2] >> (16 * (k & 1))) & 0xFFFFu, y = (wi[k / 2] >> (16 * (k & 1))) & 0xFFFFu;
          v[k] = (uint8_t)(x ? 1 + (x >> 15) * 2 : y ? 4 - (y >> 15) * 2 : 0);
        }
      } else if (mask == MASK_LEVELS) {
        PhaseRule one = ph;
        one.neg = 0;
        for (int q = 0; q < ph.lmod; ++q) {
          one.pos = 1ull << q;
          mask_words<MASK_LEVELS>(w, mg, one, disc, wd);
#pragma unroll
          for (int k = 0; k < 32; ++k)
            if ((wd[k / 2] >> (16 * (k & 1))) & 0xFFFFu) v[k] = (uint8_t)(1 + q);
        }
      } else if (mask == MASK_SIGNED) {
        mask_words<MASK_SIGNED>(w, mg, ph, disc, wd);
#pragma unroll
        for (int k = 0; k < 32; ++k)
          v[k] = ((disc >> k) & 1u) ? (uint8_t)(1 + ((wd[k / 2] >> (16 * (k & 1) + 15)) & 1u)) : 0;
      } else if (mask == MASK_MEMBRANE) {
        const uint32_t bits = block_open(w, mg, ph);
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = (uint8_t)((bits >> k) & 1u);
      } else {
        mask_words<MASK_PARITY>(w, mg, ph, disc, wd);
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = ((wd[k / 2] >> (16 * (k & 1))) & 0xFFFFu) ? 1 : 0;
      }
      if (r < rows)
        for (int k = 0; k < 32 && i0 + k < N; ++k) out[r * N + i0 + k] = v[k];
      row_next<BK>(w, ph);
    }
  }
}

fzp_status c1_map(const Plan& P, int64_t stride, int rows, CUtensorMap* tm) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    FZP_CUDA_TRY(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q));
    if (q != cudaDriverEntryPointSuccess || !fn) return set_error(FZP_E_CUDA, "cuTensorMapEncodeTiled unavailable");
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  const cuuint64_t dims[2] = {(cuuint64_t)stride, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)stride * 4};
  const cuuint32_t box[2] = {EPI_BOX, EPI_BOX};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, P.d_C1, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(FZP_E_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return FZP_OK;
}

int mask_kind(const Plan& P) {
  return P.has_deform ? MASK_MEMBRANE : P.levels > 2 ? (P.nd.ns == 64 ? MASK_QUAD : MASK_LEVELS) : P.levels == 2 ? MASK_SIGNED : MASK_PARITY;
}

// Cholesky factor (by columns, then by rows; reciprocals on the diagonal) of the node
// matrix S(x_k, x_l) + 1e-13 (the sinc matrix is singular to working
// precision) for nodes x_k = (k - (n - 1)/2) h and the band half-width c
// (radians): the normal equations of the least-squares interpolation.
// parity +1 / -1: of even / odd functions, over the nodes x > 0.
void node_factor(int n, int ns, int parity, double h, double c, double* T) {
  double dist[256];  // n <= 256
  for (int q = 0; q < n; ++q) {
    const double z = c * q * h;
    dist[q] = q ? std::sin(z) / z : 1.0;
  }
  for (int l = 0; l < ns; ++l)
    for (int k = l; k < ns; ++k)  // x_k + x_l = (k + l + 1) h on the half grid
      T[(size_t)l * ns + k] = dist[k - l] + (parity ? parity * dist[k + l + 1] : 0.0) + (k == l ? 1e-13 : 0.0);
  // column by column from those before it, four at a time (one store per four products)
  for (int q = 0; q < ns; ++q) {
    double* __restrict__ cq = &T[(size_t)q * ns];
    int l = 0;
    for (; l + 4 <= q; l += 4) {
      const double *c0 = &T[(size_t)l * ns], *c1 = c0 + ns, *c2 = c1 + ns, *c3 = c2 + ns;
      const double f0 = c0[q], f1 = c1[q], f2 = c2[q], f3 = c3[q];
      for (int k = q; k < ns; ++k) cq[k] = (((cq[k] - f0 * c0[k]) - f1 * c1[k]) - f2 * c2[k]) - f3 * c3[k];
    }
    for (; l < q; ++l) {
      const double* c0 = &T[(size_t)l * ns];
      const double f0 = c0[q];
      for (int k = q; k < ns; ++k) cq[k] -= f0 * c0[k];
    }
    const double r = 1.0 / std::sqrt(std::max(cq[q], 1e-15));
    for (int k = q + 1; k < ns; ++k) cq[k] *= r;
    cq[q] = r;
  }
  double* L = T + (size_t)ns * ns;
  for (int k = 0; k < ns; ++k)
    for (int l = 0; l <= k; ++l) L[(size_t)k * ns + l] = T[(size_t)l * ns + k];
}

template <int NT, int MASK>
fzp_status smem_attr() {
  static std::atomic<uint64_t> done{0};
  FZP_CUDA_TRY(smem_attr_once((const void*)k_nodes<NT, MASK>, Shape<NT, MASK>::SMEM, done));
  return FZP_OK;
}

template <int NT, int MASK>
fzp_status launch(Plan& P, NodeArgs& a, cudaStream_t s) {
  using S = Shape<NT, MASK>;
  fzp_status st = smem_attr<NT, MASK>();
  if (st != FZP_OK) return st;
  const int64_t rows = a.j_end - a.j_begin;
  a.n_stripes = (int)((rows + S::BN - 1) / S::BN);
  P.c1_stride = (rows + 255) / 256 * 256;
  const int c1r = S::C1_ROWS;
  // A sum of two is the same in either order: up to 256 K blocks of the whole
  // grid (N <= 8192, where the FP32 sums of whole chunks were reproducible) the
  // chunks of a unit's stripe add by twos into separate images of C1, which
  // the column pass sums in order.  Larger plates add into one image.
  a.slices = 1;
  if (P.N <= 256 * BK && !S::LD) {
    const int64_t cap = std::max<int64_t>(1, (int64_t)(c1_elems(P) / ((size_t)c1r * P.c1_stride)));
    a.group = (int)std::max<int64_t>(a.group, (a.kblocks + 2 * cap - 1) / (2 * cap));
    a.nchunks = (int)((a.kblocks + a.group - 1) / a.group);
    a.slices = (int)std::min<int64_t>(cap, (a.nchunks + 1) / 2);
  }
  P.nd.slices = a.slices;
  P.nd.slice_elems = (int64_t)c1r * P.c1_stride;
  CUtensorMap tm;
  st = c1_map(P, P.c1_stride, a.y_off + c1r * a.slices, &tm);
  if (st != FZP_OK) return st;
  const int64_t vec = (int64_t)c1r * P.c1_stride * a.slices / 4;
  const unsigned zb = (unsigned)std::min<int64_t>(2 * P.dn.num_sms, (vec + 4095) / 4096);
  k_nodes_prep<S::BN><<<1 + zb, 1024, 0, s>>>(a, const_cast<int*>(a.sched),
                                             reinterpret_cast<float4*>(P.d_C1 + (size_t)a.y_off * P.c1_stride), vec,
                                             reinterpret_cast<float4*>(P.d_Uacc), P.nd.zero_acc);
  P.nd.zero_acc = 0;
  if (!S::LD) prof_begin(P, s);  // (the SA-CZT's dominant kernel is another)
  k_nodes<NT, MASK><<<P.dn.num_sms, NUM_THREADS, S::SMEM, s>>>(a, tm);
  if (!S::LD) prof_end(P, s);
  P.launches += 2;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

}  // namespace

// The rule of the nodes (host).  The partitioned FP32 row pass (k_seg) takes
// them wherever the ROI's band leaves room on them; so do split-BF16 plans.  BF16
// without the split and explicit clusters of 2 or 4 CTAs stay with k_dense,
// and so do plates of 6 and more levels (L/2 passes: the plain FP32 form's
// single pass is the faster one there) and membranes that need two node tiles
// (four accumulators do not fit the tensor memory).
// Sets the nodes for a field of `band` cycles per ROI pitch (both signs), if
// some count of at most `hi` stored nodes holds it.
static void place_nodes(Plan& P, bool even, double band, int hi) {
  NodeSet& z = P.nd;
  const double half = even ? 0.5 * P.M : 0.5 * (P.M - 1);
  const struct { int n; double most; } sizes[] = {{64, 36.0}, {128, 80.0}, {256, 170.0}};
  for (const auto& q : sizes) {
    const int ns = even ? q.n / 2 : q.n;
    if (ns < 64 || ns > hi || 2.0 * half * band > q.most) continue;
    z.n = q.n;
    z.ns = ns;
    break;
  }
  if (!z.n) return;
  z.even = even;
  z.Mo = even ? P.M / 2 + 1 : P.M;
  z.half = half;
  z.band = band;
  z.h = 2.0 * half * 1.25 / z.n;  // node pitch in ROI pitches: a margin of a quarter
  const double centre = even ? 0.0 : 0.5 * (P.M - 1) - P.msh;
  z.delta = P.delta * z.h;
  // node k at x = (k - msh) h: the first stored node
  const double first = centre + ((even ? z.n / 2 : 0) - 0.5 * (z.n - 1)) * z.h;
  z.msh = -first / z.h;
}

// Do the nodes pay?  The interpolation runs in FP64 at two multiply-adds per clock
// and SM (0.63 million a microsecond), so on small grids with a large ROI, where it
// cannot fold (off the axis, membranes), it takes longer than all that the nodes
// save.  Microseconds of both sides, fitted to whole propagations of N = 41 to 5,401
// with either route (general / nodes):
//   FP32, membrane, 512^2, 128 nodes: N = 401 120 / 202, 801 161 / 213, 1,601 258 / 233
//   FP32, off the axis, 1024^2, 128 nodes: 801 245 / 415, 1,601 295 / 423
//   FP32, on the axis, 512^2: 41 73 / 68, 1,601 117 / 82; 64^2: 41 48 / 55
//   dense, off the axis, 1024^2, 128 nodes: 801 260 / 423, 2,401 355 / 434, 3,601 538 / 436
//   dense, membrane, 1024^2, 64 nodes: 201 310 / 340, 401 372 / 343
//   SA-CZT, off the axis, 1024^2, 128 nodes: 401 431 / 479, 801 719 / 485
// FP32 grids of 2,000 and more columns keep the nodes, whose error is the smaller one
// (N = 2,401, 512^2: 1.6e-7 of the field against 3.5e-7) and whose rows are decimated
// from about 3,000 on.
static bool nodes_pay(const Plan& P) {
  const NodeSet& z = P.nd;
  const double ns = z.ns, Mo = z.Mo, M2 = (double)P.M * P.M, N = (double)P.N;
  const bool sym = !P.has_deform;  // the field of a whole flat plate is its own transpose
  const double interp = 1.15 * (2.0 * ns * Mo * ns * (sym ? 2.0 : 1.0) + 2.0 * ns * Mo * Mo * (sym ? 0.5 : 1.0)) / 630e3;
  const double epilogue = 1e-4 * M2;  // the general one: an FP64 sine pair per sample
  if (P.form == FZP_FORM_SACZT)
    return 88.0 + interp < (P.M % 128 ? 30.0 + 0.9 * N : 148.0 + 0.45 * N) + epilogue;
  if (P.form == FZP_FORM_DENSE) {
    const double passes = P.passes.empty() ? 1.0 : (double)P.passes.size();
    const double row = P.has_deform ? 0.14 : P.M > 512 ? 0.075 : 0.045;
    return interp < (P.M > 64 ? 25.0 : 5.0) + epilogue + 70.0 * (passes - 1.0) + row * N * passes;
  }
  const double side = P.M / 1024.0, row = sym ? 0.079 * side * side : 0.284 * std::pow(side, 1.6);
  return N >= 2000.0 || interp + 7.0 < epilogue + row * N;
}

void nodes_choose(Plan& P) {
  P.nd = NodeSet{};
  const bool centred = P.msh == (double)(P.M / 2);
  if (P.form == FZP_FORM_SACZT) {
    // the propagated plane fills the padded grid, P dx wide, at the distance z_F
    if (saczt_layout(P) == FZP_OK) place_nodes(P, centred, (double)P.sa.P * P.dx * P.p / (P.lambda * P.sa.zF), 128);
    const double dist = P.sa.zF;
    if (P.nd.n > 0 && !nodes_pay(P)) P.nd = NodeSet{};
    P.nd.dist = dist;
    return;
  }
  const bool dense = P.form == FZP_FORM_DENSE && P.precision == FZP_PREC_SPLIT_BF16 && P.cluster_req <= 1 && P.levels <= 4;
  const bool seg = P.form == FZP_FORM_BLUESTEIN && P.precision == FZP_PREC_FP32 && P.conv_req != 1;
  P.nd.dist = P.f;
  if (!dense && !seg) return;
  const bool flat = !P.has_deform;
  place_nodes(P, flat && centred, 2.0 * P.R / (P.lambda * P.f) * P.p, dense && !flat ? 64 : 128);
  if (P.nd.n > 0 && !nodes_pay(P)) P.nd = NodeSet{};
  P.nd.dist = P.f;
}

bool nodes_two_masks(const Plan& P) {
  if (P.nd.n == 0 || P.form != FZP_FORM_DENSE) return false;
  const int m = mask_kind(P);
  return m == MASK_MEMBRANE || m == MASK_QUAD;
}

fzp_status nodes_layout(Plan& P, FormSizes* out) {
  NodeSet& z = P.nd;
  const int64_t ncols = P.fold ? P.c + 1 : P.N;
  z.kblocks = (ncols + BK - 1) / BK;
  out->A = (size_t)z.kblocks * (size_t)(z.ns / 64) * 2 * SUB;
  out->sched = sizeof(int) * (size_t)(3 * ((z.kblocks + 7) / 8) + 1);
  out->X = (size_t)z.ns * P.M * sizeof(double2);
  return FZP_OK;
}

// W: per plan, also in a batch (it depends on the plan's band).  An even field's
// plan also gets the matrix of all n nodes, for row ranges that are not their
// own mirror image (a batch runs whole apertures only).  Factors on the host
// (ns^3 / 6 multiply-adds), solves for all outputs on the GPU (on the host the
// two matrices of a 512^2 ROI took 0.8 ms of a plan).
fzp_status nodes_upload(Plan& P) {
  NodeSet& z = P.nd;
  const bool full = z.even && P.owns_buffers;
  const size_t nw = (size_t)z.ns * z.Mo, nf = (size_t)z.ns * z.ns * (full ? 4 : 2);
  const size_t total = nw + (full ? (size_t)z.n * P.M : 0) + nf + 2 * (size_t)P.M;
  FZP_CUDA_TRY(cudaMalloc(&z.d_W, total * sizeof(double)));
  P.device_bytes += total * sizeof(double);
  z.d_Wy = full ? z.d_W + nw : z.d_W;
  double* dL = z.d_W + (total - nf);
  z.d_chirp = reinterpret_cast<double2*>(dL - 2 * (size_t)P.M);  // 16-byte aligned: even counts throughout
  std::unique_ptr<double[]> L(new (std::nothrow) double[nf]);
  if (!L) return set_error(FZP_E_OOM, "host allocation failed");
  InterpSpec a{z.n, z.ns, P.M, z.Mo, z.even ? 1 : 0, z.h / z.half, M_PI * z.band * z.half, z.half, P.msh, P.p * P.p / (2.0 * P.lambda * z.dist)};
  node_factor(z.n, z.ns, z.even ? 1 : 0, a.h, a.c, L.get());
  if (full) node_factor(z.n, z.ns, -1, a.h, a.c, L.get() + (size_t)2 * z.ns * z.ns);
  FZP_CUDA_TRY(cudaMemcpy(dL, L.get(), nf * sizeof(double), cudaMemcpyHostToDevice));
  double* Wy = full ? z.d_Wy : nullptr;
  if (z.ns == 64) k_interp_W<2><<<(unsigned)z.Mo, full ? 64 : 32>>>(a, dL, z.d_W, Wy, z.d_chirp);
  else k_interp_W<4><<<(unsigned)z.Mo, full ? 64 : 32>>>(a, dL, z.d_W, Wy, z.d_chirp);
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status nodes_fill(Plan& P, cudaStream_t s) {
  const NodeSet& z = P.nd;
  const int64_t ncols = P.fold ? P.c + 1 : P.N;
  const int64_t threads = z.kblocks * 4 * z.ns;
  const unsigned grid = (unsigned)std::min<int64_t>(8 * P.dn.num_sms, (threads + 255) / 256);
  k_nodes_A<<<grid, 256, 0, s>>>(z.ns / 64, ncols, z.kblocks, P.fold ? 0 : P.c, P.fold ? 1 : 0, P.kappa, z.msh, z.delta,
                                 reinterpret_cast<uint8_t*>(P.dn.d_A));
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status nodes_rows(Plan& P, int64_t j0, int64_t rows, bool octant, cudaStream_t s) {
  const NodeSet& z = P.nd;
  NodeArgs a{};
  a.mg = P.mg;
  if (P.fold) a.mg.c = 0;
  a.ph = phase_rule(P, P.pass_index >= 0 ? &P.passes[P.pass_index] : nullptr);
  a.j_begin = j0;
  a.j_end = j0 + rows;
  a.octant = octant ? 1 : 0;
  a.kblocks = z.kblocks;
  a.promote = P.dn.promote_kblocks;
  // K blocks per unit: about three units per SM where the aperture is small
  // (every unit ends in a promotion of 256 KiB into C1), whole promotions where
  // it is large
  const double R = std::sqrt((double)P.mg.sR), share = (double)rows / (P.fold ? P.c + 1 : P.N);
  const double blocks = M_PI * R * R * (P.fold ? 0.25 : 1.0) * (octant ? 0.5 : 1.0) * share / (BK * 512.0);
  a.group = (int)std::min<double>(std::max(8.0, std::ceil(blocks / (3.0 * P.dn.num_sms))), (double)a.promote);
  if (a.group < 8) a.group = 8;
  a.nchunks = (int)((z.kblocks + a.group - 1) / a.group);
  a.sched = P.dn.d_sched;
  a.A = reinterpret_cast<const uint8_t*>(P.dn.d_A);
  a.err = P.d_err;
  P.dominant = "k_nodes";
  const int mask = mask_kind(P);
  if (mask == MASK_MEMBRANE) {
    a.df = deform_coef(P);
    return a.df.direct > 1 ? launch<1, MASK_DIRECT>(P, a, s) : launch<1, MASK_MEMBRANE>(P, a, s);
  }
  if (mask == MASK_QUAD) return launch<1, MASK_QUAD>(P, a, s);
  if (z.ns == 64) return mask == MASK_PARITY ? launch<1, MASK_PARITY>(P, a, s) : launch<1, MASK_SIGNED>(P, a, s);
  return mask == MASK_PARITY   ? launch<2, MASK_PARITY>(P, a, s)
         : mask == MASK_SIGNED ? launch<2, MASK_SIGNED>(P, a, s)
                               : launch<2, MASK_LEVELS>(P, a, s);
}

fzp_status nodes_table_images(Plan& P, const void* E, int64_t ncols, int64_t stride, int64_t kblocks, void* A) {
  const int64_t threads = kblocks * 4 * P.nd.ns;
  k_nodes_table<<<(unsigned)std::min<int64_t>(8 * P.dn.num_sms, (threads + 255) / 256), 256>>>(
      P.nd.ns / 64, ncols, kblocks, reinterpret_cast<const float2*>(E), stride, reinterpret_cast<uint8_t*>(A));
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status nodes_zoom_images(Plan& P, int64_t ncols, int64_t kblocks, void* A) {
  const NodeSet& z = P.nd;
  const double lz = P.lambda * z.dist;
  const int64_t threads = kblocks * 4 * z.ns;
  k_nodes_A<<<(unsigned)std::min<int64_t>(8 * P.dn.num_sms, (threads + 255) / 256), 256>>>(
      z.ns / 64, ncols, kblocks, ncols / 2, 0, P.dx2 / lz, z.msh, z.h * P.p * P.dx / lz, reinterpret_cast<uint8_t*>(A));
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status nodes_loaded_rows(Plan& P, const float* src, int64_t rows, int64_t stride, int64_t kblocks, const void* A,
                             int* sched, int part, bool lower, cudaStream_t s) {
  NodeArgs a{};
  a.j_end = rows;
  a.octant = lower ? 1 : 0;
  a.kblocks = kblocks;
  a.promote = 128;
  a.group = (int)std::min<int64_t>(64, std::max<int64_t>(8, rows / 256 * kblocks / (lower ? 2 : 1) / (3 * P.dn.num_sms)));
  a.nchunks = (int)((kblocks + a.group - 1) / a.group);
  a.sched = sched;
  a.ld_src = src;
  a.ld_stride = stride;
  a.A = reinterpret_cast<const uint8_t*>(A);
  a.err = P.d_err;
  a.y_off = part * P.nd.ns * 2;
  return P.nd.ns == 64 ? launch<1, MASK_LOADED>(P, a, s) : launch<2, MASK_LOADED>(P, a, s);
}

fzp_status nodes_epilogue(Plan& P, void* d_field, int accumulate, bool sym, cudaStream_t s) {
  const NodeSet& z = P.nd;
  const bool eveny = z.even && !z.yfull;
  const int ny = z.yfull ? z.n : z.ns, Moy = eveny ? z.Mo : P.M;
  k_interp_rows<<<dim3((unsigned)(z.ns / 32), (unsigned)Moy), 128, 0, s>>>(
      ny, z.ns, Moy, sym ? 1 : 0, z.yfull ? z.d_Wy : z.d_W, P.d_Uacc, z.d_X);
  // e^{ikf} / i: f / lambda - 1/4 turns
  const double turns = std::fmod(P.f / P.lambda, 1.0) - 0.25, amp = P.dx2 / (P.lambda * z.dist);
  InterpOut a{P.M, z.ns, Moy, eveny ? 1 : 0, z.Mo, z.even ? 1 : 0, sym ? 1 : 0,
              make_double2(amp * std::cos(2.0 * M_PI * turns), amp * std::sin(2.0 * M_PI * turns)), accumulate};
  k_interp_cols<<<dim3((unsigned)((z.Mo + ITX - 1) / ITX), (unsigned)((Moy + ITY - 1) / ITY)), 2 * ITX * ITY, 0, s>>>(
      a, z.d_W, z.d_X, z.d_chirp, reinterpret_cast<double2*>(d_field));
  P.launches += 2;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status nodes_mask(Plan& P, int64_t j0, int64_t rows, uint8_t* out, cudaStream_t s) {
  const int64_t warps = (rows + 31) / 32 * ((P.N + MASK_COLS - 1) / MASK_COLS);
  const unsigned grid = (unsigned)std::min<int64_t>((warps + 3) / 4, 65535);
  k_mask_nodes<<<grid, 128, 0, s>>>(P.mg, phase_rule(P, nullptr), mask_kind(P), P.N, j0, rows, out);
  P.launches += 1;
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

}  // namespace fzp
