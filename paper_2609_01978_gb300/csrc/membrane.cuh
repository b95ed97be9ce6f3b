// membrane.cuh -- the membrane generators' walk of the deformation phase along
// a row and the BF16 split of the mask values (dense.cu, nodes.cu).
#pragma once

#include <stdint.h>

#include "fzp_internal.cuh"

namespace fzp {

// Membrane generators: T cos(phi) and T sin(phi) of a row's columns given their
// open bits.  phi / 2 pi = 2 w / lambda in FP32: the wrinkle's turns t = di kx + dj
// ky (integer turns dropped exactly) through a hardware sine, times the taper,
// plus a Gaussian per ridge; walked along the row where the deformation is smooth
// on the columns (MembraneWalk), evaluated column by column where it is not
// (MembraneDirect).  The sum is reduced to [-1/2, 1/2] turns before one hardware
// sine or cosine (absolute error below 4e-7).
struct CxRow {
  float fjkh, fjkl, fj2, cr[3];  // row terms: dj kyh, dj kyl, dj^2, ridge offsets
};

__device__ __forceinline__ void cx_row_init(const DeformCoef& d, int64_t dj, CxRow& r) {
  const float fj = (float)dj;
  r.fjkh = fj * d.kyh;
  r.fjkl = fj * d.kyl;
  r.fj2 = fj * fj;
#pragma unroll
  for (int e = 0; e < 3; ++e) r.cr[e] = (fj - d.pj[e]) * d.ny[e] - d.pi_[e] * d.nx[e];
}

// Two FP32 values -> packed BF16 hi (RN) and lo (RN of the remainder), lower
// half from a: one cvt.rn.bf16x2 per plane (a goes to the upper half of the
// instruction's result when given first, so b is given first).
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(b), "f"(a));
  const float ah = __uint_as_float(hi << 16), bh = __uint_as_float(hi & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(b - bh), "f"(a - ah));
}

// The membrane's phase (turns, 2 w / lambda) walked along a row from column di0:
// the scaled wrinkle amp sin by its second difference, s' = s + e, e' = e - 4
// sin^2(pi kx) s (one product instead of a rotation's four, and no growth of the
// rounding at the small angles of a wrinkle), the taper by its constant second
// difference, a ridge by its ratio, kept as the ratio less one: g += g r1, r1 <-
// r1 rho - (1 - rho) (a ratio near one rounded to FP32 is off by 3e-8 and more
// each, 2e-5 of g over 32 columns).  Started exactly every 16 (k_seg, k_nodes) or
// 32 columns (k_dec).  NR ridges.  A ridge below 1e-30 at the first column is left
// out of the walk: DeformCoef::direct keeps ridges from here that could rise again
// within it.
template <int NR>
struct MembraneWalk {
  float s, e, tap, dt, ddt, z4;
  float g[NR > 0 ? NR : 1], r1[NR > 0 ? NR : 1], rho[NR > 0 ? NR : 1], eta[NR > 0 ? NR : 1];

  __device__ __forceinline__ MembraneWalk(const DeformCoef& d, const CxRow& r, int32_t di0) {
    constexpr float TWO_PI = 6.28318530717958648f;
    const float fi = (float)di0;
    const float th = fmaf(fi, d.kxh, r.fjkh);
    float tt = (th - rintf(th)) + fmaf(fi, d.kxl, r.fjkl);
    tt -= rintf(tt);
    float ws, wc;
    __sincosf(TWO_PI * tt, &ws, &wc);
    z4 = d.z4;
    s = d.amp2 * ws;
    e = d.amp2 * fmaf(0.5f * d.z4, ws, d.zs * wc);  // s minus its left neighbour
    tap = fmaf(-d.tq, fmaf(fi, fi, r.fj2), 1.0f);
    dt = -d.tq * fmaf(2.0f, fi, 1.0f);
    ddt = -2.0f * d.tq;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      g[k] = 0.0f;
      r1[k] = 0.0f;
      rho[k] = d.rho[k];
      eta[k] = d.eta[k];
      const float d0 = fmaf(fi, d.nx[k], r.cr[k]);
      const float ex = d.q[k] * d0 * d0;
      if (ex < 69.0f) {
        g[k] = d.h2[k] * __expf(-ex);
        // e^-x - 1: its series while |x| is small (wide ridges)
        const float x = d.q[k] * d.nx[k] * fmaf(2.0f, d0, d.nx[k]);
        const float p = fmaf(x, fmaf(x, fmaf(x, fmaf(x, -1.0f / 120.0f, 1.0f / 24.0f), -1.0f / 6.0f), 0.5f), -1.0f);
        r1[k] = fabsf(x) < 0.125f ? x * p : __expf(-x) - 1.0f;
      }
    }
  }
  // the phase at the column, then one column on
  __device__ __forceinline__ float next() {
    float wz = s * tap;
    e = fmaf(-z4, s, e);
    s += e;
    tap += dt;
    dt += ddt;
#pragma unroll
    for (int v = 0; v < NR; ++v) {
      wz += g[v];
      g[v] = fmaf(g[v], r1[v], g[v]);
      r1[v] = fmaf(r1[v], rho[v], -eta[v]);
    }
    return wz;
  }
};

// The same phase evaluated at the column, for ridges and wrinkles of any width.
__device__ __forceinline__ float membrane_turns(const DeformCoef& d, const CxRow& r, float fi) {
  constexpr float TWO_PI = 6.28318530717958648f;
  const float th = fmaf(fi, d.kxh, r.fjkh);
  float tt = (th - rintf(th)) + fmaf(fi, d.kxl, r.fjkl);
  tt -= rintf(tt);
  float wz = d.amp2 * __sinf(TWO_PI * tt) * fmaf(-d.tq, fmaf(fi, fi, r.fj2), 1.0f);
#pragma unroll
  for (int e = 0; e < 3; ++e)
    if (e < d.n) {
      const float dd = fmaf(fi, d.nx[e], r.cr[e]);
      wz = fmaf(d.h2[e], __expf(-d.q[e] * dd * dd), wz);
    }
  return wz;
}

struct MembraneDirect {
  const DeformCoef& d;
  const CxRow& r;
  float fi;
  __device__ __forceinline__ MembraneDirect(const DeformCoef& d_, const CxRow& r_, int32_t di0) : d(d_), r(r_), fi((float)di0) {}
  __device__ __forceinline__ float next() {
    const float wz = membrane_turns(d, r, fi);
    fi += 1.0f;
    return wz;
  }
};

struct MembraneDirect2 {
  MembraneDirect a, b;
  __device__ __forceinline__ MembraneDirect2(const MembraneDirect& a_, const MembraneDirect& b_) : a(a_), b(b_) {}
  __device__ __forceinline__ float2 next() {
    const float wa = a.next();
    return make_float2(wa, b.next());
  }
};

// Two walks side by side, every step's operations in pairs.
template <int NR>
struct MembraneWalk2 {
  float2 s, e, tap, dt, ddt, mz4;
  float2 g[NR > 0 ? NR : 1], r1[NR > 0 ? NR : 1], rho[NR > 0 ? NR : 1], meta[NR > 0 ? NR : 1];

  __device__ __forceinline__ MembraneWalk2(const MembraneWalk<NR>& a, const MembraneWalk<NR>& b) {
    s = make_float2(a.s, b.s);
    e = make_float2(a.e, b.e);
    tap = make_float2(a.tap, b.tap);
    dt = make_float2(a.dt, b.dt);
    ddt = pair2(a.ddt);
    mz4 = pair2(-a.z4);
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      g[k] = make_float2(a.g[k], b.g[k]);
      r1[k] = make_float2(a.r1[k], b.r1[k]);
      rho[k] = pair2(a.rho[k]);
      meta[k] = pair2(-a.eta[k]);
    }
  }
  __device__ __forceinline__ float2 next() {
    float2 wz = mul2(s, tap);
    e = fma2(mz4, s, e);
    s = cadd(s, e);
    tap = cadd(tap, dt);
    dt = cadd(dt, ddt);
#pragma unroll
    for (int v = 0; v < NR; ++v) {
      wz = cadd(wz, g[v]);
      g[v] = fma2(g[v], r1[v], g[v]);
      r1[v] = fma2(r1[v], rho[v], meta[v]);
    }
    return wz;
  }
};

// The sum with another phase reduced to [-1/2, 1/2] turns, in radians (|x| < 2^22).
__device__ __forceinline__ float2 reduced_rad(float2 x) {
  const float2 rint2 = pair2(12582912.0f);  // 1.5 2^23
  const float2 n = csub(cadd(x, rint2), rint2);
  return mul2(csub(x, n), pair2(6.28318530717958648f));
}

// Both masks of a membrane, T cos(phi) and T sin(phi), on the 32 columns from
// di0 (bit k of `bits`: column k open), as the row's four 16-byte parts in the
// planes cos hi, cos lo, sin hi, sin lo (`plane` bytes apart): columns k and
// k + 16 walk side by side, four at a time to the planes.
template <typename Walk2>
__device__ __forceinline__ void cx_store2_n(Walk2 walk, uint32_t bits, uint8_t* base, uint32_t plane, int sw) {
#pragma unroll 1
  for (int q = 0; q < 4; ++q, bits >>= 4) {
    uint32_t hc[2][2], lc[2][2], hs[2][2], ls[2][2];
#pragma unroll
    for (int k = 0; k < 4; k += 2) {
      float vc[2][2], vs[2][2];
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        const float2 x = reduced_rad(walk.next());
        const bool oa = (bits >> (k + z)) & 1u, ob = (bits >> (k + z + 16)) & 1u;
        vc[0][z] = oa ? __cosf(x.x) : 0.0f;
        vs[0][z] = oa ? __sinf(x.x) : 0.0f;
        vc[1][z] = ob ? __cosf(x.y) : 0.0f;
        vs[1][z] = ob ? __sinf(x.y) : 0.0f;
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        split2(vc[e][0], vc[e][1], hc[e][k / 2], lc[e][k / 2]);
        split2(vs[e][0], vs[e][1], hs[e][k / 2], ls[e][k / 2]);
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      uint8_t* o = base + ((((q >> 1) + 2 * e) ^ sw) << 4) + 8 * (q & 1);
      *reinterpret_cast<uint2*>(o) = make_uint2(hc[e][0], hc[e][1]);
      *reinterpret_cast<uint2*>(o + plane) = make_uint2(lc[e][0], lc[e][1]);
      *reinterpret_cast<uint2*>(o + 2 * plane) = make_uint2(hs[e][0], hs[e][1]);
      *reinterpret_cast<uint2*>(o + 3 * plane) = make_uint2(ls[e][0], ls[e][1]);
    }
  }
}

template <int NR>
__device__ __forceinline__ MembraneWalk2<NR> walk32(const DeformCoef& d, const CxRow& r, int32_t di0) {
  return MembraneWalk2<NR>(MembraneWalk<NR>(d, r, di0), MembraneWalk<NR>(d, r, di0 + 16));
}

// DIRECT: by column (kernels of their own: beside the walks it made them 4 % slower).
template <bool DIRECT>
__device__ __forceinline__ void cx_store2(const DeformCoef& d, const CxRow& r, int32_t di0, uint32_t bits, uint8_t* base,
                                          uint32_t plane, int sw) {
  if (DIRECT) {
    cx_store2_n(MembraneDirect2(MembraneDirect(d, r, di0), MembraneDirect(d, r, di0 + 16)), bits, base, plane, sw);
    return;
  }
  switch (d.n) {
    case 0: cx_store2_n(walk32<0>(d, r, di0), bits, base, plane, sw); break;
    case 1: cx_store2_n(walk32<1>(d, r, di0), bits, base, plane, sw); break;
    case 2: cx_store2_n(walk32<2>(d, r, di0), bits, base, plane, sw); break;
    default: cx_store2_n(walk32<3>(d, r, di0), bits, base, plane, sw); break;
  }
}

}  // namespace fzp
