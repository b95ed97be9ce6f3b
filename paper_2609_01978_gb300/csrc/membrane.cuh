// membrane.cuh -- the membrane generators' walk of the deformation phase along
// a row and the BF16 split of the mask values (dense.cu, nodes.cu).
#pragma once

#include <stdint.h>

#include "fzp_internal.cuh"

namespace fzp {

// Membrane pass: one row's T cos(phi) (or T sin(phi)) on 8-column chunks of a
// 32-column block given the block's open bits, as BF16 hi and lo planes (the
// 16-byte chunks of the 64-byte-swizzled row).  phi / 2 pi = 2 w / lambda in
// FP32, walked along the row from the first column: the wrinkle's phasor
// e^{2 pi i t} (t = di kx + dj ky, integer turns dropped exactly) turns by
// e^{2 pi i kx} per column, a ridge's g = exp(-q d^2) by its ratio r, which
// itself scales by rho = exp(-2 q nx^2); the sum is reduced to [-1/2, 1/2]
// turns before one hardware sine or cosine (absolute error below 4e-7; the
// walk adds ~1e-6 relative over 32 columns).  A ridge below 1e-30 at the
// first column stays below 1e-29 in the block (its width is hundreds of
// columns) and is left out.
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

// Both masks of a membrane, T cos(phi) and T sin(phi), on the 8-column parts
// [q0, q0 + nq) of a 32-column block: the walk above, one sine and one cosine
// per sample, each split into its hi and lo plane; NR ridges.
template <int NR>
__device__ __forceinline__ void cx_store2_n(const DeformCoef& d, const CxRow& r, int64_t di0, uint32_t bits,
                                            uint8_t* ch, uint8_t* cl, uint8_t* sh, uint8_t* sl, int sw, int q0,
                                            int nq) {
  constexpr float TWO_PI = 6.28318530717958648f;
  float fi = (float)(di0 + 8 * q0);
  const float th = fmaf(fi, d.kxh, r.fjkh);
  float tt = (th - rintf(th)) + fmaf(fi, d.kxl, r.fjkl);
  tt -= rintf(tt);
  float ws, wc;
  __sincosf(TWO_PI * tt, &ws, &wc);
  float g[NR > 0 ? NR : 1], rr[NR > 0 ? NR : 1];
#pragma unroll
  for (int e = 0; e < NR; ++e) {
    g[e] = 0.0f;
    rr[e] = 1.0f;
    const float d0 = fmaf(fi, d.nx[e], r.cr[e]);
    const float ex = d.q[e] * d0 * d0;
    if (ex < 69.0f) {
      g[e] = __expf(-ex);
      rr[e] = __expf(-d.q[e] * d.nx[e] * fmaf(2.0f, d0, d.nx[e]));
    }
  }
#pragma unroll 1
  for (int q = q0; q < q0 + nq; ++q) {
    uint32_t hc[4], lc[4], hs[4], ls[4];
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
      float vc[2], vs[2];
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        float wz = d.amp2 * ws * fmaf(-d.tq, fmaf(fi, fi, r.fj2), 1.0f);
#pragma unroll
        for (int e = 0; e < NR; ++e) {
          wz = fmaf(d.h2[e], g[e], wz);
          g[e] *= rr[e];
          rr[e] *= d.rho[e];
        }
        const float nws = fmaf(ws, d.zc, wc * d.zs);
        wc = fmaf(wc, d.zc, -ws * d.zs);
        ws = nws;
        fi += 1.0f;
        wz -= rintf(wz);
        const float x = TWO_PI * wz;
        const bool open = ((bits >> (8 * q + k + z)) & 1u) != 0;
        vc[z] = open ? __cosf(x) : 0.0f;
        vs[z] = open ? __sinf(x) : 0.0f;
      }
      split2(vc[0], vc[1], hc[k / 2], lc[k / 2]);
      split2(vs[0], vs[1], hs[k / 2], ls[k / 2]);
    }
    const int o = (q ^ sw) << 4;
    *reinterpret_cast<uint4*>(ch + o) = make_uint4(hc[0], hc[1], hc[2], hc[3]);
    *reinterpret_cast<uint4*>(cl + o) = make_uint4(lc[0], lc[1], lc[2], lc[3]);
    *reinterpret_cast<uint4*>(sh + o) = make_uint4(hs[0], hs[1], hs[2], hs[3]);
    *reinterpret_cast<uint4*>(sl + o) = make_uint4(ls[0], ls[1], ls[2], ls[3]);
  }
}

__device__ __forceinline__ void cx_store2(const DeformCoef& d, const CxRow& r, int64_t di0, uint32_t bits, uint8_t* ch,
                                          uint8_t* cl, uint8_t* sh, uint8_t* sl, int sw, int q0, int nq) {
  switch (d.n) {
    case 0: cx_store2_n<0>(d, r, di0, bits, ch, cl, sh, sl, sw, q0, nq); break;
    case 1: cx_store2_n<1>(d, r, di0, bits, ch, cl, sh, sl, sw, q0, nq); break;
    case 2: cx_store2_n<2>(d, r, di0, bits, ch, cl, sh, sl, sw, q0, nq); break;
    default: cx_store2_n<3>(d, r, di0, bits, ch, cl, sh, sl, sw, q0, nq); break;
  }
}

}  // namespace fzp
