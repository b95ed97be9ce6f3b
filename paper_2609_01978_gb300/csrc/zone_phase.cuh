// zone_phase.cuh -- the fixed-point zone phase that mask generators walk along a
// row (nodes.cu, bluestein.cu).
#pragma once

#include <cmath>

#include "fzp_internal.cuh"

namespace fzp {

// Fixed-point zone phase: phase64(s) = s K mod 2^64 (K = floor(kappa 2^63): the
// zone's parity is the top bit; more than two levels: K = floor(kappa_L / L 2^64), the
// level is floor(phase L / 2^64)).  The true phase lies less than s (in units
// of 2^-64) above it; the 32-bit walk over a block adds less than 600 units of
// 2^-32 and fl(s kappa) less than 8, so E = 640 + (s_max >> 32).
struct PhaseRule {
  uint64_t K;
  uint32_t E;
  int lmod;            // more than two levels: L
  uint64_t pos, neg;   // level sets with value +1, -1
  int open_even;       // 1: positive-centred binary plate
};

// The rule of a plan's plate; mp: the level sets of a signed-mask pass.
inline PhaseRule phase_rule(const Plan& P, const MaskPass* mp) {
  PhaseRule r{};
  r.E = 640u + (uint32_t)(P.mg.sR >> 32);
  if (P.levels > 2) {
    r.K = (uint64_t)std::floor(std::ldexp(P.kappa_mask / P.levels, 64));
    r.lmod = P.levels;
    if (mp) {
      r.pos = mp->pos;
      r.neg = mp->neg;
    }
  } else {
    r.K = (uint64_t)std::floor(std::ldexp(P.kappa_mask, 63));
    r.open_even = P.mg.centre_open;
  }
  return r;
}

// The 16 columns from di0 of row dj: upper 32 bits of the phase of the first
// column, their first and second difference.
struct Walk16 {
  uint32_t f, d, c2;
};
__device__ __forceinline__ Walk16 walk16(int64_t di0, int64_t dj2, const PhaseRule& r) {
  Walk16 w;
  w.f = (uint32_t)(((uint64_t)(dj2 + di0 * di0) * r.K + (r.open_even ? (1ull << 63) : 0ull)) >> 32);
  w.d = (uint32_t)(((uint64_t)(2 * di0 + 1) * r.K) >> 32);
  w.c2 = (uint32_t)(r.K >> 32) * 2u + (uint32_t)((r.K >> 31) & 1u);
  return w;
}

// Open bits of the binary plate on those columns (bit p: column di0 + p);
// false if a phase comes within E of a zone boundary: the caller takes the
// exact rule.
__device__ __forceinline__ bool walk_bits16(Walk16 w, const PhaseRule& r, uint32_t& bits) {
  uint32_t near = 0xFFFFFFFFu, b = 0u;
  const uint32_t e2 = 2u * r.E;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    near = min(near, (w.f << 1) + e2);
    b = __funnelshift_l(w.f, b, 1);  // the sign shifts in: column p at bit 15 - p
    w.f += w.d;
    w.d += w.c2;
  }
  bits = __brev(b) >> 16;
  return near >= 2u * e2;
}

}  // namespace fzp
