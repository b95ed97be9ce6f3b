// sums.cuh -- sums of a few partial results without the rounding of their precision.
#pragma once

namespace fzp {

// x + y = s + e exactly (Knuth's two-sum; s the rounded sum).
__host__ __device__ __forceinline__ void two_sum_f(float x, float y, float& s, float& e) {
  s = x + y;
  const float t = s - x;
  e = (x - (s - t)) + (y - t);
}

// Sum of four FP32 values to within 2^-46 of the largest, in ten FP32 additions more
// than the plain sum and three FP64 operations (four conversions and three
// additions are seven; FP64 has two lanes per SM).
__host__ __device__ __forceinline__ double sum4(const float (&v)[4]) {
  float a, b, s, ea, eb, es;
  two_sum_f(v[0], v[2], a, ea);
  two_sum_f(v[1], v[3], b, eb);
  two_sum_f(a, b, s, es);
  return (double)s + (double)((ea + eb) + es);
}
__host__ __device__ __forceinline__ double sum4(const double (&v)[4]) { return (v[0] + v[2]) + (v[1] + v[3]); }

}  // namespace fzp
