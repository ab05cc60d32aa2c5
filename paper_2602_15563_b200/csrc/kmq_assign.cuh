// Nearest stored centroid of a float32 weight, shared by the quantiser kernels.
//
// For sorted centroids the nearest one (ties to the lower, equal centroids to the lowest index) is found by counting
// the midpoints strictly below the weight.  The comparison is exact, yet made in float32: a float32 x lies above the
// real number mid = (c_i + c_{i+1}) / 2 iff it lies above the largest float32 that is not above mid.
#pragma once
#include "kmq_common.cuh"

namespace kmq {

// The midpoint of two stored centroids as an unevaluated float64 sum: (s + e) / 2 with s the rounded sum of the two
// and e its error (error-free transformation).
struct Mid {
  double s, e;
};

__device__ __forceinline__ Mid exact_mid(uint32_t a_bits, uint32_t b_bits) {
  const double a = (double)bf16_bits_to_float(a_bits), b = (double)bf16_bits_to_float(b_bits);
  Mid m;
  m.s = __dadd_rn(a, b);
  const double bb = __dadd_rn(m.s, -a);
  m.e = __dadd_rn(__dadd_rn(a, -__dadd_rn(m.s, -bb)), __dadd_rn(b, -bb));
  return m;
}

__device__ __forceinline__ bool above(double two_x, const Mid& m) {
  return two_x > m.s || (two_x == m.s && m.e < 0.0);
}

// Largest float32 that is not above the midpoint.
__device__ __forceinline__ float mid_threshold(const Mid& m) {
  const double half = __dmul_rn(0.5, m.s);
  float t = __double2float_rd(half);
  if (m.e < 0.0 && (double)t == half) {   // the midpoint itself is just below a float32: one step down
    const uint32_t u = __float_as_uint(t);
    t = __uint_as_float(t > 0.0f ? u - 1 : t < 0.0f ? u + 1 : 0x80000001u);
  }
  return t;
}

// Number of thresholds below x; monotone in the index because the centroids are sorted.
template <int BITS>
__device__ __forceinline__ int count_below(float x, const float* t) {
  int n = 0;
  if constexpr (BITS <= 2) {
#pragma unroll
    for (int i = 0; i < (1 << BITS) - 1; ++i) n += x > t[i] ? 1 : 0;
  } else {
#pragma unroll
    for (int step = 1 << (BITS - 1); step > 0; step >>= 1)
      if (x > t[n + step - 1]) n += step;
  }
  return n;
}

constexpr int kLayoutCanonical = 0, kLayoutTuned = 1, kLayoutPlanes = 2;

}  // namespace kmq
