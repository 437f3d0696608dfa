// Arithmetic of the centroids that the k-means kernels of partition.cu and kmeans_tc.cu share.
#pragma once
#include "kernels.cuh"

namespace spr {

// Mean of a group from its fixed-point sum (inv_scale = 2^-shift): the definition of an updated centroid
__device__ __forceinline__ float group_mean(i64 sum, double inv_scale, int count) { return (float)((double)sum * inv_scale / (double)count); }

// The same, to the bit, for several sums of one group: a reciprocal y of the count by Newton-Raphson steps, and quotients with one correction by
// their remainder (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990).  a / n lies at least 2^-54 / n away
// (relatively) from any midpoint between two float64 that is not itself, n < 2^31, and q + (a - q n) y, the remainder being exact, misses it by 2^-104.
struct GroupMean {
  double scale, n, y;
  __device__ __forceinline__ GroupMean(int count, double inv_scale) : scale(inv_scale), n((double)count) {
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(n));
    y = fma(y, fma(-n, y, 1.0), y);
    y = fma(y, fma(-n, y, 1.0), y);
  }
  __device__ __forceinline__ float operator()(i64 sum) const {
    const double a = (double)sum * scale, q = a * y;
    return (float)fma(fma(-q, n, a), y, q);
  }
};
// Squared norms of four rows by a warp, of each of which a lane has two columns (zeros beyond the row): in float64, rounded once.  A lane gets the
// norm of row lane / 8: at the first two levels of the butterfly it keeps half of the rows that it has.
__device__ __forceinline__ float norms_of_four(const float2 (&v)[4], int lane) {
  double s[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) s[b] = (double)v[b].x * (double)v[b].x + (double)v[b].y * (double)v[b].y;
#pragma unroll
  for (int half = 2; half > 0; half >>= 1) {
    const bool upper = lane & (8 * half);
#pragma unroll
    for (int b = 0; b < half; ++b) s[b] = (upper ? s[b + half] : s[b]) + __shfl_xor_sync(0xffffffffu, upper ? s[b] : s[b + half], 8 * half);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
  return (float)s[0];
}
// the three bf16 words of ||mu_c||^2 (all bits of a float32), then zeros: a row of the operand of the norm step
__device__ __forceinline__ uint4 norm_words(float v) {
  const __nv_bfloat16 w0 = __float2bfloat16_rn(v);
  const float v1 = v - __bfloat162float(w0);
  const __nv_bfloat16 w1 = __float2bfloat16_rn(v1), w2 = __float2bfloat16_rn(v1 - __bfloat162float(w1));
  return make_uint4((uint32_t)__bfloat16_as_ushort(w0) | ((uint32_t)__bfloat16_as_ushort(w1) << 16), __bfloat16_as_ushort(w2), 0u, 0u);
}

}  // namespace spr
