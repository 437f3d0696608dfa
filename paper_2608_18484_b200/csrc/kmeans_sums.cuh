// Device functions of the k-means that the kernels of partition.cu and kmeans_tc.cu share.
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

// Adds 32 consecutive rows of one head (phi: the first, n_rows of them valid) to the fixed-point sums [C][R] and the counts of their groups
// assign[0 .. n_rows - 1], by one warp; ids outside [0, C) are in no sum.  A row is rounded once, as in a later move of that row, so the sums stay
// exact: x 2^shift = h 2^26 + l with h = rint(x 2^(shift - 26)) and l = rint of what is left, both below 2^26 and added over up to 32 rows in
// int32.  Lane = columns lane and lane + 32, two rows in flight, one atomic per (group present in the warp, column).
__device__ __forceinline__ void add_rows_to_sums(const float* phi, int ldphi, int n_rows, int r, int R, int C, const int* assign, i64* sums, int* counts, int shift) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int cl_mine = -1;
  if (lane < n_rows) { const int c = assign[lane]; if (c >= 0 && c < C) cl_mine = c; }
  const float s_hi = __int_as_float((127 + shift - 26) << 23);
  for (int cb = 0; cb < R; cb += 64) {                         // 64 columns at a time (two passes for raw activations)
    const int col = cb + lane;
    const bool ok0 = col < r, ok1 = col + 32 < r;
    const float* p = phi + col;
    unsigned todo = __ballot_sync(FULL, cl_mine >= 0);
    while (todo) {
      const int leader = __ffs(todo) - 1;
      const int cl = __shfl_sync(FULL, cl_mine, leader);
      unsigned m = __ballot_sync(FULL, cl_mine == cl);
      todo &= ~m;
      const int n = __popc(m);
      int h0 = 0, h1 = 0, l0 = 0, l1 = 0;
      auto add = [&](float xa, float xc) {
        const float y0 = xa * s_hi, y1 = xc * s_hi;
        const int a0 = __float2int_rn(y0), a1 = __float2int_rn(y1);
        h0 += a0; h1 += a1;
        l0 += __float2int_rn((y0 - (float)a0) * 67108864.f); l1 += __float2int_rn((y1 - (float)a1) * 67108864.f);
      };
      while (m) {
        const float* pa = p + (i64)(__ffs(m) - 1) * ldphi;
        m &= m - 1;
        const float* pb = m ? p + (i64)(__ffs(m) - 1) * ldphi : nullptr;
        m &= m - 1;
        const float a0 = ok0 ? pa[0] : 0.f, a1 = ok1 ? pa[32] : 0.f;
        const float b0 = ok0 && pb ? pb[0] : 0.f, b1 = ok1 && pb ? pb[32] : 0.f;
        add(a0, a1);
        add(b0, b1);
      }
      i64* sp = sums + (i64)cl * R + col;
      if (ok0) atomicAdd(reinterpret_cast<u64*>(sp), (u64)((i64)h0 * 67108864ll + l0));
      if (ok1) atomicAdd(reinterpret_cast<u64*>(sp + 32), (u64)((i64)h1 * 67108864ll + l1));
      if (lane == 0 && cb == 0) atomicAdd(counts + cl, n);
    }
  }
}

}  // namespace spr
