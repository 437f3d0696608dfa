// The arithmetic of the centroids in csrc/kmeans_sums.cuh, on arrays in device memory: called by test_gpu_kmeans_arithmetic.py.
#include "kmeans_sums.cuh"

namespace {
__global__ void k_means(const long long* sums, const int* counts, int n, int shift, float* quick, float* divided) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double inv_scale = ldexp(1.0, -shift);
  quick[i] = spr::GroupMean(counts[i], inv_scale)(sums[i]);
  divided[i] = spr::group_mean(sums[i], inv_scale, counts[i]);
}
// rows [n][64], four rows by a warp
__global__ void k_norms(const float* rows, int n, float* out) {
  const int lane = threadIdx.x & 31, row0 = (blockIdx.x * blockDim.x + threadIdx.x) / 32 * 4;
  float2 v[4];
  for (int b = 0; b < 4; ++b) v[b] = row0 + b < n ? reinterpret_cast<const float2*>(rows + (size_t)(row0 + b) * 64)[lane] : make_float2(0.f, 0.f);
  const float norm = spr::norms_of_four(v, lane);
  if ((lane & 7) == 0 && row0 + lane / 8 < n) out[row0 + lane / 8] = norm;
}
}  // namespace

extern "C" int group_means(const long long* sums, const int* counts, int n, int shift, float* quick, float* divided) {
  k_means<<<(n + 127) / 128, 128>>>(sums, counts, n, shift, quick, divided);
  return cudaDeviceSynchronize();
}
extern "C" int row_norms(const float* rows, int n, float* out) {
  k_norms<<<(n + 15) / 16, 128>>>(rows, n, out);
  return cudaDeviceSynchronize();
}
