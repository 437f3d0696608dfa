// Response-Coupled Partitioning kernels (Section 4.1, Appendix B): sampled-query
// Gram matrix, batched Jacobi eigen-decomposition -> feature maps, response
// projections, k-means assignment/update, stable counting sort, group means.
#include <algorithm>
#include "kmeans_sums.cuh"

namespace spr {

// =============================================================================
// Gram matrices: M_K = Q_s^T Q_s / M_s (Appendix B.1) and
// M_Q = Ktilde^T Ktilde / (C_k^+ d) (Appendix B.2), float64 accumulation in order of the rows.
// Bound by latency and by conversions to float64 (16 per clock and SM; a warp alone takes 13 cycles for one): the rows of an entry are a chain of multiply-adds.
// So only the tiles on and above the diagonal are formed (the products of two mirrored entries are the same, a tile is also written mirrored), and
// they are small, 16 x 16, so that a few heads spread over the SMs.  128 threads, two neighbouring entries each; rows come a chunk ahead.
// (What the call takes for the sample / the centroids, us: 2 heads of d = 128, 256 and 38 rows, 15 / 6, 24 heads of 256 rows each 30 / 41; with 16 whole
// rows of the result per CTA 26 / 9 and 48 / 98, with tiles of 32 x 32 by two warps 34 / 17 and 48 / 184.)
// =============================================================================
constexpr int kGramChunk = 64, kGramTile = 16, kGramThreads = 128;
constexpr int gram_tiles(int d) { return (d / kGramTile) * (d / kGramTile + 1) / 2; }

template <int D> __device__ __forceinline__ void gram_tile(int t, int& i0, int& j0) {      // t-th tile by rows
  int i = 0;
  for (int left = t, n = D / kGramTile;; ++i, --n) {
    if (left < n) { i0 = i * kGramTile; j0 = (i + left) * kGramTile; return; }
    left -= n;
  }
}
// rows [kGramChunk][2][kGramTile]: the columns from i0 on, then those from j0 on
__device__ __forceinline__ void gram_accumulate(const double (*rows)[2][kGramTile], int nrows, double (&acc)[2]) {
  const int i = threadIdx.x / 8, j = threadIdx.x % 8 * 2;
#pragma unroll 8
  for (int s = 0; s < nrows; ++s) {
    const double xi = rows[s][0][i];
    const double2 xj = *reinterpret_cast<const double2*>(&rows[s][1][j]);
    acc[0] = fma(xi, xj.x, acc[0]);
    acc[1] = fma(xi, xj.y, acc[1]);
  }
}
template <int D> __device__ __forceinline__ void gram_store(double* M, int i0, int j0, const double (&acc)[2], double denom) {
  const int i = i0 + threadIdx.x / 8, j = j0 + threadIdx.x % 8 * 2;
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const double m = acc[v] / denom;
    M[i * D + j + v] = m;
    if (i0 != j0) M[(j + v) * D + i] = m;
  }
}

template <typename T, int D>
__global__ void __launch_bounds__(kGramThreads) k_sample_gram(const T* __restrict__ Q, i64 sb, i64 sh, i64 sn, int H, int N,
                                                              int Ms, u64 seed, int head0, double* __restrict__ Mout) {
  pdl_launch_dependents();                                     // (inputs of this kernel are the caller's)
  __shared__ __align__(16) double rows[kGramChunk][2][kGramTile];
  __shared__ int s_row[2][kGramChunk];                         // sampled rows of this chunk and the next
  const int bh = blockIdx.y, b = bh / H, h = bh % H, tid = threadIdx.x;
  const T* base = Q + b * sb + h * sh;
  const u64 U = sample_offset(seed, kTagQuerySample, head0 + bh);
  int i0, j0;
  gram_tile<D>(blockIdx.x, i0, j0);
  // eight columns of kOwn rows per thread and chunk
  constexpr int kOwn = kGramChunk * 2 * kGramTile / 8 / kGramThreads, kStep = kGramThreads / 4;
  const int s = tid / 4, c = tid % 4, col = c < 2 ? i0 + 8 * c : j0 + 8 * (c - 2);
  float v[kOwn][8] = {};
  const auto sample = [&](int s0) { if (tid < kGramChunk && s0 + tid < Ms) s_row[(s0 / kGramChunk) & 1][tid] = strided_row(s0 + tid, Ms, N, U); };
  const auto fetch = [&](int s0) {
#pragma unroll
    for (int u = 0; u < kOwn; ++u)
      if (s0 + s + u * kStep < Ms) load8(base + (i64)s_row[(s0 / kGramChunk) & 1][s + u * kStep] * sn + col, v[u]);
  };
  double acc[2] = {0.0, 0.0};
  sample(0);
  __syncthreads();
  fetch(0);
  for (int s0 = 0; s0 < Ms; s0 += kGramChunk) {
    sample(s0 + kGramChunk);
    __syncthreads();                                           // (the chunk before has been read)
#pragma unroll
    for (int u = 0; u < kOwn; ++u)
#pragma unroll
      for (int k = 0; k < 8; ++k) rows[s + u * kStep][c / 2][c % 2 * 8 + k] = (double)v[u][k];
    __syncthreads();
    if (s0 + kGramChunk < Ms) fetch(s0 + kGramChunk);
    gram_accumulate(rows, min(kGramChunk, Ms - s0), acc);
  }
  gram_store<D>(Mout + (i64)bh * D * D, i0, j0, acc, (double)Ms);
}

// kappa [BH][C][D] float32, n [BH][C] group sizes.  Empty groups are skipped and the
// remaining centroids are centred by their uniform mean (summed in order of the groups).
template <int D>
__global__ void __launch_bounds__(kGramThreads) k_centroid_gram(const float* __restrict__ kappa, const int* __restrict__ n, int C,
                                                                double* __restrict__ Mout) {
  pdl_wait();                                                   // the group means come from the kernel before
  pdl_launch_dependents();
  __shared__ __align__(16) double rows[kGramChunk][2][kGramTile];
  __shared__ int s_n[kMaxGroups];
  __shared__ double s_mean[2 * kGramTile];
  __shared__ int s_cnt;
  const int bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int i0, j0;
  gram_tile<D>(blockIdx.x, i0, j0);
  // lane = one of the 32 columns of the tile's rows, a warp has eight rows of a chunk
  constexpr int kOwn = kGramChunk / (kGramThreads / 32);
  const int side = lane / kGramTile, jj = lane % kGramTile;
  const float* kp = kappa + (i64)bh * C * D + (side ? j0 : i0) + jj;
  if (tid == 0) s_cnt = 0;
  __syncthreads();
  int c = 0;
  for (int g = tid; g < C; g += kGramThreads) { const int ng = n[(i64)bh * C + g]; s_n[g] = ng; c += ng > 0; }
  c = warp_sum(c);
  if (lane == 0 && c) atomicAdd(&s_cnt, c);
  __syncthreads();
  const int cplus = s_cnt;
  float x[kOwn];
  const auto fetch = [&](int g0) {
#pragma unroll
    for (int u = 0; u < kOwn; ++u) { const int g = g0 + warp * kOwn + u; x[u] = g < C && s_n[g] > 0 ? kp[(i64)g * D] : 0.f; }
  };
  // first the mean, then the products: the rows come twice
  double acc[2] = {0.0, 0.0}, m = 0.0;
  for (int pass = 0; pass < 2; ++pass) {
    const double mean = pass ? s_mean[lane] : 0.0;
    fetch(0);
    for (int g0 = 0; g0 < C; g0 += kGramChunk) {
      const int nr = min(kGramChunk, C - g0);
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kOwn; ++u) {
        const int g = g0 + warp * kOwn + u;
        rows[warp * kOwn + u][side][jj] = pass && !(g < C && s_n[g] > 0) ? 0.0 : (double)x[u] - mean;
      }
      __syncthreads();
      if (g0 + kGramChunk < C) fetch(g0 + kGramChunk);
      if (pass) {
        gram_accumulate(rows, nr, acc);
      } else if (warp == 0) {
#pragma unroll 8
        for (int u = 0; u < nr; ++u) m += rows[u][side][jj];   // (an empty group adds nothing)
      }
    }
    if (pass == 0 && warp == 0) s_mean[lane] = cplus > 0 ? m / cplus : 0.0;
    __syncthreads();
  }
  gram_store<D>(Mout + (i64)bh * D * D, i0, j0, acc, cplus > 0 ? (double)cplus * (double)D : 1.0);
}

void launch_sample_gram(int dtype, const void* Q, const i64* qs, int BH, int H, int N, int d, int Ms, u64 seed, int head0,
                        double* Mout, cudaStream_t st) {
  if (dtype == SPARSEPR_BF16) {
    if (d == 128) k_sample_gram<__nv_bfloat16, 128><<<dim3(gram_tiles(d), BH), kGramThreads, 0, st>>>((const __nv_bfloat16*)Q, qs[0], qs[1], qs[2], H, N, Ms, seed, head0, Mout);
    else k_sample_gram<__nv_bfloat16, 64><<<dim3(gram_tiles(d), BH), kGramThreads, 0, st>>>((const __nv_bfloat16*)Q, qs[0], qs[1], qs[2], H, N, Ms, seed, head0, Mout);
  } else {
    if (d == 128) k_sample_gram<float, 128><<<dim3(gram_tiles(d), BH), kGramThreads, 0, st>>>((const float*)Q, qs[0], qs[1], qs[2], H, N, Ms, seed, head0, Mout);
    else k_sample_gram<float, 64><<<dim3(gram_tiles(d), BH), kGramThreads, 0, st>>>((const float*)Q, qs[0], qs[1], qs[2], H, N, Ms, seed, head0, Mout);
  }
}
void launch_centroid_gram(const float* kappa, const int* n, int BH, int C, int d, double* Mout, cudaStream_t st) {
  if (d == 128) launch_pdl(k_centroid_gram<128>, dim3(gram_tiles(128), BH), dim3(kGramThreads), 0, st, kappa, n, C, Mout);
  else launch_pdl(k_centroid_gram<64>, dim3(gram_tiles(64), BH), dim3(kGramThreads), 0, st, kappa, n, C, Mout);
}

// =============================================================================
// Response projections: phi_K = K F_K (Eq. 6) and phi_Q = RMS-normalised Q F_Q
// (Eq. 7).  Each thread produces kRows rows of R outputs; F is staged in shared
// memory and read by broadcast.  Also tracks max |phi| per head (for the
// fixed-point centroid sums) and flags non-finite values.
// Bound by latency on small calls and by reads of F from shared memory on large ones (8 heads of 7161 rows, d = 128, 64 outputs: 224 CTAs, shared memory
// 68 % of its rate while one is on an SM, FMA pipe 38 %): multiply-adds of two columns to an instruction, and the next eight values of a row are
// fetched under those of the last eight (24 heads of 16000 rows, d = 128, 64 outputs: 261 -> 210 us).
// =============================================================================
template <typename T, int D, int R, bool RMS, int kRows>
__global__ void __launch_bounds__(128) k_project(const T* __restrict__ X, i64 sb, i64 sh, i64 sn, int H, int N, int r,
                                                 const float* __restrict__ F, float eps, float* __restrict__ phi,
                                                 int ldphi, unsigned* __restrict__ maxabs_bits, int* err) {
  __shared__ __align__(16) float Fs[D * R];
  const int bh = blockIdx.y, b = bh / H, h = bh % H;
  const float* Fh = F + (i64)bh * D * r;
  const T* base = X + b * sb + h * sh;
  const int row0 = blockIdx.x * (blockDim.x * kRows) + threadIdx.x;
  const T* p[kRows];
  float x[kRows][8];
#pragma unroll
  for (int u = 0; u < kRows; ++u) {
    const int row = row0 + u * blockDim.x;
    p[u] = base + (i64)(row < N ? row : 0) * sn;
    load8(p[u], x[u]);
  }
#pragma unroll 8
  for (int e = threadIdx.x; e < D * R; e += blockDim.x) {
    const int k = e / R, c = e % R;
    Fs[e] = c < r ? Fh[k * r + c] : 0.f;
  }
  __syncthreads();
  float2 acc2[kRows][R / 2];
#pragma unroll
  for (int u = 0; u < kRows; ++u)
#pragma unroll
    for (int c = 0; c < R / 2; ++c) acc2[u][c] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int k0 = 0; k0 < D; k0 += 8) {
    float nx[kRows][8];
    const int kn = min(k0 + 8, D - 8);
#pragma unroll
    for (int u = 0; u < kRows; ++u) load8(p[u] + kn, nx[u]);
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      const float4* f4 = reinterpret_cast<const float4*>(Fs + (k0 + kk) * R);
#pragma unroll
      for (int c = 0; c < R / 4; ++c) {
        const float4 f = f4[c];
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
          const float2 xx = make_float2(x[u][kk], x[u][kk]);
          acc2[u][2 * c] = __ffma2_rn(xx, make_float2(f.x, f.y), acc2[u][2 * c]);
          acc2[u][2 * c + 1] = __ffma2_rn(xx, make_float2(f.z, f.w), acc2[u][2 * c + 1]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kRows; ++u)
#pragma unroll
      for (int k = 0; k < 8; ++k) x[u][k] = nx[u][k];
  }
  float m = 0.f;
  bool bad = false;
#pragma unroll
  for (int u = 0; u < kRows; ++u) {
    const int row = row0 + u * blockDim.x;
    if (row >= N) continue;
    float acc[R];
#pragma unroll
    for (int c = 0; c < R; c += 2) { acc[c] = acc2[u][c / 2].x; acc[c + 1] = acc2[u][c / 2].y; }
    if (RMS) {
      float ss = 0.f;
#pragma unroll
      for (int c = 0; c < R; ++c) ss = fmaf(acc[c], acc[c], ss);
      const float inv = 1.f / fmaxf(sqrtf(ss / (float)r), eps);
#pragma unroll
      for (int c = 0; c < R; ++c) acc[c] *= inv;
    }
    float* out = phi + ((i64)bh * N + row) * ldphi;
#pragma unroll
    for (int c = 0; c < R; c += 4)      // columns r..R-1 are written as zeros (ldphi >= R)
      *reinterpret_cast<float4*>(out + c) = make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
#pragma unroll
    for (int c = 0; c < R; ++c) {
      m = fmaxf(m, fabsf(acc[c]));
      bad |= !(fabsf(acc[c]) <= 3.0e38f);
    }
  }
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) atomicMax(maxabs_bits + bh, __float_as_uint(m));
  if (bad) set_error(err, SPARSEPR_ERR_NUMERIC);
}

template <typename T, int D, int R, bool RMS>
static void project_rows(const T* X, const i64* xs, int BH, int H, int N, int r, const float* F, float eps,
                         float* phi, int ldphi, unsigned* maxabs, int* err, cudaStream_t st) {
  // One row per thread or two, which halve the reads of F per multiply-add: a call takes as long as the CTAs that one SM gets, and one more of 64 rows
  // costs 2 / 5 of one more of 256.  Measured, us, one row against two, float32, d = 128 with 64 outputs: 2 x 9251 rows (2 CTAs of 64 on an SM, 1 of 256)
  // 25.5, 29.2; 2 x 10001 (3, 1) 29.6, 28.9; 2 x 18001 (4, 1) 35.7, 29.5; 32 x 1126 (4, 2) 35.3, 43.9; 2 x 20001 (5, 2) 41.8, 43.7; 2 x 25001 (6, 2) 48.0,
  // 43.9; 8 x 10001 (9, 3) 80.8, 62.6.  d = 64 with 48: 2 x 4001 (1, 1) 12.6, 14.6; 2 x 18001 (4, 1) 19.4, 15.5; 2 x 20001 (5, 2) 21.5, 23.5; 2 x 25001 (6, 2)
  // 23.6, 23.5; with 16 outputs the two differ by a microsecond or two.
  const i64 sms = sm_count(), one = ((i64)BH * ((N + 63) / 64) + sms - 1) / sms, two = ((i64)BH * ((N + 255) / 256) + sms - 1) / sms;
  if (2 * one <= 5 * two)
    k_project<T, D, R, RMS, 1><<<dim3((N + 63) / 64, BH), 64, 0, st>>>(X, xs[0], xs[1], xs[2], H, N, r, F, eps, phi, ldphi, maxabs, err);
  else
    k_project<T, D, R, RMS, 2><<<dim3((N + 255) / 256, BH), 128, 0, st>>>(X, xs[0], xs[1], xs[2], H, N, r, F, eps, phi, ldphi, maxabs, err);
}
template <typename T, int D, bool RMS>
static void project_dispatch_r(const T* X, const i64* xs, int BH, int H, int N, int r, const float* F, float eps,
                               float* phi, int ldphi, unsigned* maxabs, int* err, cudaStream_t st) {
  if (r <= 16) project_rows<T, D, 16, RMS>(X, xs, BH, H, N, r, F, eps, phi, ldphi, maxabs, err, st);
  else if (r <= 32) project_rows<T, D, 32, RMS>(X, xs, BH, H, N, r, F, eps, phi, ldphi, maxabs, err, st);
  else if (r <= 48) project_rows<T, D, 48, RMS>(X, xs, BH, H, N, r, F, eps, phi, ldphi, maxabs, err, st);
  else project_rows<T, D, 64, RMS>(X, xs, BH, H, N, r, F, eps, phi, ldphi, maxabs, err, st);
}
void launch_project(int dtype, const void* X, const i64* xs, int BH, int H, int N, int d, int r, const float* F,
                    bool rms, float eps, float* phi, int ldphi, unsigned* maxabs, int* err, cudaStream_t st) {
#define SPR_PROJ(TT, DD)                                                                                        \
  do {                                                                                                          \
    if (rms) project_dispatch_r<TT, DD, true>((const TT*)X, xs, BH, H, N, r, F, eps, phi, ldphi, maxabs, err, st); \
    else project_dispatch_r<TT, DD, false>((const TT*)X, xs, BH, H, N, r, F, eps, phi, ldphi, maxabs, err, st);    \
  } while (0)
  if (dtype == SPARSEPR_BF16) { if (d == 128) SPR_PROJ(__nv_bfloat16, 128); else SPR_PROJ(__nv_bfloat16, 64); }
  else { if (d == 128) SPR_PROJ(float, 128); else SPR_PROJ(float, 64); }
#undef SPR_PROJ
}

// Features of the semantic reference partition (Section 3.1): the activations themselves, as float32 rows
// [BH][N][d]; also the largest magnitude per head (for the fixed-point sums) and the non-finite check.
template <typename T>
__global__ void __launch_bounds__(256) k_raw_features(const T* __restrict__ X, i64 sb, i64 sh, i64 sn, int H, int N, int d,
                                                      float* __restrict__ phi, unsigned* __restrict__ maxabs, int* __restrict__ err) {
  const int bh = blockIdx.y, b = bh / H, h = bh % H;
  const int per_row = d / 8;
  float mx = 0.f;
  bool bad = false;
  for (i64 e = (i64)blockIdx.x * 256 + threadIdx.x; e < (i64)N * per_row; e += (i64)gridDim.x * 256) {
    const int row = (int)(e / per_row), c8 = (int)(e % per_row) * 8;
    float v[8];
    load8(X + b * sb + h * sh + (i64)row * sn + c8, v);
#pragma unroll
    for (int k = 0; k < 8; ++k) { mx = fmaxf(mx, fabsf(v[k])); bad |= !isfinite(v[k]); }
    store8(phi + ((i64)bh * N + row) * d + c8, v);
  }
  mx = warp_max(mx);
  if ((threadIdx.x & 31) == 0 && mx > 0.f) atomicMax(maxabs + bh, __float_as_uint(mx));
  if (bad) set_error(err, SPARSEPR_ERR_NUMERIC);
}
void launch_raw_features(int dtype, const void* X, const i64* xs, int BH, int H, int N, int d, float* phi, unsigned* maxabs,
                         int* err, cudaStream_t st) {
  dim3 grid((unsigned)std::min<i64>(((i64)N * (d / 8) + 255) / 256, 1024), BH);
  if (dtype == SPARSEPR_BF16) k_raw_features<__nv_bfloat16><<<grid, 256, 0, st>>>((const __nv_bfloat16*)X, xs[0], xs[1], xs[2], H, N, d, phi, maxabs, err);
  else k_raw_features<float><<<grid, 256, 0, st>>>((const float*)X, xs[0], xs[1], xs[2], H, N, d, phi, maxabs, err);
}

// =============================================================================
// k-means (Section 4.1).  Assignment: a[j] = argmin_c ||x_j - mu_c||^2, ties to the
// lowest c.  Fast path in float32 via s_c = ||mu_c||^2 - 2 x.mu_c; whenever the
// gap between the best and the second-best score is inside a proven rounding
// bound the row is decided by the exact float64 evaluation (terms added in order
// of k, one multiply and one add each), so the decision always equals that
// evaluation.  Optionally accumulates order-independent fixed-point centroid sums.
// =============================================================================
__device__ __noinline__ int exact_assign(const float* __restrict__ x, const float* __restrict__ mu, int C, int r, int ldmu) {
  double best = 0.0;
  int bi = 0;
  for (int c = 0; c < C; ++c) {
    const float* m = mu + (i64)c * ldmu;
    double dsum = 0.0;
    for (int k = 0; k < r; ++k) {
      const double diff = __dsub_rn((double)x[k], (double)m[k]);
      dsum = __dadd_rn(dsum, __dmul_rn(diff, diff));
    }
    if (c == 0 || dsum < best) { best = dsum; bi = c; }
  }
  return bi;
}

constexpr int kAssignChunk = 64;   // centroids staged per shared-memory chunk

// R = padded feature width (16..128), ROWS = rows per thread (two up to 64 columns; one for the 128 columns of the
// semantic partition's raw activations, whose row already fills the registers)
template <int R, int ROWS>
__global__ void __launch_bounds__(128) k_kmeans_assign(const float* __restrict__ phi, int ldphi, int N, int r,
                                                       const float* __restrict__ mu, const float* __restrict__ mu2,
                                                       const float* __restrict__ mumax, int C, int* __restrict__ assign,
                                                       i64* __restrict__ sums, int* __restrict__ counts,
                                                       const int* __restrict__ fx_shift, int* __restrict__ recheck_count,
                                                       const int* __restrict__ prev_changed, int* __restrict__ cur_changed) {
  constexpr int kChunk = R > 64 ? 32 : kAssignChunk;
  __shared__ __align__(16) float mus[kChunk * R];
  __shared__ float mu2s[kChunk];
  const int bh = blockIdx.y;
  if (prev_changed != nullptr && prev_changed[bh] == 0) return;      // fixed point reached in the previous pass
  const float* ph = phi + (i64)bh * N * ldphi;
  const float* muh = mu + (i64)bh * C * R;
  int rows[ROWS];
  float x[ROWS][R];
  float xn2[ROWS];
#pragma unroll
  for (int t = 0; t < ROWS; ++t) {
    rows[t] = (int)(blockIdx.x * (128 * ROWS) + threadIdx.x + 128 * t);
    xn2[t] = 0.f;
    const float* p = ph + (i64)min(rows[t], N - 1) * ldphi;
#pragma unroll
    for (int k = 0; k < R; k += 4) {
      const float4 v = *reinterpret_cast<const float4*>(p + k);      // columns r..R-1 hold zeros
      x[t][k] = v.x; x[t][k + 1] = v.y; x[t][k + 2] = v.z; x[t][k + 3] = v.w;
    }
#pragma unroll
    for (int k = 0; k < R; ++k) xn2[t] = fmaf(x[t][k], x[t][k], xn2[t]);
  }
  float best[ROWS], second[ROWS];
  int bi[ROWS];
#pragma unroll
  for (int t = 0; t < ROWS; ++t) { best[t] = 3.0e38f; second[t] = 3.0e38f; bi[t] = 0; }
  for (int c0 = 0; c0 < C; c0 += kChunk) {
    const int nc = min(kChunk, C - c0);
    __syncthreads();
    for (int e = threadIdx.x; e < nc * R; e += 128) mus[e] = muh[(i64)c0 * R + e];
    if (threadIdx.x < nc) mu2s[threadIdx.x] = mu2[(i64)bh * C + c0 + threadIdx.x];
    __syncthreads();
    for (int c = 0; c < nc; ++c) {
      const float4* m4 = reinterpret_cast<const float4*>(mus + c * R);
      float dot[ROWS];
#pragma unroll
      for (int t = 0; t < ROWS; ++t) dot[t] = 0.f;
#pragma unroll
      for (int k = 0; k < R / 4; ++k) {
        const float4 m = m4[k];
#pragma unroll
        for (int t = 0; t < ROWS; ++t) {
          dot[t] = fmaf(x[t][4 * k], m.x, dot[t]); dot[t] = fmaf(x[t][4 * k + 1], m.y, dot[t]);
          dot[t] = fmaf(x[t][4 * k + 2], m.z, dot[t]); dot[t] = fmaf(x[t][4 * k + 3], m.w, dot[t]);
        }
      }
#pragma unroll
      for (int t = 0; t < ROWS; ++t) {
        const float sc = fmaf(-2.f, dot[t], mu2s[c]);
        if (sc < best[t]) { second[t] = best[t]; best[t] = sc; bi[t] = c0 + c; } else if (sc < second[t]) second[t] = sc;
      }
    }
  }
  const float mm = mumax[bh];
  const int shift = fx_shift ? fx_shift[bh] : 0;
#pragma unroll
  for (int t = 0; t < ROWS; ++t) {
    if (rows[t] >= N) continue;
    // |computed score - true score| <= E for every centroid (float32 rounding of the
    // dot product, of ||mu||^2 and of the final combination)
    const float E = 1.5f * 5.9604645e-8f * (2.f * mm * mm + (2.f * r + 2.f) * sqrtf(xn2[t]) * mm);
    int a = bi[t];
    if (!(second[t] - best[t] > 2.f * E)) {
      a = exact_assign(ph + (i64)rows[t] * ldphi, muh, C, r, R);
      if (recheck_count) atomicAdd(recheck_count, 1);
    }
    if (cur_changed != nullptr && (prev_changed == nullptr || assign[(i64)bh * N + rows[t]] != a)) atomicAdd(cur_changed + bh, 1);
    assign[(i64)bh * N + rows[t]] = a;
    if (sums) {
      i64* s = sums + ((i64)bh * C + a) * R;
      const double sc = ldexp(1.0, shift);
#pragma unroll
      for (int k = 0; k < R; ++k)
        if (k < r) atomicAdd(reinterpret_cast<u64*>(s + k), (u64)__double2ll_rn((double)x[t][k] * sc));
      atomicAdd(counts + (i64)bh * C + a, 1);
    }
  }
}

void launch_kmeans_assign(const float* phi, int ldphi, int BH, int N, int r, const float* mu, const float* mu2,
                          const float* mumax, int C, int* assign, i64* sums, int* counts, const int* fx_shift,
                          int* recheck_count, const int* prev_changed, int* cur_changed, cudaStream_t st) {
  const int R = feature_ld(r);
#define SPR_ASSIGN(RR, ROWS) k_kmeans_assign<RR, ROWS><<<dim3((N + 128 * ROWS - 1) / (128 * ROWS), BH), 128, 0, st>>>(phi, ldphi, N, r, mu, mu2, mumax, C, assign, sums, counts, fx_shift, recheck_count, prev_changed, cur_changed)
  if (R == 16) SPR_ASSIGN(16, 2); else if (R == 32) SPR_ASSIGN(32, 2); else if (R == 48) SPR_ASSIGN(48, 2);
  else if (R == 64) SPR_ASSIGN(64, 2); else SPR_ASSIGN(128, 1);
#undef SPR_ASSIGN
}

// Initial centroids = feature rows of the strided init sample; also clears the sums
// and derives the fixed-point shift of the head from max |phi|.
__global__ void k_kmeans_init(const float* __restrict__ phi, int ldphi, int N, int r, int R, int C, u64 seed, int tag, int head0,
                              float* __restrict__ mu, i64* __restrict__ sums, int* __restrict__ counts,
                              const unsigned* __restrict__ maxabs_bits, int* __restrict__ fx_shift, int* __restrict__ recheck_total) {
  pdl_wait();                                                   // the features come from the kernel before
  pdl_launch_dependents();
  const int bh = blockIdx.y;
  if (blockIdx.x == 0 && bh == 0 && threadIdx.x == 0) *recheck_total = 0;
  const u64 U = sample_offset(seed, tag, head0 + bh);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < C * R; e += gridDim.x * blockDim.x) {
    const int c = e / R, k = e % R;
    const int row = strided_row(c, C, N, U);
    mu[(i64)bh * C * R + e] = k < r ? phi[((i64)bh * N + row) * ldphi + k] : 0.f;
    sums[(i64)bh * C * R + e] = 0;
    if (k == 0) counts[(i64)bh * C + c] = 0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    // sums of up to N values of magnitude <= maxabs must stay below 2^62
    const float m = fmaxf(__uint_as_float(maxabs_bits[bh]), 1e-30f);
    int e2;
    frexpf(m, &e2);                                  // m < 2^e2
    int nb = 0;
    while ((1ll << nb) < (i64)N) ++nb;
    int sh = min(61 - nb, 50) - e2;                  // (50: what k_kmeans_group_sums adds up in int32)
    fx_shift[bh] = max(-60, min(sh, 60));
  }
}

// mu <- sums / counts for non-empty clusters (empty ones keep their centroid), then
// ||mu_c||^2 (float64 -> float32) and the largest centroid norm of the head.
// gridDim.y CTAs per head share the centroids (warp w of part y takes c = y nw + w, + nw gridDim.y, ...); the
// largest norm needs all of them and is written only when one CTA holds the whole head (mumax may be null otherwise:
// the tensor-core assignment derives the bound from ||mu_c||^2 itself).
__global__ void __launch_bounds__(1024) k_kmeans_finalize(float* __restrict__ mu, float* __restrict__ mu2,
                                                          float* __restrict__ mumax, i64* __restrict__ sums,
                                                          int* __restrict__ counts, const int* __restrict__ fx_shift,
                                                          int C, int r, int R, int update,
                                                          __nv_bfloat16* __restrict__ mh, __nv_bfloat16* __restrict__ ml,
                                                          __nv_bfloat16* __restrict__ mw, int Cpad) {
  __shared__ float red[34];
  const int bh = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  pdl_wait();                                                   // the sums come from the kernels before
  pdl_launch_dependents();
  const double inv_sc = update ? ldexp(1.0, -fx_shift[bh]) : 0.0;
  float mx = 0.f;
  auto store_words = [&](float v, int c) { *reinterpret_cast<uint4*>(mw + ((i64)bh * Cpad + c) * 8) = norm_words(v); };
  if (mw != nullptr && blockIdx.y == 0)
    for (int c = C + threadIdx.x; c < Cpad; c += blockDim.x) store_words(kKmFar, c);
  for (int c = blockIdx.y * nw + w; c < C; c += nw * gridDim.y) {
    float* m = mu + ((i64)bh * C + c) * R;
    i64* s = sums + ((i64)bh * C + c) * R;
    const int cnt = update ? counts[(i64)bh * C + c] : 0;
    double n2 = 0.0;
    for (int k = lane; k < max(R, 64); k += 32) {
      float v = 0.f;
      if (k < R) {
        v = m[k];
        if (update) {
          if (cnt > 0 && k < r) { v = group_mean(s[k], inv_sc, cnt); m[k] = v; }
          if (update == 1) s[k] = 0;
        }
        n2 += (double)v * (double)v;
      }
      if (mh != nullptr && k < 64) {
        // the two bf16 words of -2 mu for the tensor-core assignment, [C][64] with zeros beyond r
        const float x = k < r ? -2.f * v : 0.f;
        const __nv_bfloat16 hb = __float2bfloat16_rn(x);
        mh[((i64)bh * C + c) * 64 + k] = hb;
        ml[((i64)bh * C + c) * 64 + k] = __float2bfloat16_rn(x - __bfloat162float(hb));
      }
    }
    n2 = warp_sum(n2);
    __syncwarp();
    if (lane == 0) {
      mu2[(i64)bh * C + c] = (float)n2;
      if (update == 1) counts[(i64)bh * C + c] = 0;
      if (mw != nullptr) store_words((float)n2, c);
      mx = fmaxf(mx, (float)sqrt(n2) * 1.0000002f);
    }
  }
  if (gridDim.y == 1 && mumax != nullptr) {
    mx = block_max(mx, red);
    if (threadIdx.x == 0) mumax[bh] = mx;
  }
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

// Fixed-point sums and counts of the features over the groups of a partition [BH][N] (ids outside [0, C) are ignored): the
// first centroids of a warm start (Appendix C.1; a group that the previous partition left empty keeps the strided row
// k_kmeans_init gave it), and the sums after the first tensor-core assignment, which later passes only update.
// One warp per 32 consecutive rows (add_rows_to_sums).  Bound by the atomics (a warp's 32 rows fall into about 20 groups after a cold start): 67 us at
// 24 heads of 32760 rows and 64 columns, 48 us on the partition of a call before (few groups per warp).
__global__ void __launch_bounds__(256) k_kmeans_group_sums(const float* __restrict__ phi, int ldphi, int N, int r, int R, int C,
                                                           const int* __restrict__ assign, i64* __restrict__ sums,
                                                           int* __restrict__ counts, const int* __restrict__ fx_shift) {
  pdl_wait();                                                   // the assignment comes from the kernels before
  pdl_launch_dependents();
  const int bh = blockIdx.y, rowbase = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 32;
  if (rowbase >= N) return;
  const i64 row = (i64)bh * N + rowbase;
  add_rows_to_sums(phi + row * ldphi, ldphi, N - rowbase, r, R, C, assign + row, sums + (i64)bh * C * R, counts + (i64)bh * C, fx_shift[bh]);
}
void launch_kmeans_group_sums(const float* phi, int ldphi, int BH, int N, int r, int C, const int* assign, i64* sums,
                              int* counts, const int* fx_shift, cudaStream_t st) {
  const int R = feature_ld(r);
  launch_pdl(k_kmeans_group_sums, dim3((N + 255) / 256, BH), dim3(256), 0, st, phi, ldphi, N, r, R, C, assign, sums, counts, fx_shift);
}

void launch_kmeans_init(const float* phi, int ldphi, int BH, int N, int r, int C, u64 seed, int tag, int head0, float* mu,
                        i64* sums, int* counts, const unsigned* maxabs_bits, int* fx_shift, int* recheck_total, cudaStream_t st) {
  const int R = feature_ld(r);
  dim3 grid((C * R + 255) / 256, BH);
  launch_pdl(k_kmeans_init, grid, dim3(256), 0, st, phi, ldphi, N, r, R, C, seed, tag, head0, mu, sums, counts, maxabs_bits, fx_shift, recheck_total);
}
void launch_kmeans_finalize(float* mu, float* mu2, float* mumax, i64* sums, int* counts, const int* fx_shift, int BH,
                            int C, int r, int update, cudaStream_t st, __nv_bfloat16* mh, __nv_bfloat16* ml, __nv_bfloat16* mw) {
  const int R = feature_ld(r), Cpad = km_padded(C);
  if (mumax != nullptr) {
    k_kmeans_finalize<<<BH, 1024, 0, st>>>(mu, mu2, mumax, sums, counts, fx_shift, C, r, R, update, mh, ml, mw, Cpad);
  } else {
    // one warp per centroid, spread over enough CTAs to fill the GPU
    const int parts = std::max(1, std::min(32, (C + 7) / 8));
    launch_pdl(k_kmeans_finalize, dim3(BH, parts), dim3(256), 0, st, mu, mu2, (float*)nullptr, sums, counts, fx_shift, C, r, R, update, mh, ml, mw, Cpad);
  }
}

// =============================================================================
// Stable counting sort by group id (Section 4.3, group-major layout).  One CTA of
// 16 warps per head; warp w owns a contiguous segment of tokens, so that ranks
// inside a group follow the original token order.
// =============================================================================
constexpr int kSortWarps = 16;

__global__ void __launch_bounds__(kSortWarps * 32) k_group_sort(const int* __restrict__ assign, int N, int C,
                                                                 int* __restrict__ perm, int* __restrict__ inv,
                                                                 int* __restrict__ off, int* err) {
  pdl_wait();                                                   // the assignment comes from the kernels before
  pdl_launch_dependents();
  extern __shared__ int sm_sort[];
  int* hist = sm_sort;                    // [kSortWarps][C]
  int* tot = hist + kSortWarps * C;       // [C]
  __shared__ int scratch[34];
  const int bh = blockIdx.x;
  const int* a = assign + (i64)bh * N;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < kSortWarps * C; e += blockDim.x) hist[e] = 0;
  __syncthreads();
  const int L = (((N + kSortWarps - 1) / kSortWarps) + 31) / 32 * 32;
  const int s0 = w * L, s1 = min(N, s0 + L);
  for (int i = s0 + lane; i < s1; i += 32) {
    int key = a[i];
    // an id out of range (only possible after an earlier stage gave up) is recorded and counted as group 0, so that
    // the permutation stays a permutation and nothing downstream indexes out of bounds
    if (key < 0 || key >= C) { set_error(err, SPARSEPR_ERR_INVALID_ARG); key = 0; }
    atomicAdd(&hist[w * C + key], 1);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    int t = 0;
    for (int ww = 0; ww < kSortWarps; ++ww) t += hist[ww * C + c];
    tot[c] = t;
  }
  __syncthreads();
  const int total = block_exclusive_scan(tot, C, scratch);
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    int run = tot[c];
    off[(i64)bh * (C + 1) + c] = run;
    for (int ww = 0; ww < kSortWarps; ++ww) { const int t = hist[ww * C + c]; hist[ww * C + c] = run; run += t; }
  }
  if (threadIdx.x == 0) off[(i64)bh * (C + 1) + C] = total;
  __syncthreads();
  for (int i0 = s0; i0 < s1; i0 += 32) {
    const int i = i0 + lane;
    int key = i < s1 ? a[i] : -1;
    if (i < s1 && (key < 0 || key >= C)) key = 0;
    const unsigned same = __match_any_sync(0xffffffffu, key);
    const int rank = __popc(same & ((1u << lane) - 1));
    int pos = -1;
    if (key >= 0) pos = hist[w * C + key] + rank;
    __syncwarp();
    if (key >= 0 && rank == 0) hist[w * C + key] += __popc(same);
    __syncwarp();
    if (key >= 0) { perm[(i64)bh * N + pos] = i; inv[(i64)bh * N + i] = pos; }
  }
}

void launch_group_sort(const int* assign, int BH, int N, int C, int* perm, int* inv, int* off, int* err, cudaStream_t st) {
  launch_pdl(k_group_sort, dim3(BH), dim3(kSortWarps * 32), (size_t)(kSortWarps + 1) * C * sizeof(int), st, assign, N, C, perm, inv, off, err);
}
cudaError_t init_group_sort() {
  return cudaFuncSetAttribute(k_group_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)((kSortWarps + 1) * kMaxGroups * sizeof(int)));
}

// =============================================================================
// Group means in the original activation space: kappa_b (Appendix B.2) and
// theta_a (router).  One CTA per group walks its members in group-major order, eight warps on
// interleaved blocks of rows; the float32 sums have a fixed order.
// =============================================================================
template <typename T, int D>
__global__ void __launch_bounds__(256) k_group_means(const T* __restrict__ X, i64 sb, i64 sh, i64 sn, int H,
                                                     const int* __restrict__ perm, const int* __restrict__ off, int N,
                                                     int C, float* __restrict__ out, int* __restrict__ sizes) {
  pdl_wait();                                                   // the permutation comes from the kernel before
  pdl_launch_dependents();
  constexpr int LPR = D / 8;                 // lanes per row (8 elements each)
  constexpr int RPW = 32 / LPR;              // rows per warp step
  __shared__ float part[8][D];
  const int bh = blockIdx.y, b = bh / H, h = bh % H;
  const int g = blockIdx.x, w = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31, sub = lane / LPR, col = (lane % LPR) * 8;
  const T* base = X + b * sb + h * sh;
  const int* pm = perm + (i64)bh * N;
  const int p0 = off[(i64)bh * (C + 1) + g], p1 = off[(i64)bh * (C + 1) + g + 1];
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  // One CTA per group (group sizes spread over two orders of magnitude: with a warp per group the largest group set
  // the duration of the launch): warp w takes the blocks of 8 RPW rows number w, w + 8, ...; eight row loads in
  // flight per lane (the walk is bound by the latency of the index -> row chain); every sum has a fixed order, and
  // a slot beyond the group adds exact zeros
  for (int p = p0 + w * RPW * 8 + sub; p < p1; p += RPW * 8 * 8) {
    int src[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) src[j] = p + j * RPW < p1 ? pm[p + j * RPW] : -1;
    float v[8][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (src[j] >= 0) {
        load8(base + (i64)src[j] * sn + col, v[j]);
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) v[j][k] = 0.f;
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[k] += v[j][k];
  }
  // combine the RPW interleaved partial sums of the warp, then the eight warps, in a fixed order
#pragma unroll
  for (int k = 0; k < 8; ++k)
    for (int o = LPR; o < 32; o <<= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
  if (sub == 0) {
#pragma unroll
    for (int k = 0; k < 8; ++k) part[w][col + k] = acc[k];
  }
  __syncthreads();
  const int n = p1 - p0;
  if (threadIdx.x < D) {
    float t = part[0][threadIdx.x];
#pragma unroll
    for (int ww = 1; ww < 8; ++ww) t += part[ww][threadIdx.x];
    out[((i64)bh * C + g) * D + threadIdx.x] = n > 0 ? t * (1.f / (float)n) : 0.f;
  }
  if (threadIdx.x == 0 && sizes) sizes[(i64)bh * C + g] = n;
}

void launch_group_means(int dtype, const void* X, const i64* xs, int BH, int H, const int* perm, const int* off, int N,
                        int C, int d, float* out, int* sizes, cudaStream_t st) {
  dim3 grid(C, BH);
#define SPR_GM(TT, DD) launch_pdl(k_group_means<TT, DD>, grid, dim3(256), 0, st, (const TT*)X, xs[0], xs[1], xs[2], H, perm, off, N, C, out, sizes)
  if (dtype == SPARSEPR_BF16) { if (d == 128) SPR_GM(__nv_bfloat16, 128); else SPR_GM(__nv_bfloat16, 64); }
  else { if (d == 128) SPR_GM(float, 128); else SPR_GM(float, 64); }
#undef SPR_GM
}

// =============================================================================
// Row gather into the group-major layout: out[bh][p][:] = in[b,h,perm[p],:].
// =============================================================================
template <typename T, int D>
__global__ void __launch_bounds__(256) k_gather_rows(const T* __restrict__ X, i64 sb, i64 sh, i64 sn, int H,
                                                     const int* __restrict__ perm, int N, T* __restrict__ out) {
  constexpr int VEC = 16 / sizeof(T);
  constexpr int TPR = D / VEC;               // threads per row
  const int bh = blockIdx.y, b = bh / H, h = bh % H;
  const T* base = X + b * sb + h * sh;
  const i64 t = (i64)blockIdx.x * 256 + threadIdx.x;
  const int p = (int)(t / TPR), c = (int)(t % TPR) * VEC;
  if (p >= N) return;
  const int src = perm[(i64)bh * N + p];
  *reinterpret_cast<uint4*>(out + ((i64)bh * N + p) * D + c) = *reinterpret_cast<const uint4*>(base + (i64)src * sn + c);
}

void launch_gather_rows(int dtype, const void* X, const i64* xs, int BH, int H, const int* perm, int N, int d, void* out,
                        cudaStream_t st) {
  const int es = dtype == SPARSEPR_BF16 ? 2 : 4;
  const int tpr = d * es / 16;
  dim3 grid((unsigned)(((i64)N * tpr + 255) / 256), BH);
#define SPR_GA(TT, DD) k_gather_rows<TT, DD><<<grid, 256, 0, st>>>((const TT*)X, xs[0], xs[1], xs[2], H, perm, N, (TT*)out)
  if (dtype == SPARSEPR_BF16) { if (d == 128) SPR_GA(__nv_bfloat16, 128); else SPR_GA(__nv_bfloat16, 64); }
  else { if (d == 128) SPR_GA(float, 128); else SPR_GA(float, 64); }
#undef SPR_GA
}

}  // namespace spr
