// Probe-Fitted Residual Reconstruction, the per-head fit (Appendix A.3): weighted
// standardisation, weighted ridge normal equations solved by Cholesky, the
// probe-residual output subspace, and the composed affine map
//   R_hat_i = c + x_i A,  A = diag(1/s_x) B_lambda Psi_r Psi_r^T,  c = mu_R - mu_x A,
// which is algebraically Eq. 9.  Standardisation and composition are float64; the Gram matrices and the ridge
// solve are float64 for float32 tensors and float32 for 16-bit tensors.  The fit is a chain of short kernels, on the
// critical path of small calls and beside the attention kernels in large ones, where every SM it holds is lost to them:
// each stage is spread over several CTAs per head where it has the work for them.
#include "kernels.cuh"

namespace spr {

// scratch per head (doubles): Xb[M*d] Rb[M*d] G[d*d] B[d*d] S[d*d] mu_x[d] mu_R[d] s_x[d] wt[M] flag[1] failed[1]
// flag: no usable probes (k_fit_prepare); failed: a pivot of the elimination was not positive (the CTAs of k_fit_solve, all of
// which find the same one)
struct FitLayout {
  size_t Xb, Rb, G, B, S, mu_x, mu_R, s_x, wt, flag, failed, total;
  __host__ __device__ FitLayout(int M, int d) {
    size_t o = 0;
    Xb = o; o += (size_t)M * d;
    Rb = o; o += (size_t)M * d;
    G = o; o += (size_t)d * d;
    B = o; o += (size_t)d * d;
    S = o; o += (size_t)d * d;
    mu_x = o; o += d; mu_R = o; o += d; s_x = o; o += d;
    wt = o; o += M;
    flag = o; o += 1;
    failed = o; o += 1;
    total = (o + 31) / 32 * 32;
  }
};
size_t fit_scratch_doubles(int BH, int M, int d) { return FitLayout(M, d).total * BH; }

// Probe rows a head has in flight per column slice of k_fit_prepare, columns per CTA of it.
constexpr int kPrepCols = 32, kPrepSlices = 8;

// alpha, weighted means, feature scale, standardised probes, unit-mean weights.  Bound by the latency of the loads and of
// the float64 chains, so both are split: grid (d / 32, heads), thread (slice s, column j) takes the probes s, s + 8, ... of
// its column, and the eight partial sums are added in a fixed order.
// (One CTA per head with one thread per column: 26 us at M = 64, d = 128, two heads; now 6 us.)
__global__ void __launch_bounds__(kPrepCols * kPrepSlices) k_fit_prepare(FitArgs a) {
  __shared__ double red[34];
  __shared__ double part[2][kPrepSlices][kPrepCols];
  constexpr int kNt = kPrepCols * kPrepSlices;
  const int bh = blockIdx.y, M = a.M, d = a.d, tid = threadIdx.x;
  const int jl = tid % kPrepCols, sl = tid / kPrepCols, j = blockIdx.x * kPrepCols + jl;
  const FitLayout L(M, d);
  double* sc = a.scratch + (size_t)bh * L.total;
  pdl_wait();                                                   // the probe rows come from the kernel before
  pdl_launch_dependents();
  const float* X = a.X + (i64)bh * M * d;
  const float* Dn = a.Dn + (i64)bh * M * d;
  const float* w = a.w + (i64)bh * M;
  double sw = 0.0, cnt = 0.0;
  for (int p = tid; p < M; p += kNt) { sw += (double)w[p]; cnt += w[p] > 0.f ? 1.0 : 0.0; }
  sw = block_sum(sw, red);
  cnt = block_sum(cnt, red);
  if (tid == 0 && blockIdx.x == 0) {
    const bool usable = sw > 0.0 && cnt > 0.0;
    sc[L.flag] = usable ? 0.0 : 1.0;
    sc[L.failed] = 0.0;
    if (!usable) set_error(a.err, SPARSEPR_ERR_NUMERIC);
  }
  if (!(sw > 0.0)) sw = 1.0;
  const double inv_sw = 1.0 / sw;
  if (blockIdx.x == 0)
    for (int p = tid; p < M; p += kNt) sc[L.wt + p] = (double)M * (double)w[p] * inv_sw;   // unit-mean weights M w_p / sum w (Appendix A.3)
  auto total = [&](int which) {                                 // sum of the column's slices
    double t = part[which][0][jl];
#pragma unroll
    for (int s = 1; s < kPrepSlices; ++s) t += part[which][s][jl];
    return t;
  };
  double mx = 0.0, mr = 0.0;
#pragma unroll 4
  for (int p = sl; p < M; p += kPrepSlices) {
    const double al = (double)w[p], x = (double)X[p * d + j];
    mx = fma(al, x, mx);
    mr = fma(al, (double)Dn[p * d + j] - x, mr);
  }
  part[0][sl][jl] = mx; part[1][sl][jl] = mr;
  __syncthreads();
  mx = total(0) * inv_sw; mr = total(1) * inv_sw;
  __syncthreads();
  double var = 0.0;
#pragma unroll 4
  for (int p = sl; p < M; p += kPrepSlices) { const double t = (double)X[p * d + j] - mx; var = fma((double)w[p] * t, t, var); }
  part[0][sl][jl] = var;
  __syncthreads();
  const double s = sqrt(total(0) * inv_sw + (double)a.eps_std), inv_s = 1.0 / s;
  if (sl == 0) { sc[L.mu_x + j] = mx; sc[L.mu_R + j] = mr; sc[L.s_x + j] = s; }
#pragma unroll 4
  for (int p = sl; p < M; p += kPrepSlices) {
    const double x = (double)X[p * d + j];
    sc[L.Xb + (size_t)p * d + j] = (x - mx) * inv_s;
    sc[L.Rb + (size_t)p * d + j] = ((double)Dn[p * d + j] - x) - mr;
  }
}

// blockIdx.z selects G = Xb^T W Xb + lam I, B(rhs) = Xb^T W Rb, S = Rb^T W Rb; a CTA owns one kT x kT tile of it (of the
// symmetric G and S only the tiles on and above the diagonal, mirrored), a thread a 4 x 4 or 2 x 2 block.
// T = float for 16-bit tensors, double otherwise, with smaller tiles to spread it.
// The eigen-solver wants S symmetric to the bit.  With the weight on one operand, (w r_i) r_j and (w r_j) r_i round differently, so inside a
// diagonal tile, which a CTA forms in full, S_ij and S_ji become their mean.
// (One CTA per matrix with 64 entries per thread and no operand reuse in registers: 94 us at M = 64, d = 128, two heads;
// now 18 us, of which a part is the wait for the kernel before.)
template <typename T> constexpr int kGramTile = sizeof(T) == 4 ? 64 : 32;
template <typename T>
__global__ void __launch_bounds__(256) k_fit_gram(FitArgs a) {
  constexpr int kT = kGramTile<T>, kPt = kT / 16, kRows = 32;
  __shared__ __align__(16) T stage[2 * kRows * kT > kT * (kT + 1) ? 2 * kRows * kT : kT * (kT + 1)];
  T (*ls)[kT] = reinterpret_cast<T (*)[kT]>(stage), (*rs)[kT] = ls + kRows;    // weighted left and right operands
  const int bh = blockIdx.y, which = blockIdx.z, M = a.M, d = a.d;
  const int nt = d / kT, i0 = (blockIdx.x / nt) * kT, j0 = (blockIdx.x % nt) * kT;
  pdl_wait();
  pdl_launch_dependents();
  if (which != 1 && j0 < i0) return;
  const FitLayout L(M, d);
  double* sc = a.scratch + (size_t)bh * L.total;
  const double* Lm = sc + (which == 2 ? L.Rb : L.Xb) + i0;
  const double* Rm = sc + (which == 0 ? L.Xb : L.Rb) + j0;
  double* out = sc + (which == 0 ? L.G : which == 1 ? L.B : L.S);
  const int ti = (threadIdx.x / 16) * kPt, tj = (threadIdx.x % 16) * kPt;
  T acc[kPt][kPt];
#pragma unroll
  for (int u = 0; u < kPt; ++u)
#pragma unroll
    for (int v = 0; v < kPt; ++v) acc[u][v] = T(0);
  for (int p0 = 0; p0 < M; p0 += kRows) {
    const int nr = min(kRows, M - p0);
    __syncthreads();
#pragma unroll
    for (int e = threadIdx.x; e < kRows * kT; e += 256) {
      const int p = e / kT, c = e % kT;
      if (p < nr) {
        ls[p][c] = (T)(Lm[(size_t)(p0 + p) * d + c] * sc[L.wt + p0 + p]);
        rs[p][c] = (T)Rm[(size_t)(p0 + p) * d + c];
      }
    }
    __syncthreads();
    for (int p = 0; p < nr; ++p) {
      T x[kPt], y[kPt];
#pragma unroll
      for (int u = 0; u < kPt; ++u) { x[u] = ls[p][ti + u]; y[u] = rs[p][tj + u]; }
#pragma unroll
      for (int u = 0; u < kPt; ++u)
#pragma unroll
        for (int v = 0; v < kPt; ++v) acc[u][v] = fma(x[u], y[v], acc[u][v]);
    }
  }
  if (which == 2 && i0 == j0) {
    T (*tile)[kT + 1] = reinterpret_cast<T (*)[kT + 1]>(stage);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPt; ++u)
#pragma unroll
      for (int v = 0; v < kPt; ++v) tile[ti + u][tj + v] = acc[u][v];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPt; ++u)
#pragma unroll
      for (int v = 0; v < kPt; ++v) out[(size_t)(i0 + ti + u) * d + j0 + tj + v] = 0.5 * ((double)acc[u][v] + (double)tile[tj + v][ti + u]);
    return;
  }
#pragma unroll
  for (int u = 0; u < kPt; ++u)
#pragma unroll
    for (int v = 0; v < kPt; ++v) {
      const int i = i0 + ti + u, j = j0 + tj + v;
      const double g = (double)acc[u][v] + ((which == 0 && i == j) ? (double)a.lambda : 0.0);
      out[(size_t)i * d + j] = g;
      if (which != 1 && i0 != j0) out[(size_t)j * d + i] = g;
    }
}

// Ridge system (G + lam I) B = RHS by symmetric elimination G = L D L^T (no pivoting: the matrix is positive definite)
// with the right-hand sides carried along, then back substitution; T as in k_fit_gram.
// Everything stays in registers: warp w owns the rows w, w + 16, ..., lane l the columns l, l + 32, ... of [G | RHS].
// Step k: the owner of row k has published it in shared memory (two buffers, so one barrier per step); every warp takes
// its own column entries a_ik by shuffle and subtracts a_ik / a_kk times the row.  2 d barriers in all; the chain of the
// published row (update, publish, barrier, read) sets the pace.  blockIdx.y owns kRhs right-hand sides and repeats the
// elimination of G: the registers hold no more.
// (Cholesky in shared memory with three barriers per column and a dot product per row of the triangular solves: 322 us
// at d = 128 float32, 469 us float64; now 81 and 89 us, beside the eigen-solver.)
template <typename T, int D> constexpr int kSolveRhs = sizeof(T) == 4 ? 64 : 32;
template <typename T, int D>
__global__ void __launch_bounds__(512, 1) k_fit_solve(FitArgs a) {
  constexpr int kRhs = kSolveRhs<T, D>, kRpw = D / 16, kGc = D / 32, kRc = kRhs / 32, kC = kGc + kRc;
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ T rowbuf[2][kC * 32];
  __shared__ T dinv[D];                                          // 1 / pivot
  const int bh = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const FitLayout L(a.M, D);
  double* sc = a.scratch + (size_t)bh * L.total;
  const double* G = sc + L.G;
  double* Bm = sc + L.B + blockIdx.y * kRhs;
  pdl_wait();
  pdl_launch_dependents();
  T x[kRpw][kC];
#pragma unroll
  for (int r = 0; r < kRpw; ++r) {
    const int row = warp + 16 * r;
#pragma unroll
    for (int c = 0; c < kGc; ++c) x[r][c] = (T)G[row * D + lane + 32 * c];
#pragma unroll
    for (int c = 0; c < kRc; ++c) x[r][kGc + c] = (T)Bm[row * D + lane + 32 * c];
  }
  if (sc[L.flag] != 0.0) return;                                 // uniform: no usable probes (nobody writes it here)
  bool bad = false;
  if (warp == 0) {
#pragma unroll
    for (int c = 0; c < kC; ++c) rowbuf[0][lane + 32 * c] = x[0][c];
    if (lane == 0) dinv[0] = T(1) / x[0][0];
  }
#pragma unroll
  for (int ka = 0; ka < kRpw; ++ka) {
#pragma unroll 1
    for (int kw = 0; kw < 16; ++kw) {
      const int k = 16 * ka + kw;
      __syncthreads();
      const T* rb = rowbuf[k & 1];
      bad |= !(rb[k] > T(0));
      const T inv = dinv[k];
      T rv[kC];
#pragma unroll
      for (int c = ka / 2; c < kC; ++c) rv[c] = rb[lane + 32 * c];
      // the row of the next pivot first: it goes to the other buffer at once
#pragma unroll
      for (int r = ka; r < kRpw; ++r) {
        if (r > ka || warp > kw) {                               // uniform: a row below k
          const T f = __shfl_sync(FULL, x[r][ka / 2], k & 31) * inv;
#pragma unroll
          for (int c = ka / 2; c < kC; ++c) x[r][c] = fma(-f, rv[c], x[r][c]);
        }
        constexpr int kLast = kRpw - 1;
        if (r == ka || (r == ka + 1 && r <= kLast)) {
          const int kn = k + 1, rn = r == ka ? kw + 1 : 0;       // owner of row k + 1: (r, warp kw + 1), or (ka + 1, warp 0)
          if ((r == ka ? kw < 15 : kw == 15) && warp == rn) {
#pragma unroll
            for (int c = ka / 2; c < kC; ++c) rowbuf[kn & 1][lane + 32 * c] = x[r][c];
            const T piv = __shfl_sync(FULL, x[r][r / 2], kn & 31);
            if (lane == 0) dinv[kn] = T(1) / piv;
          }
        }
      }
    }
  }
  if (bad) {                                                     // uniform over the CTA: everyone saw every pivot
    if (threadIdx.x == 0) { sc[L.failed] = 1.0; set_error(a.err, SPARSEPR_ERR_NUMERIC); }
    return;
  }
  // back substitution: row k of the solution = y_k / pivot, once all rows below have been taken out of it
  __syncthreads();
  if (warp == 15) {
    const T inv = dinv[D - 1];
#pragma unroll
    for (int c = kGc; c < kC; ++c) { x[kRpw - 1][c] *= inv; rowbuf[(D - 1) & 1][lane + 32 * c] = x[kRpw - 1][c]; }
  }
#pragma unroll
  for (int kb = 0; kb < kRpw; ++kb) {
    const int ka = kRpw - 1 - kb;
#pragma unroll 1
    for (int kw = 15; kw >= 0; --kw) {
      const int k = 16 * ka + kw;
      __syncthreads();
      if (k == 0) break;
      const T* rb = rowbuf[k & 1];
      T rv[kRc];
#pragma unroll
      for (int c = 0; c < kRc; ++c) rv[c] = rb[lane + 32 * (kGc + c)];
#pragma unroll
      for (int q = 0; q <= ka; ++q) {
        const int r = ka - q;
        if (r < ka || warp < kw) {
          const T f = __shfl_sync(FULL, x[r][ka / 2], k & 31);
#pragma unroll
          for (int c = 0; c < kRc; ++c) x[r][kGc + c] = fma(-f, rv[c], x[r][kGc + c]);
        }
        if (r == ka || r == ka - 1) {
          if ((r == ka ? kw > 0 : kw == 0) && warp == (r == ka ? kw - 1 : 15)) {
            const T inv = dinv[k - 1];
#pragma unroll
            for (int c = 0; c < kRc; ++c) {
              x[r][kGc + c] *= inv;
              rowbuf[(k - 1) & 1][lane + 32 * (kGc + c)] = x[r][kGc + c];
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < kRpw; ++r)
#pragma unroll
    for (int c = 0; c < kRc; ++c) Bm[(warp + 16 * r) * D + lane + 32 * c] = (double)x[r][kGc + c];
}

// T = B Psi (d x r); A = diag(1/s_x) T Psi^T; c = mu_R - mu_x A.  float64 throughout.  Grid (d / 16 + 1, heads): CTA x
// owns 16 rows of A; the last one forms c = mu_R - ((mu_x / s_x) B) Psi Psi^T.  With `At` the map is written as the two
// (d = 64: three) bf16 words the correction pass multiplies with: At [words][BH][n][k], first words, then what their rounding dropped.
// Bound by chains of float64 latencies: four columns of A per thread at a time, quotients and loads ahead of the chains.
// (One CTA per head: 132 us at two heads of d = 128, 630 us beside the attention kernels at 24 heads; spread, one column at a time: 25 and
// 122 us; now 11 and 60 us.)
constexpr int kCompRows = 16;
__global__ void __launch_bounds__(256) k_fit_compose(FitArgs a, int r) {
  extern __shared__ __align__(16) double sm_comp[];
  const int bh = blockIdx.y, d = a.d, tid = threadIdx.x;
  const FitLayout L(a.M, d);
  const double* sc = a.scratch + (size_t)bh * L.total;
  pdl_wait();
  pdl_launch_dependents();
  const int i0 = blockIdx.x * kCompRows;
  const bool tail = i0 >= d;
  float* A = a.A + (i64)bh * d * d;
  float* cvec = a.c + (i64)bh * d;
  __nv_bfloat16* Ah = a.At ? a.At + (i64)bh * d * d : nullptr;
  __nv_bfloat16* Al = a.At ? a.At + ((i64)gridDim.y + bh) * d * d : nullptr;
  auto put = [&](int i, int j, float x) {
    if (!Ah) {
      A[(i64)i * d + j] = x;
    } else {
      const __nv_bfloat16 hb = __float2bfloat16_rn(x);
      Ah[(i64)j * d + i] = hb;
      const float rest = x - __bfloat162float(hb);
      const __nv_bfloat16 lb = __float2bfloat16_rn(rest);
      Al[(i64)j * d + i] = lb;
      if (d == 64) (Al + (i64)gridDim.y * d * d)[(i64)j * d + i] = __float2bfloat16_rn(rest - __bfloat162float(lb));
    }
  };
  if (sc[L.flag] != 0.0 || sc[L.failed] != 0.0) {                 // no usable fit: the head falls back to hard drop
    if (tail) { for (int j = tid; j < d; j += 256) cvec[j] = 0.f; }
    else for (int e = tid; e < kCompRows * d; e += 256) put(i0 + e % kCompRows, e / kCompRows, 0.f);
    return;
  }
  const double* Bm = sc + L.B;
  double* Bs = sm_comp;                    // [16][d] rows of B; tail: 256 parts of u (256 / d of them [d]), then [d] u, then [d] mu_x / s_x
  constexpr int kTailU = 256, kTailRatio = kTailU + 128;
  double* Ts = Bs + kCompRows * d;         // [16][r]
  float* Ps = reinterpret_cast<float*>(Ts + kCompRows * 64);   // [d][r + 1]
  const int ldp = r + 1;
  if (!a.full_rank) {
    const float* Psi = a.Psi + (i64)bh * d * r;
    for (int e = tid; e < d * r; e += 256) Ps[(e / r) * ldp + e % r] = Psi[e];
  }
  if (!tail) {
    for (int e = tid; e < kCompRows * d; e += 256) Bs[e] = Bm[(size_t)i0 * d + e];
    __syncthreads();
    if (!a.full_rank) {
      for (int e = tid; e < kCompRows * r; e += 256) {
        const int i = e / r, t = e % r;
        double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
        for (int k = 0; k < d; k += 2) {
          s0 = fma(Bs[i * d + k], (double)Ps[k * ldp + t], s0);
          s1 = fma(Bs[i * d + k + 1], (double)Ps[(k + 1) * ldp + t], s1);
        }
        Ts[i * r + t] = s0 + s1;
      }
      __syncthreads();
    }
    const int i = tid % kCompRows;         // one row per thread: consecutive lanes write consecutive entries of At
    const double rsx = 1.0 / sc[L.s_x + i0 + i];
    // four columns at a time: the sums over t are chains of float64 latencies (d / 16 is 4 or 8)
    for (int j0 = tid / kCompRows; j0 < d; j0 += 4 * (256 / kCompRows)) {
      double s[4] = {0.0, 0.0, 0.0, 0.0};
      if (a.full_rank) {                   // every row of B lies in the row space of the probe residuals: B Psi Psi^T = B
#pragma unroll
        for (int u = 0; u < 4; ++u) s[u] = Bs[i * d + j0 + u * (256 / kCompRows)];
      } else {
#pragma unroll 4
        for (int t = 0; t < r; ++t) {
          const double x = Ts[i * r + t];
#pragma unroll
          for (int u = 0; u < 4; ++u) s[u] = fma(x, (double)Ps[(j0 + u * (256 / kCompRows)) * ldp + t], s[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) put(i0 + i, j0 + u * (256 / kCompRows), (float)(s[u] * rsx));
    }
    return;
  }
  // c: u = (mu_x / s_x) B by 256 / d parts of the rows, t = u Psi, c = mu_R - t Psi^T
  const int parts = 256 / d, part = tid / d, k = tid % d, per = d / parts;
  double* ratio = Bs + kTailRatio;
  if (tid < d) ratio[tid] = sc[L.mu_x + tid] / sc[L.s_x + tid];
  __syncthreads();
  double u = 0.0;
#pragma unroll 16
  for (int i = part * per; i < (part + 1) * per; ++i) u = fma(ratio[i], Bm[(size_t)i * d + k], u);
  Bs[part * d + k] = u;
  __syncthreads();
  if (tid < d) {
    double t = Bs[tid];
    for (int q = 1; q < parts; ++q) t += Bs[q * d + tid];
    Bs[kTailU + tid] = t;
  }
  __syncthreads();
  const double* us = Bs + kTailU;
  if (a.full_rank) {
    if (tid < d) cvec[tid] = (float)(sc[L.mu_R + tid] - us[tid]);
    return;
  }
  if (tid < r) {
    double t = 0.0;
#pragma unroll 16
    for (int q = 0; q < d; ++q) t = fma(us[q], (double)Ps[q * ldp + tid], t);
    Ts[tid] = t;
  }
  __syncthreads();
  if (tid < d) {
    double s = 0.0;
#pragma unroll 4
    for (int t = 0; t < r; ++t) s = fma(Ts[t], (double)Ps[tid * ldp + t], s);
    cvec[tid] = (float)(sc[L.mu_R + tid] - s);
  }
}

static size_t compose_smem(int d, int r) { return ((size_t)kCompRows * d + kCompRows * 64) * sizeof(double) + (size_t)d * (r + 1) * sizeof(float); }

cudaError_t init_fit() {
  return cudaFuncSetAttribute(k_fit_compose, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)compose_smem(128, kMaxRank));
}

void launch_fit(const FitArgs& a, cudaStream_t st) {
  const int d = a.d;
  const int r = min(a.r_out, min(a.M, d));
  const FitLayout L(a.M, d);
  launch_pdl(k_fit_prepare, dim3(d / kPrepCols, a.BH), dim3(kPrepCols * kPrepSlices), 0, st, a);
  const int tile = a.precise ? kGramTile<double> : kGramTile<float>, nt = d / tile;
  const dim3 gg(nt * nt, a.BH, 3);
  if (a.precise) {
    launch_pdl(k_fit_gram<double>, gg, dim3(256), 0, st, a);
    if (d == 128) launch_pdl(k_fit_solve<double, 128>, dim3(a.BH, 128 / kSolveRhs<double, 128>), dim3(512), 0, st, a);
    else launch_pdl(k_fit_solve<double, 64>, dim3(a.BH, 64 / kSolveRhs<double, 64>), dim3(512), 0, st, a);
  } else {
    launch_pdl(k_fit_gram<float>, gg, dim3(256), 0, st, a);
    if (d == 128) launch_pdl(k_fit_solve<float, 128>, dim3(a.BH, 128 / kSolveRhs<float, 128>), dim3(512), 0, st, a);
    else launch_pdl(k_fit_solve<float, 64>, dim3(a.BH, 64 / kSolveRhs<float, 64>), dim3(512), 0, st, a);
  }
  // Psi_r: leading eigenvectors of S = Rb^T W Rb, i.e. right singular vectors of W^(1/2) Rb.
  // The solve and the first kernel of the eigen-solver both only need the Gram matrices: they run side by side.
  if (!a.full_rank) launch_eig_top(a.scratch + L.S, (i64)L.total, a.BH, d, r, 1, a.precise, a.Psi, nullptr, a.eig_ws, st, true);
  launch_pdl(k_fit_compose, dim3(d / kCompRows + 1, a.BH), dim3(256), compose_smem(d, a.full_rank ? 0 : r), st, a, r);
}

}  // namespace spr
