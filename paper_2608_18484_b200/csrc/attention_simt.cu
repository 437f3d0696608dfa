// float32 attention kernels on the CUDA cores: block-sparse attention with
// renormalised hard drop (Eq. 3) over the group-major layout, dense attention
// (Eq. 1), the residual correction (Eq. 9), and the exact probe rows with their
// retained/omitted statistics (Appendix A.1).  These are the kernels of the float32
// configuration, whose 1e-5 tolerance rules out reduced-precision tensor-core inputs.
#include <algorithm>
#include "kernels.cuh"

namespace spr {

constexpr int BM = 64;     // query rows per CTA
constexpr int BN = 64;     // keys per tile
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float row16_max(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float row16_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// =============================================================================
// Main kernel.  SPARSE: one CTA per item of a list (below): up to 64 rows of one query group against the keys of its routed
// K/V groups, streamed as one concatenated sequence (every tile of 64 keys is full except the last), or against a part of
// them.  Dense: one CTA per 64 rows over all keys.  Stores the hard-drop output at the original token index; the correction
// is a pass of its own, so that the probe rows and the fit can run beside this kernel.
//
// Bound by the FMA pipe: 128 threads, two CTAs per SM, thread (ty, tx) holds R query rows x 4 keys of the scores and
// R rows x D / 16 columns of the output, so that a 16-byte shared-memory read serves 8 to 32 multiply-adds, and all of
// them are packed two to an instruction (scores: even and odd dimensions in separate halves; output: column pairs).
// Rows are 16 bytes longer than their data, which keeps the 16-byte reads of consecutive rows in different banks.  The
// probabilities take the place of the K tile.  Tiles arrive by cp.async, V under the scores; the other CTA of the SM covers
// the latency of K.
// 8 heads, 7161 tokens, d = 128, routed density 0.24: 4040 us with 256 threads and blocks of 4 x 4 single multiply-adds, 2640 us
// with packed 8 x 4 blocks, 1610 us with equal row tiles, parts and descending order; dense 47 of the 74 TFLOP/s of the pipe.
// =============================================================================
constexpr int kFThreads = 128;
template <int D> struct F32Smem {
  static constexpr int ld = D + 4, ldp = BM + 4;
  static constexpr int q = BM * ld, k = BN * ld, v = BN * D;
  static constexpr size_t bytes = (size_t)(q + k + v) * sizeof(float) + 2 * BN * sizeof(int);
  static_assert(BN * ldp <= k, "the probabilities fit into the K tile");
};
__device__ __forceinline__ void cp16(float* dst, const float* src, bool on) {     // 16 bytes, zeros when off
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = on ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// what a CTA works on: rows row0 .. row0 + nrows of head bh against key tiles [t_begin, t_end) of L keys
struct F32Work {
  int bh, row0, nrows, L, t_begin, t_end, z, parts, slot, nroute;
  const int *ridx, *kvoff;                               // routed groups and group offsets of the head (SPARSE)
  const float *Qb, *Kb, *Vb;
  i64 qsn, ksn, vsn;
};

// R: rows per thread, ceil(nrows / 8).  Row ty R + i of the tile sits in row ty 8 + i of the shared-memory tiles, so that all R share
// one layout with aligned 16-byte rows.
template <int D, bool SPARSE, int R>
__device__ __forceinline__ void attend_f32(const AttnArgs& a, const F32Work& w, float* smem, const int* cum, int* scratch, float* __restrict__ part,
                                           int* __restrict__ counter) {
  using S = F32Smem<D>;
  float* Qs = smem;                                      // [64][D + 4]
  float* Ks = Qs + S::q;                                 // [64][D + 4], then P [64 keys][64 rows + 4]
  float* Vs = Ks + S::k;                                 // [64][D]
  int* krow = reinterpret_cast<int*>(Vs + S::v);         // [2][64] source row of every key of this / the next tile
  constexpr int OP = D / 32;                             // output column pairs per thread: columns 4 tx + 64 c + {0..3}
  constexpr int CPR = D / 4;                             // 16-byte chunks per row
  constexpr int RV = (R + 3) / 4;                        // 16-byte pieces of a thread's probabilities of one key
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int L = w.L;
#pragma unroll 4
  for (int e = tid; e < 8 * R * CPR; e += kFThreads) {
    const int r = e / CPR, c = (e % CPR) * 4;
    cp16(Qs + (r / R * 8 + r % R) * S::ld + c, w.Qb + (i64)(w.row0 + min(r, w.nrows - 1)) * w.qsn + c, r < w.nrows);
  }
  auto find_rows = [&](int t, int* dst) {                // source rows of key tile t
    if (tid < BN) {
      const int pos = t * BN + tid;
      int src = -1;
      if (pos < L) {
        if (SPARSE) {
          int lo = 0, hi = w.nroute - 1;                 // last range with cum[range] <= pos
          while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (cum[mid] <= pos) lo = mid; else hi = mid - 1; }
          src = w.kvoff[w.ridx[lo]] + (pos - cum[lo]);
        } else src = pos;
      }
      dst[tid] = src;
    }
  };
  find_rows(w.t_begin, krow);

  float2 o[R][OP];
  float m[R], l[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    m[i] = -INFINITY; l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < OP; ++c) o[i][c] = make_float2(0.f, 0.f);
  }
  const float sc = a.scale * kLog2e;
  for (int t = w.t_begin; t < w.t_end; ++t) {
    const int* kr = krow + ((t - w.t_begin) & 1) * BN;
    const int ncols = min(BN, L - t * BN);
    __syncthreads();                                     // previous tile fully consumed, rows of this one known
#pragma unroll 8
    for (int e = tid; e < BN * CPR; e += kFThreads) {
      const int r = e / CPR, c = (e % CPR) * 4, src = kr[r];
      cp16(Ks + r * S::ld + c, w.Kb + (i64)max(src, 0) * w.ksn + c, src >= 0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 8
    for (int e = tid; e < BN * CPR; e += kFThreads) {
      const int r = e / CPR, c = (e % CPR) * 4, src = kr[r];
      cp16(Vs + r * D + c, w.Vb + (i64)max(src, 0) * w.vsn + c, src >= 0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (t + 1 < w.t_end) find_rows(t + 1, krow + ((t + 1 - w.t_begin) & 1) * BN);
    asm volatile("cp.async.wait_group 1;" ::: "memory"); // Q and K
    __syncthreads();
    // scores of rows ty R + i and keys tx + 16 j
    float s[R][4];
    {
      float2 acc[R][4];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
      const float* qp = Qs + ty * 8 * S::ld;
      const float* kp = Ks + tx * S::ld;
#pragma unroll 2
      for (int k = 0; k < D; k += 4) {
        float4 kk[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) kk[j] = *reinterpret_cast<const float4*>(kp + 16 * j * S::ld + k);
        float4 q[R];
#pragma unroll
        for (int i = 0; i < R; ++i) q[i] = *reinterpret_cast<const float4*>(qp + i * S::ld + k);
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = __ffma2_rn(make_float2(q[i].x, q[i].y), make_float2(kk[j].x, kk[j].y), acc[i][j]);
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = __ffma2_rn(make_float2(q[i].z, q[i].w), make_float2(kk[j].z, kk[j].w), acc[i][j]);
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = tx + 16 * j < ncols ? (acc[i][j].x + acc[i][j].y) * sc : -INFINITY;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory"); // V
    __syncthreads();                                     // K is consumed: its place takes the probabilities
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float mx = row16_max(fmaxf(fmaxf(s[i][0], s[i][1]), fmaxf(s[i][2], s[i][3])));
      const float mn = fmaxf(m[i], mx);
      const float corr = exp2f(m[i] - mn);               // 0 on the first tile (m = -inf)
      m[i] = mn;
#pragma unroll
      for (int j = 0; j < 4; ++j) s[i][j] = exp2f(s[i][j] - mn);
      l[i] = fmaf(l[i], corr, (s[i][0] + s[i][1]) + (s[i][2] + s[i][3]));
      if (corr != 1.f) {
#pragma unroll
        for (int c = 0; c < OP; ++c) { o[i][c].x *= corr; o[i][c].y *= corr; }
      }
    }
    float* Ps = Ks;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float* pp = Ps + (tx + 16 * j) * S::ldp + ty * 8;
#pragma unroll
      for (int u = 0; u < RV; ++u)
        *reinterpret_cast<float4*>(pp + 4 * u) = make_float4(s[4 * u][j], 4 * u + 1 < R ? s[min(4 * u + 1, R - 1)][j] : 0.f,
                                                             4 * u + 2 < R ? s[min(4 * u + 2, R - 1)][j] : 0.f, 4 * u + 3 < R ? s[min(4 * u + 3, R - 1)][j] : 0.f);
    }
    __syncthreads();
#pragma unroll 4
    for (int j = 0; j < ncols; ++j) {
      float pv[4 * RV];
#pragma unroll
      for (int u = 0; u < RV; ++u) {
        const float4 p = *reinterpret_cast<const float4*>(Ps + j * S::ldp + ty * 8 + 4 * u);
        pv[4 * u] = p.x; pv[4 * u + 1] = p.y; pv[4 * u + 2] = p.z; pv[4 * u + 3] = p.w;
      }
#pragma unroll
      for (int c = 0; c < OP / 2; ++c) {
        const float4 v = *reinterpret_cast<const float4*>(Vs + j * D + 64 * c + 4 * tx);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const float2 pp = make_float2(pv[i], pv[i]);
          o[i][2 * c] = __ffma2_rn(pp, make_float2(v.x, v.y), o[i][2 * c]);
          o[i][2 * c + 1] = __ffma2_rn(pp, make_float2(v.z, v.w), o[i][2 * c + 1]);
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) l[i] = row16_sum(l[i]);
  if (SPARSE && w.parts > 1) {
    float* mine = part + (i64)(w.slot + w.z) * BM * (D + 2);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = ty * R + i;
      if (tx == 0) { mine[r] = m[i]; mine[BM + r] = l[i]; }
#pragma unroll
      for (int c = 0; c < OP / 2; ++c)
        *reinterpret_cast<float4*>(mine + 2 * BM + r * D + 64 * c + 4 * tx) = make_float4(o[i][2 * c].x, o[i][2 * c].y, o[i][2 * c + 1].x, o[i][2 * c + 1].y);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) scratch[0] = atomicAdd(counter + w.slot, 1);
    __syncthreads();
    if (scratch[0] != w.parts - 1) return;
    __threadfence();
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = ty * R + i;
      float mm = -INFINITY;
      for (int q = 0; q < w.parts; ++q) mm = fmaxf(mm, part[(i64)(w.slot + q) * BM * (D + 2) + r]);
      m[i] = mm; l[i] = 0.f;
#pragma unroll
      for (int c = 0; c < OP; ++c) o[i][c] = make_float2(0.f, 0.f);
      for (int q = 0; q < w.parts; ++q) {
        const float* pq = part + (i64)(w.slot + q) * BM * (D + 2);
        const float f = exp2f(pq[r] - mm);
        l[i] = fmaf(f, pq[BM + r], l[i]);
#pragma unroll
        for (int c = 0; c < OP / 2; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(pq + 2 * BM + r * D + 64 * c + 4 * tx);
          o[i][2 * c] = __ffma2_rn(make_float2(f, f), make_float2(v.x, v.y), o[i][2 * c]);
          o[i][2 * c + 1] = __ffma2_rn(make_float2(f, f), make_float2(v.z, v.w), o[i][2 * c + 1]);
        }
      }
    }
  }
  // ---- epilogue -------------------------------------------------------------------
  float* Ob = (float*)a.O + w.bh / a.H * a.os[0] + w.bh % a.H * a.os[1];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = ty * R + i;
    if (r >= w.nrows) continue;
    const float inv = l[i] > 0.f ? 1.f / l[i] : 0.f;
    const int dst = SPARSE ? a.q_perm[(i64)w.bh * a.N + w.row0 + r] : w.row0 + r;
#pragma unroll
    for (int c = 0; c < OP / 2; ++c) {
      const float4 v = make_float4(o[i][2 * c].x * inv, o[i][2 * c].y * inv, o[i][2 * c + 1].x * inv, o[i][2 * c + 1].y * inv);
      *reinterpret_cast<float4*>(Ob + (i64)dst * a.os[2] + 64 * c + 4 * tx) = v;
      if (a.O_sparse) *reinterpret_cast<float4*>(a.O_sparse + ((i64)w.bh * a.N + dst) * D + 64 * c + 4 * tx) = v;
    }
  }
}

template <int D>
__global__ void __launch_bounds__(kFThreads, 2) k_attention_f32_sparse(AttnArgs a, float* __restrict__ part, int* __restrict__ counter) {
  extern __shared__ __align__(16) float smem[];
  __shared__ int cum[kMaxGroups + 1];
  __shared__ int scratch[34];
  if ((int)blockIdx.x >= *a.n_items) return;
  const int4 it = a.items[blockIdx.x];
  F32Work w;
  w.bh = it.x / a.Cq; w.row0 = it.y; w.nrows = it.z & 0xFF; w.z = (it.z >> 8) & 0xFF; w.parts = it.z >> 16; w.slot = it.w;
  const int g = it.x % a.Cq;
  const int* rp = a.route_ptr + (i64)w.bh * (a.Cq + 1);
  w.ridx = a.route_idx + (i64)w.bh * a.Cq * a.Ck + rp[g];
  w.nroute = rp[g + 1] - rp[g];
  w.kvoff = a.kv_off + (i64)w.bh * (a.Ck + 1);
  for (int t = threadIdx.x; t < w.nroute; t += kFThreads) { const int bb = w.ridx[t]; cum[t] = w.kvoff[bb + 1] - w.kvoff[bb]; }
  __syncthreads();
  w.L = block_exclusive_scan(cum, w.nroute, scratch);    // ends with a barrier
  const i64 base = (i64)w.bh * a.N * D;
  w.Qb = (const float*)a.Q + base; w.Kb = (const float*)a.K + base; w.Vb = (const float*)a.V + base;
  w.qsn = w.ksn = w.vsn = D;
  const int n_tiles = (w.L + BN - 1) / BN;
  w.t_begin = (int)((i64)n_tiles * w.z / w.parts); w.t_end = (int)((i64)n_tiles * (w.z + 1) / w.parts);
  switch ((w.nrows + 7) >> 3) {
    case 1: case 2: attend_f32<D, true, 2>(a, w, smem, cum, scratch, part, counter); break;
    case 3: attend_f32<D, true, 3>(a, w, smem, cum, scratch, part, counter); break;
    case 4: attend_f32<D, true, 4>(a, w, smem, cum, scratch, part, counter); break;
    case 5: attend_f32<D, true, 5>(a, w, smem, cum, scratch, part, counter); break;
    case 6: attend_f32<D, true, 6>(a, w, smem, cum, scratch, part, counter); break;
    case 7: attend_f32<D, true, 7>(a, w, smem, cum, scratch, part, counter); break;
    default: attend_f32<D, true, 8>(a, w, smem, cum, scratch, part, counter);
  }
}
template <int D>
__global__ void __launch_bounds__(kFThreads, 2) k_attention_f32_dense(AttnArgs a) {
  extern __shared__ __align__(16) float smem[];
  F32Work w;
  w.bh = blockIdx.y; w.row0 = blockIdx.x * BM; w.nrows = min(BM, a.N - w.row0); w.L = a.N;
  w.t_begin = 0; w.t_end = (w.L + BN - 1) / BN; w.parts = 1;
  const int b = w.bh / a.H, h = w.bh % a.H;
  w.Qb = (const float*)a.Q + b * a.qs[0] + h * a.qs[1]; w.Kb = (const float*)a.K + b * a.ks[0] + h * a.ks[1];
  w.Vb = (const float*)a.V + b * a.vs[0] + h * a.vs[1];
  w.qsn = a.qs[2]; w.ksn = a.ks[2]; w.vsn = a.vs[2];
  attend_f32<D, false, 8>(a, w, smem, nullptr, nullptr, nullptr, nullptr);
}

// ---- the list of items: which rows and keys, longest first ---------------------------
// The groups of a plan differ by more than ten times in rows and in routed keys.  A group's rows are cut into tiles of equal
// size, at most 64 rows, whose CTA does the work of 8 ceil(rows / 8) rows; the keys of a tile are cut into parts of about
// `chunk` key tiles; the items are issued in descending order of their work, so that no long one is left for the end.
// Every part of a cut tile leaves (m, l, O) in `part`, and the CTA that finishes last (a counter per tile) adds them up in
// the order of the parts.  The chunk is the smallest of the series 4, 6, 8, 12, 16, 24 ... that gives at most max_items items
// (attention_f32_items) and max_slots parts of cut tiles (attention_f32_slots): fine enough for a small list to fill the GPU, and for the kernels of the probes and the fit to find
// free slots beside a large one (they would wait for the longest items of the first wave), coarse enough that the parts
// cost little.
// keys of every group's routes, in boxes of `box` rows of which only the last of a range may be short
__global__ void __launch_bounds__(1024) k_route_keys(const int* __restrict__ kv_off, const int* __restrict__ route_ptr, const int* __restrict__ route_idx, int Cq,
                                                     int Ck, int kv_div, int box, int* __restrict__ keys) {
  const int bh = blockIdx.y, g = blockIdx.x * 32 + (threadIdx.x >> 5);
  if (g >= Cq) return;
  const int* rp = route_ptr + (i64)bh * (Cq + 1);
  const int* ri = route_idx + (i64)bh * Cq * Ck;
  const int* ko = kv_off + (i64)(bh / kv_div) * (Ck + 1);
  int L = 0;
  for (int t = rp[g] + (threadIdx.x & 31); t < rp[g + 1]; t += 32) { const int b = ri[t]; L += (ko[b + 1] - ko[b] + box - 1) / box; }
  L = warp_sum(L);
  if ((threadIdx.x & 31) == 0) keys[(i64)bh * Cq + g] = L;
}
constexpr int kItemBuckets = 1024, kChunks = 15;
__device__ __forceinline__ int item_chunk(int j) { return (j & 1 ? 6 : 4) << (j >> 1); }       // 4, 6, 8 .. 512
__device__ __forceinline__ int item_parts(int nt, int j) {                                     // j = kChunks: whole
  const int c = item_chunk(j);
  return j < kChunks ? min(max((nt + c / 2) / c, 1), 255) : 1;
}
__global__ void __launch_bounds__(kItemBuckets) k_f32_items(const int* __restrict__ q_off, const int* __restrict__ keys, int BH, int Cq, int max_items, int max_slots,
                                                            int shift, int4* __restrict__ items, int* __restrict__ n_items) {
  __shared__ int hist[kItemBuckets];
  __shared__ int scratch[34];
  __shared__ int slots, sum[kChunks], cut[kChunks];
  hist[threadIdx.x] = 0;
  if (threadIdx.x == 0) slots = 0;
  if (threadIdx.x < kChunks) { sum[threadIdx.x] = 0; cut[threadIdx.x] = 0; }
  __syncthreads();
  int n_of[kChunks] = {}, n_cut[kChunks] = {}, first, n, tiles, rows, nt;
  auto group = [&](int e) {
    const int* qo = q_off + (i64)(e / Cq) * (Cq + 1) + e % Cq;
    first = qo[0]; n = qo[1] - first;
    tiles = (n + BM - 1) / BM; rows = n > 0 ? (n + tiles - 1) / tiles : 0; nt = (keys[e] + BN - 1) / BN;
    return n > 0;
  };
  for (int e = threadIdx.x; e < BH * Cq; e += kItemBuckets)
    if (group(e)) {
#pragma unroll
      for (int j = 0; j < kChunks; ++j) { const int parts = item_parts(nt, j); n_of[j] += tiles * parts; n_cut[j] += parts > 1 ? tiles * parts : 0; }
    }
#pragma unroll
  for (int j = 0; j < kChunks; ++j) {
    const int v = __reduce_add_sync(0xffffffffu, n_of[j]), c = __reduce_add_sync(0xffffffffu, n_cut[j]);
    if ((threadIdx.x & 31) == 0) { atomicAdd(&sum[j], v); atomicAdd(&cut[j], c); }
  }
  __syncthreads();
  int j = 0;
  while (j < kChunks && (sum[j] > max_items || cut[j] > max_slots)) ++j;
  int total = 0;
  for (int pass = 0; pass < 2; ++pass) {
    for (int e = threadIdx.x; e < BH * Cq; e += kItemBuckets) {
      if (!group(e)) continue;
      const int parts = item_parts(nt, j);
      const int bucket = kItemBuckets - 1 - min(kItemBuckets - 1, (((nt + parts - 1) / parts + 1) * ((rows + 7) / 8 + 1)) >> shift);
      int at = atomicAdd(&hist[bucket], tiles * parts);
      if (pass == 0) continue;
      const int slot = parts > 1 ? atomicAdd(&slots, tiles * parts) : 0;
      for (int t = 0; t < tiles; ++t)
        for (int z = 0; z < parts; ++z, ++at)
          items[at] = make_int4(e, first + t * rows, min(rows, n - t * rows) | z << 8 | parts << 16, slot + t * parts);
    }
    __syncthreads();
    if (pass == 0) total = block_exclusive_scan(hist, kItemBuckets, scratch);
  }
  if (threadIdx.x == 0) *n_items = total;
}

// Residual correction of Eq. 9 in place: O <- X + X A + c for the rows X = O (float32).  A CTA takes 32 rows of a head, thread
// (ty, tx) 4 of them x D / 16 columns, two columns to a multiply-add.  Bound by reads of shared memory (85 % of their rate, FMA pipe 64 %, at
// 8 heads of 7161 rows, d = 128): A comes through it, 16 of its rows under the arithmetic of the 16 before.  With A read through L2 and
// single multiply-adds that call took 103 us, now 45 (64 rows per CTA: 46); 2 heads of 4096 rows, d = 64, 11.6, now 4.6 (4.8).
constexpr int kCorrK = 16;
template <int D>
__global__ void __launch_bounds__(128) k_correction_f32(const float* __restrict__ A, const float* __restrict__ cvec, int H, int N,
                                                        float* __restrict__ O, i64 ob, i64 oh, i64 on) {
  constexpr int R = 4, ld = D + 4, OP = D / 32;
  __shared__ __align__(16) float xs[8 * R * ld], as[2 * kCorrK * D];
  const int bh = blockIdx.y, row0 = blockIdx.x * 8 * R, nr = min(8 * R, N - row0);
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  float* Ob = O + (bh / H) * ob + (bh % H) * oh;
  const float* Ah = A + (i64)bh * D * D;
  auto fetch = [&](int k0) {
    float* dst = as + (k0 / kCorrK & 1) * kCorrK * D;
#pragma unroll
    for (int e = tid * 4; e < kCorrK * D; e += 512) cp16(dst + e, Ah + k0 * D + e, true);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll 8
  for (int e = tid; e < 8 * R * (D / 4); e += 128) {
    const int r = e / (D / 4), c = (e % (D / 4)) * 4;
    cp16(xs + r * ld + c, Ob + (i64)(row0 + min(r, nr - 1)) * on + c, r < nr);
  }
  fetch(0);
  float2 acc[R][OP];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int c = 0; c < OP; ++c) acc[i][c] = make_float2(0.f, 0.f);
  for (int k0 = 0; k0 < D; k0 += kCorrK) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                     // this chunk is there, the one before is consumed
    if (k0 + kCorrK < D) fetch(k0 + kCorrK);
    const float* ac = as + (k0 / kCorrK & 1) * kCorrK * D + 4 * tx;
#pragma unroll 2
    for (int k = 0; k < kCorrK; k += 4) {
      float x[R][4];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(xs + (ty * R + i) * ld + k0 + k);
        x[i][0] = v.x; x[i][1] = v.y; x[i][2] = v.z; x[i][3] = v.w;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < OP / 2; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(ac + (k + u) * D + 64 * c);
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const float2 xx = make_float2(x[i][u], x[i][u]);
            acc[i][2 * c] = __ffma2_rn(xx, make_float2(v.x, v.y), acc[i][2 * c]);
            acc[i][2 * c + 1] = __ffma2_rn(xx, make_float2(v.z, v.w), acc[i][2 * c + 1]);
          }
        }
    }
  }
#pragma unroll
  for (int c = 0; c < OP / 2; ++c) {
    const float4 cv = *reinterpret_cast<const float4*>(cvec + (i64)bh * D + 64 * c + 4 * tx);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = ty * R + i;
      if (r >= nr) continue;
      const float4 x = *reinterpret_cast<const float4*>(xs + r * ld + 64 * c + 4 * tx);
      *reinterpret_cast<float4*>(Ob + (i64)(row0 + r) * on + 64 * c + 4 * tx) =
          make_float4(x.x + (cv.x + acc[i][2 * c].x), x.y + (cv.y + acc[i][2 * c].y), x.z + (cv.z + acc[i][2 * c + 1].x), x.w + (cv.w + acc[i][2 * c + 1].y));
    }
  }
}
void launch_correction_f32(const float* A, const float* c, void* O, const i64* os, int BH, int H, int N, int d, cudaStream_t st) {
  const dim3 grid((N + 31) / 32, BH);
  if (d == 128) k_correction_f32<128><<<grid, 128, 0, st>>>(A, c, H, N, (float*)O, os[0], os[1], os[2]);
  else k_correction_f32<64><<<grid, 128, 0, st>>>(A, c, H, N, (float*)O, os[0], os[1], os[2]);
}

// Items of a list at most: four rounds of CTAs on every SM slot, and twice as many as tiles.
size_t attention_f32_items(int BH, int N, int Cq) { return std::max((size_t)4 * 2 * sm_count(), (size_t)2 * BH * ((N + BM - 1) / BM + Cq)); }
// Partial states of cut tiles at most, 79 MB at d = 128 whatever the size.  (6 heads of 10224 tokens, d = 64: call 2459 us with 8 per SM, 2433
// with 16 and with 32; 8 heads of 7161 tokens, d = 128: 3335 to 3347 us with 4, 8, 16 and as many as items, which were 1.2 GB of workspace at
// 24 heads of 32760 tokens.)
size_t attention_f32_slots() { return (size_t)16 * sm_count(); }
size_t attention_f32_part_floats(int d) { return attention_f32_slots() * BM * (d + 2); }
void launch_f32_items(const int* q_off, const int* kv_off, const int* route_ptr, const int* route_idx, int BH, int N, int Cq, int Ck, int* keys, int4* items,
                      int* n_items, cudaStream_t st) {
  k_route_keys<<<dim3((Cq + 31) / 32, BH), 1024, 0, st>>>(kv_off, route_ptr, route_idx, Cq, Ck, 1, 1, keys);
  int shift = 0;
  while ((((N + BN - 1) / BN + 1) * 9) >> shift >= kItemBuckets) ++shift;
  k_f32_items<<<1, kItemBuckets, 0, st>>>(q_off, keys, BH, Cq, (int)attention_f32_items(BH, N, Cq), (int)attention_f32_slots(), shift, items, n_items);
}

// The 128-row tensor-core kernel: the tiles of a head, longest first (per head, not over all of them: tiles of one head run together
// and share its keys in L2).  Every 128 rows of a group are a tile; a last tile of at most small_rem rows is left to the
// remainder kernel.  Two lists: pairs of tiles of a group (none where cap_pairs is 0), and tiles left alone.  Item: first row, boxes of 16 keys, place of the
// group's routes in the head's list, rows << 16 | routes.
__global__ void __launch_bounds__(kItemBuckets) k_tc_items(const int* __restrict__ q_off, const int* __restrict__ route_ptr, const int* __restrict__ boxes, int Cq, int small_rem,
                                                           int shift, int cap_pairs, int cap_single, int4* __restrict__ items, int* __restrict__ n_items) {
  __shared__ int hist[kItemBuckets];
  __shared__ int scratch[34];
  const int bh = blockIdx.x, single = blockIdx.y;
  const int* qo = q_off + (i64)bh * (Cq + 1);
  const int* rp = route_ptr + (i64)bh * (Cq + 1);
  int4* out = single ? items + (i64)gridDim.x * cap_pairs + (i64)bh * cap_single : items + (i64)bh * cap_pairs;
  hist[threadIdx.x] = 0;
  __syncthreads();
  int total = 0;
  for (int pass = 0; pass < 2; ++pass) {
    for (int a = threadIdx.x; a < Cq; a += kItemBuckets) {
      const int first = qo[a], all = qo[a + 1] - first, n = all - (all % 128 <= small_rem ? all % 128 : 0), bx = boxes[(i64)bh * Cq + a];
      const int pairs = cap_pairs ? n / 256 + (n % 256 > 128 ? 1 : 0) : 0, alone = max(n - 256 * pairs, 0), mine = single ? (alone + 127) / 128 : pairs;
      if (mine == 0) continue;
      int at = atomicAdd(&hist[kItemBuckets - 1 - min(kItemBuckets - 1, bx >> shift)], mine);
      if (pass == 0) continue;
      const int r0 = rp[a], nr = rp[a + 1] - r0;
      const int size = single ? 128 : 256, from = single ? 256 * pairs : 0;
      for (int t = 0; t < mine; ++t) out[at + t] = make_int4(first + from + size * t, bx, r0, min(size, n - from - size * t) << 16 | nr);
    }
    __syncthreads();
    if (pass == 0) total = block_exclusive_scan(hist, kItemBuckets, scratch);
  }
  if (threadIdx.x == 0) n_items[single * gridDim.x + bh] = total;
}
// Two tiles per CTA where one per CTA gives the SMs 20 rounds or more (d = 64: 40): below, and above all where the longest tiles decide,
// it is better to have the tiles on as many SMs.  Attend on a kept plan, us with tiles alone and with pairs: 8 heads of 9360 tokens (4
// rounds) 233, 340; 12 of 9360 (6) 320, 371; 12 of 18720 (12) 895, 901; 8 of 49152 (21) 3795, 3767; 24 of 32760 (42) 4951, 4901; 40
// of 75600 (160) 37950, 37220.  d = 64: 16 of 17550 (15) 1235, 1272; 16 of 35100 (30) 4253, 4286; 24 of 32760 (42) 3373, 3360.
int attention_tc_pairs(int BH, int N, int d) { return (i64)BH * N >= (i64)(d == 128 ? 20 : 40) * sm_count() * 128 ? (N + 128) / 129 : 0; }      // (a pair has more than 128 rows)
int attention_tc_singles(int BH, int N, int Cq, int d) { return attention_tc_pairs(BH, N, d) ? Cq : (N + 127) / 128 + Cq; }
void launch_tc_items(const int* q_off, const int* kv_off, const int* route_ptr, const int* route_idx, int BH, int N, int Cq, int Ck, int d, int kv_div, int* boxes, int4* items,
                     int* n_items, cudaStream_t st) {
  k_route_keys<<<dim3((Cq + 31) / 32, BH), 1024, 0, st>>>(kv_off, route_ptr, route_idx, Cq, Ck, kv_div, 16, boxes);
  int shift = 0;
  while (((N + 15) / 16 + Ck) >> shift >= kItemBuckets) ++shift;
  k_tc_items<<<dim3(BH, 2), kItemBuckets, 0, st>>>(q_off, route_ptr, boxes, Cq, kRemRows, shift, attention_tc_pairs(BH, N, d), attention_tc_singles(BH, N, Cq, d), items, n_items);
}

template <int D>
static void attention_dispatch(const AttnArgs& a, float* part, int* counter, cudaStream_t st) {
  if (a.items) {
    const unsigned items = (unsigned)attention_f32_items(a.BH, a.N, a.Cq);
    cudaMemsetAsync(counter, 0, attention_f32_slots() * sizeof(int), st);
    k_attention_f32_sparse<D><<<items, kFThreads, F32Smem<D>::bytes, st>>>(a, part, counter);
  } else {
    k_attention_f32_dense<D><<<dim3((a.N + BM - 1) / BM, a.BH), kFThreads, F32Smem<D>::bytes, st>>>(a);
  }
}
void launch_attention_f32(const AttnArgs& a, float* part, int* counter, cudaStream_t st) {
  if (a.d == 128) attention_dispatch<128>(a, part, counter, st); else attention_dispatch<64>(a, part, counter, st);
}

// =============================================================================
// Probe rows (Appendix A.1-A.2).  For each probe p one pass over ALL keys keeps two
// online-softmax states: the keys retained by p's query group (Z_S, N_S) and the
// omitted ones (Z_U, N_U).  Then O_sp = N_S/Z_S and O_dense = (N_S+N_U)/(Z_S+Z_U).
// The key range is split across CTAs; partial states are merged afterwards.
// partial layout: [BH][n_split][M][2][D+2] = (m, l, N[D]) for the S and the U state.
//
// Bound by the latency of a few warps' dependent steps: two CTAs to an SM leave two warps to a scheduler, which issue in 39 % of the
// cycles (FMA pipe 43 %, shared memory 57 %, at 8 heads of 7161 tokens, d = 128).  A key belongs to one of a row's
// two states, and keys are group-major, so both states change hands only where a K/V group ends: a thread multiplies into the
// row's current state and swaps it with the other one there, which is one product with V per key instead of two.  32 rows per
// CTA (both states of four rows and the scores fit a thread's registers), packed 4 x 4 score blocks; K of the next tile
// arrives under the product with V, V under the scores.  With one block of 4 x 4 single multiply-adds per state, 64 rows per CTA
// and loads that were waited for: 2 heads of 4096 tokens, d = 64, 32 probes 60 us, now 15 us; 8 heads of 7161 tokens, d = 128,
// 64 probes (beside the attention) 200 us, now 81 us.
// =============================================================================
constexpr int kProbeRows = 32;
template <int D> struct ProbeSmem {
  static constexpr int ld = D + 4, ldp = kProbeRows + 4;
  static constexpr int q = kProbeRows * ld, k = BN * ld, v = BN * D, p = BN * ldp;
  static size_t bytes(int Ck) {
    return (size_t)(q + k + v + p) * sizeof(float) + (size_t)(kProbeRows * ((Ck + 31) / 32) + 2 * BN + Ck) * sizeof(int);
  }
};
template <int D>
__global__ void __launch_bounds__(kFThreads, 2) k_probe_rows(ProbeArgs a) {
  extern __shared__ __align__(16) float smem[];
  using S = ProbeSmem<D>;
  float* Qs = smem;                                          // [32][D + 4]
  float* Ks = Qs + S::q;                                     // [64][D + 4]
  float* Vs = Ks + S::k;                                     // [64][D]
  float* Ps = Vs + S::v;                                     // [64 keys][32 rows + 4]
  const int words = (a.Ck + 31) / 32;
  unsigned* bitmap = reinterpret_cast<unsigned*>(Ps + S::p); // [32][words] routes of every row's group
  int* kgrp = reinterpret_cast<int*>(bitmap + kProbeRows * words);   // [2][64] K/V group of every key of this / the next tile
  int* koff = kgrp + 2 * BN;                                 // [Ck]
  constexpr int OP = D / 32, CPR = D / 4, R = 4;             // output column pairs, 16-byte chunks of a row, rows per thread
  const int bh = blockIdx.z;
  const int m0 = blockIdx.y * kProbeRows, nrows = min(kProbeRows, a.M - m0);
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int* pidx = a.probe_idx + (i64)bh * a.M + m0;
  const float* Qb = (const float*)a.Qg + (i64)bh * a.N * D;
  const int* inv = a.q_inv + (i64)bh * a.N;
  const float* Kb = (const float*)a.Kg + (i64)bh * a.N * D;
  const float* Vb = (const float*)a.Vg + (i64)bh * a.N * D;
  const int* kvoff = a.kv_off + (i64)bh * (a.Ck + 1);

  // key positions of this split, in whole tiles
  const int tiles = (a.N + BN - 1) / BN;
  const int per = (tiles + a.n_split - 1) / a.n_split;
  const int k_begin = min(a.N, (int)blockIdx.x * per * BN), k_end = min(a.N, ((int)blockIdx.x + 1) * per * BN);

  auto load_keys = [&](const float* base, float* dst, int ld, int t0) {   // one commit group, empty past the last tile
    if (t0 < k_end) {
#pragma unroll 8
      for (int e = tid; e < BN * CPR; e += kFThreads) {
        const int r = e / CPR, c = (e % CPR) * 4;
        const bool on = t0 + r < k_end;
        cp16(dst + r * ld + c, base + (i64)(on ? t0 + r : 0) * D + c, on);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto find_groups = [&](int t0, int* dst) {
    if (tid < BN) {
      int lo = 0, hi = t0 + tid < k_end ? a.Ck - 1 : 0;      // last group with koff[g] <= position
      while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (koff[mid] <= t0 + tid) lo = mid; else hi = mid - 1; }
      dst[tid] = lo;
    }
  };
#pragma unroll 4
  for (int e = tid; e < kProbeRows * CPR; e += kFThreads) {
    const int r = e / CPR, c = (e % CPR) * 4;
    const int pi = r < nrows ? pidx[r] : -1;
    cp16(Qs + r * S::ld + c, Qb + (i64)(pi >= 0 ? inv[pi] : 0) * D + c, pi >= 0);
  }
  load_keys(Kb, Ks, S::ld, k_begin);                         // with Q
  load_keys(Vb, Vs, D, k_begin);
  for (int e = tid; e < kProbeRows * words; e += kFThreads) bitmap[e] = 0u;
  for (int e = tid; e < a.Ck; e += kFThreads) koff[e] = kvoff[e];
  __syncthreads();
  if ((tid >> 2) < nrows) {                                  // 4 threads per probe row
    const int r = tid >> 2, pi = pidx[r];
    if (pi >= 0) {
      const int g = a.q_assign[(i64)bh * a.N + pi];
      const int* rp = a.route_ptr + (i64)bh * (a.Cq + 1);
      const int* ri = a.route_idx + (i64)bh * a.Cq * a.Ck;
      for (int t = rp[g] + (tid & 3); t < rp[g + 1]; t += 4) atomicOr(&bitmap[r * words + (ri[t] >> 5)], 1u << (ri[t] & 31));
    }
  }
  find_groups(k_begin, kgrp);

  float2 oc[R][OP], oo[R][OP];                               // current state of every row, the other one
  float mS[R], lS[R], mU[R], lU[R];
  unsigned cur = 0;                                          // bit i: the retained state of row i is the current one
#pragma unroll
  for (int i = 0; i < R; ++i) {
    mS[i] = mU[i] = -INFINITY; lS[i] = lU[i] = 0.f;
#pragma unroll
    for (int c = 0; c < OP; ++c) oc[i][c] = oo[i][c] = make_float2(0.f, 0.f);
  }
  auto turn = [&](unsigned want) {                           // make the states `want` the current ones
    const unsigned sw = want ^ cur;
    cur = want;
    if (sw == 0) return;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int c = 0; c < OP; ++c) {
        const float2 x = oc[i][c], y = oo[i][c];
        const bool b = (sw >> i) & 1u;
        oc[i][c] = b ? y : x; oo[i][c] = b ? x : y;
      }
  };
  const unsigned* bm = bitmap + ty * R * words;
  const float sc = a.scale * kLog2e;
  int phase = 0;
  for (int t0 = k_begin; t0 < k_end; t0 += BN, phase ^= 1) {
    const int ncols = min(BN, k_end - t0);
    const int* kg = kgrp + phase * BN;
    asm volatile("cp.async.wait_group 1;" ::: "memory");     // Q and K
    __syncthreads();
    float s[R][4];
    {
      float2 acc[R][4];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
      const float* qp = Qs + ty * R * S::ld;
      const float* kp = Ks + tx * S::ld;
#pragma unroll 2
      for (int k = 0; k < D; k += 4) {
        float4 kk[4], q[R];
#pragma unroll
        for (int j = 0; j < 4; ++j) kk[j] = *reinterpret_cast<const float4*>(kp + 16 * j * S::ld + k);
#pragma unroll
        for (int i = 0; i < R; ++i) q[i] = *reinterpret_cast<const float4*>(qp + i * S::ld + k);
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = __ffma2_rn(make_float2(q[i].x, q[i].y), make_float2(kk[j].x, kk[j].y), acc[i][j]);
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = __ffma2_rn(make_float2(q[i].z, q[i].w), make_float2(kk[j].z, kk[j].w), acc[i][j]);
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = tx + 16 * j < ncols ? (acc[i][j].x + acc[i][j].y) * sc : -INFINITY;
    }
    __syncthreads();                                         // K is consumed
    load_keys(Kb, Ks, S::ld, t0 + BN);
    if (t0 + BN < k_end) find_groups(t0 + BN, kgrp + (phase ^ 1) * BN);
    int grp[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) grp[j] = kg[tx + 16 * j];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      bool ret[4];
      float mxS = -INFINITY, mxU = -INFINITY;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        ret[j] = (bm[i * words + (grp[j] >> 5)] >> (grp[j] & 31)) & 1u;
        if (ret[j]) mxS = fmaxf(mxS, s[i][j]); else mxU = fmaxf(mxU, s[i][j]);
      }
      mxS = row16_max(mxS); mxU = row16_max(mxU);
      const float nS = fmaxf(mS[i], mxS), nU = fmaxf(mU[i], mxU);
      const float cS = nS == -INFINITY ? 1.f : exp2f(mS[i] - nS), cU = nU == -INFINITY ? 1.f : exp2f(mU[i] - nU);
      mS[i] = nS; mU[i] = nU;
      float sS = 0.f, sU = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float e = s[i][j] > -INFINITY ? exp2f(s[i][j] - (ret[j] ? nS : nU)) : 0.f;   // no weight past the last key
        s[i][j] = e;
        sS += ret[j] ? e : 0.f; sU += ret[j] ? 0.f : e;
      }
      lS[i] = lS[i] * cS + sS; lU[i] = lU[i] * cU + sU;
      const bool is_s = (cur >> i) & 1u;
      const float cc = is_s ? cS : cU, co = is_s ? cU : cS;
      if (cc != 1.f || co != 1.f) {
#pragma unroll
        for (int c = 0; c < OP; ++c) { oc[i][c].x *= cc; oc[i][c].y *= cc; oo[i][c].x *= co; oo[i][c].y *= co; }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<float4*>(Ps + (tx + 16 * j) * S::ldp + ty * R) = make_float4(s[0][j], s[1][j], s[2][j], s[3][j]);
    asm volatile("cp.async.wait_group 1;" ::: "memory");     // V
    __syncthreads();
    for (int j0 = 0; j0 < ncols;) {                          // the keys of one K/V group after the other
      const int g = kg[j0];
      const int j1 = g + 1 < a.Ck ? min(ncols, koff[g + 1] - t0) : ncols;
      unsigned want = 0;
#pragma unroll
      for (int i = 0; i < R; ++i) want |= ((bm[i * words + (g >> 5)] >> (g & 31)) & 1u) << i;
      turn(want);
#pragma unroll 4
      for (int j = j0; j < j1; ++j) {
        const float4 p = *reinterpret_cast<const float4*>(Ps + j * S::ldp + ty * R);
        const float pv[R] = {p.x, p.y, p.z, p.w};
#pragma unroll
        for (int c = 0; c < OP / 2; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(Vs + j * D + 64 * c + 4 * tx);
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const float2 pp = make_float2(pv[i], pv[i]);
            oc[i][2 * c] = __ffma2_rn(pp, make_float2(v.x, v.y), oc[i][2 * c]);
            oc[i][2 * c + 1] = __ffma2_rn(pp, make_float2(v.z, v.w), oc[i][2 * c + 1]);
          }
        }
      }
      j0 = j1;
    }
    __syncthreads();                                         // V and the probabilities are consumed
    load_keys(Vb, Vs, D, t0 + BN);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");         // (a slice without keys has only fetched Q)
  turn((1u << R) - 1);
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = ty * R + i;
    const float tS = row16_sum(lS[i]), tU = row16_sum(lU[i]);
    if (r >= nrows) continue;
    float* out = a.partial + ((((i64)bh * a.n_split + blockIdx.x) * a.M + m0 + r) * 2) * (D + 2);
    if (tx == 0) { out[0] = mS[i]; out[1] = tS; out[D + 2] = mU[i]; out[D + 3] = tU; }
#pragma unroll
    for (int c = 0; c < OP; ++c) {                           // (rows of the partial states are 8-byte aligned)
      const int col = 64 * (c >> 1) + 4 * tx + 2 * (c & 1);
      *reinterpret_cast<float2*>(out + 2 + col) = oc[i][c];
      *reinterpret_cast<float2*>(out + D + 4 + col) = oo[i][c];
    }
  }
}

// merge the split states; one warp per probe row.  Bound by latency: the maxima are found by the lanes side by side, and the
// numerators of four slices are on their way at a time (on the two calls above 13 us with 16 slices -> 12 with 32, and 56 -> 32 us;
// eight at a time: 9 and 31 us, but 20 -> 26 us at 4 slices of 32 heads).
template <int D>
__global__ void __launch_bounds__(256) k_probe_merge(const float* __restrict__ partial, int n_split, int M,
                                                     float* __restrict__ X, float* __restrict__ Dn) {
  const int bh = blockIdx.y;
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (r >= M) return;
  const int lane = threadIdx.x & 31;
  constexpr int PL = D / 32;
  const float* p0 = partial + ((i64)bh * n_split * M + r) * 2 * (D + 2);   // of split 0
  const i64 step = (i64)M * 2 * (D + 2);
  float mS = -INFINITY, mU = -INFINITY;
  for (int s = lane; s < n_split; s += 32) { mS = fmaxf(mS, p0[s * step]); mU = fmaxf(mU, p0[s * step + D + 2]); }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { mS = fmaxf(mS, __shfl_xor_sync(0xffffffffu, mS, o)); mU = fmaxf(mU, __shfl_xor_sync(0xffffffffu, mU, o)); }
  float lS = 0.f, lU = 0.f, nS[PL], nU[PL];
#pragma unroll
  for (int c = 0; c < PL; ++c) nS[c] = nU[c] = 0.f;
  // a state without any key (empty key slice, or no retained / omitted key inside it) has weight 0 and its numerator may never
  // have been written: it is fetched with the others (kAhead splits at a time) but left out, not multiplied by 0
  constexpr int kAhead = 4;
  for (int s0 = 0; s0 < n_split; s0 += kAhead) {
    float xS[kAhead][PL], xU[kAhead][PL];
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const float* p = p0 + min(s0 + k, n_split - 1) * step;
#pragma unroll
      for (int c = 0; c < PL; ++c) { xS[k][c] = p[2 + lane + 32 * c]; xU[k][c] = p[D + 4 + lane + 32 * c]; }
    }
    float w = 0.f, z = 0.f;                                  // lane k, 16 + k: weight and sum of state S, U of split s0 + k
    if ((lane & 15) < kAhead && s0 + (lane & 15) < n_split) {
      const float* p = p0 + (s0 + (lane & 15)) * step + (lane < 16 ? 0 : D + 2);
      w = p[0] == -INFINITY ? 0.f : exp2f(p[0] - (lane < 16 ? mS : mU));
      z = p[1];
    }
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const float wS = __shfl_sync(0xffffffffu, w, k), wU = __shfl_sync(0xffffffffu, w, 16 + k);
      const float zS = __shfl_sync(0xffffffffu, z, k), zU = __shfl_sync(0xffffffffu, z, 16 + k);
      if (wS != 0.f) {
        lS = fmaf(zS, wS, lS);
#pragma unroll
        for (int c = 0; c < PL; ++c) nS[c] = fmaf(xS[k][c], wS, nS[c]);
      }
      if (wU != 0.f) {
        lU = fmaf(zU, wU, lU);
#pragma unroll
        for (int c = 0; c < PL; ++c) nU[c] = fmaf(xU[k][c], wU, nU[c]);
      }
    }
  }
  const float mD = fmaxf(mS, mU);
  const float eS = mS == -INFINITY ? 0.f : exp2f(mS - mD), eU = mU == -INFINITY ? 0.f : exp2f(mU - mD);
  const float zD = lS * eS + lU * eU;
#pragma unroll
  for (int c = 0; c < PL; ++c) {
    X[((i64)bh * M + r) * D + lane + 32 * c] = lS > 0.f ? nS[c] / lS : 0.f;
    Dn[((i64)bh * M + r) * D + lane + 32 * c] = zD > 0.f ? (nS[c] * eS + nU[c] * eU) / zD : 0.f;
  }
}

size_t probe_partial_floats(int BH, int n_split, int M, int d) { return (size_t)BH * n_split * M * 2 * (d + 2); }

template <int D>
static void probe_dispatch(const ProbeArgs& a, cudaStream_t st) {
  dim3 grid(a.n_split, (a.M + kProbeRows - 1) / kProbeRows, a.BH);
  k_probe_rows<D><<<grid, kFThreads, ProbeSmem<D>::bytes(a.Ck), st>>>(a);
  dim3 g2((a.M + 7) / 8, a.BH);
  k_probe_merge<D><<<g2, 256, 0, st>>>(a.partial, a.n_split, a.M, a.X, a.Dn);
}
void launch_probe_merge(const ProbeArgs& a, cudaStream_t st) {
  dim3 g2((a.M + 7) / 8, a.BH);
  if (a.d == 128) k_probe_merge<128><<<g2, 256, 0, st>>>(a.partial, a.n_split, a.M, a.X, a.Dn);
  else k_probe_merge<64><<<g2, 256, 0, st>>>(a.partial, a.n_split, a.M, a.X, a.Dn);
}
void launch_probe_rows(const ProbeArgs& a, cudaStream_t st) {
  if (a.d == 128) probe_dispatch<128>(a, st); else probe_dispatch<64>(a, st);
}

// O[b,h,probe_idx[m],:] = O_dense of the probe (Eq. 10, first case)
template <typename T>
__global__ void k_write_probe_rows(const float* __restrict__ Dn, const int* __restrict__ probe_idx, int H, int M, int d,
                                   T* __restrict__ O, i64 ob, i64 oh, i64 on) {
  const int bh = blockIdx.y, b = bh / H, h = bh % H;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < M * d; e += gridDim.x * blockDim.x) {
    const int m = e / d, c = e % d;
    const int pi = probe_idx[(i64)bh * M + m];
    if (pi >= 0) O[b * ob + h * oh + (i64)pi * on + c] = from_f32<T>(Dn[((i64)bh * M + m) * d + c]);
  }
}
void launch_write_probe_rows(int dtype, const float* Dn, const int* probe_idx, int BH, int H, int M, int d, void* O,
                             const i64* os, cudaStream_t st) {
  dim3 grid((M * d + 255) / 256, BH);
  if (dtype == SPARSEPR_BF16) k_write_probe_rows<__nv_bfloat16><<<grid, 256, 0, st>>>(Dn, probe_idx, H, M, d, (__nv_bfloat16*)O, os[0], os[1], os[2]);
  else k_write_probe_rows<float><<<grid, 256, 0, st>>>(Dn, probe_idx, H, M, d, (float*)O, os[0], os[1], os[2]);
}

cudaError_t init_attention_simt() {
  cudaError_t e;
#define SPR_ATTR(KERN, BYTES) if ((e = cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(BYTES))) != cudaSuccess) return e
  SPR_ATTR(k_attention_f32_sparse<128>, F32Smem<128>::bytes);
  SPR_ATTR(k_attention_f32_dense<128>, F32Smem<128>::bytes);
  SPR_ATTR(k_attention_f32_sparse<64>, F32Smem<64>::bytes);
  SPR_ATTR(k_attention_f32_dense<64>, F32Smem<64>::bytes);
  SPR_ATTR(k_probe_rows<128>, ProbeSmem<128>::bytes(kMaxGroups));
  SPR_ATTR(k_probe_rows<64>, ProbeSmem<64>::bytes(kMaxGroups));
#undef SPR_ATTR
  return cudaSuccess;
}

}  // namespace spr
