// k-means assignment (Section 4.1) with the score contraction on the tensor cores.
//
// score(x, c) = ||mu_c||^2 - 2 x.mu_c.  The whole score comes out of tcgen05.mma: both operands are split into two bf16
// words (x = xh + xl, -2 mu = mh + ml; the products xh.mh, xh.ml, xl.mh are accumulated in fp32 in TMEM, the dropped term is
// ~2^-16 relative), and one more k-step multiplies a constant row (1, 1, 1, 0, ...) with the three bf16 words of ||mu_c||^2
// (which holds all of its float32 bits).  Each row keeps its best and second-best score; a row whose gap is not larger than
// a conservative bound on the score error is NOT decided here but handed to the exact recheck (per-head row lists; float64
// with the operation order of the definition for every centroid that a float32 filter cannot rule out), so the final
// assignment always equals the exact float64 decision with ties to the lowest id.
//
// Persistent CTAs: each owns row tiles (128 rows) of one head; centroid chunks of 128 stream through shared memory
// (resident when C <= 256, and then four row tiles are in flight instead of two; the last chunk's product is as wide as
// its centroids).  Roles: warps 0-15 are two epilogue groups of eight warps on alternate row tiles, each with two score
// buffers of 128 columns that its chunks use in turn, warp 16 TMA producer, warps 17 and 18 MMA issuers, one per group.  In a group, warps w and
// w + 4 share the 32 rows of a TMEM quadrant and take one half of the chunk's columns each; their results meet at a named
// barrier.  With one buffer of 256 columns per group a product had to wait for the whole scan of the group's tile before,
// and scan and product ran one after the other (3100 cycles per tile against 1664 of product); now the product of a
// chunk runs while the group scans the chunk before, decides and moves rows.
// The scan needs the best score, the gap to the second best and the index of the best.  A running best / second / index
// costs five minimum, compare and select instructions per score on the half-rate ALU pipe.  Instead every score enters two
// minima, each a three-input minimum over two new scores (one instruction per score together): that of its column class
// c mod 16 (16 running minima in registers) and that of its group of 16 columns (whose running best / second / index cost
// five instructions per 16 scores).  Class and group identify a column, so the best is in the best class and the best
// group, and any other score lies in another class or in another group:
//   second best = min(second best of the class minima, second best of the group minima), exactly.
//
// Centroid sums are exact integers (fixed point, one rounding per row and column), so they are updated instead of being
// formed anew in every pass: a row that changes its group is subtracted from the old one and added to the new one.  After
// the first passes few rows move, and a pass then reads the two bf16 words of the features only.
// Measured at 24 heads of 32760 rows and 256 centroids: a pass in which no row moves 62 us (the products alone need 37, the
// two words of the features 31), the passes of one run 62 to 168 us, 1.38 ms for 16 passes where the kernel that kept best,
// second and index per score and formed the sums anew took 2.11 ms; 40 heads of 75600 rows, 591 centroids: 540 us per
// pass (958).  The early passes, in which a third of the rows move, are bound by the atomics of the sums.
#include <mutex>
#include "kmeans_sums.cuh"
#include "tc_common.cuh"

namespace spr {
namespace tc {

constexpr int kKmEpiWarps = 16;
constexpr int kKmThreads = (kKmEpiWarps + 3) * 32;   // + TMA producer, two MMA issuers
constexpr int kKmChunk = kKmChunkCols;                // centroids per MMA (N)
constexpr uint32_t kXBytes = 128 * 128;               // one [128 rows x 64 bf16] block
constexpr uint32_t kMuBytes = kKmChunk * 128;         // one [128 x 64 bf16] block
constexpr uint32_t kMwBytes = kKmChunk * 16;          // [128 x 8 bf16]: the words of ||mu_c||^2
constexpr uint32_t kMuStage = 2 * kMuBytes + kMwBytes;

// Tiles: either 4 row stages and 2 centroid stages (resident) or 2 and 4; a row stage is (hi, lo) of 128 rows, a centroid
// stage (hi, lo) and the norm words of 128 centroids.
struct KmSmem {
  static constexpr uint32_t x = 0;
  static constexpr uint32_t tiles = 2 * 2 * kXBytes + 4 * kMuStage;
  static constexpr uint32_t ones = tiles;                       // [128 x 16 bf16], unswizzled: the constant rows
  static constexpr uint32_t xchg = ones + 4096;                 // best, second, index: 3 x [2 groups][2 parities][2 halves][128]
  static constexpr uint32_t bars = xchg + 3 * 8 * 128 * 4;
  static constexpr uint32_t misc = bars + 32 * 8;
  static constexpr uint32_t total = misc + 32;
};
static_assert(4 * 2 * kXBytes + 2 * kMuStage <= KmSmem::tiles, "both stage layouts fit into the tile area");
constexpr size_t kKmSmemBytes = KmSmem::total + 1024;
static_assert(kKmSmemBytes + 256 <= 227 * 1024, "shared memory");
enum KmBar { X_FULL = 0, X_EMPTY = 4, MU_FULL = 8, MU_EMPTY = 12, ACC_FULL = 16, ACC_EMPTY = 20, KM_BARS = 24 };   // 4 each

struct KmParams {
  int N, C, r, R, n_chunks, ctas_per_head;
  const float* phi; int ldphi;          // fp32 features (for the centroid sums)
  const float* xnorm;                   // [BH][N]
  const float* mu2;                     // [BH][C]
  const __nv_bfloat16* mw;              // [BH][C padded to 128][8] words of ||mu_c||^2
  int* assign;
  const int* old;                       // [BH][N] or null: the groups whose sums `sums` holds (may be `assign`; ids outside [0, C) are in no sum)
  i64* sums; int* counts; const int* fx_shift;   // sums to be updated, or null
  int* flagged; int* flag_count;        // rows left to the exact recheck: [BH][N] row indices, [BH] their number
  int* flag_count_next;                 // [BH] or null: the counters of the next pass, zeroed here
  int* err;
  const int* prev_changed; int* cur_changed;   // [BH] or null: rows whose assignment changed in the previous / this pass
};

// one row's move between two groups, by one warp: lane = columns 2 lane and 2 lane + 1 of the row (x0, x1).  (With columns
// lane and lane + 32, whose atomics fall into half as many sectors per instruction, a pass in which most rows move takes
// twice as long.)
__device__ __forceinline__ void km_move(i64* sums, int* counts, int C, int R, int r, float scl, float2 x, int from, int to, int lane) {
  // scl = 2^shift: scaling a float32 value by a power of two is exact, so the integer is the one a float64 product gives
  const i64 v0 = __float2ll_rn(x.x * scl), v1 = __float2ll_rn(x.y * scl);
  const int c0 = 2 * lane;
  if (c0 < r) {
    atomicAdd(reinterpret_cast<u64*>(sums + (i64)to * R + c0), (u64)v0);
    if (c0 + 1 < r) atomicAdd(reinterpret_cast<u64*>(sums + (i64)to * R + c0 + 1), (u64)v1);
  }
  if (lane == 0) atomicAdd(counts + to, 1);
  if (from >= 0 && from < C) {
    if (c0 < r) {
      atomicAdd(reinterpret_cast<u64*>(sums + (i64)from * R + c0), (u64)(-v0));
      if (c0 + 1 < r) atomicAdd(reinterpret_cast<u64*>(sums + (i64)from * R + c0 + 1), (u64)(-v1));
    }
    if (lane == 0) atomicAdd(counts + from, -1);
  }
}

__device__ __forceinline__ float min3(float a, float b, float c) {
  float y;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
__device__ __forceinline__ float min16(const float* s) {
  const float a = min3(s[0], s[1], s[2]), b = min3(s[3], s[4], s[5]), c = min3(s[6], s[7], s[8]), d = min3(s[9], s[10], s[11]);
  const float e = min3(s[12], s[13], s[14]);
  return fminf(min3(a, b, s[15]), min3(c, d, e));
}

// the scores of a row tile and a chunk: ||mu||^2 + x_h mu_h + x_h mu_l + x_l mu_h; one k-step = 16 columns = 32 bytes = 2 address units
__device__ __forceinline__ void km_product(uint32_t d, uint64_t one_desc, uint64_t wd, uint64_t xh, uint64_t mh, int ksteps, uint32_t idesc) {
  const uint64_t xl = xh + (uint64_t)(kXBytes >> 4), ml = mh + (uint64_t)(kMuBytes >> 4);
  umma_bf16(d, one_desc, wd, idesc, 0);
#pragma unroll
  for (int kk = 0; kk < 4; ++kk)
    if (kk < ksteps) {
      umma_bf16(d, xh + 2 * kk, mh + 2 * kk, idesc, 1);
      umma_bf16(d, xh + 2 * kk, ml + 2 * kk, idesc, 1);
      umma_bf16(d, xl + 2 * kk, mh + 2 * kk, idesc, 1);
    }
}
// The scan of a row's scores by one thread of each half of the columns
struct KmScan {
  float cls[16];                                               // minima over the column classes c mod 16
  float gb = kKmFar, gs = kKmFar;                              // best and second best of the minima of 16 columns
  int gi = 0;                                                  // index of the best (c / 16)
  __device__ __forceinline__ KmScan() {
#pragma unroll
    for (int j = 0; j < 16; ++j) cls[j] = kKmFar;
  }
  __device__ __forceinline__ void group(float cm, int g) {
    gs = fminf(gs, fmaxf(cm, gb));
    gi = cm < gb ? g : gi;
    gb = fminf(gb, cm);
  }
  // the scores of the centroids from c0 on in this warp's lanes of tensor memory; hh: which half of the columns is this warp's
  __device__ __forceinline__ void chunk(uint32_t acc_addr, int c0, int C, int hh) {
    const int ng = (min(kKmChunk, C - c0) + 15) >> 4;          // groups of 16 columns that hold centroids
    const int ns = (ng + 1) >> 1, s_mid = (ns + 1) >> 1;       // 32-column steps; this warp's half of them
    const int s1 = hh ? ns : s_mid;
#pragma unroll 1
    for (int st = hh ? s_mid : 0; st < s1; ++st) {
      float t[32];
      tmem_ld32(acc_addr + st * 32, t);
      group(min16(t), (c0 >> 4) + 2 * st);
      if (2 * st + 1 < ng) {                                   // uniform (the product wrote no columns beyond ng groups)
        group(min16(t + 16), (c0 >> 4) + 2 * st + 1);
#pragma unroll
        for (int j = 0; j < 16; ++j) cls[j] = min3(cls[j], t[j], t[16 + j]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) cls[j] = fminf(cls[j], t[j]);
      }
    }
  }
  // best and second best score of the half and the centroid of the best: second best of the class minima (tournament) and the class of the best
  __device__ __forceinline__ void result(float& best, float& second, int& bi) const {
    float tb[8], ts[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { tb[j] = fminf(cls[2 * j], cls[2 * j + 1]); ts[j] = fmaxf(cls[2 * j], cls[2 * j + 1]); }
#pragma unroll
    for (int w = 4; w > 0; w >>= 1)
#pragma unroll
      for (int j = 0; j < w; ++j) {
        const float hi = fmaxf(tb[j], tb[j + w]);
        ts[j] = min3(hi, ts[j], ts[j + w]);
        tb[j] = fminf(tb[j], tb[j + w]);
      }
    int cj = 0;
#pragma unroll
    for (int j = 1; j < 16; ++j) cj = cls[j] == tb[0] ? j : cj;
    best = tb[0]; second = fminf(ts[0], gs);
    bi = gi * 16 + cj;
  }
};
// The results of the two halves of the columns meet: xc = this row's place of the first half, 128 floats per half, second best and index 1024
// and 2048 floats behind
__device__ __forceinline__ void km_exchange(float* xc, int hh, int barrier, float& best, float& second, int& bi) {
  xc[hh * 128] = best; xc[1024 + hh * 128] = second; reinterpret_cast<int*>(xc)[2048 + hh * 128] = bi;
  asm volatile("bar.sync %0, 64;" ::"r"(barrier) : "memory");
  const float ob = xc[(hh ^ 1) * 128], os = xc[1024 + (hh ^ 1) * 128];
  const int oi = reinterpret_cast<const int*>(xc)[2048 + (hh ^ 1) * 128];
  second = min3(fmaxf(best, ob), second, os);
  bi = ob < best ? oi : bi;
  best = fminf(best, ob);
}
// Bound on |computed score - true score|.  A bf16 rounding is off by at most 2^-8 relative, so the words of x and
// of 2 mu leave 2^-16 each and the dropped product xl.ml another 2^-16 of 2 |x| |mu|: 9.2e-5 in all.  Accumulation
// in fp32: 13 steps that add 17 terms, the largest at most 2 |x| |mu| + |mu|^2.  How the unit aligns them is not documented;
// a sum delivered in float32 keeps at least that format's places below the largest term, so each term is allowed to lose 2^-23
// of it: 2.7e-5.  (Measured with words at their worst, cancelling terms and terms just below the last place of a large one:
// at most 7e-7 of it, and 0.07 of E in all.)
__device__ __forceinline__ float km_score_error(float xn, float mm) { return 1.5e-4f * xn * mm + 2.7e-5f * mm * mm; }
// The rows of a warp's 32 that changed their group (bits of todo; phi: the first of the 32), four at a time: the latency of their features is the cost
__device__ __forceinline__ void km_moves(unsigned todo, const float* phi, int ldphi, i64* sums, int* counts, int C, int R, int r, float scl,
                                         int old_a, int bi, int lane) {
  while (todo) {
    int rr[4];
    float2 x2[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      rr[u] = todo ? __ffs(todo) - 1 : -1;
      todo &= todo - 1;
      x2[u] = make_float2(0.f, 0.f);
      if (rr[u] >= 0 && 2 * lane < r)                          // (ldphi is a multiple of 16 and columns r..ldphi-1 hold zeros)
        x2[u] = *reinterpret_cast<const float2*>(phi + (i64)rr[u] * ldphi + 2 * lane);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (rr[u] >= 0)
        km_move(sums, counts, C, R, r, scl, x2[u], __shfl_sync(0xffffffffu, old_a, rr[u]), __shfl_sync(0xffffffffu, bi, rr[u]), lane);
  }
}

__global__ void __launch_bounds__(kKmThreads, 1)
k_kmeans_assign_tc(const __grid_constant__ CUtensorMap mapXh, const __grid_constant__ CUtensorMap mapXl,
                   const __grid_constant__ CUtensorMap mapMh, const __grid_constant__ CUtensorMap mapMl, KmParams prm) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  volatile int* misc = reinterpret_cast<volatile int*>(sm + KmSmem::misc);   // [0] tmem base, [1] abort
  const uint32_t bars = base + KmSmem::bars;
  auto bar = [&](int i) { return bars + 8u * i; };
  constexpr unsigned FULLW = 0xffffffffu;
  const int tid = threadIdx.x, warp = __shfl_sync(FULLW, tid >> 5, 0), lane = tid & 31;   // (uniform, and known to be)
  const int bh = blockIdx.y, cta = blockIdx.x;

  __shared__ int s_skip;
  __shared__ float s_red[34];
  // set-up that needs nothing from the kernels before
  if (tid == 0) {
    for (int i = 0; i < KM_BARS; ++i) mbar_init(bar(i), i >= ACC_EMPTY ? 8 : (i >= MU_EMPTY && i < MU_EMPTY + 4) ? 2 : 1);
    misc[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kKmEpiWarps + 1) tmem_alloc(base + KmSmem::misc, 512);
  // the constant rows in 8 x 16-byte core matrices: row group g, k half h at g * 256 + h * 128; columns 0-2 are one
  if (tid < 256) {
    const uint32_t one2 = 0x3F803F80u;
    const bool first = (tid & 8) == 0;                      // 8 rows of 16 bytes per core matrix
    *reinterpret_cast<uint4*>(sm + KmSmem::ones + tid * 16) = first ? make_uint4(one2, 0x3F80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
  }
  fence_async_smem();
  pdl_wait();                                               // the centroids of this pass come from the kernel before
  pdl_launch_dependents();
  if (cta == 0 && tid == 0 && prm.flag_count_next) prm.flag_count_next[bh] = 0;   // last read by the recheck two kernels back
  float mu2max = 0.f;
  for (int c = tid; c < prm.C; c += kKmThreads) mu2max = fmaxf(mu2max, prm.mu2[(i64)bh * prm.C + c]);
  // a head whose previous pass changed no assignment has reached the fixed point of the iteration: skipped
  if (tid == 0) s_skip = (prm.err != nullptr && *reinterpret_cast<volatile int*>(prm.err) == SPARSEPR_ERR_TIMEOUT) ||
                         (prm.prev_changed != nullptr && prm.prev_changed[bh] == 0);
  tc_fence_before();
  // largest centroid norm of the head, rounded up: it enters the bound on the score error only
  const float mm = sqrtf(block_max(mu2max, s_red)) * 1.000001f;
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = (uint32_t)misc[0];
  volatile int* abort_flag = &misc[1];

  const int row_tiles = (prm.N + 127) / 128;
  // contiguous chunk of row tiles per CTA: CTAs that run at the same time then work on distant
  // tokens, i.e. on different clusters, and do not contend for the same centroid sums
  const int per_cta = (row_tiles + prm.ctas_per_head - 1) / prm.ctas_per_head;
  const int tile0 = cta * per_cta;
  const int my_tiles = __any_sync(0xffffffffu, s_skip) ? 0 : max(0, min(per_cta, row_tiles - tile0));
  const int n_chunks = prm.n_chunks;
  const int n_pairs = (my_tiles + 1) / 2;
  const bool resident = n_chunks <= 2;
  const int xst = resident ? 4 : 2;                         // row stages
  const int xlog = resident ? 2 : 1;
  const uint32_t mu_base = base + (uint32_t)xst * 2 * kXBytes;

  if (warp == kKmEpiWarps) {
    // =========================== TMA producer ============================================
    if (lane == 0) {
      // Step order: the row tiles are taken in pairs, and inside a pair the centroid chunks are interleaved (tile 0
      // chunk 0, tile 1 chunk 0, tile 0 chunk 1, ...), so that both tiles use the chunk that a centroid stage holds.
      // Tile t of a pair belongs to epilogue group t, and the group's k-th chunk to its buffer k mod 2: the waits on a
      // buffer's barriers follow its phases in order.  v counts the chunks loaded.
      const __nv_bfloat16* mw = prm.mw + (i64)bh * n_chunks * kKmChunk * 8;
      int v = 0;
      bool go = true;
      for (int pair = 0; pair < n_pairs && go; ++pair) {
        const int nt = min(2, my_tiles - 2 * pair);
        for (int ch = 0; ch < n_chunks && go; ++ch) {
          if (!resident || pair == 0) {
            const int ms = v & 3;
            if (!mbar_wait(bar(MU_EMPTY + ms), ((v >> 2) & 1) ^ 1, abort_flag)) { go = false; break; }
            const uint32_t dst = mu_base + ms * kMuStage;
            mbar_expect_tx(bar(MU_FULL + ms), kMuStage);
            tma_load_4d(dst, &mapMh, bar(MU_FULL + ms), 0, ch * kKmChunk, bh, 0);
            tma_load_4d(dst + kMuBytes, &mapMl, bar(MU_FULL + ms), 0, ch * kKmChunk, bh, 0);
            bulk_load(dst + 2 * kMuBytes, mw + (i64)ch * kKmChunk * 8, kMwBytes, bar(MU_FULL + ms));
            ++v;
          }
          for (int t = 0; ch == 0 && t < nt; ++t) {
            const int tl = 2 * pair + t, xs = tl & (xst - 1);
            if (!mbar_wait(bar(X_EMPTY + xs), ((tl >> xlog) & 1) ^ 1, abort_flag)) { go = false; break; }
            const int row0 = (tile0 + tl) * 128;
            mbar_expect_tx(bar(X_FULL + xs), 2 * kXBytes);
            tma_load_4d(base + KmSmem::x + xs * 2 * kXBytes, &mapXh, bar(X_FULL + xs), 0, row0, bh, 0);
            tma_load_4d(base + KmSmem::x + xs * 2 * kXBytes + kXBytes, &mapXl, bar(X_FULL + xs), 0, row0, bh, 0);
          }
        }
      }
    }
  } else if (warp > kKmEpiWarps) {
    // =========================== MMA issuers (one per group) ================================
    {
      // The whole warp walks the steps and one elected lane issues; loop control goes through votes so that it is known to
      // be uniform and descriptors stay in uniform registers.  A step costs its issuer about 500 cycles of barriers and
      // commits besides 31 per product: with one issuer for both groups the tensor pipe idled a third of the time.
      // Descriptors are built once (only their 16-byte address field moves) and the k-steps are unrolled.
      const int t = warp - (kKmEpiWarps + 1);
      const int ksteps = prm.R / 16;
      // the last chunk's product covers its centroids only (a multiple of 16 columns)
      const int n_last = min(kKmChunk, (prm.C - (n_chunks - 1) * kKmChunk + 15) & ~15);
      const uint32_t idesc_full = idesc_bf16(0, kKmChunk), idesc_last = idesc_bf16(0, n_last);
      const uint64_t x_desc0 = smem_desc(base + KmSmem::x, 16), m_desc0 = smem_desc(mu_base, 16);
      // unswizzled operands of the norm step.  A: k halves 128 bytes apart, row groups 256; B: one core matrix per 8
      // centroids, 128 bytes apart; its second k half is multiplied by zeros and reads the first one again (stride 0)
      const uint64_t one_desc = smem_desc_plain(base + KmSmem::ones, 128, 256);
      const uint64_t w_desc0 = smem_desc_plain(mu_base + 2 * kMuBytes, 0, 128);
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
      int k = 0;                                               // chunks so far
      bool go = true;
      for (int pair = 0; pair < n_pairs && go; ++pair) {
        const int tl = 2 * pair + t, xs = tl & (xst - 1);
        const bool have = tl < my_tiles;
        for (int ch = 0; ch < n_chunks; ++ch, ++k) {
          const int ms = resident ? ch : (k & 3), ab = 2 * t + (k & 1);
          if (!resident || pair == 0) go = __all_sync(FULLW, mbar_wait(bar(MU_FULL + ms), resident ? 0 : ((k >> 2) & 1), abort_flag));
          if (have && ch == 0) go = __all_sync(FULLW, go && mbar_wait(bar(X_FULL + xs), (tl >> xlog) & 1, abort_flag));
          if (have) go = __all_sync(FULLW, go && mbar_wait(bar(ACC_EMPTY + ab), ((k >> 1) & 1) ^ 1, abort_flag));
          if (!go) break;
          tc_fence_after();
          const uint32_t d = tm + (uint32_t)ab * kKmChunk;
          const uint32_t idesc = ch == n_chunks - 1 ? idesc_last : idesc_full;
          const uint64_t moff = (uint64_t)((ms * kMuStage) >> 4);
          const uint64_t mh = m_desc0 + moff, wd = w_desc0 + moff;
          const uint64_t xh = x_desc0 + (uint64_t)((xs * 2 * kXBytes) >> 4);
          if (elect_one()) {
            if (have) {
              km_product(d, one_desc, wd, xh, mh, ksteps, idesc);
              umma_commit(bar(ACC_FULL + ab));
              if (ch == n_chunks - 1) umma_commit(bar(X_EMPTY + xs));
              if (!resident) umma_commit(bar(MU_EMPTY + ms));
            } else if (!resident) {
              mbar_arrive(bar(MU_EMPTY + ms));                 // the last pair has one tile
            }
          }
          __syncwarp();
        }
      }
    }
  } else {
    // =========================== epilogue: argmin, sums =====================================
    const uint32_t FULL = 0xffffffffu;
    const int grp = warp >> 3, hh = (warp >> 2) & 1, wq = warp & 3;
    const uint32_t acc_addr0 = tmem + ((uint32_t)(wq * 32) << 16) + (uint32_t)grp * (2 * kKmChunk);
    float* xb = reinterpret_cast<float*>(sm + KmSmem::xchg);    // best; second 1024 on; index 2048 on
    const float scl = prm.sums ? __int_as_float((127 + prm.fx_shift[bh]) << 23) : 0.f;
    bool ok = true;
    for (int tl = grp, k = 0; tl < my_tiles; tl += 2) {
      const int rowbase = (tile0 + tl) * 128 + wq * 32, row = rowbase + lane;
      const i64 gr = (i64)bh * prm.N + row;
      const bool mine = row < prm.N && (lane >> 4) == hh;      // the two warps of a quadrant finish 16 of its rows each
      const float xn = mine ? prm.xnorm[gr] : 0.f;             // needed after the scores: fetched now
      const int old_a = (prm.old != nullptr && mine) ? prm.old[gr] : -1;
      KmScan scan;
      for (int ch = 0; ch < n_chunks; ++ch, ++k) {             // k: chunks of this group so far
        const int ab = 2 * grp + (k & 1);
        ok = __all_sync(FULL, ok && mbar_wait(bar(ACC_FULL + ab), (k >> 1) & 1, abort_flag));
        if (ok) {
          tc_fence_after();
          const uint32_t acc_addr = acc_addr0 + (uint32_t)(k & 1) * kKmChunk;
          scan.chunk(acc_addr, ch * kKmChunk, prm.C, hh);
          tc_fence_before();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(ACC_EMPTY + ab));
      }
      float best, second;
      int bi;
      scan.result(best, second, bi);
      km_exchange(xb + ((grp * 2 + ((tl >> 1) & 1)) * 2) * 128 + wq * 32 + lane, hh, 1 + grp * 4 + wq, best, second, bi);
      bi = min(bi, prm.C - 1);                               // (only rows of non-finite scores could point past C)
      // decide, or hand the row to the exact recheck
      bool decided = false, moved = false;
      if (ok && mine) {
        const float E = km_score_error(xn, mm);
        decided = second - best > 2.f * E;
        if (decided) {
          moved = old_a != bi;
          if (moved || prm.old != prm.assign) prm.assign[gr] = bi;
        } else {                                             // the recheck writes (and compares) this row's assignment
          const int pos = atomicAdd(prm.flag_count + bh, 1);
          prm.flagged[(i64)bh * prm.N + pos] = row;
        }
      }
      if (prm.cur_changed != nullptr) {
        const int nmoved = __popc(__ballot_sync(FULL, decided && (moved || prm.prev_changed == nullptr)));
        if (lane == 0 && nmoved) atomicAdd(prm.cur_changed + bh, nmoved);
      }
      if (prm.sums) {
        km_moves(__ballot_sync(FULL, decided && moved), prm.phi + ((i64)bh * prm.N + rowbase) * prm.ldphi, prm.ldphi, prm.sums + (i64)bh * prm.C * prm.R,
                 prm.counts + (i64)bh * prm.C, prm.C, prm.R, prm.r, scl, old_a, bi, lane);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    for (int k = 0; k < 64; ++k) __nanosleep(1000);
    if (tid == 0) set_error(prm.err, SPARSEPR_ERR_TIMEOUT);
    __syncthreads();
  }
  if (warp == kKmEpiWarps + 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// Float32 distances of row x [R] to the centroids (rows LDM floats apart) into d32 [C rounded up to 32], by one warp: 32 kJ centroids at a time; returns the smallest
template <int kJ>
__device__ __forceinline__ float recheck_distances(const float* xs, const float* mu_s, int LDM, int C, int R, float* d32, int lane) {
  const int Cp = (C + 31) & ~31;
  float best32 = INFINITY;
  for (int c0 = 0; c0 < C; c0 += 32 * kJ) {
    // packed float32 arithmetic, two columns per instruction: (m - x)^2 summed in two partial sums per centroid
    float2 acc[kJ];
    const float* mrow[kJ];
#pragma unroll
    for (int j = 0; j < kJ; ++j) { acc[j] = make_float2(0.f, 0.f); mrow[j] = mu_s + (size_t)min(c0 + 32 * j + lane, C - 1) * LDM; }
#pragma unroll 2
    for (int k = 0; k < R; k += 4) {
      const float4 xv = *reinterpret_cast<const float4*>(xs + k);
      const float2 nx0 = make_float2(-xv.x, -xv.y), nx1 = make_float2(-xv.z, -xv.w);
#pragma unroll
      for (int j = 0; j < kJ; ++j) {
        const float4 mv = *reinterpret_cast<const float4*>(mrow[j] + k);
        const float2 d0 = __fadd2_rn(make_float2(mv.x, mv.y), nx0), d1 = __fadd2_rn(make_float2(mv.z, mv.w), nx1);
        acc[j] = __ffma2_rn(d0, d0, acc[j]);
        acc[j] = __ffma2_rn(d1, d1, acc[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < kJ; ++j) {
      const int c = c0 + 32 * j + lane;
      if (c < Cp) {
        const float d = c < C ? acc[j].x + acc[j].y : INFINITY;
        d32[c] = d;
        best32 = fminf(best32, d);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) best32 = fminf(best32, __shfl_xor_sync(0xffffffffu, best32, o));
  return best32;
}
// The exact decision for one row by one warp (see the kernel below); x, centroids and the warp's scratch d32 in shared memory
__device__ __forceinline__ int recheck_row(const float* xs, const float* mu_s, int LDM, int C, int R, float* d32, int lane) {
  const unsigned FULL = 0xffffffffu;
  const float best32 = C <= 64 ? recheck_distances<2>(xs, mu_s, LDM, C, R, d32, lane) : recheck_distances<8>(xs, mu_s, LDM, C, R, d32, lane);
  const float thr = best32 * (1.f + 4.f * (float)(R + 4) * 5.9604645e-8f) + 1e-30f;
  // candidates: normally one, and then the decision is made (the definition is a chain of float64 additions, about 9 cycles per term,
  // behind conversions)
  int ncand = 0, cand = -1;
  for (int c = lane; c < C; c += 32)                         // (never past C: with a NaN row thr is +inf, and so are the pad entries)
    if (d32[c] <= thr) { ++ncand; cand = c; }
  const int total_cand = __reduce_add_sync(FULL, ncand);
  int bi;
  if (total_cand == 1) {
    bi = __reduce_max_sync(FULL, cand);
  } else if (total_cand == 0) {
    bi = 0;                                                  // every distance is NaN (non-finite input, reported elsewhere): group 0
  } else {
    double best = 0.0;
    bi = -1;
    for (int c = lane; c < C; c += 32) {
      if (d32[c] <= thr) {
        const float* m = mu_s + (size_t)c * LDM;
        double dsum = 0.0;
#pragma unroll 8
        for (int k = 0; k < R; ++k) {
          const double diff = __dsub_rn((double)xs[k], (double)m[k]);
          dsum = __dadd_rn(dsum, __dmul_rn(diff, diff));
        }
        if (bi < 0 || dsum < best) { best = dsum; bi = c; }    // a lane meets its centroids in increasing order
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(FULL, best, o);
      const int oi = __shfl_xor_sync(FULL, bi, o);
      if (oi >= 0 && (bi < 0 || ob < best || (ob == best && oi < bi))) { best = ob; bi = oi; }
    }
  }
  return min(max(bi, 0), C - 1);
}

// Exact decision for the rows the fast path could not prove (a few thousand per pass at N = 32760 and 24 heads).
// The definition is the squared distance in float64 with the terms added in order of k (the zero padding of columns
// r..R-1 adds exact zeros), ties to the lowest id.  Every such row needs all C centroids of its head, so the rows of a
// head share them: grid (G, BH); a CTA brings the head's centroids to shared memory once and its eight warps take the
// head's flagged rows in turn.  Per row:
//   1. float32 distances to all centroids (lane = centroid, 8 at a time; rows of mu padded by 4 floats, so that the
//      16-byte reads of consecutive centroids fall into different banks).  Every term is non-negative, hence the
//      float32 value is within (R + 3) 2^-24 of the true distance, relatively;
//   2. only centroids within 4 (R + 4) 2^-24 of the float32 minimum (relative, plus a denormal's worth) can hold the
//      float64 minimum: those few (normally one or two) are evaluated by the definition, one lane each.
__global__ void __launch_bounds__(256) k_assign_recheck_staged(const int* __restrict__ flagged, const int* __restrict__ flag_count,
                                                               const float* __restrict__ phi, int ldphi, int N, int r, int R,
                                                               const float* __restrict__ mu, int C, int* __restrict__ assign,
                                                               i64* __restrict__ sums, int* __restrict__ counts,
                                                               const int* __restrict__ fx_shift, int* __restrict__ recheck_total,
                                                               const int* __restrict__ old, int count_all, int* __restrict__ cur_changed) {
  extern __shared__ __align__(16) float rs_smem[];
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bh = blockIdx.y;
  pdl_wait();                                                  // the row lists come from the assignment kernel before
  pdl_launch_dependents();
  const int n = flag_count[bh];
  if (blockIdx.x == 0 && bh == 0 && tid == 0 && recheck_total) {
    int total = 0;
    for (int h = 0; h < (int)gridDim.y; ++h) total += flag_count[h];
    *recheck_total = total;
  }
  if ((int)blockIdx.x * 8 >= n) return;                        // no row for this CTA
  const int LDM = R + 4, Cp = (C + 31) & ~31;
  float* mu_s = rs_smem;                                       // [C][R + 4]
  float* d32_all = mu_s + (size_t)C * LDM;                     // [8 warps][Cp]
  float* xs_all = d32_all + 8 * Cp;                            // [8 warps][R]
  {
    const float4* src = reinterpret_cast<const float4*>(mu + (i64)bh * C * R);
    const int q = R / 4;
    for (int e = tid; e < C * q; e += 256) {
      const int c = e / q, k4 = e - c * q;
      *reinterpret_cast<float4*>(mu_s + (size_t)c * LDM + 4 * k4) = src[e];
    }
  }
  __syncthreads();
  float* d32 = d32_all + warp * Cp;
  float* xs = xs_all + warp * R;
  for (int i = blockIdx.x * 8 + warp; i < n; i += gridDim.x * 8) {
    const int row = flagged[(i64)bh * N + i];
    const i64 gr = (i64)bh * N + row;
    const float* x = phi + gr * ldphi;
    __syncwarp();
    for (int k = lane; k < R; k += 32) xs[k] = x[k];
    __syncwarp();
    const int bi = recheck_row(xs, mu_s, LDM, C, R, d32, lane);
    const int old_a = old != nullptr ? old[gr] : -1;
    __syncwarp();                                              // everyone has read it (`old` may be `assign`)
    if (lane == 0) {
      if (cur_changed != nullptr && (count_all || old_a != bi)) atomicAdd(cur_changed + bh, 1);
      assign[gr] = bi;
    }
    if (sums && old_a != bi) {
      const float scl = __int_as_float((127 + fx_shift[bh]) << 23);
      km_move(sums + (i64)bh * C * R, counts + (i64)bh * C, C, R, r, scl, 2 * lane < R ? *reinterpret_cast<const float2*>(xs + 2 * lane) : make_float2(0.f, 0.f), old_a, bi, lane);
    }
  }
}
// shared memory of the kernel above
static size_t recheck_staged_smem(int C, int R) { return ((size_t)C * (R + 4) + 8 * (size_t)((C + 31) & ~31) + 8 * (size_t)R) * sizeof(float); }

// All passes of a k-means run in one kernel, for at most 256 centroids: a cluster of CTAs per head, each with a contiguous run of the head's row tiles.
// A pass of the kernels above is three dependent launches, 16 us at two heads of 4770 rows; here it is
//   centroids from the sums, by every CTA for itself, straight into the operands in shared memory
//   -> products, scan, decisions as above -> exact recheck of the CTA's own undecided rows -> sums -> barrier of the cluster.
// The sums stay in global memory (atomics, read past the first-level cache); a second barrier of the cluster keeps them from changing before everyone
// has read them.  (Centroids dealt out to the CTAs and handed round through the cluster's shared memory: stores to other CTAs move 8 bytes per cycle
// and SM, 2 to 5 k cycles a pass more than forming all of them.)  Up to four row tiles of at most 128 centroids stay in shared memory for all passes.
// What an SM sends to the sums is bound by its atomics (a row is 16 sectors of 32 bytes per sum), so the rows that move are listed, and where they are
// many they are sorted by group, so that a warp adds up rows of one group; in a first pass, all rows in windows of the list's length.
// Every thread of the cluster meets the same barriers whatever happens: an abort only skips the work in between, and the end of the iteration is read
// from a counter that all of them see behind a barrier.
// A pass at two heads of 4770 rows is 15 k cycles: centroids 3, products and decisions of three tiles 5.5, recheck of a row or two 3, barriers 3; its
// first pass 25.  Runs of eight passes, us, in separate launches and here: 2 heads of 4770 rows and 38 centroids 132, 72; 2 of 4096 float32 rows and 64
// centroids 143, 76; 8 of 7161 rows and 112 centroids 228, 176.
constexpr int kKmRunList = 2048;                     // moved rows of a pass that are listed (the others go to the sums at once)
constexpr int kKmRunSort = 48;                       // listed rows from which they are sorted
constexpr int kKmRunTiles = 64;                      // row tiles per CTA (a row has 14 bits in the list)
struct KmRunParams {
  int N, C, r, R, T, n_chunks, per_cta;
  const float* phi; int ldphi;
  const float* xnorm;
  const float* mu;
  int from_sums;
  const int* old;
  int* assign;
  i64* sums; int* counts; const int* fx_shift;
  int* flagged; int* recheck_total; int* err;
  int* changed; int ld_changed;
};
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// A moved row in the list: row (from the CTA's first), group before (511: none) and group now
constexpr int kKmNone = 511;
__device__ __forceinline__ unsigned km_entry(int row, int was, int is) { return (unsigned)row | (unsigned)was << 14 | (unsigned)is << 23; }
// The moves of a sorted list by one warp: elements lo .. hi - 1, the place of an entry and, in the top bit, whether its row leaves its old group or joins its new one
__device__ __forceinline__ void km_move_sorted(const unsigned* entries, const unsigned short* list, int lo, int hi, const float* phi, int ldphi,
                                               i64* sums, int* counts, int R, int r, float scl, int lane) {
  constexpr int kRows = 8;                                     // rows in flight
  const int c0 = 2 * lane;
  const float* at = phi + (c0 < r ? c0 : 0);                   // (without a condition on the loads, so that they go out together)
  i64 s0 = 0, s1 = 0;
  int group = -1, count = 0;
  const auto flush = [&] {
    if (group >= 0) {
      if (s0 != 0 && c0 < r) atomicAdd(reinterpret_cast<u64*>(sums + (i64)group * R + c0), (u64)s0);
      if (s1 != 0 && c0 + 1 < r) atomicAdd(reinterpret_cast<u64*>(sums + (i64)group * R + c0 + 1), (u64)s1);
      if (lane == 0 && count != 0) atomicAdd(counts + group, count);
    }
    s0 = s1 = 0; count = 0;
  };
  for (int i0 = lo; i0 < hi; i0 += kRows) {
    int g[kRows];                                              // group, leaving: - 1 - group
    float2 x[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const int l = list[min(i0 + u, hi - 1)];
      const unsigned e = entries[l & 0x7FFF];
      g[u] = l & 0x8000 ? -1 - (int)((e >> 14) & 511u) : (int)(e >> 23);
      x[u] = *reinterpret_cast<const float2*>(at + (i64)(e & 0x3FFFu) * ldphi);
    }
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      if (i0 + u >= hi) break;                                 // (uniform)
      const int sign = g[u] >> 31, gu = g[u] ^ sign;           // 0 or -1
      if (gu != group) { flush(); group = gu; }
      const float signed_scale = sign ? -scl : scl;            // (rounded as in km_move)
      s0 += __float2ll_rn(x[u].x * signed_scale);
      s1 += __float2ll_rn(x[u].y * signed_scale);
      count += 1 + 2 * sign;
    }
  }
  flush();
}

__global__ void __launch_bounds__(kKmThreads, 1)
k_kmeans_run(const __grid_constant__ CUtensorMap mapXh, const __grid_constant__ CUtensorMap mapXl, KmRunParams prm) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  volatile int* misc = reinterpret_cast<volatile int*>(sm + KmSmem::misc);   // [0] tmem base, [1] abort
  const uint32_t bars = base + KmSmem::bars;
  auto bar = [&](int i) { return bars + 8u * i; };
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int kWarps = kKmThreads / 32;
  const int tid = threadIdx.x, warp = __shfl_sync(FULL, tid >> 5, 0), lane = tid & 31;
  const int bh = blockIdx.y, cta = blockIdx.x, C = prm.C, R = prm.R, LDM = R + 4, n_chunks = prm.n_chunks;
  // four row stages and one chunk of centroids, or two and two: operands, then float32 values
  const int xst = n_chunks == 1 ? 4 : 2, xlog = n_chunks == 1 ? 2 : 1;
  const uint32_t mu_area = (uint32_t)xst * 2 * kXBytes, val_area = mu_area + (uint32_t)n_chunks * kMuStage;
  static_assert(2 * 2 * kXBytes + 4 * kMuStage <= KmSmem::tiles && 4 * 2 * kXBytes + 2 * kMuStage <= KmSmem::tiles && kKmChunk * (64 + 4) * 4 <= kMuStage, "layouts");
  static_assert(kKmRunList * 4 <= KmSmem::bars - KmSmem::xchg && kKmEpiWarps * (kKmChunk + 64) * 4 <= KmSmem::bars - KmSmem::xchg, "sorted list, recheck scratch");
  __shared__ unsigned s_list[kKmRunList];
  __shared__ float s_max[kWarps];
  __shared__ int s_start[2 * kKmChunk + 1];
  __shared__ int s_flagged, s_moved, s_left, s_skip;
  if (tid == 0) {
    for (int i = 0; i < KM_BARS; ++i) mbar_init(bar(i), i >= ACC_EMPTY ? 8 : 1);
    misc[1] = 0;
    s_flagged = 0; s_moved = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kKmEpiWarps + 1) tmem_alloc(base + KmSmem::misc, 512);
  if (tid < 256) {                                             // the constant rows (see k_kmeans_assign_tc)
    const uint32_t one2 = 0x3F803F80u;
    *reinterpret_cast<uint4*>(sm + KmSmem::ones + tid * 16) = (tid & 8) == 0 ? make_uint4(one2, 0x3F80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
  }
  // operands of the places beyond C: zeros, and a norm larger than any score
  for (uint32_t e = tid * 16; e < n_chunks * kMuStage; e += kKmThreads * 16)
    *reinterpret_cast<uint4*>(sm + mu_area + e) = e % kMuStage < 2 * kMuBytes ? make_uint4(0u, 0u, 0u, 0u) : norm_words(kKmFar);
  pdl_wait();                                                  // features, first centroids and sums come from the kernels before
  if (tid == 0) s_skip = prm.err != nullptr && *reinterpret_cast<volatile int*>(prm.err) == SPARSEPR_ERR_TIMEOUT;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = (uint32_t)misc[0];
  volatile int* abort_flag = &misc[1];
  const int row_tiles = (prm.N + 127) / 128, tile0 = cta * prm.per_cta;
  const int my_tiles = __any_sync(FULL, s_skip) ? 0 : max(0, min(prm.per_cta, row_tiles - tile0));
  const bool keep = my_tiles <= xst && n_chunks == 1;          // the row tiles stay in shared memory
  const int row0 = tile0 * 128, my_rows = max(0, min(my_tiles * 128, prm.N - row0));
  const i64 hrow0 = (i64)bh * prm.N + row0;                    // (rows count from the CTA's first below)
  const float* phi = prm.phi + hrow0 * prm.ldphi;
  int* assign = prm.assign + hrow0;
  int* flagged = prm.flagged + hrow0;
  const float scl = __int_as_float((127 + prm.fx_shift[bh]) << 23);
  const double inv_sc = ldexp(1.0, -prm.fx_shift[bh]);
  i64* sums = prm.sums + (i64)bh * C * R;
  int* counts = prm.counts + (i64)bh * C;
  float* values = reinterpret_cast<float*>(sm + val_area);
  int tiles = my_tiles;                                        // 0 once a wait has run out
  int kc = 0;                                                  // chunks of this warp's group so far (issuers and epilogue)
  for (int t = 1;; ++t) {
    // ---- centroids: words of -2 mu, words of the norm, float32 values
    const bool from_sums = t > 1 || prm.from_sums;
    float mx = 0.f;
    constexpr int kB = 4;                                      // centroids of a warp in flight
    for (int c0 = warp; c0 < C; c0 += kB * kWarps) {
      const int k = 2 * lane;
      int cnt[kB];
      longlong2 sv[kB];
      float2 v[kB];
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int c = c0 + b * kWarps;
        cnt[b] = 0;
        v[b] = make_float2(0.f, 0.f);
        sv[b] = make_longlong2(0, 0);
        if (c < C && k < R) {                                  // (columns r to R - 1 hold zeros)
          if (from_sums) { cnt[b] = __ldcg(counts + c); sv[b] = __ldcg(reinterpret_cast<const longlong2*>(sums + (i64)c * R + k)); }
          v[b] = t > 1 ? *reinterpret_cast<const float2*>(values + c * LDM + k) : *reinterpret_cast<const float2*>(prm.mu + ((i64)bh * C + c) * R + k);
        }
      }
#pragma unroll
      for (int b = 0; b < kB; ++b) {                           // (no branches: the chains of the four run side by side)
        const GroupMean mean(max(cnt[b], 1), inv_sc);
        const float mx0 = mean(sv[b].x), mx1 = mean(sv[b].y);
        v[b].x = cnt[b] > 0 ? mx0 : v[b].x; v[b].y = cnt[b] > 0 ? mx1 : v[b].y;
      }
      const float n2 = norms_of_four(v, lane);                 // of centroid lane / 8 of the four
      mx = fmaxf(mx, n2);
      if ((lane & 7) == 0 && c0 + lane / 8 * kWarps < C) {
        const int c = c0 + lane / 8 * kWarps;
        *reinterpret_cast<uint4*>(sm + mu_area + (c / kKmChunk) * kMuStage + 2 * kMuBytes + c % kKmChunk * 16) = norm_words(n2);
      }
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int c = c0 + b * kWarps;
        if (c >= C) break;                                     // (uniform)
        if (k < R) *reinterpret_cast<float2*>(values + c * LDM + k) = v[b];
        const uint32_t hi = pack_bf16x2(-2.f * v[b].x, -2.f * v[b].y), lo = pack_bf16x2_rest(-2.f * v[b].x, -2.f * v[b].y, hi);
        unsigned char* st = sm + mu_area + (c / kKmChunk) * kMuStage;
        const int cc = c % kKmChunk, off = cc * 128 + (((k >> 3) ^ (cc & 7)) << 4) + (k & 7) * 2;      // rows of 128 bytes, 128-byte swizzle
        *reinterpret_cast<uint32_t*>(st + off) = hi;
        *reinterpret_cast<uint32_t*>(st + kMuBytes + off) = lo;
      }
    }
    mx = warp_max(mx);
    if (lane == 0) s_max[warp] = mx;
    fence_async_smem();                                        // the tensor cores read the operands
    __syncthreads();
    // Every warp has read the sums; they may change once all CTAs have.  One warp's release carries the reads of all, which lie before the barrier
    // above: that of the producer, which has nothing to load in most passes.  The others wait for the cluster when their first product is under way
    // or read: in front of the moves, and of the prefetches for the recheck (waiting empties the first-level cache).  Runs of keys and queries, us, so,
    // with the wait behind all products, and with a release and the wait in front of them: 2 heads of 4770 rows 72 and 78, 73 and 80, 73 and 80; 8 of
    // 7161 float32 rows 168 and 184, 171 and 186, 173 and 190; 16 of 17550 rows, d = 64, 344 and 363, 344 and 364, 352 and 375.
    if (warp == kKmEpiWarps) cluster_arrive(); else cluster_arrive_relaxed();
    bool may_move = false;                                     // this warp has waited for the cluster
    const auto wait_for_cluster = [&] {
      __syncwarp();
      if (!may_move) cluster_wait();                           // (uniform)
      may_move = true;
    };
    float mm = s_max[0];                                       // largest centroid norm of the head, rounded up
#pragma unroll
    for (int w = 1; w < kWarps; ++w) mm = fmaxf(mm, s_max[w]);
    mm = sqrtf(mm) * 1.000001f;
    const bool upd = t < prm.T;                                // the last pass needs no sums
    const int* old = t > 1 ? assign : prm.old != nullptr ? prm.old + hrow0 : nullptr;
    const bool first = old == nullptr;                         // no row is in a group yet: the sums are formed from all rows behind the pass
    const int loads = keep ? 0 : (t - 1) * my_tiles;           // row tiles loaded in the passes before
    if (warp == kKmEpiWarps) {
      // =========================== TMA producer ============================================
      if (lane == 0 && (!keep || t == 1)) {
        for (int tl = 0; tl < tiles; ++tl) {
          const int n = loads + tl, xs = n & (xst - 1);
          if (!mbar_wait(bar(X_EMPTY + xs), ((n >> xlog) & 1) ^ 1, abort_flag)) break;
          mbar_expect_tx(bar(X_FULL + xs), 2 * kXBytes);
          tma_load_4d(base + KmSmem::x + xs * 2 * kXBytes, &mapXh, bar(X_FULL + xs), 0, row0 + tl * 128, bh, 0);
          tma_load_4d(base + KmSmem::x + xs * 2 * kXBytes + kXBytes, &mapXl, bar(X_FULL + xs), 0, row0 + tl * 128, bh, 0);
        }
      }
      wait_for_cluster();
    } else if (warp > kKmEpiWarps) {
      // =========================== MMA issuers (one per group) ================================
      const int g = warp - (kKmEpiWarps + 1), ksteps = R / 16;
      const int n_last = min(kKmChunk, (C - (n_chunks - 1) * kKmChunk + 15) & ~15);
      const uint32_t idesc_full = idesc_bf16(0, kKmChunk), idesc_last = idesc_bf16(0, n_last);
      const uint64_t x_desc0 = smem_desc(base + KmSmem::x, 16), m_desc0 = smem_desc(base + mu_area, 16);
      const uint64_t one_desc = smem_desc_plain(base + KmSmem::ones, 128, 256), w_desc0 = smem_desc_plain(base + mu_area + 2 * kMuBytes, 0, 128);
      const uint32_t tm = __shfl_sync(FULL, tmem, 0);
      bool go = true;
      for (int tl = g; tl < tiles && go; tl += 2) {
        const int n = loads + tl, xs = n & (xst - 1);
        if (!keep || t == 1) go = __all_sync(FULL, mbar_wait(bar(X_FULL + xs), (n >> xlog) & 1, abort_flag));
        for (int ch = 0; ch < n_chunks; ++ch, ++kc) {
          const int ab = 2 * g + (kc & 1);
          go = __all_sync(FULL, go && mbar_wait(bar(ACC_EMPTY + ab), ((kc >> 1) & 1) ^ 1, abort_flag));
          if (!go) break;
          tc_fence_after();
          const bool last = ch == n_chunks - 1;
          const uint64_t moff = (uint64_t)((ch * kMuStage) >> 4);
          if (elect_one()) {
            km_product(tm + (uint32_t)ab * kKmChunk, one_desc, w_desc0 + moff, x_desc0 + (uint64_t)((xs * 2 * kXBytes) >> 4), m_desc0 + moff, ksteps,
                       last ? idesc_last : idesc_full);
            umma_commit(bar(ACC_FULL + ab));
            if (last && !keep) umma_commit(bar(X_EMPTY + xs));
          }
          __syncwarp();
        }
        wait_for_cluster();
      }
    } else {
      // =========================== epilogue: argmin ===========================================
      const int grp = warp >> 3, hh = (warp >> 2) & 1, wq = warp & 3;
      const uint32_t acc_addr0 = tmem + ((uint32_t)(wq * 32) << 16) + (uint32_t)grp * (2 * kKmChunk);
      float* xb = reinterpret_cast<float*>(sm + KmSmem::xchg);
      int n_changed = 0;
      bool ok = true;
      // a row's norm and group are fetched a tile ahead; the two warps of a quadrant finish 16 of its rows each
      const auto is_mine = [&](int tl) { return tl < tiles && tl * 128 + wq * 32 + lane < my_rows && (lane >> 4) == hh; };
      const auto norm_of = [&](int tl) { return is_mine(tl) ? prm.xnorm[hrow0 + tl * 128 + wq * 32 + lane] : 0.f; };
      const auto group_of = [&](int tl) { return !first && is_mine(tl) ? old[tl * 128 + wq * 32 + lane] : -1; };
      float xn_next = norm_of(grp);
      int old_next = group_of(grp);
      for (int tl = grp; tl < tiles; tl += 2) {
        const int rowbase = tl * 128 + wq * 32, row = rowbase + lane;
        const bool mine = is_mine(tl);
        const float xn = xn_next;
        const int was = old_next >= 0 && old_next < C ? old_next : kKmNone;
        xn_next = norm_of(tl + 2);
        old_next = group_of(tl + 2);
        KmScan scan;
        for (int ch = 0; ch < n_chunks; ++ch, ++kc) {
          const int ab = 2 * grp + (kc & 1);
          ok = __all_sync(FULL, ok && mbar_wait(bar(ACC_FULL + ab), (kc >> 1) & 1, abort_flag));
          if (ok) {
            tc_fence_after();
            scan.chunk(acc_addr0 + (uint32_t)(kc & 1) * kKmChunk, ch * kKmChunk, C, hh);
            tc_fence_before();
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(ACC_EMPTY + ab));
        }
        float best, second;
        int bi;
        wait_for_cluster();
        scan.result(best, second, bi);
        km_exchange(xb + ((grp * 2 + ((tl >> 1) & 1)) * 2) * 128 + wq * 32 + lane, hh, 1 + grp * 4 + wq, best, second, bi);
        bi = min(bi, C - 1);                                   // (only rows of non-finite scores could point past C)
        const bool decided = ok && mine && second - best > 2.f * km_score_error(xn, mm), moved = decided && was != bi;
        if (decided) {
          if (moved || t == 1) assign[row] = bi;
        } else if (ok && mine) {                               // the recheck decides this row
          flagged[atomicAdd(&s_flagged, 1)] = row;
          asm volatile("prefetch.global.L1 [%0];" ::"l"(phi + (i64)row * prm.ldphi));
          asm volatile("prefetch.global.L1 [%0];" ::"l"(phi + (i64)row * prm.ldphi + prm.ldphi - 16));
        }
        n_changed += __popc(__ballot_sync(FULL, t == 1 ? decided : moved));
        const unsigned mask = __ballot_sync(FULL, moved);
        if (mask && upd && !first) {
          int at = 0;
          if (lane == 0) at = atomicAdd(&s_moved, __popc(mask));
          at = __shfl_sync(FULL, at, 0) + __popc(mask & ((1u << lane) - 1));
          if (moved && at < kKmRunList) s_list[at] = km_entry(row, was, bi);
          const unsigned over = __ballot_sync(FULL, moved && at >= kKmRunList);
          if (over) km_moves(over, phi + (i64)rowbase * prm.ldphi, prm.ldphi, sums, counts, C, R, prm.r, scl, was, bi, lane);
        }
      }
      if (lane == 0 && n_changed) atomicAdd(prm.changed + (i64)t * prm.ld_changed + bh, n_changed);
    }
    __syncthreads();
    if (*abort_flag) tiles = 0;                                // (the same for all threads: nobody waits now)
    wait_for_cluster();
    const int n_flagged = tiles ? s_flagged : 0, n_moved = tiles ? min(s_moved, kKmRunList) : 0;
    const bool sorted = n_moved > kKmRunSort;
    // ---- exact decisions for the rows that are left, by the epilogue warps; moves row by row, the last warps first
    if (warp < kKmEpiWarps && n_flagged > 0) {
      // scratch of a warp: behind the row stages' use (more than 128 centroids, whose tiles are not kept), else where the halves of the columns meet
      const int Cp = (C + 31) & ~31;
      float *d32 = reinterpret_cast<float*>(sm + (n_chunks == 1 ? KmSmem::xchg : KmSmem::x)) + warp * (Cp + R), *xs = d32 + Cp;
      for (int i = warp; i < n_flagged; i += kKmEpiWarps) {
        const int row = flagged[i], o = first ? -1 : old[row], was = o >= 0 && o < C ? o : kKmNone;
        __syncwarp();
        for (int k = lane; k < R; k += 32) xs[k] = phi[(i64)row * prm.ldphi + k];
        __syncwarp();                                          // (everyone has read the old group, which may lie in `assign`)
        const int bi = recheck_row(xs, values, LDM, C, R, d32, lane);
        if (lane == 0) {
          assign[row] = bi;
          if (t == 1 || was != bi) atomicAdd(prm.changed + (i64)t * prm.ld_changed + bh, 1);
        }
        if (upd && !first && was != bi)
          km_move(sums, counts, C, R, prm.r, scl, 2 * lane < R ? *reinterpret_cast<const float2*>(xs + 2 * lane) : make_float2(0.f, 0.f), was == kKmNone ? -1 : was, bi, lane);
      }
    }
    if (t == prm.T) {
      if (tid == 0 && prm.recheck_total != nullptr && n_flagged) atomicAdd(prm.recheck_total, n_flagged);
      break;
    }
    if (!first && !sorted) {
      for (int i = kWarps - 1 - warp; i < n_moved; i += kWarps) {
        const unsigned e = s_list[i];
        const int row = e & 0x3FFFu, was = (e >> 14) & 511u;
        const float2 x = 2 * lane < prm.r ? *reinterpret_cast<const float2*>(phi + (i64)row * prm.ldphi + 2 * lane) : make_float2(0.f, 0.f);
        km_move(sums, counts, C, R, prm.r, scl, x, was == kKmNone ? -1 : was, e >> 23, lane);
      }
    } else {
      __syncthreads();                                         // the recheck's groups and scratch
      unsigned short* list = reinterpret_cast<unsigned short*>(sm + KmSmem::xchg);           // sorted: up to two elements per entry
      const int in_pass = first ? (tiles ? my_rows : 0) : n_moved;
      for (int w0 = 0; w0 < in_pass; w0 += kKmRunList) {       // (one round where rows have moved)
        const int n = min(kKmRunList, in_pass - w0);
        for (int g = tid; g <= C; g += kKmThreads) s_start[g] = 0;
        if (first) for (int i = tid; i < n; i += kKmThreads) s_list[i] = km_entry(w0 + i, kKmNone, assign[w0 + i]);
        __syncthreads();
        for (int i = tid; i < n; i += kKmThreads) {
          const unsigned e = s_list[i];
          atomicAdd(s_start + (e >> 23), 1);
          if (((e >> 14) & 511u) != kKmNone) atomicAdd(s_start + ((e >> 14) & 511u), 1);
        }
        __syncthreads();
        if (warp == 0) {                                       // exclusive prefix sums over up to 256 groups, total behind them
          int c[8], sum = 0;
#pragma unroll
          for (int u = 0; u < 8; ++u) { c[u] = 8 * lane + u < C ? s_start[8 * lane + u] : 0; sum += c[u]; }
          int inc = sum;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) { const int up = __shfl_up_sync(FULL, inc, o); if (lane >= o) inc += up; }
          int at = inc - sum;
#pragma unroll
          for (int u = 0; u < 8; ++u) { if (8 * lane + u < C) s_start[8 * lane + u] = at; at += c[u]; }
          if (lane == 31) s_start[C] = inc;
        }
        __syncthreads();
        for (int i = tid; i < n; i += kKmThreads) {
          const unsigned e = s_list[i];
          list[atomicAdd(s_start + (e >> 23), 1)] = (unsigned short)i;
          if (((e >> 14) & 511u) != kKmNone) list[atomicAdd(s_start + ((e >> 14) & 511u), 1)] = (unsigned short)(i | 0x8000);
        }
        __syncthreads();
        const int total = s_start[C];
        km_move_sorted(s_list, list, total * warp / kWarps, total * (warp + 1) / kWarps, phi, prm.ldphi, sums, counts, R, prm.r, scl, lane);
        if (w0 + kKmRunList < in_pass) __syncthreads();        // the list is filled again
      }
    }
    // a pass that changes nothing has reached the fixed point of the iteration
    __syncwarp();
    cluster_arrive();
    cluster_wait();                                            // the sums and the counter of this pass are complete
    if (tid == 0) { s_left = __ldcg(prm.changed + (i64)t * prm.ld_changed + bh); s_flagged = 0; s_moved = 0; }
    fence_async_smem();                                        // (scratch in the row stages, which are filled again)
    __syncthreads();
    if (s_left == 0) break;                                    // (the same for the whole cluster)
  }
  pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    for (int k = 0; k < 64; ++k) __nanosleep(1000);
    if (tid == 0) set_error(prm.err, SPARSEPR_ERR_TIMEOUT);
    __syncthreads();
  }
  if (warp == kKmEpiWarps + 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// The same decision without staging, for centroid tables that do not fit into shared memory: grid (X, BH), one CTA per
// row, one thread per centroid, float64 throughout.
__global__ void __launch_bounds__(256) k_assign_recheck(const int* __restrict__ flagged, const int* __restrict__ flag_count,
                                                        const float* __restrict__ phi, int ldphi, int N, int r, int R,
                                                        const float* __restrict__ mu, int C, int* __restrict__ assign,
                                                        i64* __restrict__ sums, int* __restrict__ counts,
                                                        const int* __restrict__ fx_shift, int* __restrict__ recheck_total,
                                                        const int* __restrict__ old, int count_all, int* __restrict__ cur_changed) {
  __shared__ double s_best[8];
  __shared__ int s_bi[8];
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bh = blockIdx.y;
  const int n = flag_count[bh];
  if (blockIdx.x == 0 && bh == 0 && tid == 0 && recheck_total) {
    int total = 0;
    for (int h = 0; h < (int)gridDim.y; ++h) total += flag_count[h];
    *recheck_total = total;
  }
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const i64 gr = (i64)bh * N + flagged[(i64)bh * N + i];
    const float4* x4 = reinterpret_cast<const float4*>(phi + gr * ldphi);
    const float* muh = mu + (i64)bh * C * R;
    double best = 0.0;
    int bi = -1;
    for (int c = tid; c < C; c += 256) {
      const float4* m4 = reinterpret_cast<const float4*>(muh + (i64)c * R);
      double dsum = 0.0;
      for (int k4 = 0; k4 < R / 4; k4 += 4) {               // R is a multiple of 16: four vector loads in flight
        float4 xv[4], mv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { xv[u] = x4[k4 + u]; mv[u] = m4[k4 + u]; }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float xs[4] = {xv[u].x, xv[u].y, xv[u].z, xv[u].w}, ms[4] = {mv[u].x, mv[u].y, mv[u].z, mv[u].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const double diff = __dsub_rn((double)xs[e], (double)ms[e]);
            dsum = __dadd_rn(dsum, __dmul_rn(diff, diff));
          }
        }
      }
      if (bi < 0 || dsum < best) { best = dsum; bi = c; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(FULL, best, o);
      const int oi = __shfl_xor_sync(FULL, bi, o);
      if (oi >= 0 && (bi < 0 || ob < best || (ob == best && oi < bi))) { best = ob; bi = oi; }
    }
    if (lane == 0) { s_best[warp] = best; s_bi[warp] = bi; }
    __syncthreads();
    best = s_best[0]; bi = s_bi[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) {
      const double ob = s_best[w];
      const int oi = s_bi[w];
      if (oi >= 0 && (bi < 0 || ob < best || (ob == best && oi < bi))) { best = ob; bi = oi; }
    }
    const int old_a = old != nullptr ? old[gr] : -1;
    __syncthreads();                                           // everyone has read it (`old` may be `assign`)
    if (tid == 0) {
      if (cur_changed != nullptr && (count_all || old_a != bi)) atomicAdd(cur_changed + bh, 1);
      assign[gr] = bi;
    }
    if (sums && old_a != bi && warp == 0) {
      const float* x = phi + gr * ldphi;
      const float scl = __int_as_float((127 + fx_shift[bh]) << 23);
      km_move(sums + (i64)bh * C * R, counts + (i64)bh * C, C, R, r, scl, 2 * lane < R ? *reinterpret_cast<const float2*>(x + 2 * lane) : make_float2(0.f, 0.f), old_a, bi, lane);
    }
    __syncthreads();
  }
}

// phi fp32 [rows][ld] -> hi/lo bf16 [rows][64] (zero padded) and the row norms
__global__ void __launch_bounds__(256) k_split_bf16(const float* __restrict__ x, int ld, i64 rows, int r,
                                                    __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                                    float* __restrict__ norm) {
  pdl_wait();                                                   // the features come from the kernels before
  pdl_launch_dependents();
  const i64 t = (i64)blockIdx.x * 256 + threadIdx.x;
  const i64 row = t >> 3;
  const int c0 = (int)(t & 7) * 8;
  if (row >= rows) return;
  float v[8], h[8], l[8];
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    v[k] = c0 + k < r ? x[row * ld + c0 + k] : 0.f;
    const __nv_bfloat16 hb = __float2bfloat16_rn(v[k]);
    h[k] = __bfloat162float(hb);
    l[k] = v[k] - h[k];
    ss = fmaf(v[k], v[k], ss);
  }
  store8(hi + row * 64 + c0, h);
  store8(lo + row * 64 + c0, l);
  if (norm) {
    ss += __shfl_xor_sync(0xffffffffu, ss, 1);
    ss += __shfl_xor_sync(0xffffffffu, ss, 2);
    ss += __shfl_xor_sync(0xffffffffu, ss, 4);
    if ((t & 7) == 0) norm[row] = sqrtf(ss) * 1.000001f;
  }
}

}  // namespace tc

constexpr size_t kRecheckSmemMax = 200 * 1024;
cudaError_t init_kmeans_tc() {
  cudaError_t e = cudaFuncSetAttribute(tc::k_assign_recheck_staged, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRecheckSmemMax);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(tc::k_kmeans_assign_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::kKmSmemBytes);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(tc::k_kmeans_run, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::kKmSmemBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(tc::k_kmeans_run, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}
bool kmeans_tc_supported() { return tc::tma_available(); }

void launch_split_bf16(const float* x, int ld, i64 rows, int r, __nv_bfloat16* hi, __nv_bfloat16* lo, float* norm,
                       cudaStream_t st) {
  launch_pdl(tc::k_split_bf16, dim3((unsigned)((rows * 8 + 255) / 256)), dim3(256), 0, st, x, ld, rows, r, hi, lo, norm);
}

// Clusters of s CTAs that run side by side on the current device (0: none), s = 1 .. 16
static const int* run_clusters() {
  static int table[64][17];
  static std::once_flag once[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { static const int none[17] = {}; return none; }
  std::call_once(once[dev], [dev] {
    for (int s = 1; s <= 16; ++s) {
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(s, 1); cfg.blockDim = dim3(tc::kKmThreads); cfg.dynamicSmemBytes = tc::kKmSmemBytes;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = s; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cfg.attrs = at; cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, tc::k_kmeans_run, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
      table[dev][s] = n;
    }
  });
  return table[dev];
}
// CTAs per head for a run in one kernel, 0 where separate passes are faster.  One head's CTAs form a cluster, and all clusters have to be on the GPU at
// once: the largest that BH heads leave room for.  Of clusters of an odd number of CTAs the last ones that should fit often do not (they share pairs of
// SMs with others: 25 and 26 clusters of 5 where 26 are promised, 42 to 45 of 3 where 45 are), hence the margin there.
// A pass in one kernel saves 8 us and 0.45 us per head, measured; clusters leave SMs idle, and a row tile more per CTA than the separate launches
// have costs 0.9 us for its rows and as much for 256 centroids; the line below is drawn a little to the safe side of that.  Plans in one kernel / separately, us: 2 heads of 4096 rows
// (32 centroids) 582 / 707, 16 of 17408 (136) 1523 / 1622, 33 of 16384 (128) 1956 / 2372; on the other side 1 of 32768 (256) 1308 / 1025, 16 of 32768
// 2655 / 2514, 24 of 32768 3242 / 3263.
int kmeans_run_ctas(int BH, int N, int C, int r) {
  if (C > 2 * tc::kKmChunk || r > kMaxRank || !kmeans_tc_supported()) return 0;
  const int row_tiles = (N + 127) / 128, *fit = run_clusters();
  int s = 0;
  for (int k = 1; k <= 16 && k <= row_tiles; ++k) if (fit[k] - (k & 1 ? fit[k] / 11 : 0) >= BH) s = k;
  if (s == 0) return 0;
  const int per = (row_tiles + s - 1) / s, alone = (int)(((i64)row_tiles * BH + sm_count() - 1) / sm_count());
  if (per > tc::kKmRunTiles || (per - alone) * (256 + C) > 2000 + 110 * BH) return 0;
  return (row_tiles + per - 1) / per;
}
bool launch_kmeans_run(const KmeansRunArgs& a, cudaStream_t st) {
  using namespace tc;
  CUtensorMap mxh, mxl;
  if (!make_map(&mxh, a.xh, 64, a.N, a.BH, 1, 0, (i64)a.N * 64, 64, 128) || !make_map(&mxl, a.xl, 64, a.N, a.BH, 1, 0, (i64)a.N * 64, 64, 128)) return false;
  const int s = kmeans_run_ctas(a.BH, a.N, a.C, a.r), row_tiles = (a.N + 127) / 128;
  KmRunParams p{};
  p.N = a.N; p.C = a.C; p.r = a.r; p.R = a.R; p.T = a.T; p.n_chunks = (a.C + kKmChunk - 1) / kKmChunk; p.per_cta = (row_tiles + s - 1) / s;
  p.phi = a.phi; p.ldphi = a.ldphi; p.xnorm = a.xnorm; p.mu = a.mu; p.from_sums = a.from_sums; p.old = a.old; p.assign = a.assign;
  p.sums = a.sums; p.counts = a.counts; p.fx_shift = a.fx_shift; p.flagged = a.flagged; p.recheck_total = a.recheck_total; p.err = a.err;
  p.changed = a.changed; p.ld_changed = a.ld_changed;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(s, a.BH); cfg.blockDim = dim3(kKmThreads); cfg.dynamicSmemBytes = kKmSmemBytes; cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = s; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_kmeans_run, mxh, mxl, p) == cudaSuccess;
}

// One assignment pass.  xh/xl: bf16 [BH][N][64]; mh/ml: bf16 [BH][C][64]; sums may be null (no update wanted), else they
// hold the sums over the groups `old`, which may be `assign` itself.
bool launch_kmeans_assign_tc(const KmeansTcArgs& a, cudaStream_t st) {
  using namespace tc;
  CUtensorMap mxh, mxl, mmh, mml;
  if (!make_map(&mxh, a.xh, 64, a.N, a.BH, 1, 0, (i64)a.N * 64, 64, 128) || !make_map(&mxl, a.xl, 64, a.N, a.BH, 1, 0, (i64)a.N * 64, 64, 128) ||
      !make_map(&mmh, a.mh, 64, a.C, a.BH, 1, 0, (i64)a.C * 64, 64, kKmChunk) || !make_map(&mml, a.ml, 64, a.C, a.BH, 1, 0, (i64)a.C * 64, 64, kKmChunk))
    return false;
  KmParams p{};
  p.N = a.N; p.C = a.C; p.r = a.r; p.R = a.R; p.n_chunks = (a.C + kKmChunk - 1) / kKmChunk;
  const int row_tiles = (a.N + 127) / 128;
  // CTAs per head: one CTA fills an SM and works through its row tiles one after the other, so the launch takes
  // (rounds of CTAs over the SMs) x (tiles per CTA, plus about three tiles' worth of set-up).  With heads x CTAs below
  // the SM count a single round can leave many SMs idle (40 heads x 3 CTAs on 148 SMs); several rounds of shorter
  // CTAs are then faster, as long as a chunk keeps 24 tiles or more so that the set-up remains small.
  {
    const int sms = sm_count();
    int best_k = 1;
    long best_cost = -1;
    for (int k = 1; k <= row_tiles; ++k) {
      const int per = (row_tiles + k - 1) / k;
      if ((long)k * a.BH > sms && per < 24) break;          // several rounds only with chunks of 24 tiles or more
      const long rounds = ((long)k * a.BH + sms - 1) / sms;
      const long cost = rounds * (per + 3);
      if (best_cost < 0 || cost < best_cost) { best_cost = cost; best_k = k; }
    }
    p.ctas_per_head = best_k;
  }
  p.phi = a.phi; p.ldphi = a.ldphi; p.xnorm = a.xnorm; p.mu2 = a.mu2; p.assign = a.assign;
  p.sums = a.sums; p.counts = a.counts; p.fx_shift = a.fx_shift; p.flagged = a.flagged; p.flag_count = a.flag_count; p.err = a.err;
  p.old = a.old; p.mw = a.mw; p.prev_changed = a.prev_changed; p.cur_changed = a.cur_changed; p.flag_count_next = a.flag_count_next;
  // the three kernels of a pass (assignment, exact recheck, new centroids) follow each other with programmatic
  // dependent launches: 48 short dependent launches per k-means run otherwise pay their launch latency one by one
  launch_pdl(k_kmeans_assign_tc, dim3(p.ctas_per_head, a.BH), dim3(kKmThreads), kKmSmemBytes, st, mxh, mxl, mmh, mml, p);
  const size_t rs = recheck_staged_smem(a.C, a.R);
  const int per_head = std::max(1, 2 * sm_count() / a.BH);
  if (rs <= kRecheckSmemMax)
    launch_pdl(k_assign_recheck_staged, dim3(per_head, a.BH), dim3(256), rs, st, a.flagged, a.flag_count, a.phi, a.ldphi, a.N, a.r, a.R, a.mu, a.C,
               a.assign, a.sums, a.counts, a.fx_shift, a.recheck_total, a.old, (int)(a.prev_changed == nullptr), a.cur_changed);
  else
    k_assign_recheck<<<dim3(std::max(1, 4 * sm_count() / a.BH), a.BH), 256, 0, st>>>(a.flagged, a.flag_count, a.phi, a.ldphi, a.N, a.r, a.R, a.mu, a.C,
                                                                                     a.assign, a.sums, a.counts, a.fx_shift, a.recheck_total,
                                                                                     a.old, (int)(a.prev_changed == nullptr), a.cur_changed);
  return true;
}

}  // namespace spr
