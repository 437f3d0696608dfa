// Block-sparse / dense attention on the sm_100a tensor cores (bf16, D = d = d_v = 64 or 128).  At D = 64 the probabilities keep the
// float32 precision that the CUDA-core kernels of this head dimension gave them: they enter P V as two bf16 words (two products, as
// long together as the one at D = 128; tensor memory has the room), every exponential takes ex2.approx, and the product of a key
// tile is a sum of its own that the softmax threads add up in float32 (the accumulator of the tensor cores drops what does not fit
// when a term is added: 1.0e-5 with one running sum).  Error of the hard-drop rows against float64 at 17550 tokens: 4.8e-7; with one
// word 2.0e-4, of the CUDA-core kernels 1.2e-6.  Attention stage of 16 such heads: 1.12 ms (one word 0.90, CUDA cores 12.2).
//
// One CTA processes one 128-row query tile, or two of the same query group (of one query group, Eq. 3; or of the whole
// head for dense attention, Eq. 1).  With one tile, roles:
//   warps 0-7  softmax: warps w and w+4 share the 32 rows of TMEM quadrant w and split the
//              128 scores of a row in two halves (keys 0-63 / 64-127 of the tile)
//   warp  8    TMA producer of Q and the key tiles (+ tile meta ring)
//   warp  9    issues Q K^T (one elected lane); owns the TMEM allocation
//   warp  10   TMA producer of the value tiles
//   warp  11   issues P V (one elected lane)
// The routed keys/values arrive as one concatenated sequence of 16-row boxes (tiles of 128 keys, only
// range ends are ragged); consecutive boxes of one key range are fetched by one copy per set bit of their
// number (tensor maps with 16-, 32-, 64- and 128-row boxes).  Data path per key tile i:
//   S_b = Q K_i^T        tcgen05.mma, smem x smem -> TMEM (fp32), two score buffers b = i mod 2; a buffer is
//                        released as soon as the softmax threads hold its scores in registers, so the product
//                        runs two tiles ahead of the softmax
//   P_b = exp2(.)        softmax threads: tcgen05.ld their half row of S_b, row maximum (the two halves meet
//                        through shared memory), bf16 P to TMEM columns of its own (two buffers as well);
//                        3 of every 8 exponentials are a cubic on the FMA pipe, the others use ex2.approx (D = 64: all of them)
//   O  += P V_i          tcgen05.mma with the A operand read from TMEM; O stays in TMEM
// A single issuing thread shares its warp scheduler with two softmax warps that rarely leave it an issue slot:
// this is why the two products have a thread each on different schedulers, why the producers issue few, large
// copies, and why the barrier polls of a tile are grouped.
// The reference maximum of a row moves only when it grows by more than 2^8 (then O is rescaled).
// Two tiles (PAIR): the K and V tiles serve 256 rows, which halves the traffic from L2 (64 KB per key tile; all SMs together
// read 9.1 to 10.4 TB/s from L2, 0.95 us per 64 KB and SM, and one tile per CTA takes 1.1 us per key tile).  Every tile has its
// own four softmax warps, one row per thread, and its own issuer of both products; P takes the place of S (the
// accumulators leave no other), so a tile alternates between the tensor cores and its softmax warps, while the other tile does
// the opposite.  Bound by that chain; the account was taken while three pairs of eight went to the polynomial (one does now, 6 %
// faster): product 845 cycles (512 and what the other tile has queued), fetch and maximum 500, exponentials 1200, P V and its
// completion 750, 3300 cycles per key tile for both, where one tile takes 2010.  The threads have
// 224 registers (setmaxnreg).  One pair of eight by polynomial instead of three: a warp alone is short of issue slots, not of
// the special-function unit (dense, 12 heads of 18944 tokens: 1726 us with three, 1662 with two, 1630 with one, 1644 with none).
// Dense, 24 heads of 32760 tokens, one call after the other: 12.7 -> 11.0 ms (the clock falls to 1.6 GHz under the power limit); the
// same two tiles left to themselves fall into step (3900 cycles per key tile).
// Epilogue: O / l, stored as bf16 at the original token index (inverse permutation).  The residual correction of
// Eq. 9 is a pass of its own (correction_tc.cu) so that the fit can overlap this kernel; for that pass the part of
// every element that the bf16 rounding dropped is stored as a second bf16 word (O_lo), so that the corrected output
// is, in effect, rounded to bf16 only once.  D = 64: the two words are the halves of the float32 value itself.
// A tile with at most 64 valid rows (the remainder of a query group) holds every row TWICE, at lanes r and r + 64:
// the softmax threads of lanes 64-127 would otherwise spend a full tile's worth of exponentials on rows that do not
// exist (the loop is bound by the throughput of those instructions).  The four threads that then sit on a row (two
// lanes x two halves) take 32 of its 128 scores each; the copy at lane r accumulates the keys [0,32) and [64,96) of
// every tile, the copy at lane r + 64 the others, and the epilogue adds the two accumulators.  The products
// themselves are unchanged (the tile was padded to 128 rows anyway).
// Every mbarrier wait is bounded; on expiry the CTA records SPARSEPR_ERR_TIMEOUT and leaves.
#include <cuda.h>
#include <mutex>
#include "kernels.cuh"
#include "tc_common.cuh"

namespace spr {

namespace tc {

constexpr int kThreads = 384;
constexpr int kTile = 128;            // rows per query tile (one or two per CTA), keys per tile
constexpr int kSub = 16;              // rows per TMA box of the K/V stream
constexpr int kSubPerTile = kTile / kSub;
constexpr uint32_t kHalfBytes = kTile * 128;          // one [128 rows x 64 bf16] swizzled block
template <int D> constexpr uint32_t kTileBytes = (D / 64) * kHalfBytes;      // 32 KB at D = 128, 16 KB at D = 64
constexpr uint32_t kSubBytes = kSub * 128;            // 2 KB per box
constexpr int kPolyOf8 = 3;            // pairs of every 8 whose exponential is a polynomial on the FMA pipe
constexpr int kPairPolyOf8 = 1;        // the same with two query tiles per CTA
template <int D> constexpr bool kTwoWords = D == 64;   // P as two bf16 words
constexpr int kKStages = 2;            // K tiles in flight (consumed by Q K^T)
constexpr int kVStages = 2;            // V tiles in flight (consumed by P V)
constexpr int kSoftmaxRegs = 224, kOtherRegs = 56;     // registers per thread after the split: 128 (2 x 224 + 56) = the 384 x 168 of the launch

template <int D, bool PAIR> struct Smem {         // offsets from a 1024-byte aligned base
  static constexpr uint32_t q = 0;
  static constexpr uint32_t k = q + (PAIR ? 2 : 1) * kTileBytes<D>;
  static constexpr uint32_t v = k + kKStages * kTileBytes<D>;
  static constexpr uint32_t ranges = v + kVStages * kTileBytes<D>;
  static constexpr uint32_t xchg = ranges + kMaxGroups * 8;     // float [2 tile parities][2 halves][128] row maxima; float [2][128] row sums
  static constexpr uint32_t meta = xchg + 6 * 128 * 4;            // uint2[8]: ring of per-tile box counts
  static constexpr uint32_t bars = meta + 8 * 8;                  // kNumBars mbarriers
  static constexpr uint32_t misc = bars + 32 * 8;                 // tmem base, abort flag, counters
  static constexpr uint32_t dst = misc + 64;                      // int per row: where the rows of this CTA go (original token index)
  static constexpr uint32_t total = dst + (PAIR ? 2 : 1) * kTile * 4;
};
template <int D, bool PAIR> constexpr size_t kSmemBytes = Smem<D, PAIR>::total;                        // the dynamic segment is 1024-byte aligned and the only shared memory

enum Bar { Q_FULL = 0, K_FULL = 1, K_EMPTY = K_FULL + kKStages, V_FULL = K_EMPTY + kKStages, V_EMPTY = V_FULL + kVStages,
           S_FULL = V_EMPTY + kVStages, S_FREE = S_FULL + 2, P_FULL = S_FREE + 2, P_EMPTY = P_FULL + 2, O_DONE = P_EMPTY + 2, META_FULL,
           // two query tiles x: P of the keys [0, 96) and [96, 128) is in tensor memory; P V is complete (P and O at rest)
           P_PART = META_FULL + 8, PV_DONE = P_PART + 4, kNumBars = PV_DONE + 2 };
static_assert(kNumBars <= 32, "barrier area");

struct Params {
  int BH, H, N, Cq, Ck, sparse;
  int kv_div;                      // query heads per K/V head: K/V tensors, their maps and kv_off are indexed by head / kv_div
  float scale_log2;
  const int *kv_off, *route_idx, *q_perm;
  const int4* items; const int* n_items;       // block-sparse: the tiles of a head (launch_tc_items)
  __nv_bfloat16* O; i64 os[3];
  float* O_sparse;
  __nv_bfloat16* O_lo;             // optional [BH][N][D], original order: second word for the correction pass, o - bf16(o); D = 64: lower half of float32 o
  int* err;
};

struct Maps { CUtensorMap m[4]; };      // the same tensor with boxes of 16, 32, 64 and 128 rows

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) { return pack_bf16x2(a, b); }

template <int D, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
k_attention_tc(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapQ64,
               const __grid_constant__ Maps mapsK, const __grid_constant__ Maps mapsV, Params prm) {
  using SM = Smem<D, PAIR>;
  constexpr int kRows = PAIR ? 2 * kTile : kTile;                          // query rows of a CTA
  constexpr int kHalves = D / 64;                                          // 64-column blocks of a row
  constexpr int kOc = D / 2;                                               // output columns of a thread
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  unsigned char* sm = smem_raw;
  int2* ranges = reinterpret_cast<int2*>(sm + SM::ranges);
  float* xmax = reinterpret_cast<float*>(sm + SM::xchg);                 // [2][2][128] half-row maxima of the current / next tile
  float* xsum = xmax + 4 * 128;                                            // [2][128] half-row sums (end)
  uint2* meta = reinterpret_cast<uint2*>(sm + SM::meta);
  volatile int* misc = reinterpret_cast<volatile int*>(sm + SM::misc);   // [0] tmem base, [1] abort, [3] leave
  const uint32_t bars = base + SM::bars;
  auto bar = [&](int i) { return bars + 8u * i; };

  constexpr uint32_t FULLW = 0xffffffffu;
  const int tid = threadIdx.x, warp = __shfl_sync(FULLW, tid >> 5, 0), lane = tid & 31;   // (uniform, and known to be)
  const int bh = blockIdx.y, b = bh / prm.H, h = bh % prm.H;
  // ---- which query tile ---------------------------------------------------------------
  // Few dependent global reads before the first copy can start: the item (rows, place of the routes), the routed groups,
  // their ranges.  (Looking the tile up in prefix sums over the query groups took two reads more and two barriers, 5400 cycles
  // of a CTA's 130000 at 480p-like size; with that and tiles in group order: attend on a kept plan, 12 heads of 25200 tokens,
  // 1446 us, now 1417; call with 16 heads of d = 64 and 17550 tokens 2540 us, now 2494.)
  // Once any CTA has recorded a timeout the remaining CTAs of the launch leave at once (also if the
  // shared-memory base is not aligned as the swizzled tiles require).
  int4 item = make_int4((int)blockIdx.x * kRows, 0, 0, (min(kRows, prm.N - (int)blockIdx.x * kRows) << 16) | 1);
  bool none = false;
  if (prm.sparse) {
    none = (int)blockIdx.x >= prm.n_items[bh];                 // beyond this head's tiles
    item = prm.items[(i64)bh * gridDim.x + blockIdx.x];
  }
  if (tid == 0) {
    misc[3] = (prm.err != nullptr && *reinterpret_cast<volatile int*>(prm.err) == SPARSEPR_ERR_TIMEOUT) || (base & 1023u) != 0;
    if ((base & 1023u) != 0) set_error(prm.err, SPARSEPR_ERR_CUDA);
    misc[1] = 0;
  }
  __syncthreads();
  if (misc[3] || none) return;
  const int row0 = item.x, nrows = item.w >> 16, nroute = item.w & 0xFFFF;
  const bool dup = !PAIR && prm.sparse && nrows <= kTile / 2;           // every row twice: lanes r and r + 64 (see the header)
  // destination rows of the tile, fetched now so that the epilogue does not wait for them
  int* dsts = reinterpret_cast<int*>(sm + SM::dst);
  if (tid < kRows) dsts[tid] = tid < nrows ? (prm.sparse ? prm.q_perm[(i64)bh * prm.N + row0 + tid] : row0 + tid) : -1;

  // ---- set-up: barriers, TMEM, key ranges ---------------------------------------------------
  if (warp == 8 && lane == 0) {
    for (int i = 0; i < kNumBars; ++i)
      mbar_init(bar(i), i >= S_FREE && i < P_EMPTY ? 256 : i >= P_PART && i < PV_DONE ? 128
                        : PAIR && i >= K_EMPTY && i < S_FULL && (i < V_FULL || i >= V_EMPTY) ? 2 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) tmem_alloc(base + SM::misc, 512);
  if (warp == 10 && lane < 8) prefetch_map(lane < 4 ? &mapsK.m[lane] : &mapsV.m[lane - 4]);
  int boxes = 0;
  if (prm.sparse) {
    const int* kvo = prm.kv_off + (i64)(bh / prm.kv_div) * (prm.Ck + 1);
    const int* ridx = prm.route_idx + (i64)bh * prm.Cq * prm.Ck + item.z;
    for (int t = tid; t < nroute; t += kThreads) {
      const int g = ridx[t], start = kvo[g];
      ranges[t] = make_int2(start, kvo[g + 1] - start);
    }
    boxes = item.y;
  } else {
    if (tid == 0) ranges[0] = make_int2(0, prm.N);
    boxes = (prm.N + kSub - 1) / kSub;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(FULLW, (uint32_t)misc[0], 0);
  const int total_boxes = __shfl_sync(FULLW, boxes, 0);
  const int n_tiles = (total_boxes + kSubPerTile - 1) / kSubPerTile;
  volatile int* abort_flag = &misc[1];

  if (warp >= 8) {
  if constexpr (PAIR) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
  if (warp == 8 || warp == 10) {
    // =========================== TMA producers ==========================================
    // warp 8 streams Q and the key tiles, warp 10 the value tiles.  All lanes of a producer walk
    // the concatenated key ranges together (uniform); lane j issues the copies of box j.
    if (n_tiles > 0) {
      const bool is_k = warp == 8;
      const int c3 = prm.sparse ? 0 : b;
      const int c2 = (prm.sparse ? bh : h) / prm.kv_div;       // K/V head (group-major copies: [BH / kv_div]; originals: [B][H / kv_div])
      if (is_k && lane == 0) {
        const int q2 = prm.sparse ? bh : h;
        mbar_expect_tx(bar(Q_FULL), kRows / kTile * kTileBytes<D>);
        if (dup) {
          // the same 64 rows into both halves of the tile (rows 64-127 of a [128 x 64] block start 8 KB in)
          for (int part = 0; part < 2; ++part) {
            for (int c = 0; c < kHalves; ++c)
              tma_load_4d(base + SM::q + c * kHalfBytes + part * (kHalfBytes / 2), &mapQ64, bar(Q_FULL), 64 * c, row0, q2, c3);
          }
        } else {
          for (int x = 0; x < kRows / kTile; ++x)
            for (int c = 0; c < kHalves; ++c)
              tma_load_4d(base + SM::q + x * kTileBytes<D> + c * kHalfBytes, &mapQ, bar(Q_FULL), 64 * c, row0 + x * kTile, q2, c3);
        }
      }
      const int nst = is_k ? kKStages : kVStages;
      const int full0 = is_k ? K_FULL : V_FULL, empty0 = is_k ? K_EMPTY : V_EMPTY;
      const uint32_t buf0 = base + (is_k ? SM::k : SM::v);
      const Maps* maps = is_k ? &mapsK : &mapsV;
      int ri = 0, off = 0;
      bool ok = true;
      for (int i = 0; i < n_tiles && ok; ++i) {
        const int s = i % nst;
        const uint32_t ph = ((i / nst) & 1) ^ 1;             // empty barriers: the first pass completes immediately
        // the tile takes up to 8 boxes of 16 rows; consecutive boxes of one key range form a segment, and a segment
        // of n boxes is fetched by one copy per set bit of n (128, 64, 32 or 16 rows), largest first
        int my_start = 0, my_t = 0, my_n = 0, nsub = 0;
        uint32_t cnt_bits = 0;
        while (nsub < kSubPerTile && ri < nroute) {
          const int2 rg = ranges[ri];
          const int left = rg.y - off, nb = (left + kSub - 1) / kSub;
          const int n = min(kSubPerTile - nsub, nb);
          if (lane >= nsub && lane < nsub + n) { my_t = lane - nsub; my_n = n; my_start = rg.x + off + my_t * kSub; }
          uint32_t bits = n == 8 ? 0xFFFFFFFFu : ((1u << (4 * n)) - 1u);      // valid rows of every box, minus one
          if (n == nb) {                                                       // the range ends here: its last box may be short
            const int sh = 4 * (n - 1);
            bits = (bits & ~(0xFu << sh)) | ((uint32_t)(left - (n - 1) * kSub - 1) << sh);
            ++ri; off = 0;
          } else {
            off += n * kSub;
          }
          cnt_bits |= bits << (4 * nsub);
          nsub += n;
        }
        int my_k = -1;                                                         // log2 of the boxes this lane's copy spans
#pragma unroll
        for (int kb = 0; kb < 4; ++kb)
          if (lane < nsub && ((my_n >> kb) & 1) && my_t == ((my_n >> (kb + 1)) << (kb + 1))) my_k = kb;
        ok = __all_sync(0xffffffffu, mbar_wait(bar(empty0 + s), ph, abort_flag));
        if (!ok) break;
        if (lane == 0) {
          if (is_k) {
            // the key producer runs at most four tiles ahead of the last reader of meta[i]: ring of 8
            meta[i & 7] = make_uint2(cnt_bits, (uint32_t)nsub);
            mbar_arrive(bar(META_FULL + (i & 7)));
          }
          mbar_expect_tx(bar(full0 + s), nsub * kHalves * kSubBytes);
        }
        __syncwarp();
        if (my_k >= 0) {
          const uint32_t dst = buf0 + s * kTileBytes<D> + lane * kSubBytes;
#pragma unroll
          for (int c = 0; c < kHalves; ++c) tma_load_4d(dst + c * kHalfBytes, &maps->m[my_k], bar(full0 + s), 64 * c, my_start, c2, c3);
        }
      }
    }
  } else if constexpr (PAIR) {
    // =========================== two query tiles: issuer of both products of tile x (warps 9 and 11) =======
    // TMEM columns: S_x [128 x, 128 x + 128), P_x over its first 64 (second words: over the others) once the scores are in registers,
    // O_x [256 + 128 x, ... + D).
    // (As below, the whole warp walks the tiles and one elected lane issues.)
    if (n_tiles > 0) {
      const int x = warp == 9 ? 0 : 1;
      const uint32_t idesc_qk = idesc_bf16(0, 128), idesc_pv = idesc_bf16(1, D);
      const uint64_t q_desc = smem_desc(base + SM::q + x * kTileBytes<D>, 16), k_desc = smem_desc(base + SM::k, 16), v_desc = smem_desc(base + SM::v, kHalfBytes);
      const uint32_t sx = tmem + 128u * x, ox = tmem + 256u + 128u * x;
      bool ok = __all_sync(FULLW, mbar_wait(bar(Q_FULL), 0, abort_flag));
      for (int i = 0; i < n_tiles && ok; ++i) {
        const int s = i & 1;
        ok = mbar_wait(bar(K_FULL + s), (i >> 1) & 1, abort_flag);
        if (i > 0) ok = ok && mbar_wait(bar(PV_DONE + x), (i - 1) & 1, abort_flag);     // P of tile i - 1 lies in the score columns
        if (!__all_sync(FULLW, ok)) break;
        tc_fence_after();
        const uint64_t kd = k_desc + (uint64_t)(s * (kTileBytes<D> >> 4)), vd = v_desc + (uint64_t)(s * (kTileBytes<D> >> 4));
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint64_t koff = (uint64_t)((kk >> 2) * (kHalfBytes >> 4) + (kk & 3) * 2);     // compile-time constant
            umma_bf16(sx, q_desc + koff, kd + koff, idesc_qk, kk > 0);
          }
          umma_commit(bar(K_EMPTY + s));
          umma_commit(bar(S_FULL + x));
        }
        __syncwarp();
        ok = mbar_wait(bar(META_FULL + (i & 7)), (i >> 3) & 1, abort_flag);
        const int nsub = __shfl_sync(FULLW, (int)meta[i & 7].y, 0);
        ok = ok && mbar_wait(bar(V_FULL + s), (i >> 1) & 1, abort_flag);
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          ok = __all_sync(FULLW, ok && mbar_wait(bar(P_PART + 2 * x + part), i & 1, abort_flag));   // these P in TMEM, O rescaled if needed
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int kk = part ? 6 : 0; kk < (part ? 8 : 6); ++kk)
              if (kk < nsub) {
                umma_bf16_ts(ox, sx + kk * 8, vd + (uint64_t)(kk * (kSubBytes >> 4)), idesc_pv, (!kTwoWords<D> && i > 0) || kk > 0 ? 1u : 0u);
                if constexpr (kTwoWords<D>) umma_bf16_ts(ox, sx + 64u + kk * 8, vd + (uint64_t)(kk * (kSubBytes >> 4)), idesc_pv, 1u);
              }
            if (part == 1) { umma_commit(bar(V_EMPTY + s)); umma_commit(bar(PV_DONE + x)); }
          }
          __syncwarp();
        }
      }
    }
  } else if (warp == 9) {
    // =========================== Q K^T issuer ============================================
    // TMEM columns: S_0 [0,128), S_1 [128,256), P_0 [256,320) and P_1 [448,512) (two bf16 per column), O [320,320+D); D = 64: O_0 [320,384),
    // O_1 [384,448), of tiles in turn.  The second words
    // of P_b take the place of its scores: a thread's 32 columns of them lie over the 64 scores that only it reads, so the next
    // product into the buffer waits for P V instead of the scores' way into registers (the products still run a tile ahead).
    // The two products are issued by two threads on different warp schedulers: an issuing thread shares its
    // scheduler with two softmax warps that rarely leave it a slot, and the score tile two steps ahead must not
    // queue behind the P V of the current one.
    // The whole warp walks the tiles and one elected lane issues; loop control goes through votes, so that it is known
    // to be uniform and the descriptors stay in uniform registers.  With a loop in one thread (divergent exits) an
    // instruction cost its issuer about 70 cycles instead of 31: dense launch 12.7 -> 11.9 ms, block-sparse stage of the
    // 480p-like call 4.95 -> 4.43 ms.
    if (n_tiles > 0) {
      const uint32_t idesc_qk = idesc_bf16(0, 128);
      // descriptors are built once; inside the loops only their address field moves (in 16-byte units)
      const uint64_t q_desc = smem_desc(base + SM::q, 16);
      const uint64_t k_desc0 = smem_desc(base + SM::k, 16);
      bool ok = __all_sync(FULLW, mbar_wait(bar(Q_FULL), 0, abort_flag));
      for (int i = 0; i < n_tiles && ok; ++i) {
        const int s = i % kKStages;
        // score buffer i mod 2 is free once every softmax thread holds tile i - 2 in registers (second words: once they are consumed)
        if (i >= 2) ok = mbar_wait(bar((kTwoWords<D> ? P_EMPTY : S_FREE) + (i & 1)), ((i - 2) >> 1) & 1, abort_flag);
        ok = __all_sync(FULLW, ok && mbar_wait(bar(K_FULL + s), (i / kKStages) & 1, abort_flag));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(i & 1) * 128u;
        const uint64_t kd = k_desc0 + (uint64_t)(s * (kTileBytes<D> >> 4));
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint64_t koff = (uint64_t)((kk >> 2) * (kHalfBytes >> 4) + (kk & 3) * 2);     // compile-time constant
            umma_bf16(d, q_desc + koff, kd + koff, idesc_qk, kk > 0);
          }
          umma_commit(bar(K_EMPTY + s));
          umma_commit(bar(S_FULL + (i & 1)));
        }
        __syncwarp();
      }
    }
  } else if (warp == 11) {
    // =========================== P V issuer ==============================================
    if (n_tiles > 0) {
      const uint32_t idesc_pv = idesc_bf16(1, D);
      const uint64_t v_desc0 = smem_desc(base + SM::v, kHalfBytes);
      bool ok = true;
      for (int i = 0; i < n_tiles && ok; ++i) {
        const int s = i % kVStages;
        ok = mbar_wait(bar(META_FULL + (i & 7)), (i >> 3) & 1, abort_flag);
        const int nsub = __shfl_sync(FULLW, (int)meta[i & 7].y, 0);
        ok = ok && mbar_wait(bar(V_FULL + s), (i / kVStages) & 1, abort_flag);
        ok = __all_sync(FULLW, ok && mbar_wait(bar(P_FULL + (i & 1)), (i >> 1) & 1, abort_flag));   // P(i) in TMEM, O rescaled if needed
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem + 320u + (kTwoWords<D> ? (uint32_t)(i & 1) * 64u : 0u);
        const uint32_t pa = tmem + ((i & 1) ? 448u : 256u);
        const uint64_t vd = v_desc0 + (uint64_t)(s * (kTileBytes<D> >> 4));
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < kSubPerTile; ++kk)
            if (kk < nsub) {
              umma_bf16_ts(d, pa + kk * 8, vd + (uint64_t)(kk * (kSubBytes >> 4)), idesc_pv, (!kTwoWords<D> && i > 0) || kk > 0 ? 1u : 0u);
              if constexpr (kTwoWords<D>)
                umma_bf16_ts(d, tmem + (uint32_t)(i & 1) * 128u + (kk >> 2) * 64 + (kk & 3) * 8, vd + (uint64_t)(kk * (kSubBytes >> 4)), idesc_pv, 1u);
            }
          umma_commit(bar(V_EMPTY + s));
          umma_commit(bar(P_EMPTY + (i & 1)));
        }
        __syncwarp();
      }
      if (ok && elect_one()) umma_commit(bar(O_DONE));
    }
  }
  } else if constexpr (PAIR) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftmaxRegs));
    // =========================== two query tiles: softmax ===================================
    // Warps 4 x .. 4 x + 3 own tile x, a thread one row of it.
    const int x = warp >> 2, row = (warp & 3) * 32 + lane;
    const uint32_t s_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 128u * (uint32_t)x, o_addr = s_addr + 256u;
    const float sc = prm.scale_log2;
    float m_ref = -INFINITY, l = 0.f;
    float oa[kTwoWords<D> ? D : 1];                              // the row's sum of the tiles before (D = 64)
#pragma unroll
    for (float& v : oa) v = 0.f;
    auto take = [&] {                                            // ... plus the last one's share
#pragma unroll
      for (int q = 0; q < D / 32; ++q) {
        float t[32];
        tmem_ld32(o_addr + q * 32, t);
        add_share(oa + q * 32, t, 1.f, 1.f, true);
      }
    };
    bool ok = true;
    // The warps of the two tiles that share a scheduler take turns with their exponentials (barriers 1 + w and 5 + w: tile 0,
    // tile 1 may go): left to themselves the tiles fall into step, and then wait for the tensor cores together and compete
    // for the scheduler together.  Every turn is taken and passed on whatever happened.
    const int turn_mine = 1 + warp, turn_other = 1 + (warp ^ 4);
    if (x == 1) asm volatile("bar.arrive %0, 64;" ::"r"(turn_other) : "memory");
    for (int i = 0; i < n_tiles; ++i) {
      // the two barriers are polled back to back (their shared-memory round trips overlap)
      const bool t_meta = mbar_try(bar(META_FULL + (i & 7)), (i >> 3) & 1), t_s = mbar_try(bar(S_FULL + x), i & 1);
      if (!t_meta) ok = ok && mbar_wait(bar(META_FULL + (i & 7)), (i >> 3) & 1, abort_flag);
      if (!t_s) ok = ok && mbar_wait(bar(S_FULL + x), i & 1, abort_flag);
      ok = __all_sync(FULLW, ok);
      float s[4][32];
      float corr = 1.f, mneg = 0.f;
      if (ok) {
        tc_fence_after();
        const uint2 mt = meta[i & 7];
        if constexpr (kTwoWords<D>) { if (i > 0) take(); }       // (the previous P V is complete: S_FULL says so)
#pragma unroll
        for (int q = 0; q < 4; ++q) tmem_ld32_nowait(s_addr + 32 * q, s[q]);
        tmem_ld_wait();
        if (!(mt.x == 0xFFFFFFFFu && mt.y == 8u)) {              // (uniform)
          // only the boxes that end a key range (or lie beyond the stream) have columns to mask
#pragma unroll
          for (int bx = 0; bx < 8; ++bx) {
            const int lim = bx < (int)mt.y ? (int)((mt.x >> (4 * bx)) & 15u) : -1;      // last valid column of the box
            if (lim != 15) {
#pragma unroll
              for (int c = 0; c < 16; ++c) s[bx >> 1][(bx & 1) * 16 + c] = (c <= lim) ? s[bx >> 1][(bx & 1) * 16 + c] : -INFINITY;
            }
          }
        }
        float m8[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) m8[c] = -INFINITY;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int c = 0; c < 32; c += 2) m8[(c >> 1) & 7] = max3(m8[(c >> 1) & 7], s[q][c], s[q][c + 1]);
        const float mx = max3(max3(m8[0], m8[1], m8[2]), max3(m8[3], m8[4], m8[5]), fmaxf(m8[6], m8[7]));
        const bool move = (mx - m_ref) * sc > 8.f;               // true on the first tile (m_ref = -inf)
        const float m_new = move ? mx : m_ref;
        corr = move ? ex2((m_ref - m_new) * sc) : 1.f;           // 0 on the first tile
        mneg = -m_new * sc;
        m_ref = m_new;
        if (i > 0 && __any_sync(FULLW, move)) {                  // rescale the rows of this warp (rare); the previous P V is complete: S_FULL says so
          if constexpr (kTwoWords<D>) {
#pragma unroll
            for (float& v : oa) v *= corr;
          } else
#pragma unroll 1
          for (int q = 0; q < D / 32; ++q) {
            float t[32];
            tmem_ld32(o_addr + q * 32, t);
#pragma unroll
            for (int c = 0; c < 32; ++c) t[c] *= corr;
            tmem_st32(o_addr + q * 32, t);
          }
        }
      }
      asm volatile("bar.sync %0, 64;" ::"r"(turn_mine) : "memory");
      if (ok) {
        // probabilities, 32 at a time; P V starts on the first 96 while the others are computed
        float2 ps2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const float2 sc2 = make_float2(sc, sc), mneg2 = make_float2(mneg, mneg);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t w[16], wl[kTwoWords<D> ? 16 : 1];
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            float2 e = __ffma2_rn(make_float2(s[q][2 * c], s[q][2 * c + 1]), sc2, mneg2);
            if (!kTwoWords<D> && (c & 7) < kPairPolyOf8) e = ex2_poly2(e);
            else { e.x = ex2(e.x); e.y = ex2(e.y); }
            ps2[c & 1] = __fadd2_rn(ps2[c & 1], e);
            w[c] = pack_bf16(e.x, e.y);
            if constexpr (kTwoWords<D>) wl[c] = pack_bf16x2_rest(e.x, e.y, w[c]);
          }
          tmem_st16u_nowait(s_addr + 16 * q, w);
          if constexpr (kTwoWords<D>) tmem_st16u_nowait(s_addr + 64 + 16 * q, wl);
          if (q >= 2) {
            tmem_st_wait();
            tc_fence_before();
            mbar_arrive(bar(P_PART + 2 * x + (q - 2)));
          }
        }
        l = l * corr + ((ps2[0].x + ps2[0].y) + (ps2[1].x + ps2[1].y));
      }
      asm volatile("bar.arrive %0, 64;" ::"r"(turn_other) : "memory");
    }
    // ---- normalise, store ------------------------------------------------------------------------
    if (n_tiles > 0) ok = __all_sync(FULLW, ok && mbar_wait(bar(PV_DONE + x), (n_tiles - 1) & 1, abort_flag));
    const float inv = l > 0.f ? 1.f / l : 0.f;
    const int rows = min(kTile, nrows - x * kTile);
    const int* dst = dsts + x * kTile;
    tc_fence_after();
    if constexpr (kTwoWords<D>) { if (ok && n_tiles > 0) take(); }   // (uniform)
    // Coalesced stores, as below, but a warp stages and writes its own rows, one of the two words at a time, in the place
    // of its query rows (the other tile may still be reading the rings); 16-byte pieces are permuted within a row by the
    // row number, so that a quarter warp meets different banks both ways.
    unsigned char* stage = sm + SM::q + x * kTileBytes<D>;
    constexpr int kLpr = D / 8, kRpi = 32 / kLpr;                // pieces (lanes) per row, rows per step of a warp
#pragma unroll 1
    for (int word = 0; word < (prm.O_lo ? 2 : 1); ++word) {
#pragma unroll (kTwoWords<D> ? D / 32 : 1)
      for (int q = 0; q < D / 32; ++q) {
        float t[32];
        if constexpr (kTwoWords<D>) {
#pragma unroll
          for (int c = 0; c < 32; ++c) t[c] = oa[q * 32 + c];
        } else {
          if (ok && n_tiles > 0) tmem_ld32(o_addr + q * 32, t);  // (uniform)
        }
#pragma unroll
        for (int c = 0; c < 32; ++c) t[c] = ok && n_tiles > 0 && inv != 0.f ? t[c] * inv : 0.f;
        if (word == 0 && prm.O_sparse && ok && row < rows) {
          float* sp = prm.O_sparse + ((i64)bh * prm.N + dst[row]) * D + q * 32;
#pragma unroll
          for (int c = 0; c < 32; c += 4) *reinterpret_cast<float4*>(sp + c) = make_float4(t[c], t[c + 1], t[c + 2], t[c + 3]);
        }
        if (kTwoWords<D> && prm.O_lo) {
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            uint32_t h[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float a0 = t[8 * ch + 2 * k], a1 = t[8 * ch + 2 * k + 1];
              h[k] = word ? lower_halves(a0, a1) : upper_halves(a0, a1);
            }
            *reinterpret_cast<uint4*>(stage + row * 2 * D + (((q * 4 + ch) ^ (row & 7)) * 16)) = make_uint4(h[0], h[1], h[2], h[3]);
          }
          continue;
        }
        if (word == 1) {
#pragma unroll
          for (int c = 0; c < 32; ++c) t[c] -= __bfloat162float(__float2bfloat16_rn(t[c]));     // what the rounding of the first word dropped
        }
#pragma unroll
        for (int ch = 0; ch < 4; ++ch)
          *reinterpret_cast<uint4*>(stage + row * 2 * D + (((q * 4 + ch) ^ (row & 7)) * 16)) =
              make_uint4(pack_bf16(t[8 * ch], t[8 * ch + 1]), pack_bf16(t[8 * ch + 2], t[8 * ch + 3]), pack_bf16(t[8 * ch + 4], t[8 * ch + 5]), pack_bf16(t[8 * ch + 6], t[8 * ch + 7]));
      }
      __syncwarp();
#pragma unroll 4
      for (int it = 0; it < 32 / kRpi; ++it) {
        const int r = (warp & 3) * 32 + kRpi * it + lane / kLpr, ch = lane % kLpr;
        if (ok && r < rows) {
          const uint4 vh = *reinterpret_cast<const uint4*>(stage + r * 2 * D + ((ch ^ (r & 7)) * 16));
          __nv_bfloat16* op = word == 0 ? prm.O + b * prm.os[0] + h * prm.os[1] + (i64)dst[r] * prm.os[2] : prm.O_lo + ((i64)bh * prm.N + dst[r]) * D;
          *reinterpret_cast<uint4*>(op + ch * 8) = vh;
        }
      }
      __syncwarp();
    }
  } else {
    // =========================== softmax (warps 0-7) =======================================
    // Thread (half hh, quadrant wq, lane) owns the 64 scores of keys [64 hh, 64 hh + 64) of query row
    // 32 wq + lane; warps wq and wq + 4 meet at the named barrier 1 + wq to agree on the row maximum.
    const int hh = warp >> 2, wq = warp & 3;
    const int row = wq * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
    const uint32_t FULL = 0xffffffffu;
    const uint32_t p_addr0 = tmem + lane_addr + 256u + (uint32_t)hh * 32u;      // P of even tiles; odd tiles 192 columns on
    const uint32_t o_addr = tmem + lane_addr + 320u + (uint32_t)(hh * kOc);
    float m_ref = -INFINITY, l = 0.f;
    bool ok = true;
    const float sc = prm.scale_log2;
    // D = 64: sum of the tiles but the last two, whose shares lie in tensor memory; corr_prev: the rescaling since the one before the last
    float oa[kTwoWords<D> ? kOc : 1], corr_prev = 1.f;
#pragma unroll
    for (float& v : oa) v = 0.f;
    auto take = [&](int i, float fo, float ft) {                 // the share of tile i
      float t[32];
      tmem_ld32(o_addr + (uint32_t)(i & 1) * 64u, t);
      add_share(oa, t, fo, ft, __all_sync(FULL, fo == 1.f && ft == 1.f));
    };
    auto take_last = [&] {
      if (n_tiles > 1) take(n_tiles - 2, 1.f, corr_prev);
      take(n_tiles - 1, 1.f, 1.f);
    };
    // the finished output columns [kOc hh, kOc hh + kOc) of tile row r: bf16 at the original token index, the part that
    // the rounding dropped as a second word, float32 on request
    auto store_row = [&](int r, const float (&o)[kOc]) {
      const int dst = prm.sparse ? prm.q_perm[(i64)bh * prm.N + row0 + r] : row0 + r;
      __nv_bfloat16* op = prm.O + b * prm.os[0] + h * prm.os[1] + (i64)dst * prm.os[2] + hh * kOc;
      if (kTwoWords<D> && prm.O_lo) {                          // the two halves of the float32 value
        __nv_bfloat16* lp = prm.O_lo + ((i64)bh * prm.N + dst) * D + hh * kOc;
#pragma unroll
        for (int ch = 0; ch < kOc / 8; ++ch) {
          const float* v = o + ch * 8;
          *reinterpret_cast<uint4*>(op + ch * 8) = make_uint4(upper_halves(v[0], v[1]), upper_halves(v[2], v[3]), upper_halves(v[4], v[5]), upper_halves(v[6], v[7]));
          *reinterpret_cast<uint4*>(lp + ch * 8) = make_uint4(lower_halves(v[0], v[1]), lower_halves(v[2], v[3]), lower_halves(v[4], v[5]), lower_halves(v[6], v[7]));
        }
      } else {
#pragma unroll
        for (int ch = 0; ch < kOc / 8; ++ch) {
          float v8[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) v8[k] = o[ch * 8 + k];
          store8(op + ch * 8, v8);
        }
      }
      if (!kTwoWords<D> && prm.O_lo) {                         // what the bf16 rounding above dropped
        __nv_bfloat16* lp = prm.O_lo + ((i64)bh * prm.N + dst) * D + hh * kOc;
#pragma unroll
        for (int ch = 0; ch < kOc / 8; ++ch) {
          float v8[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) v8[k] = o[ch * 8 + k] - __bfloat162float(__float2bfloat16_rn(o[ch * 8 + k]));
          store8(lp + ch * 8, v8);
        }
      }
      if (prm.O_sparse) {
        float* sp = prm.O_sparse + ((i64)bh * prm.N + dst) * D + hh * kOc;
#pragma unroll
        for (int ch = 0; ch < kOc / 8; ++ch) {
          float v8[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) v8[k] = o[ch * 8 + k];
          store8(sp + ch * 8, v8);
        }
      }
    };
    if (dup) {
      // ================= at most 64 valid rows: four threads per row, 32 scores each ==================
      const int u = wq >> 1, q0 = wq & 1;                        // copy of the row (lane r or r + 64); pair of quadrants
      const int vr = q0 * 32 + lane;                             // the row, 0..63
      const int cb = 64 * hh + 32 * u;                           // this thread's keys of a tile: [cb, cb + 32)
      const int slot = 2 * hh + u;
      for (int i = 0; i < n_tiles; ++i) {
        const bool t_meta = mbar_try(bar(META_FULL + (i & 7)), (i >> 3) & 1);
        const bool t_s = mbar_try(bar(S_FULL + (i & 1)), (i >> 1) & 1);
        const bool t_pe = i > 1 ? mbar_try(bar(P_EMPTY + (i & 1)), ((i - 2) >> 1) & 1) : true;
        {
          bool w = ok;
          if (!t_meta) w = w && mbar_wait(bar(META_FULL + (i & 7)), (i >> 3) & 1, abort_flag);
          if (!t_s) w = w && mbar_wait(bar(S_FULL + (i & 1)), (i >> 1) & 1, abort_flag);
          ok = __all_sync(FULL, w);
        }
        float s[32];
        float mx = -INFINITY;
        if (ok) {
          tc_fence_after();
          const uint2 mt = meta[i & 7];
          tmem_ld32_nowait(tmem + lane_addr + (uint32_t)(i & 1) * 128u + (uint32_t)cb, s);
          tmem_ld_wait();
          if constexpr (!kTwoWords<D>) {
            tc_fence_before();
            mbar_arrive(bar(S_FREE + (i & 1)));                     // the scores are in registers
          }
          if (!(mt.x == 0xFFFFFFFFu && mt.y == 8u)) {
#pragma unroll
            for (int bx = 0; bx < 2; ++bx) {
              const int box = (cb >> 4) + bx;
              const int lim = box < (int)mt.y ? (int)((mt.x >> (4 * box)) & 15u) : -1;    // last valid column of the box
              if (lim != 15) {
#pragma unroll
                for (int c = 0; c < 16; ++c) s[bx * 16 + c] = (c <= lim) ? s[bx * 16 + c] : -INFINITY;
              }
            }
          }
          float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int c = 0; c < 32; c += 8) {
            mx4[0] = max3(mx4[0], s[c], s[c + 1]); mx4[1] = max3(mx4[1], s[c + 2], s[c + 3]);
            mx4[2] = max3(mx4[2], s[c + 4], s[c + 5]); mx4[3] = max3(mx4[3], s[c + 6], s[c + 7]);
          }
          mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
        }
        // the four threads of a row exchange their maxima (four warps meet: both halves of quadrants q0 and q0 + 2)
        float* xm = xmax + (i & 1) * 256;
        xm[slot * 64 + vr] = mx;
        asm volatile("bar.sync %0, 128;" ::"r"(1 + q0) : "memory");
        mx = fmaxf(fmaxf(xm[vr], xm[64 + vr]), fmaxf(xm[128 + vr], xm[192 + vr]));
        const bool move = (mx - m_ref) * sc > 8.f;
        const float m_new = move ? mx : m_ref;
        const float corr = move ? ex2((m_ref - m_new) * sc) : 1.f;
        const float mneg = -m_new * sc;
        m_ref = m_new;
        if (!__all_sync(FULL, t_pe)) {
          ok = __all_sync(FULL, ok && (t_pe || mbar_wait(bar(P_EMPTY + (i & 1)), ((i - 2) >> 1) & 1, abort_flag)));
          tc_fence_after();
        }
        if (!ok) continue;
        if constexpr (kTwoWords<D>) {
          if (i > 1) take(i - 2, corr, corr_prev * corr);        // (its product is complete: P_EMPTY says so)
          corr_prev = corr;
        } else if (i > 0 && __any_sync(FULL, move)) {            // rescale this half of the lane's accumulator (rare)
          ok = __all_sync(FULL, mbar_wait(bar(P_EMPTY + ((i - 1) & 1)), ((i - 1) >> 1) & 1, abort_flag));
          if (!ok) continue;
          tc_fence_after();
#pragma unroll
          for (int q = 0; q < kOc / 32; ++q) {
            float t[32];
            tmem_ld32(o_addr + q * 32, t);
#pragma unroll
            for (int c = 0; c < 32; ++c) t[c] *= corr;
            tmem_st32(o_addr + q * 32, t);
          }
        }
        float2 ps2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const float2 sc2 = make_float2(sc, sc), mneg2 = make_float2(mneg, mneg);
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          float2 x = __ffma2_rn(make_float2(s[2 * q], s[2 * q + 1]), sc2, mneg2);
          if (!kTwoWords<D> && (q & 7) < kPolyOf8) x = ex2_poly2(x);
          else { x.x = ex2(x.x); x.y = ex2(x.y); }
          s[2 * q] = x.x; s[2 * q + 1] = x.y;
          ps2[q & 1] = __fadd2_rn(ps2[q & 1], x);
        }
        l = l * corr + ((ps2[0].x + ps2[0].y) + (ps2[1].x + ps2[1].y));
        // P of this lane and half: this thread's 32 probabilities -> 16 columns, zeros in the 16 columns of the keys
        // that the other copy of the row takes
        {
          uint32_t w[16], z[16];
#pragma unroll
          for (int c = 0; c < 16; ++c) { w[c] = pack_bf16(s[2 * c], s[2 * c + 1]); z[c] = 0u; }
          const uint32_t pa = p_addr0 + (uint32_t)(i & 1) * 192u;
          tmem_st16u_nowait(pa + 16u * (uint32_t)u, w);
          tmem_st16u_nowait(pa + 16u * (uint32_t)(1 - u), z);
          if constexpr (kTwoWords<D>) {
#pragma unroll
            for (int c = 0; c < 16; ++c) w[c] = pack_bf16x2_rest(s[2 * c], s[2 * c + 1], w[c]);
            const uint32_t pl = tmem + lane_addr + (uint32_t)(i & 1) * 128u + (uint32_t)hh * 64u;
            tmem_st16u_nowait(pl + 16u * (uint32_t)u, w);
            tmem_st16u_nowait(pl + 16u * (uint32_t)(1 - u), z);
          }
          tmem_st_wait();
        }
        tc_fence_before();
        mbar_arrive(bar(P_FULL + (i & 1)));
      }
      // ---- row sums of the four threads, sum of the two accumulators, normalise, store -----------------
      if (n_tiles > 0) ok = __all_sync(FULL, ok && mbar_wait(bar(O_DONE), 0, abort_flag));
      xsum[slot * 64 + vr] = l;
      float o[kOc];
#pragma unroll
      for (int c = 0; c < kOc; ++c) o[c] = 0.f;
      if (ok && n_tiles > 0) {
        tc_fence_after();
        if constexpr (kTwoWords<D>) {
          take_last();
#pragma unroll
          for (int c = 0; c < kOc; ++c) o[c] = oa[c];
        } else
#pragma unroll
        for (int q = 0; q < kOc / 32; ++q) {
          float t[32];
          tmem_ld32(o_addr + q * 32, t);
#pragma unroll
          for (int c = 0; c < 32; ++c) o[q * 32 + c] = t[c];
        }
      }
      // the copy at lane r + 64 hands its accumulator over through the Q tile's shared memory (every product that
      // reads it has completed): [half][column][row], conflict-free for consecutive rows
      float* ex = reinterpret_cast<float*>(sm + SM::q);
      if (u == 1) {
#pragma unroll
        for (int c = 0; c < kOc; ++c) ex[(hh * kOc + c) * 64 + vr] = o[c];
      }
      asm volatile("bar.sync %0, 128;" ::"r"(1 + q0) : "memory");
      if (u == 0) {
        const float ltot = (xsum[vr] + xsum[64 + vr]) + (xsum[128 + vr] + xsum[192 + vr]);
        const float inv = ltot > 0.f ? 1.f / ltot : 0.f;
#pragma unroll
        for (int c = 0; c < kOc; ++c) o[c] = inv != 0.f ? (o[c] + ex[(hh * kOc + c) * 64 + vr]) * inv : 0.f;
        if (ok && vr < nrows) store_row(vr, o);
      }
    } else {
    for (int i = 0; i < n_tiles; ++i) {
      // the three barriers of this tile are polled back to back (their shared-memory round trips overlap); the P
      // buffer of this parity was consumed by the product two tiles back and is normally free long before
      const bool t_meta = mbar_try(bar(META_FULL + (i & 7)), (i >> 3) & 1);
      const bool t_s = mbar_try(bar(S_FULL + (i & 1)), (i >> 1) & 1);
      const bool t_pe = i > 1 ? mbar_try(bar(P_EMPTY + (i & 1)), ((i - 2) >> 1) & 1) : true;
      {
        bool w = ok;
        if (!t_meta) w = w && mbar_wait(bar(META_FULL + (i & 7)), (i >> 3) & 1, abort_flag);
        if (!t_s) w = w && mbar_wait(bar(S_FULL + (i & 1)), (i >> 1) & 1, abort_flag);
        ok = __all_sync(FULL, w);
      }
      float s[64];
      float mx = -INFINITY;
      if (ok) {
        tc_fence_after();
        const uint2 mt = meta[i & 7];
        const uint32_t s_addr = tmem + lane_addr + (uint32_t)(i & 1) * 128u + (uint32_t)hh * 64u;
        tmem_ld32_nowait(s_addr, *reinterpret_cast<float(*)[32]>(&s[0]));
        tmem_ld32_nowait(s_addr + 32, *reinterpret_cast<float(*)[32]>(&s[32]));
        tmem_ld_wait();
        if constexpr (!kTwoWords<D>) {
          tc_fence_before();
          mbar_arrive(bar(S_FREE + (i & 1)));                       // the scores are in registers
        }
        if (!(mt.x == 0xFFFFFFFFu && mt.y == 8u)) {
          // only the boxes that end a key range (or lie beyond the stream) have columns to mask; the test is uniform
#pragma unroll
          for (int bx = 0; bx < 4; ++bx) {
            const int box = hh * 4 + bx;
            const int lim = box < (int)mt.y ? (int)((mt.x >> (4 * box)) & 15u) : -1;      // last valid column of the box
            if (lim != 15) {
#pragma unroll
              for (int c = 0; c < 16; ++c) s[bx * 16 + c] = (c <= lim) ? s[bx * 16 + c] : -INFINITY;
            }
          }
        }
        float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < 64; c += 8) {
          mx4[0] = max3(mx4[0], s[c], s[c + 1]); mx4[1] = max3(mx4[1], s[c + 2], s[c + 3]);
          mx4[2] = max3(mx4[2], s[c + 4], s[c + 5]); mx4[3] = max3(mx4[3], s[c + 6], s[c + 7]);
        }
        mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      }
      // the two halves of the row exchange their maxima (buffer of this tile's parity; executed whatever happened)
      float* xm = xmax + (i & 1) * 256;
      xm[hh * 128 + row] = mx;
      asm volatile("bar.sync %0, 64;" ::"r"(1 + wq) : "memory");
      mx = fmaxf(mx, xm[(hh ^ 1) * 128 + row]);
      const bool move = (mx - m_ref) * sc > 8.f;                 // true on the first tile (m_ref = -inf); same in both halves
      const float m_new = move ? mx : m_ref;
      const float corr = move ? ex2((m_ref - m_new) * sc) : 1.f; // 0 on the first tile
      const float mneg = -m_new * sc;
      m_ref = m_new;
      // the P buffer of this parity must have been consumed by the product two tiles back
      if (!__all_sync(FULL, t_pe)) {
        ok = __all_sync(FULL, ok && (t_pe || mbar_wait(bar(P_EMPTY + (i & 1)), ((i - 2) >> 1) & 1, abort_flag)));
        tc_fence_after();
      }
      if (!ok) continue;                                         // warp-uniform; the pair barrier above has been passed
      if constexpr (kTwoWords<D>) {
        if (i > 1) take(i - 2, corr, corr_prev * corr);          // (its product is complete: P_EMPTY says so)
        corr_prev = corr;
      } else if (i > 0 && __any_sync(FULL, move)) {              // rescale this half of the warp's O rows (rare)
        // O must be at rest: the product of the previous tile has to be complete as well
        ok = __all_sync(FULL, mbar_wait(bar(P_EMPTY + ((i - 1) & 1)), ((i - 1) >> 1) & 1, abort_flag));
        if (!ok) continue;
        tc_fence_after();
#pragma unroll
        for (int q = 0; q < kOc / 32; ++q) {
          float t[32];
          tmem_ld32(o_addr + q * 32, t);
#pragma unroll
          for (int c = 0; c < 32; ++c) t[c] *= corr;
          tmem_st32(o_addr + q * 32, t);
        }
      }
      // exponentials: kPolyOf8 of every 8 pairs on the FMA pipe, the others on the special-function unit
      float2 ps2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      const float2 sc2 = make_float2(sc, sc), mneg2 = make_float2(mneg, mneg);
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        float2 x = __ffma2_rn(make_float2(s[2 * q], s[2 * q + 1]), sc2, mneg2);
        if (!kTwoWords<D> && (q & 7) < kPolyOf8) x = ex2_poly2(x);
        else { x.x = ex2(x.x); x.y = ex2(x.y); }
        s[2 * q] = x.x; s[2 * q + 1] = x.y;
        ps2[q & 1] = __fadd2_rn(ps2[q & 1], x);
      }
      l = l * corr + ((ps2[0].x + ps2[0].y) + (ps2[1].x + ps2[1].y));
      // P (bf16, two per 32-bit column): this half's 64 probabilities -> 32 columns
      {
        uint32_t w[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) w[c] = pack_bf16(s[2 * c], s[2 * c + 1]);
        tmem_st32u(p_addr0 + (uint32_t)(i & 1) * 192u, w);
        if constexpr (kTwoWords<D>) {
#pragma unroll
          for (int c = 0; c < 32; ++c) w[c] = pack_bf16x2_rest(s[2 * c], s[2 * c + 1], w[c]);
          tmem_st32u(tmem + lane_addr + (uint32_t)(i & 1) * 128u + (uint32_t)hh * 64u, w);
        }
      }
      tc_fence_before();
      mbar_arrive(bar(P_FULL + (i & 1)));
    }
    // ---- row sums of the two halves, normalise, store ------------------------------------------
    if (n_tiles > 0) ok = __all_sync(FULL, ok && mbar_wait(bar(O_DONE), 0, abort_flag));
    xsum[hh * 128 + row] = l;
    asm volatile("bar.sync %0, 64;" ::"r"(1 + wq) : "memory");
    const float ltot = l + xsum[(hh ^ 1) * 128 + row];
    const float inv = ltot > 0.f ? 1.f / ltot : 0.f;
    // this thread finishes output columns [kOc hh, kOc hh + kOc) of its row
    float o[kOc];
#pragma unroll
    for (int c = 0; c < kOc; ++c) o[c] = 0.f;
    if (ok && n_tiles > 0) {
      tc_fence_after();
      if constexpr (kTwoWords<D>) {
        take_last();
#pragma unroll
        for (int c = 0; c < kOc; ++c) o[c] = inv != 0.f ? oa[c] * inv : 0.f;
      } else
#pragma unroll
      for (int q = 0; q < kOc / 32; ++q) {
        float t[32];
        tmem_ld32(o_addr + q * 32, t);
#pragma unroll
        for (int c = 0; c < 32; ++c) o[q * 32 + c] = inv != 0.f ? t[c] * inv : 0.f;
      }
    }
    if (prm.O_sparse) {
      if (ok && row < nrows) store_row(row, o);
    } else {
      // Coalesced stores: a thread holds half the columns of one row, and storing them directly makes every 16-byte store
      // of a warp touch 32 different lines.  The tile is staged in shared memory instead (the K and V rings are idle:
      // every product has completed), rows 16 bytes more than their length apart so that the 16-byte accesses of a
      // quarter warp fall into different banks, and written out with 16 (D = 64: 8) lanes per row.
      constexpr uint32_t kPitch = 2 * D + 16;
      static_assert(kTile * kPitch <= 2 * kTileBytes<D>, "the rings hold the staged tile");
      unsigned char* st_hi = sm + SM::k;
      unsigned char* st_lo = sm + SM::v;
      {
        uint4* ph = reinterpret_cast<uint4*>(st_hi + row * kPitch + hh * D);
        uint4* pl = reinterpret_cast<uint4*>(st_lo + row * kPitch + hh * D);
#pragma unroll
        for (int ch = 0; ch < kOc / 8; ++ch) {
          uint32_t wh[4], wl[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float a0 = o[ch * 8 + 2 * k], a1 = o[ch * 8 + 2 * k + 1];
            if (kTwoWords<D> && prm.O_lo) { wh[k] = upper_halves(a0, a1); wl[k] = lower_halves(a0, a1); continue; }
            wh[k] = pack_bf16(a0, a1);
            wl[k] = pack_bf16(a0 - __bfloat162float(__float2bfloat16_rn(a0)), a1 - __bfloat162float(__float2bfloat16_rn(a1)));
          }
          ph[ch] = make_uint4(wh[0], wh[1], wh[2], wh[3]);
          if (prm.O_lo) pl[ch] = make_uint4(wl[0], wl[1], wl[2], wl[3]);
        }
      }
      asm volatile("bar.sync 6, 256;" ::: "memory");
      constexpr int kLpr = D / 8, kRpi = 32 / kLpr;               // lanes per row, rows per step of a warp
      const int c16 = lane % kLpr;
#pragma unroll
      for (int it = 0; it < 16 / kRpi; ++it) {
        const int r = warp * 16 + kRpi * it + lane / kLpr;
        const int dst = dsts[r];
        if (ok && r < nrows) {
          const uint4 vh = *reinterpret_cast<const uint4*>(st_hi + r * kPitch + c16 * 16);
          *reinterpret_cast<uint4*>(prm.O + b * prm.os[0] + h * prm.os[1] + (i64)dst * prm.os[2] + c16 * 8) = vh;
          if (prm.O_lo) {
            const uint4 vl = *reinterpret_cast<const uint4*>(st_lo + r * kPitch + c16 * 16);
            *reinterpret_cast<uint4*>(prm.O_lo + ((i64)bh * prm.N + dst) * D + c16 * 8) = vl;
          }
        }
      }
    }
    }
  }
  // ---- teardown ----------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies that may still be in flight time to land before the shared memory is released
    for (int k = 0; k < 64; ++k) __nanosleep(1000);
    if (tid == 0) set_error(prm.err, SPARSEPR_ERR_TIMEOUT);
    __syncthreads();
  }
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ---- tensor maps (driver entry point fetched through the runtime; libcuda is not linked) -------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
std::once_flag g_encode_once;

EncodeTiledFn encode_fn() {
  std::call_once(g_encode_once, [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  });
  return g_encode;
}

bool tma_available() { return encode_fn() != nullptr; }

bool make_map(CUtensorMap* m, const void* ptr, int cols, int rows, int H, int B, i64 sb, i64 sh, i64 sn, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const i64 hstride = H > 1 ? sh : (i64)rows * sn;
  const i64 bstride = B > 1 ? sb : (i64)H * hstride;
  const cuuint64_t dims[4] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)H, (cuuint64_t)B};
  const cuuint64_t strides[3] = {(cuuint64_t)sn * 2, (cuuint64_t)hstride * 2, (cuuint64_t)bstride * 2};
  const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tc

cudaError_t init_attention_tc() {
  cudaError_t e = cudaSuccess;
  const auto set = [&](auto kernel, size_t bytes) { if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); };
  set(tc::k_attention_tc<128, false>, tc::kSmemBytes<128, false>);
  set(tc::k_attention_tc<64, false>, tc::kSmemBytes<64, false>);
  set(tc::k_attention_tc<128, true>, tc::kSmemBytes<128, true>);
  set(tc::k_attention_tc<64, true>, tc::kSmemBytes<64, true>);
  return e;
}

bool attention_tc_supported(const AttnArgs& a) {
  return a.dtype == SPARSEPR_BF16 && (a.d == 64 || a.d == 128) && tc::tma_available();
}

bool launch_attention_tc(const AttnArgs& a, cudaStream_t st, bool pairs) {
  using namespace tc;
  const int d = a.d;
  CUtensorMap mq, mq64;
  Maps mk, mv;
  const bool sparse = a.route_ptr != nullptr;
  const int B = a.BH / a.H;
  const int kvd = a.kv_div < 1 ? 1 : a.kv_div;
  bool ok;
  if (sparse) {
    ok = make_map(&mq, a.Q, d, a.N, a.BH, 1, 0, (i64)a.N * d, d, kTile) &&
         make_map(&mq64, a.Q, d, a.N, a.BH, 1, 0, (i64)a.N * d, d, kTile / 2);
    for (int k = 0; k < 4 && ok; ++k)
      ok = make_map(&mk.m[k], a.K, d, a.N, a.BH / kvd, 1, 0, (i64)a.N * d, d, kSub << k) &&
           make_map(&mv.m[k], a.V, d, a.N, a.BH / kvd, 1, 0, (i64)a.N * d, d, kSub << k);
  } else {
    ok = make_map(&mq, a.Q, d, a.N, a.H, B, a.qs[0], a.qs[1], a.qs[2], kTile) &&
         make_map(&mq64, a.Q, d, a.N, a.H, B, a.qs[0], a.qs[1], a.qs[2], kTile / 2);
    for (int k = 0; k < 4 && ok; ++k)
      ok = make_map(&mk.m[k], a.K, d, a.N, a.H / kvd, B, a.ks[0], a.ks[1], a.ks[2], kSub << k) &&
           make_map(&mv.m[k], a.V, d, a.N, a.H / kvd, B, a.vs[0], a.vs[1], a.vs[2], kSub << k);
  }
  if (!ok) return false;
  Params p{};
  p.BH = a.BH; p.H = a.H; p.N = a.N; p.Cq = a.Cq; p.Ck = a.Ck; p.sparse = sparse; p.kv_div = kvd;
  p.scale_log2 = a.scale * 1.4426950408889634f;
  p.kv_off = a.kv_off; p.route_idx = a.route_idx; p.q_perm = a.q_perm; p.items = a.items + (pairs ? 0 : (i64)a.BH * attention_tc_pairs(a.BH, a.N, d)); p.n_items = a.n_items + (pairs ? 0 : a.BH);
  p.O = (__nv_bfloat16*)a.O; for (int i = 0; i < 3; ++i) p.os[i] = a.os[i];
  p.O_sparse = a.O_sparse; p.O_lo = (__nv_bfloat16*)a.O_lo; p.err = a.err;
  const auto run = [&](auto kernel, int ctas, size_t bytes) { kernel<<<dim3(ctas, a.BH), kThreads, bytes, st>>>(mq, mq64, mk, mv, p); };
  // Two query tiles per CTA for dense calls: a pair takes about 1.6 times as long as one tile (D = 64, whose two words of P keep the
  // tensor cores twice as long: 1.8 times), so that it pays unless the CTAs of one tile leave SMs idle (or fill their last round where
  // the pairs do not).  8 heads of 4096 tokens, two rounds of tiles, one of pairs: 79 us with tiles alone, 66 with pairs (D = 64: 96, 86);
  // 24 heads of 32760 tokens 12.7 ms, 11.0 (D = 64: 13.8, 13.3); 2 heads of 4770 tokens, one round of tiles, 49 us, which pairs on
  // half the SMs would lengthen.
  const int tiles = (a.N + kTile - 1) / kTile, sms = sm_count();
  const auto rounds = [&](int per_head) { return ((i64)per_head * a.BH + sms - 1) / sms; };
  if (sparse ? pairs : 100 * rounds(tiles) > (d == 128 ? 164 : 180) * rounds((tiles + 1) / 2)) {
    const int ctas = sparse ? attention_tc_pairs(a.BH, a.N, d) : (tiles + 1) / 2;
    if (d == 128) run(k_attention_tc<128, true>, ctas, kSmemBytes<128, true>);
    else run(k_attention_tc<64, true>, ctas, kSmemBytes<64, true>);
  } else {
    const int ctas = sparse ? attention_tc_singles(a.BH, a.N, a.Cq, d) : tiles;
    if (d == 128) run(k_attention_tc<128, false>, ctas, kSmemBytes<128, false>);
    else run(k_attention_tc<64, false>, ctas, kSmemBytes<64, false>);
  }
  return true;
}

}  // namespace spr
