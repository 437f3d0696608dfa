// Residual correction of Eq. 9 as a pass of its own on the sm_100a tensor cores:
//   O <- X + X A + c     (in place, bf16, D = d_v = 64 or 128; A, c = composed affine map of one head)
// It runs after the block-sparse kernels, so that the probe rows and the fit (which produce A and c) can execute
// on a second stream while those kernels are busy.  The block-sparse kernels hand over the hard-drop rows X = O^sp
// as two bf16 words, X = X_h + X_l: X_h is what they stored in O, X_l the part that rounding dropped (2^-17
// relative together), so that the corrected output is rounded to bf16 once -- a one-word hand-over rounds twice,
// which shows in the largest elements.  At D = 64, where the fused pass of the CUDA-core kernels had X and A in float32, the words
// are the two halves of float32 X; the epilogue warps first make the other two bf16 words of the product out of them (three words hold
// all of X) and then add X itself; A enters in three words too, with the six products that reach float32.  (Share of the outputs
// that are not the rounded float64 value at 1333 tokens and 130 probes, ridge 10: 1.3e-3; with two words each 2.9e-3 and up, with
// probabilities in bf16 besides 0.23; fused float32 pass 6e-4.  44 us instead of 32 for 16 heads of 17550 rows.)  A enters the product as two bf16 words as well, A = A_h + A_l: with few probes
// (M < d_v) and a small ridge the fitted map can have a norm of ~10, and one word of A then costs up to 0.012 of
// the 0.02 that the output may differ from the oracle (the products are X_h A_h + X_l A_h + X_h A_l; X_l A_l is
// below 2^-17 of the result).
// The pass is bandwidth bound: each 128-row tile is read once (4 D bytes per row) and written once (2 D), 93 us at the copy rate for
// 24 heads of 32760 rows.  One CTA per SM walks a run of consecutive tiles, of one head mostly, whose map stays in shared
// memory; two tiles are in work, so that the loads of one, the products (24 instructions, 0.8 us) and the epilogue of the other
// overlap, and the result leaves as a bulk store of the whole tile from the place of X_h.  (A CTA per two tiles, which loaded,
// multiplied and stored, row by row, one after the other: 194 us; now 112.)
//   warps 0-7  warps w and w + 4: 32 rows, half of the columns each: (D = 64: words of X,) X A from TMEM, X from the two swizzled tiles, + c, back to X_h
//   warp  8    TMA loads (X_h, X_l of a tile; the words of A^T when the head changes)
//   warp  9    3 D / 16 (D = 64: 6 D / 16) tcgen05.mma per tile, TMEM owner
// Every mbarrier wait is bounded; on expiry the CTA records SPARSEPR_ERR_TIMEOUT and leaves.
#include <cuda.h>
#include <algorithm>
#include "kernels.cuh"
#include "tc_common.cuh"

namespace spr {
namespace tc {

constexpr int kCorrThreads = 320;
constexpr int kCorrTile = 128;
constexpr uint32_t kCorrHalf = kCorrTile * 128;      // one [128 rows x 64 bf16] swizzled block
template <int D> constexpr uint32_t kCorrTileBytes = (D / 64) * kCorrHalf;
template <int D> constexpr uint32_t kCorrMapHalf = D * 128;                   // [D rows x 64 bf16]
template <int D> struct CorrSmem {
  static constexpr uint32_t xh = 0;                        // stage u at xh + 2 u kCorrTileBytes<D>, its second words one tile further
  static constexpr uint32_t xl = xh + kCorrTileBytes<D>;
  static constexpr uint32_t a = xh + 4 * kCorrTileBytes<D>;
  static constexpr uint32_t map_bytes = (D / 64) * kCorrMapHalf<D>;             // one word of A^T
  static constexpr uint32_t xc = a + map_words(D) * map_bytes;                  // D = 64: second and third words of X, [2 stages][2]
  static constexpr uint32_t bars = xc + (D == 64 ? 4 * kCorrTileBytes<D> : 0);
  static constexpr uint32_t misc = bars + 88;
  static constexpr uint32_t total = misc + 16;
};
static_assert(CorrSmem<128>::total <= 227 * 1024, "shared memory");

// a stage is loaded; stored and free; multiplied (product u in TMEM); the product has been read; the words of X are made; the map is loaded
enum CorrBar { C_FULL = 0, C_EMPTY = 2, C_DONE = 4, C_READ = 6, C_CONV = 8, C_MAP = 10, kCorrBars };
struct CorrParams {
  int BH, H, N;
  const float* c;                  // [BH][D]
  int* err;
};

template <int D>
__global__ void __launch_bounds__(kCorrThreads)
k_correction_tc(const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapL,
                const __grid_constant__ CUtensorMap mapA, CorrParams prm) {
  using SM = CorrSmem<D>;
  constexpr int kHalves = D / 64;
  constexpr uint32_t kMapHalf = kCorrMapHalf<D>;
  constexpr bool kHalvesOfX = D == 64;                           // X_h and the tile beside it are the halves of float32 X
  constexpr uint32_t FULLW = 0xffffffffu;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  volatile int* misc = reinterpret_cast<volatile int*>(smem_raw + SM::misc);   // [0] tmem base, [1] abort, [2] skip
  const auto bar = [&](int i) { return base + SM::bars + 8u * i; };
  const int tid = threadIdx.x, warp = __shfl_sync(FULLW, tid >> 5, 0), lane = tid & 31;
  const int n_tiles = (prm.N + kCorrTile - 1) / kCorrTile;
  const i64 total = (i64)prm.BH * n_tiles;
  const int g0 = (int)(total * blockIdx.x / gridDim.x), count = (int)(total * (blockIdx.x + 1) / gridDim.x) - g0;    // this CTA's tiles
  if (tid == 0) {
    misc[2] = (prm.err != nullptr && *reinterpret_cast<volatile int*>(prm.err) == SPARSEPR_ERR_TIMEOUT) || (base & 1023u) != 0;
    if ((base & 1023u) != 0) set_error(prm.err, SPARSEPR_ERR_CUDA);
    for (int i = 0; i < kCorrBars; ++i) mbar_init(bar(i), i >= C_READ && i < C_MAP ? 256 : 1);     // C_READ, C_CONV
    misc[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (misc[2]) return;
  if (warp == 9) tmem_alloc(base + SM::misc, 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(FULLW, (uint32_t)misc[0], 0);
  volatile int* abort_flag = &misc[1];

  if (warp == 8) {
    int head = -1;
    for (int k = 0; k < count; ++k) {
      const int u = k & 1, bh = (g0 + k) / n_tiles, row0 = ((g0 + k) % n_tiles) * kCorrTile;
      if (!__all_sync(FULLW, mbar_wait(bar(C_EMPTY + u), ((k >> 1) & 1) ^ 1, abort_flag))) break;     // (the first pass completes at once)
      if (lane == 0) {
        const uint32_t xb = base + SM::xh + u * 2 * kCorrTileBytes<D>;
        mbar_expect_tx(bar(C_FULL + u), 2 * kCorrTileBytes<D>);
        for (int c = 0; c < kHalves; ++c) {
          tma_load_4d(xb + c * kCorrHalf, &mapO, bar(C_FULL + u), 64 * c, row0, bh % prm.H, bh / prm.H);
          tma_load_4d(xb + kCorrTileBytes<D> + c * kCorrHalf, &mapL, bar(C_FULL + u), 64 * c, row0, bh, 0);
        }
      }
      __syncwarp();
      if (bh != head) {                                          // the products with the map before must be complete
        if (k > 0 && !__all_sync(FULLW, mbar_wait(bar(C_DONE + (u ^ 1)), ((k - 1) >> 1) & 1, abort_flag))) break;
        head = bh;
        if (lane == 0) {
          mbar_expect_tx(bar(C_MAP), map_words(D) * SM::map_bytes);
          for (int w = 0; w < map_words(D); ++w)
            for (int c = 0; c < kHalves; ++c) tma_load_4d(base + SM::a + w * SM::map_bytes + c * kMapHalf, &mapA, bar(C_MAP), 64 * c, 0, w * prm.BH + bh, 0);
        }
        __syncwarp();
      }
    }
  } else if (warp == 9) {
    // (the whole warp walks the tiles and one elected lane issues: see attention_tc.cu)
    const uint64_t ad = smem_desc(base + SM::a, 16);
    const uint32_t idesc = idesc_bf16(0, D);
    int head = -1, maps = 0;
    bool ok = true;
    for (int k = 0; k < count && ok; ++k) {
      const int u = k & 1, bh = (g0 + k) / n_tiles;
      if (bh != head) { ok = mbar_wait(bar(C_MAP), maps & 1, abort_flag); head = bh; ++maps; }
      ok = ok && mbar_wait(bar(C_READ + u), ((k >> 1) & 1) ^ 1, abort_flag);
      ok = __all_sync(FULLW, ok && mbar_wait(bar((kHalvesOfX ? C_CONV : C_FULL) + u), (k >> 1) & 1, abort_flag));
      if (!ok) break;
      tc_fence_after();
      const uint64_t hd = smem_desc(base + SM::xh + u * 2 * kCorrTileBytes<D>, 16);
      const uint64_t ld = smem_desc(base + (kHalvesOfX ? SM::xc + u * 2 * kCorrTileBytes<D> : SM::xl + u * 2 * kCorrTileBytes<D>), 16);
      const uint32_t d = tmem + 128u * u;
      if (elect_one()) {
        auto product = [&](uint64_t xd, int word, bool first) {          // (X A)[m][n] = sum_k X[m][k] At[n][k]
          const uint64_t wd = ad + (uint64_t)(word * (SM::map_bytes >> 4));
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint64_t koff = (uint64_t)((kk >> 2) * (kCorrHalf >> 4) + (kk & 3) * 2), aoff = (uint64_t)((kk >> 2) * (kMapHalf >> 4) + (kk & 3) * 2);
            umma_bf16(d, xd + koff, wd + aoff, idesc, !first || kk > 0);
          }
        };
        if constexpr (kHalvesOfX) {                                      // smallest first
          product(hd, 2, true);
          product(ld, 1, false);
          product(ld + (uint64_t)(kCorrTileBytes<D> >> 4), 0, false);
          product(hd, 1, false);
          product(ld, 0, false);
          product(hd, 0, false);
        } else {
          product(hd, 0, true);
          product(ld, 0, false);
          product(hd, 1, false);
        }
        umma_commit(bar(C_DONE + u));
      }
      __syncwarp();
    }
  } else {
    // ---- epilogue: a thread takes half the columns of a row -----------------------------------------------------
    const int wq = warp & 3, hh = warp >> 2, row = wq * 32 + lane;
    bool ok = true;
    for (int k = 0; k < count; ++k) {
      const int u = k & 1, bh = (g0 + k) / n_tiles, row0 = ((g0 + k) % n_tiles) * kCorrTile;
      if constexpr (kHalvesOfX) {
        ok = __all_sync(FULLW, ok && mbar_wait(bar(C_FULL + u), (k >> 1) & 1, abort_flag));
        if (ok) {
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            const uint32_t at = row * 128 + (((hh * 4 + ch) ^ (row & 7)) << 4);
            const uint4 rh = *reinterpret_cast<const uint4*>(smem_raw + SM::xh + u * 2 * kCorrTileBytes<D> + at);
            const uint4 rl = *reinterpret_cast<const uint4*>(smem_raw + SM::xl + u * 2 * kCorrTileBytes<D> + at);
            const uint32_t h[4] = {rh.x, rh.y, rh.z, rh.w}, l[4] = {rl.x, rl.y, rl.z, rl.w};
            uint32_t w[4], w2[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float r0 = __uint_as_float(__byte_perm(l[e], h[e], 0x5410)) - __uint_as_float(h[e] << 16);
              const float r1 = __uint_as_float(__byte_perm(l[e], h[e], 0x7632)) - __uint_as_float(h[e] & 0xFFFF0000u);
              w[e] = pack_bf16x2(r0, r1);
              w2[e] = pack_bf16x2_rest(r0, r1, w[e]);
            }
            unsigned char* xw = smem_raw + SM::xc + u * 2 * kCorrTileBytes<D> + at;
            *reinterpret_cast<uint4*>(xw) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4*>(xw + kCorrTileBytes<D>) = make_uint4(w2[0], w2[1], w2[2], w2[3]);
          }
          fence_async_smem();                                            // the product reads what was written
          mbar_arrive(bar(C_CONV + u));
        }
      }
      ok = __all_sync(FULLW, ok && mbar_wait(bar(C_DONE + u), (k >> 1) & 1, abort_flag));
      tc_fence_after();
      const float* cv = prm.c + (i64)bh * D;
      unsigned char* hrow = smem_raw + SM::xh + u * 2 * kCorrTileBytes<D> + row * 128;
      const unsigned char* lrow = hrow + kCorrTileBytes<D>;
#pragma unroll
      for (int q2 = 0; q2 < D / 64; ++q2) {
        if (!ok) break;
        const int q = hh * (D / 64) + q2;
        float t[32];
        tmem_ld32(tmem + ((uint32_t)(wq * 32) << 16) + 128u * u + q * 32, t);
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          const int j = (q & 1) * 4 + ch;                                // 16-byte chunk of the 128-byte row
          const uint32_t so = (q >> 1) * kCorrHalf + ((j ^ (row & 7)) << 4);
          const uint4 rh = *reinterpret_cast<const uint4*>(hrow + so);
          const uint4 rl = *reinterpret_cast<const uint4*>(lrow + so);
          const __nv_bfloat162* hp = reinterpret_cast<const __nv_bfloat162*>(&rh);
          const __nv_bfloat162* lp = reinterpret_cast<const __nv_bfloat162*>(&rl);
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float2 x;
            if constexpr (kHalvesOfX) {
              const uint32_t h = reinterpret_cast<const uint32_t*>(&rh)[e], l = reinterpret_cast<const uint32_t*>(&rl)[e];
              x = make_float2(__uint_as_float(__byte_perm(l, h, 0x5410)), __uint_as_float(__byte_perm(l, h, 0x7632)));
            } else {
              const float2 fh = __bfloat1622float2(hp[e]), fl = __bfloat1622float2(lp[e]);
              x = make_float2(fh.x + fl.x, fh.y + fl.y);
            }
            const int col = q * 32 + ch * 8 + 2 * e;
            w[e] = pack_bf16x2(x.x + t[ch * 8 + 2 * e] + cv[col], x.y + t[ch * 8 + 2 * e + 1] + cv[col + 1]);
          }
          *reinterpret_cast<uint4*>(hrow + so) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      tc_fence_before();
      mbar_arrive(bar(C_READ + u));
      fence_async_smem();                                                // the copy below reads what was written above
      asm volatile("bar.sync 1, 256;" ::: "memory");                     // (passed whatever happened)
      if (tid == 0 && ok) {                                                    // rows past the end of the tensor are not written
        const uint32_t xb = base + SM::xh + u * 2 * kCorrTileBytes<D>;
        for (int c = 0; c < kHalves; ++c) tma_store_4d(&mapO, xb + c * kCorrHalf, 64 * c, row0, bh % prm.H, bh / prm.H);
        bulk_store_wait_read();
        mbar_arrive(bar(C_EMPTY + u));
      }
      __syncwarp();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    for (int k = 0; k < 64; ++k) __nanosleep(1000);      // let copies that may still be in flight land
    if (tid == 0) set_error(prm.err, SPARSEPR_ERR_TIMEOUT);
    __syncthreads();
  }
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

// Self-test of the bounded wait: one warp waits on an mbarrier that nobody arrives at (no copy in flight, no
// tensor memory held), with a limit of 2^16 cycles; the wait gives up, the error word receives
// SPARSEPR_ERR_TIMEOUT, the kernel returns normally and the context stays usable.
__global__ void k_selftest_bounded_wait(int* err, long long limit) {
  __shared__ __align__(8) unsigned long long sbar;
  __shared__ int abort_flag;
  const uint32_t bar = smem_u32(&sbar);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const bool ok = mbar_wait_limit(bar, 0, &abort_flag, limit);
  __syncthreads();
  if (threadIdx.x == 0 && (!ok || abort_flag)) set_error(err, SPARSEPR_ERR_TIMEOUT);
}

}  // namespace tc

void launch_selftest_bounded_wait(int* err, cudaStream_t st) { tc::k_selftest_bounded_wait<<<1, 32, 0, st>>>(err, 1ll << 16); }

cudaError_t init_correction_tc() {
  const cudaError_t e = cudaFuncSetAttribute(tc::k_correction_tc<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::CorrSmem<128>::total);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(tc::k_correction_tc<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::CorrSmem<64>::total);
}

bool launch_correction_tc(const float* c, const __nv_bfloat16* At, const void* O_lo, void* O, const i64* os, int BH,
                          int H, int N, int d, int* err, cudaStream_t st) {
  using namespace tc;
  CUtensorMap mo, ml, ma;
  if (!make_map(&mo, O, d, N, H, BH / H, os[0], os[1], os[2], kCorrTile) ||
      !make_map(&ml, O_lo, d, N, BH, 1, 0, (i64)N * d, d, kCorrTile) ||
      !make_map(&ma, At, d, d, map_words(d) * BH, 1, 0, (i64)d * d, d, d))
    return false;
  CorrParams p{};
  p.BH = BH; p.H = H; p.N = N; p.c = c; p.err = err;
  const int grid = (int)std::min<i64>(sm_count(), (i64)BH * ((N + kCorrTile - 1) / kCorrTile));
  if (d == 128) k_correction_tc<128><<<grid, kCorrThreads, CorrSmem<128>::total, st>>>(mo, ml, ma, p);
  else k_correction_tc<64><<<grid, kCorrThreads, CorrSmem<64>::total, st>>>(mo, ml, ma, p);
  return true;
}

}  // namespace spr
