// Small-batch tensor-core scan of 4-bit codes (Sec. II-B step 5 as a skinny
// GEMM): vectors on the MMA's M dimension (128 per tile), queries on N (16 or
// 32 columns), the decoded fp16 centroids as the A operand in tensor memory.
//
// What bounds it.  A batch of up to 32 queries reads each code once, so HBM
// bounds it from below (767 MB at 999,000 x 1536: 115 us at 6.7 TB/s).  The
// shared-memory datapath (128 bytes per cycle per SM) is the nearer limit: per
// 128-vector tile at d = 1536 the codes come in by TMA (768 cycles) and are
// read once (768), one 4-byte lookup per packed byte turns them into two fp16
// centroids (3,072), and the MMAs read the query block (N = 16: 384; 32: 768):
// about 5,000 cycles per tile, 124 us at 999,000 vectors.  The decoded values
// go from registers to tensor memory (tcgen05.st), so they cross shared memory
// neither when written nor when the MMA reads them; decoding into shared
// memory instead (k_scan_mma) adds 4 bytes per packed byte each way, and its
// register decode costs about 21 integer instructions per 8 codes, at 64 lanes
// per cycle and SM.  The query block of the whole contraction stays in shared
// memory for the kernel's life (N x d fp16), so no query bytes are re-read per
// tile.  (Decoding a quarter of the words with byte permutes instead of lookups,
// to relieve that datapath, was slower, 185 us against 170: with 27 warps the
// decoders are as close to the issue rate.)  Measured at 999,000 x 1536, whole
// searches: one query, top-5, 217 us (lookup scan) -> 162; 32 queries 484 us
// (k_scan_mma) -> 216; four queries of 1,000 tenants 857 -> 175; eight queries over
// 250,007 rows 425 -> 79.
//
// Two uses:
//  * BOUND = false, 16 <= nq <= 32: the scores themselves, fp16 products with
//    float32 accumulation, the same operand rounding as k_scan_mma.
//  * BOUND = true, nq < 16: an exact float32 search.  The scan computes, per
//    vector, an upper bound U of the score the lookup scan would give: the
//    fp16 score plus a bound of everything it leaves out (the rounding of both
//    operands, summed exactly per query and codebook, and the accumulation
//    error).  Each CTA keeps the 32 best by U; k_rescore then takes the lookup
//    scan's float32 score of every candidate that can still be among the k
//    best and sorts by that.  The lists are checked: if a vector that a full
//    list dropped could still be among the k best, or anything is not finite,
//    the query's gate opens and the lookup scan runs for it after all.  Scores
//    and ids are those of the lookup scan, bit for bit.
//
// Roles (27 warps): 0-15 decoders in four groups of four warps (one warp per
// TMEM lane quarter; group g takes the 128-coordinate blocks it = g, g + 4,
// ...; block it goes to TMEM stage it % 6); 16-23 epilogue in two groups (one
// vector per thread, all queries); 24 code producer (TMA); 25, 26 MMA issuers.
// Waits are bounded as in every pipeline here.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>

#include "tq_internal.h"
#include "tq_kernels.h"
#include "tq_wait.cuh"
#include "tq_tc.cuh"
#include "tq_topk.cuh"

namespace tq {
namespace {

constexpr int TM_M = 128;                 // vectors per tile
constexpr int TM_GROUPS = 4;              // decoder groups
constexpr int TM_STAGES = 6;              // decoded blocks in tensor memory
constexpr int TM_ISSUERS = 2;             // MMA warps: block it goes to warp it % 2 and that warp's accumulator
constexpr int TM_DEC_WARPS = 4 * TM_GROUPS;
constexpr int TM_EPI0 = TM_DEC_WARPS, TM_PROD = TM_EPI0 + 8, TM_MMA = TM_PROD + 1;
constexpr int TM_THREADS = (TM_MMA + TM_ISSUERS) * 32;
constexpr int TM_BLK = 128;               // coordinates per decoded block (64 TMEM columns)
constexpr int TM_RAW = TM_M * 128;        // a raw code tile: 128 rows x 128 bytes, two blocks
constexpr int TM_MAX_CST = 8;
constexpr uint32_t TM_LUT = 256 * 256;    // entry (byte, lane) at byte * 256 + lane * 4
constexpr uint32_t TM_SMEM_MAX = 232448;  // 227 KB per block
// The upper half of each 256-byte table row is free (a byte permute makes the
// entry's address only with that row size): 8,192 words, of which 2 * N * 128
// hold two tiles' candidate scores (and with 16 columns 2 * 128 their |scale|).
constexpr int TM_TILE_LIST = 2 * 16 * TM_M + 2 * TM_M;  // first word of the tile list (16 columns)
constexpr int TM_MAX_TILES = 8192 - TM_TILE_LIST;
constexpr int TM_LIST = kTmMaxK;          // entries of a query's list in a CTA (one per lane)
constexpr uint32_t TM_A_COL = 128;        // TMEM: two sets of two accumulators of N <= 32 columns, then the stages
// misc area (after the raw tiles): per-query values, masks, barriers
struct TmMisc {
  static constexpr uint32_t th = 0, bias = 128, err = 256, us = 384;  // float [32] each
  static constexpr uint32_t mask = 512;                               // uint32 [2][N][4], at most 1,024 bytes
  static constexpr uint32_t bars = 1536;                              // 35 mbarriers
  static constexpr uint32_t slot = bars + 36 * 8;                     // TMEM address, abort flag
  static constexpr uint32_t any = slot + 16;                          // uint32 [2][4]: queries with a candidate, by warp
  static constexpr uint32_t tiles = any + 32;                         // int: tiles in the list
  static constexpr uint32_t total = tiles + 4;
};
static_assert(TmMisc::total <= 2048, "misc area");

__host__ __device__ constexpr uint32_t tm_b_bytes(int d, int N) { return (uint32_t)(d / 64) * N * 128; }

// Raw code stages that fit (even, so that a stage always serves the same two
// decoder groups, which makes the parity waits sound), 0 if fewer than two do.
int tm_stages(int d, int N) {
  const int64_t left = (int64_t)TM_SMEM_MAX - 1024 - 2048 - TM_LUT - tm_b_bytes(d, N);
  if (left < 2 * TM_RAW) return 0;
  return (int)std::min<int64_t>(TM_MAX_CST, left / TM_RAW) & ~1;
}

__host__ __device__ constexpr uint32_t tm_idesc(int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TM_M >> 4) << 24);
}

// warp_wait whose usual case, a phase already complete, is one poll per lane.
__device__ __forceinline__ bool all_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err,
                                         int where) {
  if (__all_sync(FULL, mbar_try_wait(bar, parity))) return true;
  return warp_wait(bar, parity, abort_flag, err, where);
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

// Magnitudes the bounds are derived for (no product below over- or underflows).
constexpr float TM_BIG = 0x1p60f, TM_SMALL = 0x1p-50f, TM_SMALL_SCALE = 0x1p-40f;

// Sorts one key per lane across the warp, best first.
__device__ __noinline__ uint64_t warp_sort_keys(uint64_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int size = 2; size <= 32; size <<= 1)
#pragma unroll 1
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const uint64_t o = __shfl_xor_sync(FULL, x, stride);
      x = (o > x) == (((lane & stride) == 0) == ((lane & size) == 0)) ? o : x;  // the better, or the worse
    }
  return x;
}

// The 32 best of a sorted list and another one held in reverse (lane 31 the best).
__device__ __forceinline__ uint64_t list_merge(uint64_t list, uint64_t reversed) {
  const int lane = threadIdx.x & 31;
  list = reversed > list ? reversed : list;  // the 32 best, as a bitonic sequence
#pragma unroll
  for (int stride = 16; stride; stride >>= 1) {
    const uint64_t o = __shfl_xor_sync(FULL, list, stride);
    list = (o > list) == ((lane & stride) == 0) ? o : list;
  }
  return list;
}

// A warp's sorted list of 32 keys (one per lane, best first) takes up to 32
// candidates (one per lane, 0 where there is none; `mask`: the lanes that hold
// one).  A few go in one by one (rank by ballot, shift by shuffle); more are
// sorted and merged.
__device__ __noinline__ uint64_t list_add(uint64_t list, uint64_t cand, uint32_t mask) {
  const int lane = threadIdx.x & 31;
  if (__popc(mask) <= 4) {
    while (mask) {
      const uint64_t c = __shfl_sync(FULL, cand, __ffs(mask) - 1);
      mask &= mask - 1;
      const int pos = __popc(__ballot_sync(FULL, list > c));
      const uint64_t up = __shfl_up_sync(FULL, list, 1);
      list = lane > pos ? up : lane == pos ? c : list;
    }
    return list;
  }
#pragma unroll
  for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const uint64_t o = __shfl_xor_sync(FULL, cand, stride);
      const bool up = ((lane & stride) == 0) == ((lane & size) == 0);  // keeps the better of the two
      cand = (o > cand) == up ? o : cand;
    }
  return list_merge(list, __shfl_sync(FULL, cand, 31 - lane));
}

template <int N, bool BOUND, bool MASKED>
__global__ void __launch_bounds__(TM_THREADS, 1)
k_scan_tm(const __grid_constant__ CUtensorMap codes_map, const float* __restrict__ qrot,
          const float* __restrict__ centroids, const float* __restrict__ scale, const uint32_t* __restrict__ del,
          const uint32_t* __restrict__ dense, const uint32_t* __restrict__ allow_bits, int words,
          const uint32_t* __restrict__ bmask, int mask_words, int fblock, const float* __restrict__ bias, int n,
          int nq, int d, int k, int C, int cst, float* __restrict__ cand_s,
          int* __restrict__ cand_i, int* __restrict__ err, int* __restrict__ force, uint32_t* __restrict__ gth,
          float* __restrict__ lows) {
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* base = smem_dyn + ((1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u);
  unsigned char* lut = base;
  unsigned char* sB = base + TM_LUT;
  unsigned char* sRaw = sB + tm_b_bytes(d, N);
  unsigned char* misc = sRaw + (size_t)cst * TM_RAW;
  float* s_th = reinterpret_cast<float*>(misc + TmMisc::th);
  float* s_bias = reinterpret_cast<float*>(misc + TmMisc::bias);
  float* s_err = reinterpret_cast<float*>(misc + TmMisc::err);
  float* s_us = reinterpret_cast<float*>(misc + TmMisc::us);
  uint32_t* s_mask = reinterpret_cast<uint32_t*>(misc + TmMisc::mask);
  uint32_t* s_any = reinterpret_cast<uint32_t*>(misc + TmMisc::any);
  uint64_t* bars = reinterpret_cast<uint64_t*>(misc + TmMisc::bars);
  uint64_t* cfull = bars;            // [cst] raw code tile landed
  uint64_t* cempty = bars + 8;       // [cst] raw code tile read
  uint64_t* dec = bars + 16;         // [7] decoded block in tensor memory
  uint64_t* tfree = bars + 23;       // [7] MMAs done with the decoded block
  uint64_t* acc_full = bars + 30;    // [2] accumulator complete
  uint64_t* acc_empty = bars + 32;   // [2] accumulator read out
  uint64_t* fin = bars + 34;         // every MMA of this CTA complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc + TmMisc::slot);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + TmMisc::slot + 4);
  auto gapw = [&](int w) { return lut + ((uint32_t)w >> 5) * 256u + 128u + ((uint32_t)w & 31u) * 4u; };

  const int tid = threadIdx.x, warp = __shfl_sync(FULL, tid >> 5, 0), lane = tid & 31;
  const int ntiles = row_tiles(n, TM_M);
  const int all_tiles = (int)blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int raws = d >> 8;        // raw code tiles per vector tile
  const int blks = d / TM_BLK;    // decoded blocks per vector tile
  // With block masks (MASKED: BOUND searches with a filter) the CTA walks the tiles
  // that hold a filter block some query allows (Sec. III-B: skipped before any
  // code byte is read), listed behind the candidate slots.
  int my_tiles = all_tiles;  // (MASKED: set when the list is complete)
  int* s_tiles = reinterpret_cast<int*>(misc + TmMisc::tiles);
  auto tile_at = [&](int i) {
    return MASKED ? *reinterpret_cast<const int*>(gapw(TM_TILE_LIST + i))
                          : (int)blockIdx.x + i * (int)gridDim.x;
  };

  griddep_launch_dependents();
  if (tid == 0) {
    for (int s = 0; s < cst; ++s) {
      mbar_init(cfull + s, 1);
      mbar_init(cempty + s, 8);  // the two groups' warps
    }
    for (int s = 0; s < TM_STAGES; ++s) {
      mbar_init(dec + s, 4);
      mbar_init(tfree + s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(acc_full + s, TM_ISSUERS);
      mbar_init(acc_empty + s, 4);
    }
    mbar_init(fin, TM_ISSUERS);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == TM_PROD) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto issue = [&](int ld) {
    const int s = ld % cst;
    const int t = tile_at(ld / raws);
    mbar_arrive_expect_tx(cfull + s, TM_RAW);
    tma_load_2d(sRaw + (size_t)s * TM_RAW, &codes_map, (ld % raws) * 128, t * TM_M, cfull + s);
  };
  int issued = 0;
  if (warp == TM_PROD && lane == 0 && !MASKED)  // the first code tiles go out before the tables are built
    for (; issued < cst && issued < all_tiles * raws; ++issued) issue(issued);

  // the codebook in fp16: BOUND scales it by a power of two to [1, 2) at its
  // largest centroid and takes the largest rounding error
  float cmax = 0.f, cerr = 0.f, cs = 1.f;
  if (BOUND) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float v = fabsf(__ldg(centroids + i));
      cmax = v > cmax || isnan(v) ? v : cmax;  // a NaN stays
    }
    if (cmax >= TM_SMALL && cmax <= TM_BIG) cs = pow2f(-exp2_of(cmax));
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float v = __ldg(centroids + i) * cs;
      cerr = fmaxf(cerr, fabsf(v - __half2float(__float2half_rn(v))));
    }
  }
  for (int i = tid; i < 256 * 8; i += TM_THREADS) {  // four lanes' copies at a time
    const int x = i >> 3;
    const __half2 h = __floats2half2_rn(__ldg(centroids + (x & 15)) * cs, __ldg(centroids + (x >> 4)) * cs);
    const uint32_t v = *reinterpret_cast<const uint32_t*>(&h);
    *reinterpret_cast<uint4*>(lut + x * 256 + (i & 7) * 16) = make_uint4(v, v, v, v);
  }
  for (int i = tid; i < 2 * N * 4; i += TM_THREADS) s_mask[i] = 0u;
  if (tid == 0) *s_tiles = 0;
  if (MASKED) __syncthreads();
  griddep_wait();  // the rotated queries (and allow bitmaps, TQ+ terms) are written
  if (MASKED) {
    const int per = TM_M / fblock;  // 2 or 4 filter blocks a tile, in one mask word
    for (int i = tid; i < all_tiles; i += TM_THREADS) {
      const int t = (int)blockIdx.x + i * (int)gridDim.x, b = t * per;
      uint32_t any = 0;
      for (int q = 0; q < nq; ++q) any |= __ldg(bmask + (size_t)q * mask_words + (b >> 5));
      if ((any >> (b & 31)) & ((1u << per) - 1u))
        *reinterpret_cast<int*>(gapw(TM_TILE_LIST + atomicAdd(s_tiles, 1))) = t;
    }
  }
  // The query block: a warp per column, d fp16 values, K-major with the
  // 128-byte swizzle in blocks of 64 coordinates; columns past nq are zero.
  for (int q = warp; q < N; q += TM_THREADS / 32) {
    const float4* src = reinterpret_cast<const float4*>(qrot + (size_t)q * d);
    float qs = 1.f, l1 = 0.f, mx = 0.f, dq = 0.f;
    bool fine = true;
    if (BOUND && q < nq) {
#pragma unroll 6
      for (int c = lane; c < d / 4; c += 32) {
        const float4 v = src[c];
        const float m = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
        mx = fmaxf(mx, m);
        l1 += (fabsf(v.x) + fabsf(v.y)) + (fabsf(v.z) + fabsf(v.w));
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
        l1 += __shfl_xor_sync(FULL, l1, o);
      }
      // (a NaN query leaves l1 NaN; comparisons with it are false)
      const float qc = l1 * cmax;
      fine = cmax <= TM_BIG && cmax >= TM_SMALL && (mx == 0.f || mx >= TM_SMALL) && l1 <= TM_BIG && qc <= TM_BIG &&
             (mx == 0.f || qc >= 0x1p-60f);
      if (fine && mx > 0.f) qs = pow2f(13 - exp2_of(mx));
    }
#pragma unroll 3
    for (int c = lane; c < d / 8; c += 32) {
      uint32_t o[4] = {0, 0, 0, 0};
      if (q < nq) {
        const float4 a = src[2 * c], b = src[2 * c + 1];
        const float f[8] = {a.x * qs, a.y * qs, a.z * qs, a.w * qs, b.x * qs, b.y * qs, b.z * qs, b.w * qs};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const __half2 h = __floats2half2_rn(f[2 * j], f[2 * j + 1]);
          o[j] = *reinterpret_cast<const uint32_t*>(&h);
          if (BOUND) dq += fabsf(f[2 * j] - __low2float(h)) + fabsf(f[2 * j + 1] - __high2float(h));
        }
      }
      *reinterpret_cast<uint4*>(sB + (c >> 3) * (N * 128) + sw128_offset(q, c & 7)) =
          make_uint4(o[0], o[1], o[2], o[3]);
    }
    float e = 0.f, us = 1.f, bq = 0.f;
    if (q < nq) bq = bias ? bias[q] : 0.f;
    if (BOUND && q < nq) {
#pragma unroll
      for (int o = 16; o; o >>= 1) dq += __shfl_xor_sync(FULL, dq, o);
      fine = fine && fabsf(bq) <= TM_BIG;
      if (fine) {
        // |fp16 score - lookup score| <= sum |q16 c16 - q c| (operand
        // rounding) + accumulation: the MMAs add d products to a float32 sum
        // in d / 16 steps.  How a step rounds is not documented; if it aligns
        // its 17 terms to the largest and cuts below its last bit, as was
        // measured on earlier tensor cores (Fasi, Higham, Mikaitis and Pranesh,
        // "Numerical behavior of NVIDIA tensor cores", 2021), d * 2^-23 of
        // sum |q c| covers it twice over.  On GB300 the largest error of
        // products far apart in magnitude, d = 256 and 2,048, was 0.025 of
        // that (test_gpu_scan_tm.py).  2^-17 covers the lookup scan's own
        // float32 rounding and the additions and products here.
        const float de = dq / qs, ce = cerr / cs;
        e = (l1 + de) * ce + de * cmax + l1 * cmax * ((float)d * 0x1p-23f + 0x1p-17f) + fabsf(bq) * 0x1p-20f;
        e *= 1.0001f;
        us = 1.0f / (qs * cs);
      } else if (lane == 0) {
        atomicExch(force, 1);
      }
    }
    if (lane == 0) {
      s_th[q] = -INFINITY;
      s_bias[q] = bq;
      s_err[q] = e;
      s_us[q] = us;
    }
  }
  fence_proxy_async();  // the query block is read by the MMAs
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (MASKED) my_tiles = *s_tiles;
  const int total_ld = my_tiles * raws, total_it = my_tiles * blks;

  if (warp == TM_PROD) {
    // ------------------------------------------------- code tiles (TMA, HBM)
    if (lane == 0) {
      for (; issued < total_ld; ++issued) {
        const int s = issued % cst, use = issued / cst;
        if (use > 0 && !mbar_wait(cempty + s, (use - 1) & 1, abort_flag, err, 61)) break;
        issue(issued);
      }
      // never leave with copies in flight: wait (bounded) for the last one of each stage
      for (int s = 0; s < cst && s < issued; ++s) mbar_wait_drain(cfull + s, ((issued - 1 - s) / cst) & 1);
    }
  } else if (warp >= TM_MMA) {
    // --------------------------------------------------------- MMA issuers
    // The whole warp runs the loop and one elected lane issues, so that the
    // descriptors stay in uniform registers (14 cycles per MMA; 46 from a
    // single-lane branch).  With the waits and commits a block of 8 MMAs still
    // takes one warp about 240 cycles, more than half of a block's share of
    // the tile, so two warps take turns, each with its own accumulator (the
    // epilogue adds them).  Waiting by parity is sound: stage it % 6 always
    // serves the same issuer.
    const int w = warp - TM_MMA;
    const uint64_t b0 = sw128_desc(__shfl_sync(FULL, smem_u32(sB), 0));
    const uint32_t tm = __shfl_sync(FULL, tmem, 0);
    int kb = w, tile_i = 0, st = w, par = 0;
    for (int it = w; it < total_it; it += TM_ISSUERS) {
      const int set = tile_i & 1;
      if (kb == w && tile_i >= 2 && !all_wait(acc_empty + set, ((tile_i >> 1) - 1) & 1, abort_flag, err, 62)) break;
      if (!all_wait(dec + st, par, abort_flag, err, 63)) break;
      tc_fence_after();
      const uint32_t at = tm + TM_A_COL + (uint32_t)st * 64u, dt = tm + (uint32_t)((set * TM_ISSUERS + w) * N);
      const uint64_t bd = b0 + (uint64_t)((uint32_t)kb * (2u * N * 128u >> 4));
      const uint32_t more = kb != w;
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < TM_BLK / 16; ++kk)
          mma_f16_ta(dt, at + (uint32_t)kk * 8u, bd + (uint64_t)((kk >> 2) * (N * 8) + (kk & 3) * 2), tm_idesc(N),
                     kk ? 1u : more);
        mma_commit(tfree + st);
        if (kb + TM_ISSUERS >= blks) mma_commit(acc_full + set);
      }
      __syncwarp();
      if ((kb += TM_ISSUERS) >= blks) {
        kb = w;
        ++tile_i;
      }
      if ((st += TM_ISSUERS) >= TM_STAGES) {
        st = w;
        par ^= 1;
      }
    }
    if (elect_one()) {
      mma_commit(fin);
      mbar_wait_drain(fin, 0);
    }
    __syncwarp();
  } else if (warp < TM_DEC_WARPS) {
    // ------------------------------------------------------------ decoders
    const int g = warp >> 2, quarter = warp & 3, row = quarter * 32 + lane;
    const uint32_t lane4 = (uint32_t)lane * 4u;
    const uint32_t tq = tmem + ((uint32_t)(quarter * 32) << 16) + TM_A_COL;
    // Waiting for block it - 6's MMAs by parity is sound: the group's own
    // block it - 4 waited for block it - 10 of the same issuer, so block
    // it - 12, the stage's use before, is long complete.
    for (int it = g; it < total_it; it += TM_GROUPS) {
      const int ld = it >> 1, sb = it & 1, s = ld % cst;
      const int st = it % TM_STAGES;
      const uint32_t ta = tq + (uint32_t)st * 64u;
      if (!all_wait(cfull + s, (ld / cst) & 1, abort_flag, err, 64)) break;
      const unsigned char* rp = sRaw + (size_t)s * TM_RAW + row * 128;
      uint4 w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        w[j] = *reinterpret_cast<const uint4*>(rp + (((sb * 4 + j) ^ (row & 7)) << 4));
      __syncwarp();
      if (lane == 0) mbar_arrive(cempty + s);  // (releases after the warp's reads)
      bool ok = true;
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // 64 coordinates: 32 bytes, 32 TMEM columns
        uint32_t o[32];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint32_t x[4] = {w[2 * h + j].x, w[2 * h + j].y, w[2 * h + j].z, w[2 * h + j].w};
#pragma unroll
          for (int i = 0; i < 16; ++i)
            o[j * 16 + i] = *reinterpret_cast<const uint32_t*>(
                lut + __byte_perm(x[i >> 2], lane4, 0x5504u | ((uint32_t)(i & 3) << 4)));
        }
        if (h == 0) {
          ok = it < TM_STAGES || all_wait(tfree + st, ((it / TM_STAGES) - 1) & 1, abort_flag, err, 65);
          if (!ok) break;
          tc_fence_after();
        }
        tmem_st32(ta + (uint32_t)h * 32u, o);
      }
      if (!ok) break;
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(dec + st);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // Two groups of four warps take turns on tiles (group p the accumulators
    // of set p).  One vector per thread: its scores against every query are
    // compared with the queries' thresholds; those that reach theirs go to the
    // group's slots (one word per vector and query) with a bit each.  After a
    // barrier each warp takes the candidates of its N / 4 queries (q = 4 j + e),
    // up to 32 at a time, into the group's lists: 32 entries, one per lane,
    // best first, in registers.  (Inserting them one by one into a list in
    // shared memory took about 50 us for the first tile alone; with one group
    // the lists of 32 queries took longer than the tiles' decoding: 250 us
    // for 32 queries over 999,000 rows.)
    const int grp = (warp - TM_EPI0) >> 2, e = warp & 3, row = e * 32 + lane;
    const uint32_t qmask = nq >= 32 ? 0xFFFFFFFFu : (1u << nq) - 1u;
    uint64_t lst[N / 4];
    float smax[BOUND ? N / 4 : 1];  // BOUND: per lane, the largest |scale| of the list's candidates so far
#pragma unroll
    for (int j = 0; j < N / 4; ++j) {
      lst[j] = rank_key(-INFINITY, INT_MAX);
      if (BOUND) smax[j] = 0.f;
    }
    bool odd_scale = false;
    // the next tile's scale (and tenant) of this thread's vector, loaded a tile ahead
    float sc_next = 0.f;
    uint32_t tn_next = 0;
    auto fetch = [&](int tile_i) {
      const int v = tile_i < my_tiles ? tile_at(tile_i) * TM_M + row : n;
      const bool in = v < n;
      sc_next = in ? (scale ? __ldg(scale + v) : 1.0f) : 0.f;
      tn_next = in && allow_bits ? __ldg(dense + v) : 0u;
    };
    fetch(grp);
    for (int tile_i = grp; tile_i < my_tiles; tile_i += 2) {
      const int t = tile_at(tile_i);
      const int v = t * TM_M + row;
      const bool valid = v < n;
      const float sc = sc_next, asc = fabsf(sc);
      const uint32_t tn = tn_next;
      fetch(tile_i + 2);
      if (BOUND && !(asc <= TM_BIG && (sc == 0.f || asc >= TM_SMALL_SCALE))) odd_scale = true;
      const bool ok = all_wait(acc_full + grp, (tile_i >> 1) & 1, abort_flag, err, 66);
      uint32_t any_all = 0;
      if (ok) {
        tc_fence_after();
        const uint32_t tb = tmem + ((uint32_t)(32 * e) << 16) + (uint32_t)(grp * TM_ISSUERS * N);
#pragma unroll
        for (int c = 0; c < N; c += 16) {
          float r[16];
          {
            uint32_t ra[16], rb[16];
            tmem_ld16_issue(tb + (uint32_t)c, ra);
            tmem_ld16_issue(tb + (uint32_t)(N + c), rb);
            tmem_wait16(ra);
            tmem_wait16(rb);
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] = __uint_as_float(ra[i]) + __uint_as_float(rb[i]);
          }
          if (c + 16 == N) {  // the accumulators are read out
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty + grp);
          }
          uint32_t m = 0;  // bit i: query c + i
#pragma unroll
          for (int q = 0; q < 16; q += 4) {
            if (c + q >= nq) break;
            const float4 th4 = *reinterpret_cast<const float4*>(s_th + c + q);
            const float4 b4 = *reinterpret_cast<const float4*>(s_bias + c + q);
            const float th[4] = {th4.x, th4.y, th4.z, th4.w}, bq[4] = {b4.x, b4.y, b4.z, b4.w};
            if constexpr (BOUND) {
              const float4 u4 = *reinterpret_cast<const float4*>(s_us + c + q);
              const float4 e4 = *reinterpret_cast<const float4*>(s_err + c + q);
              const float us[4] = {u4.x, u4.y, u4.z, u4.w}, ee[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
              for (int j = 0; j < 4; ++j) r[q + j] = fmaf(asc, ee[j], fmaf(r[q + j], us[j], bq[j]) * sc);
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j) r[q + j] = (r[q + j] + bq[j]) * sc;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) m |= (r[q + j] >= th[j] ? 1u : 0u) << (q + j);
          }
          m = valid ? m & (qmask >> c) : 0u;
          if (!__any_sync(FULL, m != 0u)) continue;
          if (m && tombstoned(del, v)) m = 0u;  // a deleted row never enters a list
          if (allow_bits) {                     // nor does one of a tenant the query does not allow (Sec. III-B)
            uint32_t left = m;
            while (left) {
              const int q = __ffs(left) - 1;
              left &= left - 1;
              if (!((__ldg(allow_bits + (size_t)(c + q) * words + (tn >> 5)) >> (tn & 31)) & 1u)) m &= ~(1u << q);
            }
          }
          __syncwarp();
          const uint32_t any = __reduce_or_sync(FULL, m);
          any_all |= any << c;
          if (BOUND && m) *reinterpret_cast<float*>(gapw((2 * N + grp) * TM_M + row)) = asc;
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            if (!((any >> q) & 1u)) continue;  // the same for the whole warp
            const bool has = (m >> q) & 1u;
            const unsigned b = __ballot_sync(FULL, has);
            if (has) *reinterpret_cast<float*>(gapw((grp * N + c + q) * TM_M + row)) = r[q];
            if (lane == 0) s_mask[(grp * N + c + q) * 4 + e] = b;
          }
        }
      }
      if (lane == 0) s_any[grp * 4 + e] = any_all;
      // all four warps take the same decision, so none is left at a barrier
      int all_ok;
      asm volatile(
          "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n bar.red.and.pred q, %2, 128, p;\n"
          " selp.s32 %0, 1, 0, q;\n}"
          : "=r"(all_ok)
          : "r"(ok ? 1 : 0), "r"(1 + grp)
          : "memory");
      if (!all_ok) break;
      const uint4 ay = *reinterpret_cast<const uint4*>(s_any + grp * 4);
      const uint32_t todo = ay.x | ay.y | ay.z | ay.w;
      if (todo) {
        if (lane < N / 4 && 4 * lane + e < nq) {  // take the best threshold any CTA has published
          const uint32_t g = __ldcg(gth + 4 * lane + e);
          if (g && ordered(g) > s_th[4 * lane + e]) s_th[4 * lane + e] = ordered(g);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < N / 4; ++j) {
          const int q = 4 * j + e;
          if (!((todo >> q) & 1u)) continue;  // the same for the whole warp
          uint4* mp = reinterpret_cast<uint4*>(s_mask + (grp * N + q) * 4);
          const uint4 mm = *mp;
          __syncwarp();
          if (lane == 0) *mp = make_uint4(0, 0, 0, 0);
          uint64_t lj = lst[j];
#pragma unroll 1
          for (int i = 0; i < 4; ++i) {
            const uint32_t wv = i == 0 ? mm.x : i == 1 ? mm.y : i == 2 ? mm.z : mm.w;
            if (!wv) continue;
            const int r0 = i * 32 + lane;
            uint64_t cand = 0;
            if ((wv >> lane) & 1u) {
              cand = rank_key(*reinterpret_cast<const float*>(gapw((grp * N + q) * TM_M + r0)), t * TM_M + r0);
              if (BOUND) smax[j] = fmaxf(smax[j], *reinterpret_cast<const float*>(gapw((2 * N + grp) * TM_M + r0)));
            }
            lj = list_add(lj, cand, wv);
          }
          lst[j] = lj;
          // the k-th best score (BOUND: a lower bound of the k-th best float32
          // score: the k-th best U less twice the largest error bound): what
          // cannot reach it is not among the k best, in any CTA
          const uint64_t kk = __shfl_sync(FULL, lj, k - 1);
          float th = key_id(kk) == INT_MAX ? -INFINITY : key_score(kk);
          if (BOUND) {
            float sm = smax[j];
#pragma unroll
            for (int o = 16; o; o >>= 1) sm = fmaxf(sm, __shfl_xor_sync(FULL, sm, o));
            th -= 2.0002f * s_err[q] * sm;
            th -= fabsf(th) * 0x1p-22f;
          }
          float own = th;
          if (BOUND) own = fmaxf(own, key_score(__shfl_sync(FULL, lj, C - 1)));  // a full list takes only better ones
          if (lane == 0 && own > s_th[q]) {
            if (th > s_th[q]) atomicMax(gth + q, order_bits(th));
            s_th[q] = own;
          }
        }
      }
      // no slot is written for the group's next tile before all of this one's are read
      asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
    }
    if (BOUND && odd_scale) atomicExch(force, 1);
    // group 1 hands its lists to group 0 through its own (now idle) slots
    const int hand = N * TM_M;
    if (grp == 1) {
#pragma unroll
      for (int j = 0; j < N / 4; ++j) {
        const int w = hand + ((4 * j + e) * 32 + lane) * 2;  // 64-bit words stay within a 128-byte gap
        *reinterpret_cast<uint64_t*>(gapw(w)) = lst[j];
        if (BOUND) *reinterpret_cast<float*>(gapw(hand + N * 64 + (4 * j + e) * 32 + lane)) = smax[j];
      }
    }
    asm volatile("bar.sync 3, 256;" ::: "memory");
    if (grp == 0) {
#pragma unroll
      for (int j = 0; j < N / 4; ++j) {
        const int q = 4 * j + e;
        if (q >= nq) break;
        lst[j] = list_merge(lst[j], *reinterpret_cast<const uint64_t*>(gapw(hand + (q * 32 + 31 - lane) * 2)));
        if (lane < C) {
          const size_t o = ((size_t)q * gridDim.x + blockIdx.x) * C + lane;
          cand_s[o] = key_score(lst[j]);
          cand_i[o] = key_id(lst[j]);
        }
        if (BOUND) {  // lower bounds of the list's best and of its k-th best float32 score
          float sm = fmaxf(smax[j], *reinterpret_cast<const float*>(gapw(hand + N * 64 + q * 32 + lane)));
#pragma unroll
          for (int o = 16; o; o >>= 1) sm = fmaxf(sm, __shfl_xor_sync(FULL, sm, o));
          const float lo = key_score(lst[j]) - 2.0002f * s_err[q] * sm;
          const float l = key_id(lst[j]) == INT_MAX ? -INFINITY : lo - fabsf(lo) * 0x1p-22f;
          const size_t o = (size_t)q * gridDim.x + blockIdx.x;
          if (lane == 0) lows[o] = l;
          if (lane == k - 1) lows[(size_t)nq * gridDim.x + o] = l;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == TM_PROD) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// The float32 score of candidate rows and the query's result (BOUND scans).
// One block per query.  T, a lower bound of the k-th best score: the k-th best
// lane maximum of the lists' head lower bounds (k distinct candidates), or the
// best lower bound of any one list's k-th entry, whichever is better; `lows`
// holds both per list ([2][nq][nl]).  Every candidate with U >= T is scored as the lookup scan does
// (k_scan_stream's operations in its order) and the k best of those are the
// result, unless a full list's last U reaches the k-th best score: a vector
// that list dropped might belong to the result, so the gate opens.
//
// The keys sorted at the end hold, below ~id (whose top bit is always set and
// left out), whether the score is -0: zeros of either sign rank by id, as in the
// lookup scan, and come out as they were.
__device__ __forceinline__ uint64_t result_key(float s, int id) {
  return (rank_key(s, 0) & 0xFFFFFFFF00000000u) | ((uint32_t)~id << 1) |
         (__float_as_uint(s) == 0x80000000u ? 1u : 0u);
}
__device__ __forceinline__ float result_score(uint64_t key) {
  const float s = key_score(key);
  return s == 0.f && (key & 1u) ? -0.f : s;
}
__device__ __forceinline__ int result_id(uint64_t key) { return (int)~(((uint32_t)key >> 1) | 0x80000000u); }

constexpr int RS_NT = 1024;
constexpr int RS_CAP = 1024;  // candidates one block scores
constexpr int RS_PER = 5;     // list entries per thread: 152 lists of 32

// (The kernel is one short block per query, so its time is latency: few
// dependent round trips, rolled loops, since the instructions come from L2 too
// (the unrolled form took 12 us for one query), and 32 warps, so that the usual
// number of candidates is scored in one go (16 warps: 2 us more).)
__global__ void __launch_bounds__(RS_NT)
k_rescore(const float* __restrict__ qrot, int d, const float* __restrict__ centroids,
          const uint8_t* __restrict__ codes, const float* __restrict__ scale, int k, int C, int nl,
          const float* __restrict__ cand_s, const int* __restrict__ cand_i, const float* __restrict__ lows,
          const int* __restrict__ force, int* __restrict__ gate, const uint64_t* __restrict__ ext,
          int64_t* __restrict__ out_ids, float* __restrict__ out_scores, const float* __restrict__ bias) {
  __shared__ uint64_t key[RS_CAP];
  __shared__ int si[RS_CAP];
  __shared__ __align__(16) float sq[2048];
  __shared__ float ctab[16];
  __shared__ int nsv, drop;
  const int q = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nchunks = d >> 4;
  griddep_launch_dependents();
  if (tid < 16) ctab[tid] = __ldg(centroids + tid);
  if (tid == 0) {
    nsv = 0;
    drop = 0;
  }
  griddep_wait();
  const float* cs = cand_s + (size_t)q * nl * C;
  const int* ci = cand_i + (size_t)q * nl * C;
  // one round trip: the force word, the query, every list's two bounds and the lists
  const int forced = __ldcg(force);
  const float bq = bias ? bias[q] : 0.f;
  if (tid < d / 4)
    reinterpret_cast<float4*>(sq)[tid] = __ldcg(reinterpret_cast<const float4*>(qrot + (size_t)q * d) + tid);
  float hl = -INFINITY, kl = -INFINITY;  // of the lists l = lane, lane + 32, ... (every warp alike)
#pragma unroll 5
  for (int l = lane; l < nl; l += 32) {
    hl = fmaxf(hl, __ldcg(lows + (size_t)q * nl + l));
    kl = fmaxf(kl, __ldcg(lows + (size_t)(gridDim.x + q) * nl + l));
  }
  float u[RS_PER];
  int id[RS_PER];
#pragma unroll
  for (int i = 0; i < RS_PER; ++i) {
    const int c = tid + i * RS_NT;
    u[i] = c < nl * C ? __ldcg(cs + c) : -INFINITY;
    id[i] = c < nl * C ? __ldcg(ci + c) : INT_MAX;
  }
  const float hk = key_score(__shfl_sync(FULL, warp_sort_keys(rank_key(hl, 0)), k - 1));
#pragma unroll 1
  for (int o = 16; o; o >>= 1) kl = fmaxf(kl, __shfl_xor_sync(FULL, kl, o));
  const float T = fmaxf(kl, nl >= k ? hk : -INFINITY);
  __syncthreads();  // nsv is zero, the query is in shared memory
#pragma unroll
  for (int i = 0; i < RS_PER; ++i)
    if (id[i] != INT_MAX && u[i] >= T) {
      const int p = atomicAdd(&nsv, 1);
      if (p < RS_CAP) si[p] = id[i];
    }
#pragma unroll 1
  for (int c = RS_PER * RS_NT + tid; c < nl * C; c += RS_NT) {  // (more lists than a GB300 has SMs)
    const int v = __ldcg(ci + c);
    if (v != INT_MAX && __ldcg(cs + c) >= T) {
      const int p = atomicAdd(&nsv, 1);
      if (p < RS_CAP) si[p] = v;
    }
  }
  __syncthreads();
  const int ns = nsv;
  if (forced || ns > RS_CAP) {  // values the bounds do not cover, or too many candidates: the lookup scan runs
    if (tid == 0) gate[q] = 1;
    return;
  }
#pragma unroll 1
  for (int p = warp; p < ns; p += RS_NT / 32) {
    const int v = si[p];
    const uint8_t* row = codes + (size_t)v * (d / 2);
    uint2 w[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int chunk = lane + 32 * s;
      w[s] = chunk < nchunks ? __ldg(reinterpret_cast<const uint2*>(row + chunk * 8)) : make_uint2(0u, 0u);
    }
    const float sc = scale ? __ldg(scale + v) : 1.0f;
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int s = 0; s < 4; ++s) {  // (the lookup scan's zero chunks past d add nothing: skipped)
      const int chunk = lane + 32 * s;
      if (chunk >= nchunks) break;
      const float2* q2 = reinterpret_cast<const float2*>(sq) + chunk * 8;
      uint64_t x = (uint64_t)w[s].x | ((uint64_t)w[s].y << 32);
#pragma unroll 2
      for (int b = 0; b < 8; ++b) {
        acc = __ffma2_rn(q2[b], make_float2(ctab[x & 15u], ctab[(x >> 4) & 15u]), acc);
        x >>= 8;
      }
    }
    __syncwarp();
    float tot = acc.x + acc.y;
#pragma unroll
    for (int o = 16; o; o >>= 1) tot += __shfl_xor_sync(FULL, tot, o);
    if (lane == 0) key[p] = result_key((tot + bq) * sc, v);
  }
  int P = 32;
  while (P < ns) P <<= 1;
  const uint64_t none = result_key(-INFINITY, INT_MAX);
  for (int i = ns + tid; i < P; i += RS_NT) key[i] = none;
  __syncthreads();
  if (P == 32) {
    if (warp == 0) key[lane] = warp_sort_keys(key[lane]);
  } else {
#pragma unroll 1
    for (int size = 2; size <= P; size <<= 1)
#pragma unroll 1
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int t = tid; t < P / 2; t += RS_NT) {
          const int i = 2 * t - (t & (stride - 1)), j = i + stride;
          const uint64_t a = key[i], b = key[j];
          if ((b > a) == ((i & size) == 0)) {
            key[i] = b;
            key[j] = a;
          }
        }
        __syncthreads();
      }
  }
  __syncthreads();
  if (tid < k) {
    const int v = result_id(key[tid]);
    const bool empty = v == INT_MAX;
    out_ids[(size_t)q * k + tid] = empty ? -1 : ext ? (int64_t)__ldg(ext + v) : (int64_t)v;
    out_scores[(size_t)q * k + tid] = empty ? -INFINITY : result_score(key[tid]);
  }
  const float kth = key_score(key[k - 1]);
  // each thread still holds the lists' last entries it loaded
#pragma unroll
  for (int i = 0; i < RS_PER; ++i)
    if ((tid + i * RS_NT) % C == C - 1 && id[i] != INT_MAX && u[i] >= kth) drop = 1;
#pragma unroll 1
  for (int c = RS_PER * RS_NT + tid; c < nl * C; c += RS_NT)
    if (c % C == C - 1 && __ldcg(ci + c) != INT_MAX && __ldcg(cs + c) >= kth) drop = 1;
  __syncthreads();
  if (tid == 0) gate[q] = drop;
}

}  // namespace

// Batches the scan takes: up to 16 columns for the exact search (BOUND), up
// to 32 for the fp16 one.  The exact search pays for its table, its query block
// and two more kernels (about 20 us), so it starts where that is earned back;
// measured (us, this / the lookup scan, one query, d = 1536, k = 10): 2,048 rows
// 28.2 / 25.1, 10,000 28.5 / 29.4, 50,000 36.6 / 40.3, 200,000 61.9 / 72.7; two
// queries 5,000 rows 30.2 / 29.8, 10,000 31.4 / 33.1; four 10,000 35.8 / 42.2; 15
// queries 2,048 rows 66.6 / 72.8.  With k = 32 the first tiles put more into the
// lists: one query 50,000 rows 57.9 / 55.0, 300,000 102 / 118; four 50,000 87 / 103.
// The fp16 scan is faster than the batched one (which makes each CTA decode
// 256-vector tiles and stream its queries) at every size: 16 queries 2,048 rows
// 46 / 120, 100,000 67 / 187.
// With a filter a tile is read when any query allows one of its blocks, so one
// query, whose lookup scan skips 32-row steps, stays there; from two on the
// tiles are read once for all of them.
bool scan_tm_supported(int64_t nq, int64_t n, int d, int bits, int k, bool bound, bool filtered) {
  if (bits != 4 || d % 256 != 0 || d > 2048 || k > TM_LIST || nq < 1) return false;
  if (bound && nq >= kMmaMinBatch) return false;
  if (filtered && bound)
    return nq >= 2 && n * d * nq >= (int64_t)1 << 26 &&
           (n + TM_M - 1) / TM_M <= (int64_t)TM_MAX_TILES * device_sm_count();
  if (bound) return n >= kTmMinRows && n * d * nq >= (k <= kTmSmallK ? (int64_t)1 << 24 : (int64_t)1 << 27);
  return nq <= kTmMaxBatch;
}

int scan_tm_list(int k, bool bound) { return bound ? TM_LIST : k; }

int scan_tm_grid_x(int64_t n) {
  return (int)std::min<int64_t>((n + TM_M - 1) / TM_M, (int64_t)device_sm_count());
}

cudaError_t launch_scan_tm(const float* qrot, int64_t nq, int d, const float* centroids, const uint8_t* codes,
                           const float* scale, int64_t n, const uint32_t* del, const uint32_t* dense,
                           const uint32_t* allow_bits, int words, const uint32_t* bmask, int mask_words, int fblock,
                           const float* bias, int k, bool bound, float* cand_s, int32_t* cand_i, int* err, int* force,
                           uint32_t* gth, float* lows, cudaStream_t s, cudaEvent_t ev0,
                           cudaEvent_t ev1) {
  if (nq == 0) return cudaSuccess;
  PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const int N = nq <= 16 ? 16 : 32;
  const int cst = tm_stages(d, N), C = scan_tm_list(k, bound);
  if (cst < 2 || C > TM_LIST || k > C || (bound && N != 16)) return cudaErrorInvalidValue;
  CUtensorMap map;
  const cuuint64_t gdim[2] = {(cuuint64_t)(d / 2), (cuuint64_t)n};
  const cuuint64_t gstride[1] = {(cuuint64_t)(d / 2)};
  const cuuint32_t box[2] = {128, (cuuint32_t)TM_M};
  const cuuint32_t estride[2] = {1, 1};
  if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(codes), gdim, gstride, box, estride,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const size_t smem = 1024 + 2048 + TM_LUT + tm_b_bytes(d, N) + (size_t)cst * TM_RAW;
  const dim3 grid((unsigned)scan_tm_grid_x(n)), block(TM_THREADS);
  const bool pdl = s != nullptr && ev0 == nullptr;
  cudaError_t e;
  if (ev0 && (e = cudaEventRecord(ev0, s)) != cudaSuccess) return e;
  auto go = [&](auto kernel) {
    const cudaError_t r = set_max_dynamic_smem(reinterpret_cast<const void*>(kernel), (int)smem);
    if (r != cudaSuccess) return r;
    return launch_maybe_pdl(pdl, kernel, grid, block, smem, s, map, qrot, centroids, scale, del, dense, allow_bits,
                            words, bmask, mask_words, fblock, bias, (int)n, (int)nq, d, k, C, cst, cand_s, cand_i, err,
                            force, gth, lows);
  };
  e = bound ? (bmask ? go(k_scan_tm<16, true, true>) : go(k_scan_tm<16, true, false>))
            : N == 16 ? go(k_scan_tm<16, false, false>) : go(k_scan_tm<32, false, false>);
  if (e != cudaSuccess) return e;
  if (ev1 && (e = cudaEventRecord(ev1, s)) != cudaSuccess) return e;
  return cudaSuccess;
}

cudaError_t launch_rescore(const float* qrot, int64_t nq, int d, const float* centroids, const uint8_t* codes,
                           const float* scale, int64_t n, int k, const float* cand_s, const int32_t* cand_i,
                           const float* lows, const int* force, int* gate, const uint64_t* ext, int64_t* out_ids,
                           float* out_scores, const float* bias, cudaStream_t s) {
  if (nq == 0) return cudaSuccess;
  const int C = scan_tm_list(k, true), nl = scan_tm_grid_x(n);
  return launch_maybe_pdl(s != nullptr, k_rescore, dim3((unsigned)nq), dim3(RS_NT), 0, s, qrot, d, centroids, codes,
                          scale, k, C, nl, cand_s, cand_i, lows, force, gate, ext, out_ids, out_scores, bias);
}

}  // namespace tq
