// Tensor-core encode in fp16 (Sec. II-B steps 1-5): the rotation Y = X R^T on
// tcgen05 with a three-product fp16 split, for callers that give the encoder a
// workspace (tq_encode_planned without one uses TF32, tq_encode_tc.cu).
//
// Precision.  fp16 keeps 10 explicit mantissa bits, as TF32 does, and its MMA
// rate is twice TF32's.  What it lacks is exponent range, so every row of X is
// scaled by a power of two to a norm in [2^14, 2^15) and every row of R to a
// largest entry in [2^13, 2^14): then x = x_hi + x_lo and r = r_hi + r_lo lose
// at most 2^-22 of each entry (or 2^-38 of the row's largest, where a low part
// falls below fp16's normal range), and
//   x . r  ~  x_hi . r_hi + x_hi . r_lo + x_lo . r_hi
// is accumulated in float32, in half as many MMAs as the TF32 form, which cuts
// the accumulation error, the largest one here.  The scales are exact and are
// undone exactly.
//
// What bounds it: 3 * 2 d^2 fp16 flops per row (14.1 TFLOP for 999,000 x 1536:
// 7.3 ms at 1,936 TFLOP/s), under the power cap at that rate (the SM clock falls
// to 1.65-1.95 GHz); with the loads, the split and the read-out taken out the
// kernel takes 7.1 ms and the norms' pass over X 0.95.  On top come X's way to
// the SMs, once per chunk (about 2 ms), its split, which 8 warps just keep up
// with (2.4 ms), and R's tiles (1 ms).  Measured at 999,000 x 1536, 4-bit: 20.1 ms
// (TF32) -> 12.4 ms; 1,000 rows 375 -> 48 us; 40,003 x 768 at 8 bits 444 -> 181 us.
// Two accumulators of 192 columns hide the read-out behind the next chunk; with
// one of 256 it took 12.9 ms and 211 us.  Four converter groups (72 registers,
// the epilogue spills) 14.0 ms; separate rings of 3 X and 5 R stages 13.7 ms.
//
// Work.  The items are (128-row panel, chunk of N output coordinates), panel by
// panel; each CTA takes an equal run of items, so the SMs finish together
// whatever the number of panels (with one panel per CTA and turn, 40,003 rows
// took three turns for 2.06 turns of work, and 1,000 rows used 8 SMs).  A panel
// whose chunks fall to several CTAs gets its scalars from the last of them.
// Per K-block a stage holds the raw X tile (128 x 32 fp32, 128-byte swizzle) and
// the R_hi, R_lo tiles (N x 32 fp16, 64-byte swizzle); the split X goes to
// tensor memory (A operand).  K-blocks are walked alternately forwards and
// backwards, by the 192-coordinate block a chunk lies in, so that a chunk
// starts on the X tiles the previous one read last, and an output coordinate's
// sum does not depend on N.  Roles (18 warps): 0-7 converters (two groups of
// four, alternate K-blocks), 8 producer, 9 MMA issuer, 10-17 epilogue (lane
// quarter x column half).  Every wait is bounded; timeouts go to the plan's
// status word.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "tq_internal.h"
#include "tq_kernels.h"
#include "tq_tc.cuh"
#include "tq_topk.cuh"

namespace tq {
namespace {

constexpr int HM = 128;                     // rows of X per panel (MMA M)
constexpr int HK = 32;                      // coordinates per K-block
constexpr int H_MAXN = 192;                 // output coordinates per chunk (MMA N): 192, 96 or 64
constexpr int H_STAGES = 4;
constexpr int HX_BYTES = HM * HK * 4;       // 16 KB
constexpr int HR_BYTES = H_MAXN * HK * 2;   // 12 KB: room for an R_hi or R_lo tile
constexpr int H_STAGE_BYTES = HX_BYTES + 2 * HR_BYTES;
constexpr int H_CONV = 8, H_PROD = 8, H_MMA = 9, H_EPI0 = 10, H_EPI = 8;
constexpr int H_THREADS = (H_EPI0 + H_EPI) * 32;  // 576
constexpr uint32_t H_TM_A = 2 * H_MAXN;     // TMEM: two accumulators, then per stage x_hi (16 columns) and x_lo
constexpr size_t kPlanHead = 256;           // the plan: status word, then R_hi, R_lo in fp32 (tq_encode_tc.cu)

struct HSmem {
  static constexpr uint32_t bnd = H_STAGES * H_STAGE_BYTES;  // [512] floats (one copy per bank up to 4 bits)
  static constexpr uint32_t cen = bnd + 512 * 4;             // [512] floats
  static constexpr uint32_t cell = cen + 512 * 4;            // [2048] (boundary, code below it) by cell
  static constexpr uint32_t part = cell + 2048 * 8;          // [2][128] double: the second column half's sums
  static constexpr uint32_t bars = part + 2 * HM * 8;        // 21 mbarriers
  static constexpr uint32_t misc = bars + 22 * 8;            // TMEM address, abort flag, last flag
  static constexpr uint32_t total = misc + 16;
};
constexpr uint32_t kHSmem = HSmem::total + 1024;
static_assert(kHSmem <= 232448, "encoder shared memory");

// Workspace: R_hi, R_lo in fp16 [2d][d] | 1 / scale of R's rows [d] | scale and
// norm of X's rows [n] each | arrivals per panel | partial row sums of split
// panels, [CTA][first, last][128] pairs of doubles.
struct HWs {
  size_t r16, rinv, xs, nrm, cnt, part, total;
};
HWs h_ws(int64_t n, int d) {
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  HWs w;
  const size_t panels = (size_t)((n + HM - 1) / HM);
  w.r16 = 0;
  w.rinv = up((size_t)2 * d * d * 2);
  w.xs = w.rinv + up((size_t)d * 4);
  w.nrm = w.xs + up((size_t)n * 4);
  w.cnt = w.nrm + up((size_t)n * 4);
  w.part = w.cnt + up(panels * 4);
  w.total = w.part + (size_t)device_sm_count() * 2 * HM * 16;
  return w;
}

__device__ __forceinline__ void h_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// Before the encode: blocks 0 .. d-1 scale and convert a row of the plan's
// R_hi and R_lo (TF32 values, so the conversions are exact up to the low
// range); the others take a row of X per warp: its norm (step 1; float
// partials per 16 values, double across them) and power-of-two scale.
__global__ void __launch_bounds__(256)
k_encode_prep(const float* __restrict__ X, int64_t n, int d, const unsigned char* __restrict__ plan,
              __half* __restrict__ r16, float* __restrict__ rinv, float* __restrict__ xs, float* __restrict__ nrm,
              int* __restrict__ cnt, int64_t panels) {
  griddep_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if ((int)blockIdx.x < d) {
    __shared__ float red[8];
    const float4* hi = reinterpret_cast<const float4*>(plan + kPlanHead) + (size_t)blockIdx.x * (d / 4);
    const float4* lo = hi + (size_t)d * (d / 4);
    float mx = 0.f;
    for (int c = tid; c < d / 4; c += 256) {
      const float4 v = hi[c];
      mx = fmaxf(mx, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    for (int w = 0; w < 8; ++w) mx = fmaxf(mx, red[w]);
    // (a row of zeros, or one out of float32's middle range, is converted as it is)
    const float s = mx >= 0x1p-100f && mx <= 0x1p100f ? pow2f(13 - exp2_of(mx)) : 1.0f;
    if (tid == 0) rinv[blockIdx.x] = 1.0f / s;
    uint2* oh = reinterpret_cast<uint2*>(r16 + (size_t)blockIdx.x * d);
    uint2* ol = reinterpret_cast<uint2*>(r16 + ((size_t)d + blockIdx.x) * d);
    auto pack = [&](float4 v) {
      const __half2 a = __floats2half2_rn(v.x * s, v.y * s), b = __floats2half2_rn(v.z * s, v.w * s);
      return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    };
    for (int c = tid; c < d / 4; c += 256) {
      oh[c] = pack(hi[c]);
      ol[c] = pack(lo[c]);
    }
    for (int64_t i = (int64_t)blockIdx.x * 256 + tid; i < panels; i += (int64_t)d * 256) cnt[i] = 0;
    return;
  }
  const int64_t row = (int64_t)(blockIdx.x - d) * 8 + warp;
  if (row >= n) return;
  const float4* x = reinterpret_cast<const float4*>(X + row * d);
  double ss = 0.0;
  for (int c0 = lane; c0 < d / 4; c0 += 128) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = c0 + 32 * u < d / 4 ? __ldg(x + c0 + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
    float p[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      p[0] = fmaf(v[u].x, v[u].x, p[0]);
      p[1] = fmaf(v[u].y, v[u].y, p[1]);
      p[2] = fmaf(v[u].z, v[u].z, p[2]);
      p[3] = fmaf(v[u].w, v[u].w, p[3]);
    }
    ss += (double)((p[0] + p[1]) + (p[2] + p[3]));
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(FULL, ss, o);
  if (lane == 0) {
    const float nr = (float)sqrt(ss);
    nrm[row] = nr;
    // 0 for a zero row; also where the norm is not finite (its 1/norm is 0, and
    // a value that is not finite still gives NaN)
    xs[row] = nr > 0.f && nr < INFINITY ? pow2f(14 - max(exp2_of(nr), -100)) : 0.f;
  }
}

template <int BITS, bool CAL>
__global__ void __launch_bounds__(H_THREADS, 1)
k_encode_h(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap rmap, int n, int d, int N,
           const float* __restrict__ centroids, const float* __restrict__ boundaries, int scale_mode,
           const float* __restrict__ cal_mu, const float* __restrict__ cal_a, const float* __restrict__ rinv,
           const float* __restrict__ xs, const float* __restrict__ nrm, int* __restrict__ cnt,
           double2* __restrict__ part, uint8_t* __restrict__ codes, float* __restrict__ scale, int* __restrict__ err) {
  constexpr int L = 1 << BITS;
  constexpr int REP = BITS <= 4 ? 32 : 1;  // copies of each table entry (one per bank)
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* base = smem_dyn + ((1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u);
  float* sBnd = reinterpret_cast<float*>(base + HSmem::bnd);
  float* sCen = reinterpret_cast<float*>(base + HSmem::cen);
  float2* sCell = reinterpret_cast<float2*>(base + HSmem::cell);
  double* sPart = reinterpret_cast<double*>(base + HSmem::part);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + HSmem::bars);
  uint64_t* full = bars;             // [4] X and R tiles landed
  uint64_t* conv = bars + 4;         // [4] X tile split into tensor memory
  uint64_t* empty = bars + 8;        // [4] MMAs done with the stage
  uint64_t* acc_full = bars + 12;    // [2] accumulator complete
  uint64_t* acc_empty = bars + 19;   // [2] accumulator read out
  uint64_t* part_ready = bars + 14;  // the second column half's row sums of a panel written
  uint64_t* part_free = bars + 15;   // and read
  uint64_t* fin = bars + 16;
  uint64_t* cut_written = bars + 17; // a split panel's part written by the four warps
  uint64_t* cut_known = bars + 18;   // whether this CTA was the last of the panel's
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + HSmem::misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base + HSmem::misc + 4);
  volatile int* s_last = reinterpret_cast<volatile int*>(base + HSmem::misc + 8);

  const int tid = threadIdx.x, warp = __shfl_sync(FULL, tid >> 5, 0), lane = tid & 31;
  const int KB = d / HK, C = (d + N - 1) / N;
  const int64_t T = (int64_t)((n + HM - 1) / HM) * C, G = gridDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * T / G, i1 = ((int64_t)blockIdx.x + 1) * T / G;  // this CTA's items
  const int stage_tx = HX_BYTES + 2 * N * HK * 2;

  for (int i = tid; i < 512; i += H_THREADS) {
    const int e = i / REP;
    sCen[i] = e < L ? centroids[e] : 0.f;
    sBnd[i] = e < L - 1 ? boundaries[e] : INFINITY;
  }
  // The code of z by cells: the boundaries' range is cut into MC equal cells, few
  // enough apart that a cell holds at most one boundary; then the code is the
  // count of boundaries in lower cells plus a comparison with the cell's own.
  // One lookup instead of a search of BITS dependent ones, with the same
  // result for every z (the cell is a monotone function of z, evaluated alike
  // for z and the boundaries).  Where a cell would hold two (or the range is not
  // finite), the search stays.
  constexpr int MC = BITS <= 4 ? 128 : 2048;           // cells
  constexpr int CREP = BITS <= 4 ? 16 : 1;             // copies (8-byte lookups: one per bank pair)
  const float lo_b = __ldg(boundaries), hi_b = __ldg(boundaries + L - 2);
  const float cs = (float)(MC - 3) / (hi_b - lo_b), co = 1.0f - lo_b * cs;
  auto cell_of = [&](float z) {
    const float f = fminf(fmaxf(fmaf(z, cs, co), 0.f), (float)(MC - 1));  // (NaN: 0)
    return __float_as_int(f + 8388608.0f) & 0xFFFF;                      // rounded to the nearest
  };
  bool cells_ok = hi_b > lo_b && cs < 0x1p60f && fabsf(co) < 0x1p60f;
  for (int i = tid; i < L; i += H_THREADS) {  // cells above the boundary before, up to boundary i's
    const int prev = i == 0 ? -1 : cell_of(__ldg(boundaries + i - 1));
    const float b = i < L - 1 ? __ldg(boundaries + i) : INFINITY;
    const int c = i < L - 1 ? cell_of(b) : MC - 1;
    if (i < L - 1 && c <= prev) cells_ok = false;
    for (int j = prev + 1; j <= c; ++j)
      for (int r = 0; r < CREP; ++r)
        sCell[j * CREP + r] = make_float2(j == c && i < L - 1 ? b : INFINITY, __int_as_float(i));
  }
  cells_ok = __syncthreads_and(cells_ok);
  if (tid == 0) {
    for (int s = 0; s < H_STAGES; ++s) {
      mbar_init(full + s, 1);
      mbar_init(conv + s, 4);
      mbar_init(empty + s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(acc_full + s, 1);
      mbar_init(acc_empty + s, H_EPI);
    }
    mbar_init(part_ready, HM);
    mbar_init(part_free, 4);
    mbar_init(fin, 1);
    mbar_init(cut_written, 4);
    mbar_init(cut_known, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == H_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  griddep_wait();  // the converted R, the rows' scales and norms, the zeroed counters

  if (warp == H_PROD) {
    // ------------------------------------------------ X, R_hi, R_lo tiles (TMA)
    if (lane == 0) {
      int64_t it = 0;
      bool ok = true;
      for (int64_t item = i0; item < i1 && ok; ++item) {
        const int panel = (int)(item / C), c = (int)(item % C);
        const bool back = (c * N / H_MAXN) & 1;
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = (int)(it % H_STAGES);
          const int64_t use = it / H_STAGES;
          if (use > 0 && !mbar_wait(empty + s, (uint32_t)((use - 1) & 1), abort_flag, err, 71)) {
            ok = false;
            break;
          }
          const int kc = back ? KB - 1 - kb : kb;
          unsigned char* st = base + s * H_STAGE_BYTES;
          mbar_arrive_expect_tx(full + s, (uint32_t)stage_tx);
          tma_load_2d(st, &xmap, kc * HK, panel * HM, full + s);
          // in a partial last chunk the rows past d are R_lo rows or zero fill; their columns are not read
          tma_load_2d(st + HX_BYTES, &rmap, kc * HK, c * N, full + s);
          tma_load_2d(st + HX_BYTES + HR_BYTES, &rmap, kc * HK, d + c * N, full + s);
        }
      }
      // never leave with copies in flight: wait (bounded) for the last one of each stage
      for (int s = 0; s < H_STAGES && s < it; ++s)
        mbar_wait_drain(full + s, (uint32_t)(((it - 1 - s) / H_STAGES) & 1));
    }
  } else if (warp == H_MMA) {
    // ------------------------------------------------------------ MMA issuer
    const uint32_t idesc = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(HM >> 4) << 24);
    const uint64_t r0 = sw64_desc(__shfl_sync(FULL, smem_u32(base), 0) + HX_BYTES);
    const uint32_t tm = __shfl_sync(FULL, tmem, 0);
    const int64_t chunks = i1 - i0;
    int s = 0, par = 0;
    bool ok = true;
    for (int64_t cs = 0; cs < chunks && ok; ++cs) {
      const int set = (int)(cs & 1);
      const uint32_t dt = tm + (uint32_t)(set * H_MAXN);
      if (cs >= 2 && !warp_wait(acc_empty + set, (uint32_t)(((cs >> 1) - 1) & 1), abort_flag, err, 72)) break;
      for (int kb = 0; kb < KB; ++kb) {
        if (!warp_wait(conv + s, (uint32_t)par, abort_flag, err, 73)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t rh = r0 + (uint64_t)((uint32_t)s * (H_STAGE_BYTES >> 4)), rl = rh + (HR_BYTES >> 4);
        const uint32_t ah = tm + H_TM_A + (uint32_t)s * 32u, al = ah + 16u;
        const uint32_t more = kb != 0;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < HK / 16; ++kk) {  // 16 values: 32 bytes of each R row, 8 TMEM columns of x
            mma_f16_ta(dt, ah + kk * 8u, rh + kk * 2u, idesc, kk ? 1u : more);
            mma_f16_ta(dt, ah + kk * 8u, rl + kk * 2u, idesc, 1u);
            mma_f16_ta(dt, al + kk * 8u, rh + kk * 2u, idesc, 1u);
          }
          mma_commit(empty + s);
          if (kb == KB - 1) mma_commit(acc_full + set);
        }
        __syncwarp();
        if (++s == H_STAGES) {
          s = 0;
          par ^= 1;
        }
      }
    }
    if (elect_one()) {
      mma_commit(fin);
      mbar_wait_drain(fin, 0);
    }
    __syncwarp();
  } else if (warp < H_CONV) {
    // ------------------------------------------------------------- converters
    // Thread t of a group owns row t of the tile; part q of row t sits at part
    // q ^ (t & 7) of the 128-byte swizzle, so a warp's reads are free of bank
    // conflicts.
    const int g = warp >> 2, quarter = warp & 3, t = quarter * 32 + lane;
    const uint32_t ta0 = tmem + ((uint32_t)(quarter * 32) << 16) + H_TM_A;
    int64_t it = 0;
    bool ok = true;
    int panel = -1;
    float sx = 0.f;
    for (int64_t item = i0; item < i1 && ok; ++item) {
      if ((int)(item / C) != panel) {
        panel = (int)(item / C);
        const int64_t row = (int64_t)panel * HM + t;
        sx = row < n ? __ldg(xs + row) : 0.f;
      }
      for (int kb = 0; kb < KB; ++kb, ++it) {
        if ((int)(it & 1) != g) continue;
        const int s = (int)(it % H_STAGES);
        if (!warp_wait(full + s, (uint32_t)((it / H_STAGES) & 1), abort_flag, err, 74)) {
          ok = false;
          break;
        }
        // The stage's copies were queued after the MMAs of its last use had read
        // this stage's columns of tensor memory (commit -> empty -> producer ->
        // full); the fence orders the stores below behind that chain.  (A
        // wait for `empty` here as well costs a fifth: 12.5 -> 15.2 ms, 999,000 x 1536.)
        tc_fence_after();
        const unsigned char* xt = base + s * H_STAGE_BYTES + t * 128;
        uint32_t hv[16], lv[16];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 v = *reinterpret_cast<const float4*>(xt + ((uint32_t)(q ^ (t & 7)) << 4));
          const float a = v.x * sx, b = v.y * sx, c = v.z * sx, e = v.w * sx;
          const __half2 h0 = __floats2half2_rn(a, b), h1 = __floats2half2_rn(c, e);
          const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
          const __half2 l0 = __floats2half2_rn(a - f0.x, b - f0.y), l1 = __floats2half2_rn(c - f1.x, e - f1.y);
          hv[2 * q] = *reinterpret_cast<const uint32_t*>(&h0);
          hv[2 * q + 1] = *reinterpret_cast<const uint32_t*>(&h1);
          lv[2 * q] = *reinterpret_cast<const uint32_t*>(&l0);
          lv[2 * q + 1] = *reinterpret_cast<const uint32_t*>(&l1);
        }
        h_st16(ta0 + (uint32_t)s * 32u, hv);
        h_st16(ta0 + (uint32_t)s * 32u + 16u, lv);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(conv + s);
      }
    }
  } else {
    // --------------------------------------------------------------- epilogue
    const int quarter = warp & 3;          // TMEM lane quarter this warp may read
    const int h = (warp - H_EPI0) >> 2;    // column half of the chunk
    const int row = quarter * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(h * (N / 2));
    const int64_t rbytes = (int64_t)d * BITS / 8;
    const int rl = lane & (REP - 1);       // this lane's copy of the tables
    float inv = 0.f, nr = 0.f;
    double c2 = 0.0, yc = 0.0;  // the row's sums over this thread's columns (float per 16, then double)
    int64_t grow = 0;
    // 16 consecutive accumulator columns (coordinates j0 .. j0+15) of this row
    const float2* my_cell = sCell + (lane & (CREP - 1));
    auto group = [&](const uint32_t (&r)[16], int j0, auto by_cell) {
      if (j0 >= d) return;  // columns of a partial last chunk (d is a multiple of 32)
      uint64_t packed = 0;  // 2-, 3- and 4-bit codes, little-endian bit stream
      uint32_t p8[4] = {0, 0, 0, 0};
      float g2 = 0.f, gy = 0.f;
#pragma unroll
      for (int u = 0; u < 16; u += 4) {
        const float4 ri = __ldg(reinterpret_cast<const float4*>(rinv + j0 + u));
        const float rs[4] = {ri.x, ri.y, ri.z, ri.w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const int t = u + w;
          const float y = __uint_as_float(r[t]) * rs[w] * inv;  // (the scales are powers of two)
          float z = y, mu = 0.f, a = 1.f;
          if constexpr (CAL) {
            mu = __ldg(cal_mu + j0 + t);
            a = __ldg(cal_a + j0 + t);
            z = (y - mu) * (1.0f / a);
          }
          int code = 0;
          if constexpr (decltype(by_cell)::value) {
            const float2 e = my_cell[cell_of(z) * CREP];
            code = __float_as_int(e.y) + (z > e.x ? 1 : 0);
          } else {
#pragma unroll
            for (int step = L / 2; step >= 1; step >>= 1)
              if (z > sBnd[(code + step - 1) * REP + rl]) code += step;
          }
          const float cc = sCen[code * REP + rl];
          const float cv = CAL ? fmaf(a, cc, mu) : cc;
          g2 = fmaf(cv, cv, g2);
          gy = fmaf(y, cv, gy);
          if constexpr (BITS == 8) p8[t >> 2] |= (uint32_t)code << (8 * (t & 3));
          else packed |= (uint64_t)code << (BITS * t);
        }
      }
      c2 += (double)g2;
      yc += (double)gy;
      if (grow >= n) return;
      uint8_t* dst = codes + grow * rbytes + (int64_t)j0 * BITS / 8;
      if constexpr (BITS == 8) {
        *reinterpret_cast<uint4*>(dst) = make_uint4(p8[0], p8[1], p8[2], p8[3]);
      } else if constexpr (BITS == 4) {
        *reinterpret_cast<uint2*>(dst) = make_uint2((uint32_t)packed, (uint32_t)(packed >> 32));
      } else if constexpr (BITS == 2) {
        *reinterpret_cast<uint32_t*>(dst) = (uint32_t)packed;
      } else {  // 48 bits at an even byte offset (j0 / 16 * 6)
        uint16_t* d16 = reinterpret_cast<uint16_t*>(dst);
        d16[0] = (uint16_t)packed;
        d16[1] = (uint16_t)(packed >> 16);
        d16[2] = (uint16_t)(packed >> 32);
      }
    };
    int64_t done = 0;  // panels (or parts of one) finished
    int cuts = 0;      // split panels among them
    for (int64_t item = i0; item < i1; ++item) {
      const int64_t panel = item / C, cs = item - i0;
      const int c = (int)(item - panel * C);
      if (item == i0 || c == 0) {
        grow = panel * HM + row;
        nr = grow < n ? __ldg(nrm + grow) : 0.f;
        const float sx = grow < n ? __ldg(xs + grow) : 0.f;
        inv = nr > 0.f && sx > 0.f ? (1.0f / nr) * (1.0f / sx) : 0.f;  // 1 / norm, exactly scaled
        c2 = 0.0;
        yc = 0.0;
      }
      const int set = (int)(cs & 1);
      if (!warp_wait(acc_full + set, (uint32_t)((cs >> 1) & 1), abort_flag, err, 75)) break;
      tc_fence_after();
      const int jb = c * N + h * (N / 2);
      const uint32_t ts = tl + (uint32_t)(set * H_MAXN);
      const int G16 = N / 32;  // 16-column groups of this half
      auto read_out = [&](auto by_cell) {
        uint32_t ra[16], rb[16];
        tmem_ld16_issue(ts, ra);
        tmem_wait16(ra);
#pragma unroll 1
        for (int g = 0; g < G16; g += 2) {
          const bool two = g + 1 < G16, more = g + 2 < G16;
          if (two) tmem_ld16_issue(ts + (uint32_t)(16 * g + 16), rb);
          group(ra, jb + 16 * g, by_cell);
          if (!two) break;
          tmem_wait16(rb);
          if (more) tmem_ld16_issue(ts + (uint32_t)(16 * g + 32), ra);
          group(rb, jb + 16 * g + 16, by_cell);
          if (more) tmem_wait16(ra);
        }
      };
      if (cells_ok) read_out(std::true_type{});
      else read_out(std::false_type{});
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty + set);
      if (c != C - 1 && item != i1 - 1) continue;
      // the panel's scalar (step 5), or this CTA's part of it: the second
      // column half hands its sums to the first, row by row
      if (h == 1) {
        if (done > 0 && !warp_wait(part_free, (uint32_t)((done - 1) & 1), abort_flag, err, 76)) break;
        sPart[row] = c2;
        sPart[HM + row] = yc;
        mbar_arrive(part_ready);
        ++done;
        continue;
      }
      if (!warp_wait(part_ready, (uint32_t)(done & 1), abort_flag, err, 77)) break;
      c2 += sPart[row];
      yc += sPart[HM + row];
      __syncwarp();
      if (lane == 0) mbar_arrive(part_free);
      ++done;
      const int64_t p0 = panel * C, p1 = p0 + C;  // the panel's items
      bool write = true;
      if (p0 < i0 || p1 > i1) {  // other CTAs hold the rest: the last to arrive adds the parts in CTA order
        part[((int64_t)blockIdx.x * 2 + (panel == i0 / C ? 0 : 1)) * HM + row] = make_double2(c2, yc);
        __threadfence();
        __syncwarp();
        if (lane == 0) mbar_arrive(cut_written);
        const int64_t b0 = ((p0 + 1) * G - 1) / T, b1 = (p1 * G - 1) / T;  // CTAs of the panel's first and last item
        if (warp == H_EPI0) {
          if (!warp_wait(cut_written, (uint32_t)(cuts & 1), abort_flag, err, 78)) break;
          if (lane == 0) {
            int prev;
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(prev) : "l"(cnt + panel) : "memory");
            *s_last = prev == (int)(b1 - b0);
            mbar_arrive(cut_known);
          }
          __syncwarp();
        }
        if (!warp_wait(cut_known, (uint32_t)(cuts & 1), abort_flag, err, 79)) break;
        ++cuts;
        write = *s_last != 0;  // (written again only after all four warps' next part)
        __threadfence();
        if (write) {
          c2 = 0.0;
          yc = 0.0;
          for (int64_t b = b0; b <= b1; ++b) {
            const int64_t first = b * T / G / C;  // CTA b's first panel
            const double2 v = __ldcg(part + (b * 2 + (panel == first ? 0 : 1)) * HM + row);
            c2 += v.x;
            yc += v.y;
          }
        }
      }
      if (write && grow < n) {
        const float tc2 = (float)c2, tyc = (float)yc;
        float sv = 0.f;
        if (nr > 0.f) {
          if (scale_mode == TQ_SCALE_NONE) {
            sv = nr;
          } else if (scale_mode == TQ_SCALE_NORM) {
            const float cn = sqrtf(tc2);
            sv = cn > 0.f ? nr / cn : 0.f;
          } else {
            sv = tyc != 0.f ? nr / tyc : 0.f;
          }
        }
        scale[grow] = sv;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == H_MMA) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// Output coordinates per chunk: the N that the fewest cycles are expected of.
// A K-block takes as long as its MMAs (3 N cycles), its tiles' way from L2
// (16 KB of X and 128 N bytes of R at about 55 bytes per cycle) or its
// conversion (about 350); an SM takes ceil(items / SMs) of them in turn.
int encode_h_chunk(int64_t n, int d) {
  const int64_t panels = (n + HM - 1) / HM, sms = device_sm_count();
  int best = H_MAXN;
  double best_t = 1e300;
  for (const int N : {192, 96, 64}) {
    const int64_t items = panels * ((d + N - 1) / N);
    const double kb = std::max({350.0, 3.0 * N, (16384.0 + 128.0 * N) / 55.0});
    const double t = (double)((items + sms - 1) / sms) * kb;
    if (t < best_t) {
      best_t = t;
      best = N;
    }
  }
  return best;
}

}  // namespace

// Where the fp16 encoder runs: a matter of agreement with the TF32 encoder's
// bytes, not of accuracy (against 64 bits it was the closer of the two wherever
// measured).  The two decide about 2 in 100,000
// coordinates, those next to a boundary, differently, and one such coordinate
// moves its row's scalar by (c1^2 - c0^2) / 2, at the outermost boundary up to
// 1.04 / d of its value for 2-bit, 1.4 / d for 3-bit, 1.6 / d for 4-bit codes,
// times its calibration squared.  Over 999,000 rows the largest change of a
// scalar measured was 4.1e-3 at d = 768, 3.0e-3 at 1024, 2.1e-3 at 1536.  The
// outer boundaries of 8-bit codes are rarely reached (2.2e-3 at d = 768, the one
// d measured).  Below these d rows encoded now and rows encoded before
// keep agreeing as closely as rows of the TF32 encoder do: its codes stay.
bool encode_h_applies(int d, int bits) { return encode_tc_supported(d) && d >= (bits == 8 ? 768 : 1024); }

size_t encode_h_workspace(int64_t n, int d) { return encode_h_applies(d, 8) ? h_ws(n, d).total : 256; }

cudaError_t launch_encode_h(const float* X, int64_t n, int d, const void* plan, const float* centroids,
                            const float* boundaries, int bits, int scale_mode, const float* cal_mu,
                            const float* cal_a, uint8_t* codes, float* scale, void* ws, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  if (!encode_h_applies(d, bits)) return cudaErrorInvalidValue;
  PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const HWs w = h_ws(n, d);
  unsigned char* wp = static_cast<unsigned char*>(ws);
  __half* r16 = reinterpret_cast<__half*>(wp + w.r16);
  float* rinv = reinterpret_cast<float*>(wp + w.rinv);
  float* xs = reinterpret_cast<float*>(wp + w.xs);
  float* nrm = reinterpret_cast<float*>(wp + w.nrm);
  int* cnt = reinterpret_cast<int*>(wp + w.cnt);
  double2* part = reinterpret_cast<double2*>(wp + w.part);
  const int64_t panels = (n + HM - 1) / HM;
  const int N = encode_h_chunk(n, d);
  CUtensorMap xmap, rmap;
  const cuuint32_t estride[2] = {1, 1};
  {
    const cuuint64_t gdim[2] = {(cuuint64_t)d, (cuuint64_t)n};
    const cuuint64_t gstride[1] = {(cuuint64_t)d * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)HK, (cuuint32_t)HM};
    if (enc(&xmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(X), gdim, gstride, box, estride,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  {
    const cuuint64_t gdim[2] = {(cuuint64_t)d, (cuuint64_t)2 * d};
    const cuuint64_t gstride[1] = {(cuuint64_t)d * sizeof(__half)};
    const cuuint32_t box[2] = {(cuuint32_t)HK, (cuuint32_t)N};
    if (enc(&rmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, r16, gdim, gstride, box, estride,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  int* err = reinterpret_cast<int*>(const_cast<void*>(plan));
  const int64_t items = panels * ((d + N - 1) / N);
  const dim3 grid((unsigned)std::min<int64_t>(items, device_sm_count())), block(H_THREADS);
  const dim3 pgrid((unsigned)(d + (n + 7) / 8));
  k_encode_prep<<<pgrid, 256, 0, s>>>(X, n, d, static_cast<const unsigned char*>(plan), r16, rinv, xs, nrm, cnt,
                                      panels);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  auto go = [&](auto kernel) {
    const cudaError_t r = set_max_dynamic_smem(reinterpret_cast<const void*>(kernel), (int)kHSmem);
    if (r != cudaSuccess) return r;
    return launch_maybe_pdl(s != nullptr, kernel, grid, block, (size_t)kHSmem, s, xmap, rmap, (int)n, d, N, centroids,
                            boundaries, scale_mode, cal_mu, cal_a, (const float*)rinv, (const float*)xs,
                            (const float*)nrm, cnt, part, codes, scale, err);
  };
  const bool cal = cal_mu != nullptr;
  switch (bits) {
    case 2: return cal ? go(k_encode_h<2, true>) : go(k_encode_h<2, false>);
    case 3: return cal ? go(k_encode_h<3, true>) : go(k_encode_h<3, false>);
    case 4: return cal ? go(k_encode_h<4, true>) : go(k_encode_h<4, false>);
    case 8: return cal ? go(k_encode_h<8, true>) : go(k_encode_h<8, false>);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace tq
