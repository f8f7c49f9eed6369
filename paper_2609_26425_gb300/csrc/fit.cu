// fit.cu -- k-means centroids of one chunk per head (Sec. 2: the
// centroid-residual form of QVG with centroids kept in BF16, App. D.1).
//
// Lloyd's algorithm with the arithmetic of its plain definition: initial
// centroid j = token floor(j*N/C); each iteration assigns every token to its
// Euclidean-nearest centroid, the distance being the fp32 sum in channel order
// of the rounded squares of the rounded differences (ties to the lower
// index), then replaces each non-empty cluster by the fp32 rounding of its
// fp64 member mean; the result is rounded to bf16.  Per iteration:
//
//   fit_assign  (persistent, one CTA per SM, tcgen05).  A 128-token tile
//     arrives by TMA and two MMAs per K step accumulate
//     P = X mu_hi^T + X mu_lo^T in TMEM (mu_hi = bf16(mu), mu_lo =
//     bf16(mu - mu_hi): mu to 2^-18 relative; bf16 x bf16 products are exact);
//     one more MMA, a column of ones against -|mu_j|^2 / 2 in two bf16 parts,
//     makes it s_j = P_j - |mu_j|^2 / 2, so that |x|^2 - 2 s_j is the distance
//     and the row's nearest centroid its largest s_j, which the TMEM load
//     reduces on its way.  ||x|^2 - 2 s_j - d_j| stays below
//     E_j = c (|x|^2 + |mu_j|^2), c = 2^-13, for the sequential fp32 distance
//     d_j: fp32 accumulation of 256 products at two ulps of the running
//     absolute sum each, 2^-13 |x| |mu_j|; the operand split 2^-18 and the
//     norm's 2^-17, the fp32 norms and the sequential sum's own rounding
//     2^-16, all relative to |x|^2 + |mu_j|^2: 0.75 c.  With k the largest
//     computed s and j the exact argmin, E_j + E_k bounds 2 (s_k - s_j), and
//     both centroids are within (|x| + sqrt(d))^2 <= 2 (|x|^2 + d) of the origin
//     squared, d = |x|^2 - 2 s_k the distance found (+ E): so every j with
//     s_j > s_k - c (|x|^2 + 2.02 (|x|^2 + d)) is a candidate for the exact
//     argmin.  A row with a single candidate is decided, the others are
//     rescored with the sequential fp32 distance.  Columns past C hold -inf;
//     heads with values from 2^59 up are not screened (kMaxExp).
//   fit_means   (four warps per centroid): exact member sums (bf16 values of
//     ordinary range add exactly, so the order does not matter) from the list of
//     members that the assignment leaves per centroid, the mean, and the next
//     iteration's operand images and norm; the last iteration's launch writes the
//     bf16 result.
// Each launch is a programmatic dependent of the one before it (its prologue
// overlaps that one's tail).
#include <mutex>

#include "ptx_sm103.cuh"
#include "qwm_internal.cuh"

namespace qwm {
namespace {

using namespace ptx;

constexpr int AT = 128;                       // tokens per tile
constexpr int AEW = 16;                       // epilogue warps: rows 32 (w & 3) + lane, column quarter w >> 2
constexpr int ANT = (AEW + 1) * 32;           // + one producer / MMA warp
constexpr int kPairCap = 2048;                // (token, centroid) pairs waiting to be rescored
constexpr int kRowCapList = kPairCap / 2;     // tokens they belong to (two or more candidates each)
constexpr int kRowCap = 8;                    // candidates per row
constexpr int A_X = 0;                        // 2 token tiles, each 2 x [128 rows][128 B] bf16
constexpr int A_IMG = 65536;                  // operand images hi, lo: 2 x 2 x [Npad][128 B]
constexpr int A_ONE = A_IMG + 131072;         // ones: [128 rows][16] bf16 operand (columns 0 and 1), no swizzle
constexpr int A_NRM = A_ONE + 4096;           // -|mu_j|^2 / 2 in two bf16 parts: [256 rows][16], no swizzle
constexpr int A_PJ = A_NRM + 8192;            // waiting pairs' centroids (u8) [kPairCap]
constexpr int A_ROW = A_PJ + kPairCap;        // waiting tokens: tile of the run << 7 | row [kRowCapList]
constexpr int A_RPJ = A_ROW + kRowCapList * 4;   // their first pair << 4 | number of pairs [kRowCapList] (u16)
constexpr int A_MIN = A_RPJ + kRowCapList * 2;         // [4 quarters][128] partial maxima of s
constexpr int A_CNT = A_MIN + 4 * AT * 4;     // [4 quarters][128] candidate count | first candidate << 8
constexpr int A_CND = A_CNT + 4 * AT * 4;     // [128][4 quarters][kRowCap] candidates (u8)
constexpr int A_BAR = A_CND + AT * 4 * kRowCap;   // mbarriers, pair counter, flag, TMEM slot
constexpr int A_SMEM = A_BAR + 128 + 1024;
static_assert(A_SMEM <= 232448, "shared memory of the assignment kernel");
constexpr uint32_t kPadNorm = 0x0000FF80u;    // bf16 -inf | 0 << 16: a padding column never wins, whatever the data
// The screening holds where no product, norm or sum of it leaves the fp32
// range: token values below 2^59 (this bf16 exponent field), so that |x|^2 and
// |mu|^2 stay below 2^125.  A head with a larger value, an infinity or a NaN
// among its tokens has every row searched centroid by centroid: there a
// centroid may be inf or NaN, which the sequential search orders as the
// definition does (a NaN never replaces a distance, and centroid 0's is kept).
constexpr int kMaxExp = 185;

// Operand block of rows of 16 two-byte values without swizzle: 8 rows x 16
// bytes contiguous, the second half of the values 128 bytes on, row groups 256
// bytes apart.
__device__ __forceinline__ uint64_t desc_k16(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(128u >> 4) << 16;
  d |= (uint64_t)(256u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
__device__ __forceinline__ int k16_off(int row) { return (row >> 3) * 256 + (row & 7) * 16; }

// -n2 / 2 as two bf16 parts (the first in the low half-word).
__device__ __forceinline__ uint32_t half_norm(float n2) {
  const float v = -0.5f * n2;
  const __nv_bfloat16 hi = __float2bfloat16_rn(v);
  return pack_bf16(v, v - __bfloat162float(hi));
}

// Byte offset of 16-byte chunk `ch` (channels 8ch..8ch+7) of row `row` in two
// 128-byte-swizzled blocks of `rows` rows x 64 two-byte elements.
__device__ __forceinline__ int sw_off(int rows, int row, int ch) {
  return (ch >> 3) * rows * 128 + row * 128 + (((ch & 7) ^ (row & 7)) << 4);
}

// The sequential fp32 distance of the definition: channel order, the
// difference, its square and the running sum each rounded on its own.
// (One thread: for rows left to the search of every centroid.  mu is read by
// ordinary loads: fit_means may still be writing it when the assignment's
// launch starts, so it is no read-only data of that kernel.)
__device__ __noinline__ float exact_dist(const __nv_bfloat16* x, const float* mu) {
  float acc = 0.0f;
#pragma unroll 1
  for (int ch = 0; ch < 16; ++ch) {
    const float4 ma = reinterpret_cast<const float4*>(mu)[2 * ch], mb = reinterpret_cast<const float4*>(mu)[2 * ch + 1];
    const uint4 xr = __ldg(reinterpret_cast<const uint4*>(x) + ch);
    const uint32_t xw[4] = {xr.x, xr.y, xr.z, xr.w};
    const float ms[8] = {ma.x, ma.y, ma.z, ma.w, mb.x, mb.y, mb.z, mb.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float xe = (e & 1) ? __uint_as_float(xw[e >> 1] & 0xFFFF0000u) : __uint_as_float(xw[e >> 1] << 16);
      const float t = __fsub_rn(xe, ms[e]);
      acc = __fadd_rn(acc, __fmul_rn(t, t));
    }
  }
  return acc;
}

// The same sum for two centroids by a warp: lane l squares channels 4 l .. 4 l
// + 3 (the rows fetched at once), then the running sums pass through the lanes
// in order.  Every lane gets the results.  (Its own function: inlined, its
// registers spilled under those of the kernel's tile loop.)
__device__ __noinline__ float2 exact_dist2(uint2 xv, const float* mu0, const float* mu1) {
  const int lane = threadIdx.x & 31;
  const float xf[4] = {__uint_as_float(xv.x << 16), __uint_as_float(xv.x & 0xFFFF0000u), __uint_as_float(xv.y << 16),
                       __uint_as_float(xv.y & 0xFFFF0000u)};
  const float4 ma = reinterpret_cast<const float4*>(mu0)[lane], mb = reinterpret_cast<const float4*>(mu1)[lane];
  const float m0[4] = {ma.x, ma.y, ma.z, ma.w}, m1[4] = {mb.x, mb.y, mb.z, mb.w};
  float s0[4], s1[4], d0 = 0.0f, d1 = 0.0f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float t0 = __fsub_rn(xf[e], m0[e]), t1 = __fsub_rn(xf[e], m1[e]);
    s0[e] = __fmul_rn(t0, t0);
    s1[e] = __fmul_rn(t1, t1);
  }
  // step l leaves lane l with the sum over the channels up to its own (the lanes
  // after it with values that later steps replace)
#pragma unroll 4
  for (int l = 0; l < 32; ++l) {
    float a = __shfl_up_sync(0xFFFFFFFFu, d0, 1), b = __shfl_up_sync(0xFFFFFFFFu, d1, 1);
    a = lane == 0 ? 0.0f : a;
    b = lane == 0 ? 0.0f : b;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      a = __fadd_rn(a, s0[e]);
      b = __fadd_rn(b, s1[e]);
    }
    d0 = a;
    d1 = b;
  }
  return make_float2(__shfl_sync(0xFFFFFFFFu, d0, 31), __shfl_sync(0xFFFFFFFFu, d1, 31));
}

// Operand images and norm of centroid j of head h from its fp32 row (one
// warp, lane = channels 4 lane .. 4 lane + 3).
__device__ __forceinline__ void emit_row(const FitArgs& a, int h, int j, float4 m, int lane) {
  const int c0 = 4 * lane;
  const __nv_bfloat162 h01 = __floats2bfloat162_rn(m.x, m.y), h23 = __floats2bfloat162_rn(m.z, m.w);
  const float2 f01 = __bfloat1622float2(h01), f23 = __bfloat1622float2(h23);
  const __nv_bfloat162 l01 = __floats2bfloat162_rn(m.x - f01.x, m.y - f01.y);
  const __nv_bfloat162 l23 = __floats2bfloat162_rn(m.z - f23.x, m.w - f23.y);
  const size_t off = (size_t)sw_off(a.Npad, j, c0 >> 3) + (size_t)(c0 & 7) * 2;
  uint8_t* hi = a.img + (size_t)h * 2 * a.Npad * 256;
  uint8_t* lo = hi + (size_t)a.Npad * 256;
  *reinterpret_cast<uint2*>(hi + off) =
      make_uint2(*reinterpret_cast<const uint32_t*>(&h01), *reinterpret_cast<const uint32_t*>(&h23));
  *reinterpret_cast<uint2*>(lo + off) =
      make_uint2(*reinterpret_cast<const uint32_t*>(&l01), *reinterpret_cast<const uint32_t*>(&l23));
  float n2 = fmaf(m.x, m.x, fmaf(m.y, m.y, fmaf(m.z, m.z, m.w * m.w)));
#pragma unroll
  for (int o = 16; o; o >>= 1) n2 += __shfl_xor_sync(0xFFFFFFFFu, n2, o);
  if (lane == 0) a.nrm[(size_t)h * a.Npad + j] = half_norm(n2);
}

__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Initial centroids (token floor(j N / C)) and their images; padding rows
// j in [C, Npad) get zero images and norm; the counters start at zero.  One
// warp per (head, row).
__global__ void __launch_bounds__(512) fit_prep(const FitArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= (int64_t)a.H * a.Npad) return;
  const int h = (int)(w / a.Npad), j = (int)(w % a.Npad);
  if (lane == 0) {
    if (w == 0) *a.status = 0;
    if (j == 0) a.emax[h] = 0;
    if (j < a.C) a.counts[(size_t)h * a.C + j] = 0;
  }
  if (j >= a.C) {
    const size_t off = (size_t)sw_off(a.Npad, j, lane >> 1) + (size_t)(lane & 1) * 8;
    uint8_t* hi = a.img + (size_t)h * 2 * a.Npad * 256;
    *reinterpret_cast<uint2*>(hi + off) = make_uint2(0, 0);
    *reinterpret_cast<uint2*>(hi + (size_t)a.Npad * 256 + off) = make_uint2(0, 0);
    if (lane == 0) a.nrm[(size_t)h * a.Npad + j] = kPadNorm;
    return;
  }
  const int64_t src = ((int64_t)j * a.N) / a.C;
  const uint2 xv = __ldg(reinterpret_cast<const uint2*>(a.x + ((size_t)src * a.H + h) * 128 + 4 * lane));
  const float4 m = make_float4(__uint_as_float(xv.x << 16), __uint_as_float(xv.x & 0xFFFF0000u),
                               __uint_as_float(xv.y << 16), __uint_as_float(xv.y & 0xFFFF0000u));
  reinterpret_cast<float4*>(a.cent + ((size_t)h * a.C + j) * 128)[lane] = m;
  emit_row(a, h, j, m, lane);
}

// Assignment of every token (see the file comment).  Units are (head, tile)
// in head-major order, split into contiguous runs over the CTAs.  Warp 16 loads
// (TMA) and multiplies (tcgen05) tile t + 1 into the second token buffer and
// TMEM accumulator while warps 0-15 finish tile t: four warps per row, one per
// column quarter of the accumulator (at most 64 columns, read once and kept in
// registers), meeting in shared memory.  The rows that need the exact distance
// wait in a list until the run's end (or until it may not hold another tile's):
// rescored tile by tile, a handful of rows each, their latency was a third of
// the kernel's time.
__global__ void __launch_bounds__(ANT, 1)
    fit_assign(const FitArgs a, const __grid_constant__ CUtensorMap tm, int tiles, int units) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int C = a.C, Npad = a.Npad;
  uint8_t* sPJ = sm + A_PJ;
  uint32_t* sRow = reinterpret_cast<uint32_t*>(sm + A_ROW);
  uint16_t* sRpj = reinterpret_cast<uint16_t*>(sm + A_RPJ);
  float* sMin = reinterpret_cast<float*>(sm + A_MIN);
  int* sCnt = reinterpret_cast<int*>(sm + A_CNT);
  uint8_t* sCnd = sm + A_CND;
  const uint32_t bars = smem_u32(sm + A_BAR);
  auto bar_tma = [&](int b) { return bars + 8 * b; };          // token tile b landed
  auto bar_mma = [&](int b) { return bars + 16 + 8 * b; };     // accumulator b complete
  auto bar_free = [&](int b) { return bars + 32 + 8 * b; };    // tile b and accumulator b consumed
  const uint32_t bar_img = bars + 48;
  int* s_np = reinterpret_cast<int*>(sm + A_BAR + 64);   // pairs waiting; s_np[3]: tokens waiting
  volatile int* s_err = reinterpret_cast<volatile int*>(sm + A_BAR + 68);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + A_BAR + 72);
  uint32_t ncols = 32;
  while ((int)ncols < Npad) ncols <<= 1;
  const int Nm = (Npad + 31) & ~31;

  if (warp == 0) {
    tmem_alloc(smem_u32(tslot), 2 * ncols);
    tmem_relinquish();
  }
  // the ones operand; the norm operand's unused columns; the image rows from
  // Npad to the MMA width Nm (a multiple of 32: the loads read whole chunks)
  for (int i = tid; i < 128 * 2; i += ANT)
    *reinterpret_cast<uint4*>(sm + A_ONE + i * 16) = make_uint4((i & 8) ? 0u : 0x3F803F80u, 0u, 0u, 0u);
  for (int i = tid; i < 256 * 2; i += ANT)
    *reinterpret_cast<uint4*>(sm + A_NRM + i * 16) = make_uint4((i & 8) ? 0u : kPadNorm, 0u, 0u, 0u);
  for (int i = tid; i < 4 * (Nm - Npad) * 8; i += ANT)
    *reinterpret_cast<uint4*>(sm + A_IMG + (i / ((Nm - Npad) * 8)) * Nm * 128 + Npad * 128 + (i % ((Nm - Npad) * 8)) * 16) =
        make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async_smem();
  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_tma(b), 1);
      mbar_init(bar_mma(b), 1);
      mbar_init(bar_free(b), AEW);
    }
    mbar_init(bar_img, 1);
    fence_mbar_init();
    s_np[0] = s_np[3] = 0;
    *s_err = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_launch();
  pdl_wait();   // the images, norms and member lists of the launches before
  const uint32_t tbase = *tslot;
  const int u0 = (int)((int64_t)blockIdx.x * units / gridDim.x);
  const int u1 = (int)((int64_t)(blockIdx.x + 1) * units / gridDim.x);
  const int T = u1 - u0;

  if (warp == AEW) {
    // ---------------- producer / MMA issuer
    const uint32_t id = idesc_f16(128, Nm, false, true);
    const uint32_t aI = smem_u32(sm + A_IMG);
    int cur_h = -1;
    uint32_t images = 0;       // heads' images loaded
    bool go = true;
    int loads = 0, mmas = 0;   // tiles loaded, tiles multiplied
    auto load_tile = [&](int t) {
      ++loads;
      const int u = u0 + t, h = u / tiles, b = t & 1;
      const uint32_t aX = smem_u32(sm + A_X + b * 32768);
      if (lane == 0) {
        mbar_arrive_expect_tx(bar_tma(b), 32768u);
        tma_load_3d(aX, &tm, 0, h, (u - h * tiles) * 128, bar_tma(b));
        tma_load_3d(aX + 16384, &tm, 64, h, (u - h * tiles) * 128, bar_tma(b));
      }
    };
    if (T > 0) load_tile(0);
    for (int t = 0; t < T; ++t) {
      const int h = (u0 + t) / tiles, b = t & 1;
      if (h != cur_h) {
        // the previous head's MMAs read the images and norms: wait for them, then load this head's
        if (t >= 1) go = __all_sync(0xFFFFFFFFu, mbar_wait(bar_mma((t - 1) & 1), ((t - 1) >> 1) & 1));
        if (go) {
          if (lane == 0) {
            mbar_arrive_expect_tx(bar_img, (uint32_t)Npad * 512u);
#pragma unroll
            for (int q = 0; q < 4; ++q)   // hi, lo x channels [0, 64), [64, 128)
              bulk_g2s(aI + q * Nm * 128, a.img + ((size_t)h * 4 + q) * Npad * 128, (uint32_t)Npad * 128u, bar_img);
          }
          for (int j = lane; j < Npad; j += 32)
            *reinterpret_cast<uint32_t*>(sm + A_NRM + k16_off(j)) = a.nrm[(size_t)h * Npad + j];
          fence_proxy_async_smem();
          go = mbar_wait(bar_img, images & 1);
          ++images;
          cur_h = h;
        }
      }
      go = go && mbar_wait(bar_tma(b), (t >> 1) & 1);
      go = go && (t < 2 || mbar_wait(bar_free(b), ((t >> 1) - 1) & 1));
      go = __all_sync(0xFFFFFFFFu, go);
      if (!go) break;
      tc_fence_after();
      if (lane == 0) {
        const uint32_t aX = smem_u32(sm + A_X + b * 32768);
        const uint32_t tD = tbase + (uint32_t)b * ncols;
#pragma unroll
        for (int half = 0; half < 2; ++half)
#pragma unroll
          for (int kb = 0; kb < 2; ++kb)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              umma_ss(tD, desc_sw128(aX + kb * 16384 + ks * 32), desc_sw128(aI + (half * 2 + kb) * Nm * 128 + ks * 32),
                      id, (half | kb | ks) != 0);
        umma_ss(tD, desc_k16(smem_u32(sm + A_ONE)), desc_k16(smem_u32(sm + A_NRM)), id, 1u);
        umma_commit(bar_mma(b));
      }
      ++mmas;
      __syncwarp();
      // the next tile's copy, once the MMAs of the tile before this one have left its buffer
      if (t + 1 < T) {
        if (t >= 1) go = __all_sync(0xFFFFFFFFu, mbar_wait(bar_mma(b ^ 1), ((t - 1) >> 1) & 1));
        if (!go) break;
        load_tile(t + 1);
      }
    }
    if (!go) *s_err = 1;
    // no copy and no MMA outlives the CTA's memory, also where a wait ran out
    if (loads) mbar_wait(bar_tma((loads - 1) & 1), ((loads - 1) >> 1) & 1);
    if (images) mbar_wait(bar_img, (images - 1) & 1);
    if (mmas) mbar_wait(bar_mma((mmas - 1) & 1), ((mmas - 1) >> 1) & 1);
  } else {
    // ---------------- epilogue: warps 0-15
    const int qt = warp >> 2, row = (warp & 3) * 32 + lane;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;
    const int nchunk = (Npad + 31) >> 5;
    const int ch0 = (qt * nchunk) >> 2, ch1 = ((qt + 1) * nchunk) >> 2;   // this quarter's 32-column chunks
    // A token's assignment.  Its place among its centroid's members comes back
    // from an atomic count; it is listed one call later, when that has long arrived.
    int pl_rank = 0, pl_tok = -1;
    size_t pl_cent = 0;
    auto list_member = [&]() {
      if (pl_tok < 0 || pl_rank >= a.cap) return;
      const size_t at = pl_cent * a.cap + pl_rank;
      if (a.wide) reinterpret_cast<int32_t*>(a.list)[at] = pl_tok;
      else reinterpret_cast<uint16_t*>(a.list)[at] = (uint16_t)pl_tok;
    };
    auto assign = [&](int h, int64_t n, int j) {
      a.asg[(size_t)h * a.N + n] = (uint8_t)j;
      list_member();
      pl_cent = (size_t)h * C + j;
      pl_tok = (int)n;
      pl_rank = atomicAdd(a.counts + pl_cent, 1);
    };
    // the waiting tokens' exact distances, a warp each: ascending centroids, the
    // lower one keeps a tie (called by all epilogue threads, the list complete)
    auto rescore = [&]() {
      const int nr = s_np[3];
#pragma unroll 1
      for (int r = warp; r < nr; r += AEW) {
        const int u = u0 + (int)(sRow[r] >> 7), h = u / tiles;
        const int64_t n = (int64_t)(u - h * tiles) * 128 + (sRow[r] & 127u);
        const int p0 = sRpj[r] >> 4, np = sRpj[r] & 15;
        const uint2 xv = __ldg(reinterpret_cast<const uint2*>(a.x + ((size_t)n * a.H + h) * 128) + lane);
        float bd = 0.0f;
        int best = -1;
#pragma unroll 1
        for (int p = 0; p < np; p += 2) {
          const int j0 = sPJ[p0 + p], j1 = sPJ[p0 + min(p + 1, np - 1)];
          const float* cent = a.cent + (size_t)h * C * 128;
          const float2 d = exact_dist2(xv, cent + j0 * 128, cent + j1 * 128);
          if (best < 0 || d.x < bd) {
            bd = d.x;
            best = j0;
          }
          if (d.y < bd) {
            bd = d.y;
            best = j1;
          }
        }
        if (lane == 0) assign(h, n, best);
      }
    };
    for (int t = 0; t < T; ++t) {
      const int u = u0 + t, h = u / tiles, tile = u - h * tiles, b = t & 1;
      const uint32_t tD = tbase + (uint32_t)b * ncols;
      const int64_t n = (int64_t)tile * 128 + row;
      const bool valid = n < a.N;
      const float kx = valid ? a.xn2[(size_t)h * a.N + n] : 0.0f;
      const bool in_range = a.emax[h] <= kMaxExp;
      const bool ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar_mma(b), (t >> 1) & 1));
      tc_fence_after();
      // s_j of this quarter's columns and the largest
      constexpr float kC = 1.220703125e-4f;   // c
      float v[64];
      float mx = -INFINITY;
      const bool any = ok && ch0 < ch1;
      if (any) {
        const int cb2 = ch0 + 1 < ch1 ? ch0 + 1 : ch0;  // a lone chunk is read twice
        mx = tmem_ld64_max(tD + lrow + ch0 * 32, tD + lrow + cb2 * 32, v);
      }
      sMin[qt * AT + row] = mx;
      tc_fence_before();
      if (lane == 0) mbar_arrive(bar_free(b));   // the accumulator is in registers
      // one vote, so that every epilogue warp leaves the loop together
      if (!named_bar_and(1, AEW * 32, ok)) {
        *s_err = 1;
        break;
      }
      const bool full = s_np[0] > kPairCap - AT * kRowCap;   // the list may not hold this tile's pairs
      mx = fmaxf(fmaxf(sMin[row], sMin[AT + row]), fmaxf(sMin[2 * AT + row], sMin[3 * AT + row]));
      const float dist = fmaxf(fmaf(-2.0f, mx, kx), 0.0f);
      const float thr = fmaf(-kC, fmaf(2.02f, kx + dist, kx), mx) - 1e-30f;
      const bool fin = ok && in_range && thr > -INFINITY && thr < INFINITY;
      // this quarter's candidates, ascending (bit 31 - e of a mask: column e)
      int cnt = 0;
      uint32_t word = 0xFFu;   // count (0xFF: every centroid), first candidate << 8
      uint8_t* cand = sCnd + (row * 4 + qt) * kRowCap;
      if (fin) {
        uint32_t mk[2] = {0u, 0u};
        if (any) {
#pragma unroll
          for (int e = 0; e < 64; ++e) mk[e >> 5] = __funnelshift_l(__float_as_uint(thr - v[e]), mk[e >> 5], 1);
          if (ch0 + 1 >= ch1) mk[1] = 0u;
        }
        cnt = __popc(mk[0]) + __popc(mk[1]);
        const int first = mk[0] ? __clz((int)mk[0]) : 32 + __clz((int)mk[1]);
        word = (uint32_t)cnt | ((uint32_t)(ch0 * 32 + first) << 8);
        if (cnt > 1) {
          int k = 0;
#pragma unroll
          for (int hb = 0; hb < 2; ++hb)
            for (uint32_t m = mk[hb]; m && k < kRowCap;) {
              const int e = __clz((int)m);
              m &= ~(0x80000000u >> e);
              cand[k++] = (uint8_t)((ch0 + hb) * 32 + e);
            }
        }
      }
      sCnt[qt * AT + row] = (int)word;
      named_bar_sync(1, AEW * 32);
      if (full) {
        rescore();
        named_bar_sync(1, AEW * 32);
        if (tid == 0) s_np[0] = s_np[3] = 0;
        named_bar_sync(1, AEW * 32);
      }
      // the row owner (quarter 0) merges: one candidate decides, a few wait for their exact distances
      if (qt == 0 && valid) {
        uint32_t cw[4];
        int tot = 0, best = 0;
        bool bad = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          cw[q] = (uint32_t)sCnt[q * AT + row];
          bad = bad || (cw[q] & 0xFFu) == 0xFFu;
          tot += (int)(cw[q] & 0xFFu);
          if (cw[q] & 0xFFu) best = (int)(cw[q] >> 8);
        }
        if (bad || tot == 0 || tot > kRowCap) {   // every centroid, sequentially
          const __nv_bfloat16* xr = a.x + ((size_t)n * a.H + h) * 128;
          float bd = 0.0f;
          for (int j = 0; j < C; ++j) {
            const float dj = exact_dist(xr, a.cent + ((size_t)h * C + j) * 128);
            if (j == 0 || dj < bd) {
              bd = dj;
              best = j;
            }
          }
          tot = 1;
        }
        if (tot == 1) {
          assign(h, n, best);
        } else {
          const int p0 = atomicAdd(s_np, tot), r = atomicAdd(s_np + 3, 1);
          int k = p0;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int n2 = (int)(cw[q] & 0xFFu);
            for (int c2 = 0; c2 < n2; ++c2)
              sPJ[k++] = n2 == 1 ? (uint8_t)(cw[q] >> 8) : sCnd[(row * 4 + q) * kRowCap + c2];
          }
          sRow[r] = ((uint32_t)t << 7) | (uint32_t)row;
          sRpj[r] = (uint16_t)((p0 << 4) | tot);
        }
      }
      if (t == T - 1) {
        named_bar_sync(1, AEW * 32);
        rescore();
      }
    }
    list_member();
  }
  if (tid == 0 && *s_err) atomicCAS(a.status, 0, (int)QWM_ERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tbase, 2 * ncols);
  }
}

// Largest bf16 exponent field over each head's tokens, which fixes the unit
// 2^U of the exact fixed-point member sums (U = emax - 134 - room), and |x|^2
// of every token, which sizes the screening bound.
__global__ void __launch_bounds__(256) fit_scale(const FitArgs a) {
  pdl_launch();
  pdl_wait();
  const int h = blockIdx.y, lane = threadIdx.x & 31;
  uint32_t mx = 0;
  for (int64_t n = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); n < a.N; n += (int64_t)gridDim.x * 8) {
    const uint2 xv = __ldg(reinterpret_cast<const uint2*>(a.x + ((size_t)n * a.H + h) * 128 + 4 * lane));
    mx = max(mx, max(max((xv.x >> 7) & 0xFFu, (xv.x >> 23) & 0xFFu), max((xv.y >> 7) & 0xFFu, (xv.y >> 23) & 0xFFu)));
    const float x0 = __uint_as_float(xv.x << 16), x1 = __uint_as_float(xv.x & 0xFFFF0000u);
    const float x2 = __uint_as_float(xv.y << 16), x3 = __uint_as_float(xv.y & 0xFFFF0000u);
    float n2 = fmaf(x0, x0, fmaf(x1, x1, fmaf(x2, x2, x3 * x3)));
#pragma unroll
    for (int o = 16; o; o >>= 1) n2 += __shfl_xor_sync(0xFFFFFFFFu, n2, o);
    if (lane == 0) a.xn2[(size_t)h * a.N + n] = n2;
  }
  mx = __reduce_max_sync(0xFFFFFFFFu, mx);
  if (lane == 0) atomicMax(a.emax + h, (int)mx);
}

// New centroid j of head h: the fp32 rounding of the fp64 member mean (kept
// when the cluster is empty); then its images and norm.  One warp each, lane =
// four channels, member rows read four at a time.
//   The member sum is exact and independent of order.  A normal bf16 value is
//   (128 + f) 2^(e - 134); with U = emax - 134 - room every member is the
//   integer (128 + f) << (e - 134 - U) < 2^(8 + room) in units of 2^U, and N
//   of them add in int64 without overflow.  A member outside that grid (tiny,
//   subnormal, inf or NaN) sends the cluster to fp64 sums instead.
//   The mean RN32(RN64(S / n)): S and 1 / n as pairs of fp32 values (S to 2^-48,
//   1 / n to 2^-46 relative) and one product of pairs give S / n to 2^-44;
//   its high part is the result unless the true quotient may lie within 2^-40
//   relative of a point halfway between two fp32 values (which also covers the
//   rounding to fp64 in between), or leaves the fp32 normal range: there the
//   fp64 division decides.  (fp64 operations run at 1/64 of the fp32 rate.)
__device__ __forceinline__ float mean_of(long long k, int U, float rh, float rl, double dc) {
  const float kh = __ll2float_rn(k);
  const float kl = __ll2float_rn(k - __float2ll_rn(kh));
  const float ph = __fmul_rn(kh, rh);
  const float pe = fmaf(kh, rl, fmaf(kl, rh, fmaf(kh, rh, -ph)));
  const float q = __fadd_rn(ph, pe);
  const float e = __fsub_rn(pe, __fsub_rn(q, ph));          // exact: |pe| is far below |ph|
  const uint32_t qb = __float_as_uint(q) & 0x7FFFFFFFu;
  const int ex = (int)(qb >> 23) + U;                        // exponent field of the mean
  const float ulp = __uint_as_float((qb & 0x7F800000u) - (23u << 23));   // of q (|q| >= 2^-24: k is an integer)
  // half an ulp, a quarter just below a power of two, less 2^-16 of it
  const float lim = ulp * ((qb & 0x7FFFFFu) ? 0.49999237f : 0.24999619f);
  if (k != 0 && (!(fabsf(e) < lim) || ex < 1 || ex > 254))
    return __double2float_rn(__ddiv_rn(ldexp((double)k, U), dc));
  return k == 0 ? 0.0f : __uint_as_float(__float_as_uint(q) + ((uint32_t)U << 23));
}

// Four warps per centroid (the largest clusters hold many times the average,
// and with one warp each they set the launch's time): batches of eight members
// go round the warps, whose int64 sums meet in shared memory; warp 0 finishes.
// The members are the centroid's list where the assignment had room for all of
// them (twice the average cluster), else they are picked out of the head's
// assignment bytes, kPick tokens at a time.
constexpr int kPick = 4096;
__global__ void __launch_bounds__(128) fit_means(const FitArgs a, int last) {
  __shared__ uint16_t s_list[kPick];
  __shared__ long long s_sum[4][128];
  __shared__ int s_n, s_ok;
  pdl_launch();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t w = blockIdx.x;
  const int h = (int)(w / a.C), j = (int)(w % a.C);
  if (tid == 0) {
    s_n = 0;
    s_ok = 1;
  }
  pdl_wait();
  const int cnt = a.counts[w];
  const int U = a.emax[h] - 134 - a.room;
  float4* cr = reinterpret_cast<float4*>(a.cent + (size_t)w * 128) + lane;
  float4 m = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (warp == 0) m = *cr;
  __syncthreads();
  // Exact member sums.  A member value in units of 2^U, y = (128 + f) 2^(e - 134
  // - U) < 2^48 (room <= 40), has 8 significant bits.  Two additions of 3 2^54
  // and 3 2^38 split it exactly into fp32 limbs that are multiples of 2^32 and
  // 2^16 and a remainder below 2^15; 32 such limbs add exactly in fp32 (below
  // 2^21 units each), and every 32 members the three limb sums go to int64.  A
  // value off the grid (tiny, subnormal, inf, NaN) or a unit beyond the fp32
  // range sends the cluster to fp64 sums.
  const float unit = U >= -127 ? __uint_as_float((uint32_t)(127 - U) << 23) : 0.0f;   // 2^-U
  const float C32 = 5.4043195528445952e16f;   // 3 * 2^54
  const float C16 = 8.24633720832e11f;        // 3 * 2^38
  int64_t k0 = 0, k1 = 0, k2 = 0, k3 = 0;
  uint32_t least = 0xFFFFFFFFu, most = 0u;    // smallest magnitude - 1 (zero wraps) and largest, of bf16 pairs
  float l2[4] = {}, l1[4] = {}, l0[4] = {};
  auto limb = [&](float x, int ch) {
    const float y = __fmul_rn(x, unit);
    const float hi = __fsub_rn(__fadd_rn(y, C32), C32);
    const float r1 = __fsub_rn(y, hi);
    const float mid = __fsub_rn(__fadd_rn(r1, C16), C16);
    l2[ch] = __fadd_rn(l2[ch], hi);
    l1[ch] = __fadd_rn(l1[ch], mid);
    l0[ch] = __fadd_rn(l0[ch], __fsub_rn(r1, mid));
  };
  auto pair = [&](uint32_t v, int ch) {
    const uint32_t mag = v & 0x7FFF7FFFu;
    least = vmin_u16x2(least, vadd_u16x2(mag, 0xFFFFFFFFu));
    most = vmax_u16x2(most, mag);
    limb(__uint_as_float(v << 16), ch);
    limb(__uint_as_float(v & 0xFFFF0000u), ch + 1);
  };
  auto flush = [&](int64_t& k, int ch) {
    k += ((int64_t)__float2int_rn(l2[ch] * 2.3283064365386963e-10f) << 32) +
         ((int64_t)__float2int_rn(l1[ch] * 1.52587890625e-05f) << 16) + (int64_t)__float2int_rn(l0[ch]);
    l2[ch] = l1[ch] = l0[ch] = 0.0f;
  };
  auto flush_all = [&]() {
    flush(k0, 0);
    flush(k1, 1);
    flush(k2, 2);
    flush(k3, 3);
  };
  // batches warp, warp + 4, ... of n members, token(m) the m-th: lane 8 i + k
  // reads the token of row k of the i-th of four batches
  auto rows = [&](int n, auto token) {
    for (int b0 = 8 * warp; b0 < n; b0 += 128) {
      const int mine = b0 + 32 * (lane >> 3) + (lane & 7);
      const int64_t tk = mine < n ? token(mine) : -1;
#pragma unroll 1
      for (int i = 0; i < 4 && b0 + 32 * i < n; ++i) {
        uint2 xv[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int64_t tok = __shfl_sync(0xFFFFFFFFu, tk, 8 * i + k);
          xv[k] = make_uint2(0, 0);
          if (tok >= 0 && tok < a.N)  // every member, unless a timed-out assignment left stale entries
            xv[k] = __ldg(reinterpret_cast<const uint2*>(a.x + ((size_t)tok * a.H + h) * 128 + 4 * lane));
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          pair(xv[k].x, 0);
          pair(xv[k].y, 2);
        }
      }
      flush_all();   // after at most 32 members
    }
  };
  const uint8_t* asg = a.asg + (size_t)h * a.N;
  if (cnt <= a.cap) {
    const size_t at = (size_t)w * a.cap;
    if (a.wide) rows(cnt, [&](int i) { return (int64_t)reinterpret_cast<const int32_t*>(a.list)[at + i]; });
    else rows(cnt, [&](int i) { return (int64_t)reinterpret_cast<const uint16_t*>(a.list)[at + i]; });
  } else {
    const uint32_t jj = (uint32_t)j * 0x01010101u;
    const int lead = (int)(reinterpret_cast<uintptr_t>(asg) & 15u);   // the head's bytes start inside a 16-byte word
    for (int64_t c0 = 0; c0 < a.N; c0 += kPick) {
      const int64_t c1 = c0 + kPick < a.N ? c0 + kPick : a.N;
      // whole words over tokens [c0, c1) (kPick is a multiple of 16)
      for (int64_t o = c0 - lead + 16 * tid; o < c1; o += 16 * 128) {
        const uint4 v = *reinterpret_cast<const uint4*>(asg + o);
        const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t mk = __vcmpeq4(w4[q], jj) & 0x01010101u;
          while (mk) {
            const int64_t t = o + 4 * q + ((__ffs((int)mk) - 1) >> 3);
            mk &= mk - 1;
            if (t >= c0 && t < c1) s_list[atomicAdd(&s_n, 1)] = (uint16_t)(t - c0);
          }
        }
      }
      __syncthreads();
      const int n = s_n;
      rows(n, [&](int i) { return c0 + (int64_t)s_list[i]; });
      __syncthreads();
      if (tid == 0) s_n = 0;
      __syncthreads();
    }
  }
  s_sum[warp][4 * lane] = k0;
  s_sum[warp][4 * lane + 1] = k1;
  s_sum[warp][4 * lane + 2] = k2;
  s_sum[warp][4 * lane + 3] = k3;
  {
    const uint32_t lim = ((uint32_t)(U + 134) << 7) - 1u;   // magnitude - 1 of the smallest value on the grid
    const bool on_grid = most == 0u || (U >= -127 && min(least & 0xFFFFu, least >> 16) >= lim &&
                                        max(most & 0xFFFFu, most >> 16) < 0x7F80u);
    if (!on_grid) s_ok = 0;
  }
  __syncthreads();
  if (warp != 0) return;

  if (cnt > 0) {
    const double dc = (double)cnt;
    bool ok = s_ok != 0 && cnt <= (1 << 24);
    if (ok) {
      auto total = [&](int ch) {
        return s_sum[0][4 * lane + ch] + s_sum[1][4 * lane + ch] + s_sum[2][4 * lane + ch] + s_sum[3][4 * lane + ch];
      };
      const float n = (float)cnt;   // exact: cnt <= 2^24
      const float rh = __frcp_rn(n), rl = __fmul_rn(fmaf(-n, rh, 1.0f), rh);
      bool rep = true;   // every sum exact in fp64, as the definition's is
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        const long long t = total(ch);
        rep = rep && ((t < (1LL << 53) && t > -(1LL << 53)) || (long long)(double)t == t);
      }
      ok = __all_sync(0xFFFFFFFFu, rep);
      if (ok)
        m = make_float4(mean_of(total(0), U, rh, rl, dc), mean_of(total(1), U, rh, rl, dc),
                        mean_of(total(2), U, rh, rl, dc), mean_of(total(3), U, rh, rl, dc));
    }
    if (!ok) {  // fp64 sums in token order (exact for members of ordinary range)
      double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      for (int64_t n0 = 0; n0 < a.N; n0 += 32) {
        uint32_t mk = __ballot_sync(0xFFFFFFFFu, n0 + lane < a.N && asg[n0 + lane] == (uint8_t)j);
        for (; mk; mk &= mk - 1) {
          const int64_t tok = n0 + __ffs((int)mk) - 1;
          const uint2 xv = __ldg(reinterpret_cast<const uint2*>(a.x + ((size_t)tok * a.H + h) * 128 + 4 * lane));
          s0 += (double)__uint_as_float(xv.x << 16);
          s1 += (double)__uint_as_float(xv.x & 0xFFFF0000u);
          s2 += (double)__uint_as_float(xv.y << 16);
          s3 += (double)__uint_as_float(xv.y & 0xFFFF0000u);
        }
      }
      m = make_float4(__double2float_rn(__ddiv_rn(s0, dc)), __double2float_rn(__ddiv_rn(s1, dc)),
                      __double2float_rn(__ddiv_rn(s2, dc)), __double2float_rn(__ddiv_rn(s3, dc)));
    }
    *cr = m;
  }
  if (last) {
    // the bf16 result; NaN everywhere if a wait inside an assignment ran out
    const bool bad = *a.status != 0;
    const uint32_t nan2 = 0x7FFF7FFFu;
    reinterpret_cast<uint2*>(a.out + (size_t)w * 128)[lane] =
        bad ? make_uint2(nan2, nan2) : make_uint2(pack_bf16(m.x, m.y), pack_bf16(m.z, m.w));
    return;
  }
  emit_row(a, h, j, m, lane);
  if (lane == 0) a.counts[w] = 0;  // ready for the next assignment
}

// bf16 output of the initial centroids (no iteration).
__global__ void fit_out(const FitArgs a) {
  const int64_t n = (int64_t)a.H * a.C * 128;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    a.out[i] = __float2bfloat16_rn(a.cent[i]);
}

int sm_count() {
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) !=
                                                 cudaSuccess || nsm < 1)
    return 1;
  return nsm;
}

}  // namespace

static int npad_of(int C) { return C < 16 ? 16 : (C + 15) & ~15; }

size_t fit_workspace_bytes(int H, int d, int C, int64_t N) {
  const int Np = npad_of(C);
  size_t b = 256;                                               // status
  b += (size_t)round_up((int64_t)H * C * d * 4, 256);           // cent
  b += (size_t)round_up((int64_t)H * Np * 512, 256);            // images
  b += (size_t)round_up((int64_t)H * Np * 4, 256);              // norms
  b += 2 * (size_t)round_up((int64_t)H * 4, 256);               // largest exponent (and a reserved field)
  b += 2 * (size_t)round_up((int64_t)H * C * 4, 256);           // counts (and a reserved field)
  b += (size_t)round_up((int64_t)H * N, 256);                   // assignment
  b += (size_t)round_up((int64_t)H * N * 4, 256);               // token norms
  b += (size_t)round_up((int64_t)H * N * 4, 256);               // member lists
  return b;
}

void fit_carve(FitArgs& a, uint8_t* ws) {
  a.Npad = npad_of(a.C);
  uint8_t* p = ws;
  auto take = [&](int64_t bytes) {
    uint8_t* q = p;
    p += round_up(bytes, 256);
    return q;
  };
  a.status = reinterpret_cast<int32_t*>(take(256));
  a.cent = reinterpret_cast<float*>(take((int64_t)a.H * a.C * a.d * 4));
  a.img = take((int64_t)a.H * a.Npad * 512);
  a.nrm = reinterpret_cast<uint32_t*>(take((int64_t)a.H * a.Npad * 4));
  take((int64_t)a.H * 4);   // reserved
  a.emax = reinterpret_cast<int32_t*>(take((int64_t)a.H * 4));
  // member sums of at most N values below 2^(8 + room) each stay below 2^61, and
  // each value below 2^48 units
  int lg = 0;
  while (((int64_t)1 << lg) < a.N + 1) ++lg;
  a.room = 53 - lg < 40 ? 53 - lg : 40;  // values below 2^48 units: three fp32 limbs (fit_means)
  a.counts = reinterpret_cast<int32_t*>(take((int64_t)a.H * a.C * 4));
  take((int64_t)a.H * a.C * 4);   // reserved
  a.asg = take((int64_t)a.H * a.N);
  a.xn2 = reinterpret_cast<float*>(take((int64_t)a.H * a.N * 4));
  a.list = reinterpret_cast<int32_t*>(take((int64_t)a.H * a.N * 4));
  // members listed per centroid: twice the average where a token's index fits 16 bits
  a.wide = a.N > 65536;
  a.cap = (int32_t)((a.wide ? a.N : 2 * a.N) / a.C);
}

namespace {
// A launch that may start its prologue before the one in front of it has ended.
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t lc{};
  lc.gridDim = grid;
  lc.blockDim = dim3((unsigned)threads);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, k, static_cast<P>(args)...);
}
}  // namespace

cudaError_t launch_fit(const FitArgs& a, cudaStream_t st) {
  cudaError_t e;
  const int64_t prep_warps = (int64_t)a.H * a.Npad;
  fit_prep<<<(unsigned)((prep_warps + 15) / 16), 512, 0, st>>>(a);
  if (a.iters == 0) {
    const int64_t n = (int64_t)a.H * a.C * a.d;
    fit_out<<<(unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, st>>>(a);
    return cudaGetLastError();
  }
  CUtensorMap tm;
  if (!make_token_map(&tm, a.x, a.N, a.H, 128)) return cudaErrorInvalidValue;
  if ((e = cudaFuncSetAttribute(fit_assign, cudaFuncAttributeMaxDynamicSharedMemorySize, A_SMEM)) != cudaSuccess)
    return e;
  const int tiles = (int)((a.N + 127) / 128);
  const int units = a.H * tiles;
  const int sms = sm_count();
  const int grid = units < sms ? units : sms;
  const int64_t sb = (a.N + 7) / 8;
  e = launch_pdl(fit_scale, dim3((unsigned)(sb < 64 ? sb : 64), (unsigned)a.H), 256, 0, st, a);
  for (int it = 0; it < a.iters && e == cudaSuccess; ++it) {
    e = launch_pdl(fit_assign, dim3((unsigned)grid), ANT, A_SMEM, st, a, tm, tiles, units);
    if (e == cudaSuccess)
      e = launch_pdl(fit_means, dim3((unsigned)((int64_t)a.H * a.C)), 128, 0, st, a, (int)(it + 1 == a.iters));
  }
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace qwm

namespace qwm {

// ----------------------------------------------------------------------------
// Allocation-free variant of qwm_fit_centroids.
//
// Some callers cannot hand the library a scratch buffer: a plain C host
// program that only owns the input and output tensors it was given, or an
// inference engine whose device memory is already reserved by its own pool
// and which must not call cudaMalloc/cudaFree in the middle of generation
// (those calls can synchronise the whole device).  For them the k-means
// scratch (fp32 centroids, MMA operand images, norms, counts, assignment and
// member lists) lives in this file-scope device array instead.
// ----------------------------------------------------------------------------
namespace {

constexpr size_t kNoAllocFitScratchBytes = (size_t)16 << 20;  // 16 MiB per GPU that loads the library
static __device__ __align__(256) uint8_t g_fit_scratch[kNoAllocFitScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_fit_scratch_mutex;
void* g_fit_scratch_addr[kMaxDevices] = {};

}  // namespace
}  // namespace qwm

extern "C" QWM_API qwm_status qwm_fit_centroids_noalloc(const qwm_config* cfg, const void* x, int64_t N,
                                                        void* centroids, void* stream) {
  using namespace qwm;
  if (!cfg || !x || !centroids || N < 1) return QWM_ERR_INVALID_ARG;
  if (!config_supported(cfg)) return QWM_ERR_UNSUPPORTED;  // the same set qwm_fit_centroids accepts
  if (N > (int64_t)1 << 31) return QWM_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(x) & 15u) || (reinterpret_cast<uintptr_t>(centroids) & 15u))
    return QWM_ERR_INVALID_ARG;
  const size_t need = fit_workspace_bytes(cfg->num_heads, cfg->head_dim, cfg->num_centroids, N);
  if (need > kNoAllocFitScratchBytes) return QWM_ERR_CAPACITY;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return QWM_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return QWM_ERR_UNSUPPORTED;
  uint8_t* ws = nullptr;
  {
    // First call on a device: look up the device address of the array there
    // (in host code its name is only a host-side stand-in).
    std::lock_guard<std::mutex> lock(g_fit_scratch_mutex);
    if (!g_fit_scratch_addr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_fit_scratch) != cudaSuccess || !p) return QWM_ERR_CUDA;
      g_fit_scratch_addr[dev] = p;
    }
    ws = static_cast<uint8_t*>(g_fit_scratch_addr[dev]);
  }
  FitArgs a{};
  a.H = cfg->num_heads; a.d = cfg->head_dim; a.C = cfg->num_centroids; a.iters = cfg->kmeans_iters;
  a.N = N;
  a.x = static_cast<const __nv_bfloat16*>(x);
  a.out = static_cast<__nv_bfloat16*>(centroids);
  fit_carve(a, ws);
  // launch_fit clears the status word, the counts and the largest exponents
  // and writes every centroid, image and norm before reading it, so nothing
  // depends on what an earlier call left in the array.
  return launch_fit(a, static_cast<cudaStream_t>(stream)) == cudaSuccess ? QWM_OK : QWM_ERR_CUDA;
}

