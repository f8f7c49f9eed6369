// qstats.cu -- historical Query statistics and the principal Query basis on
// the GPU (Sec. 4.1 Eq. 6 and 8, Sec. 4.2 Eq. 15, App. C.3 cold start,
// App. D.1: per-head statistics kept incrementally, the basis recomputed at
// chunk boundaries, no past Query kept).
//
//   gram_kernel   S_h += Q_h^T Q_h for one chunk of Queries.  A tile of 64
//                 tokens x 128 channels is staged by TMA (128-byte swizzle,
//                 token rows) and serves as both MMA operands read MN-major:
//                 M = N = 128 channels, K = 16 tokens per tcgen05.mma, the
//                 fp32 accumulator in TMEM.  A cluster of S CTAs splits the
//                 tokens of one head; the S partial sums meet in distributed
//                 shared memory and are added to S_h in rank order, so the
//                 result does not depend on timing.
//   basis_kernel  w from the diagonal of S (Eq. 8) and the eigenvalues and
//                 leading eigenvectors of M = S / count in fp32 (Eq. 15):
//                 Householder tridiagonalisation, multisection, inverse
//                 iteration, back-transformation; one CTA per head.
#include <type_traits>

#include "qwm_internal.cuh"
#include "ptx_sm103.cuh"

namespace qwm {
namespace {
using namespace ptx;

constexpr int kStatsHeader = 256;   // status word, count, solver steps; then the sums

// ------------------------------------------------------------------ Gram sums
constexpr int kGTok = 64;                        // tokens per stage
constexpr int kGStages = 6;
constexpr int kGStage = kGTok * 256;             // two 8 KB boxes: channels [0,64) and [64,128)
constexpr int kGThreads = 128;
constexpr int kGBarOff = kGStages * kGStage;     // the [128][128] fp32 partial reuses the stages
constexpr int kGBarBytes = (2 * kGStages + 1) * 8;
constexpr int kGSmem = kGBarOff + kGBarBytes + 8 + 1024;   // barriers, TMEM slot, flag, alignment slack
static_assert(kGStages * kGStage >= 128 * 128 * 4, "partial sum buffer");

__global__ void __launch_bounds__(kGThreads) gram_kernel(const __grid_constant__ CUtensorMap tm, uint8_t* stats,
                                                         int64_t N, int S) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t base = smem_u32(sm);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + kGBarOff);  // full[kGStages], empty[kGStages], done
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + kGBarOff + kGBarBytes);
  volatile int* s_err = reinterpret_cast<volatile int*>(sm + kGBarOff + kGBarBytes + 4);
  auto bar = [&](int i) { return smem_u32(bars + i); };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int h = blockIdx.y;
  const int rank = (int)cluster_rank();
  const int64_t ntile = (N + kGTok - 1) / kGTok;
  const int my = (int)((ntile - rank + S - 1) / S);  // tiles rank, rank + S, ...; >= 1 as S <= ntile

  if (tid == 0) {
    for (int i = 0; i < 2 * kGStages + 1; ++i) mbar_init(bar(i), 1);
    *s_err = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tslot), 128);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tD = *tslot;

  // rows [rank R, rank R + R) of the running sum S_h, which this CTA updates
  // at the end: loaded now, while the tiles stream in
  const int R = 128 / S;                                  // S in {1, 2, 4, 8}
  float4* gS = reinterpret_cast<float4*>(stats + kStatsHeader) + (size_t)h * (128 * 32);
  float4 acc[32];                                         // R * 32 / 128 <= 32 items per thread
  const int nit = R / 4;
#pragma unroll
  for (int m = 0; m < 32; ++m)
    if (m < nit) acc[m] = gS[rank * R * 32 + tid + 128 * m];

  if (warp == 0) {
    if (lane == 0) {  // TMA producer
      prefetch_tmap(&tm);
      for (int k = 0; k < my; ++k) {
        const int s = k % kGStages;
        if (k >= kGStages && !mbar_wait(bar(kGStages + s), ((k / kGStages) - 1) & 1)) {
          *s_err = 1;
          break;
        }
        const int n0 = (int)(((int64_t)rank + (int64_t)k * S) * kGTok);
        const uint32_t dst = base + s * kGStage;
        mbar_arrive_expect_tx(bar(s), kGStage);
        tma_load_3d(dst, &tm, 0, h, n0, bar(s));
        tma_load_3d(dst + kGStage / 2, &tm, 64, h, n0, bar(s));
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer: D[c][e] += sum over the tile's tokens of q_c q_e
      constexpr uint32_t id = idesc_f16_mn(128, 128, true);
      for (int k = 0; k < my; ++k) {
        const int s = k % kGStages;
        if (!mbar_wait(bar(s), (k / kGStages) & 1)) {
          *s_err = 1;
          break;
        }
        tc_fence_after();
        const uint32_t a = base + s * kGStage;
#pragma unroll
        for (int ks = 0; ks < kGTok / 16; ++ks) {
          const uint64_t dsc = desc_sw128_mn(a + ks * 2048, kGStage / 2);
          umma_ss(tD, dsc, dsc, id, (k | ks) != 0);
        }
        umma_commit(bar(kGStages + s));
      }
      umma_commit(bar(2 * kGStages));  // every MMA issued above has completed
    }
    __syncwarp();
  }

  // ---- this CTA's partial sum: TMEM -> shared memory, row c = TMEM lane c,
  // float4 chunks XOR-swizzled by c % 8 (conflict-free stores and loads)
  bool ok = mbar_wait(bar(2 * kGStages), 0);
  ok = __all_sync(0xFFFFFFFFu, ok);
  tc_fence_after();
  float4* red = reinterpret_cast<float4*>(sm);
  const int row = warp * 32 + lane;
#pragma unroll 1
  for (int cb = 0; cb < 4; ++cb) {
    float v[32];
    if (ok) {
      tmem_ld32(tD + ((uint32_t)(warp * 32) << 16) + (uint32_t)(cb * 32), v);
    } else {
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = 0.0f;
    }
#pragma unroll
    for (int e4 = 0; e4 < 8; ++e4) {
      const int c4 = cb * 8 + e4;
      red[row * 32 + (c4 ^ (row & 7))] = make_float4(v[4 * e4], v[4 * e4 + 1], v[4 * e4 + 2], v[4 * e4 + 3]);
    }
  }
  if (!ok && lane == 0) *s_err = 1;
  tc_fence_before();
  cluster_sync();
  tc_fence_after();

  // ---- the running sum plus the partials of ranks 0, 1, ..., S-1, in that
  // order; the loads of all ranks for a row are issued before the adds
  const uint32_t red_s = smem_u32(red);
#pragma unroll
  for (int m = 0; m < 32; ++m) {
    if (m < nit) {
      const int i = tid + 128 * m;
      const int r = rank * R + (i >> 5), c4 = i & 31;
      const uint32_t off = red_s + (uint32_t)((r * 32 + (c4 ^ (r & 7))) * 16);
      float4 p[8];
#pragma unroll
      for (int src = 0; src < 8; ++src)
        if (src < S) p[src] = ld_dsmem_f4(mapa(off, (uint32_t)src));
#pragma unroll
      for (int src = 0; src < 8; ++src)
        if (src < S) {
          acc[m].x += p[src].x;
          acc[m].y += p[src].y;
          acc[m].z += p[src].z;
          acc[m].w += p[src].w;
        }
      gS[rank * R * 32 + i] = acc[m];
    }
  }
  cluster_sync();  // no CTA leaves while its partial is still being read
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tD, 128);
  if (tid == 0) {
    if (*s_err) atomicCAS(reinterpret_cast<int*>(stats), 0, (int)QWM_ERR_TIMEOUT);
    if (h == 0 && rank == 0) *reinterpret_cast<unsigned long long*>(stats + 8) += (unsigned long long)N;
  }
}

// ------------------------------------------------------------------ Query basis
constexpr int kBThreads = 512;
constexpr int kVecs = 32;                        // eigenvectors kept at most (the largest PSAC rank)
constexpr int kXs = kVecs + 1;                   // row stride of the vectors [128][kXs]
// shared memory, in floats
constexpr int Q_HV = 0;                          // Householder vectors [126][128], unnormalised
constexpr int Q_LU = Q_HV + 126 * 128;           // tridiagonal LU factors [4][128][kVecs]
constexpr int Q_X = Q_LU + 4 * 128 * kVecs;      // right-hand sides, vectors [128][kXs]
constexpr int Q_HC = Q_X + 128 * kXs;            // Householder scales [128]
constexpr int Q_D = Q_HC + 128;                  // T: diagonal, off-diagonal, its square [128] each
constexpr int Q_E = Q_D + 128;
constexpr int Q_E2 = Q_E + 128;
constexpr int Q_LAM = Q_E2 + 128;                // eigenvalues, decreasing
constexpr int Q_XB = Q_LAM + 128;                // two buffers of 128
constexpr int Q_RED = Q_XB + 256;                // [32]
constexpr int Q_CNT = Q_RED + 32;                // counts at the grid points [512]
constexpr int Q_ORD = Q_CNT + 512;               // order of a diagonal matrix [128]
constexpr int kBasisSmem = (Q_ORD + 128) * 4;
constexpr int kIter = 2;                         // steps of inverse iteration, at least
constexpr int kMaxIter = 30;                     // at most (a basis that took as many has not converged)
constexpr float kResidual = 7.6293945e-6f;       // 2^-17 of the norm: largest entry of T y - lambda y
constexpr float kTinyPivot = 1.1920929e-7f;      // 2^-23 of the matrix norm

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  return x;
}

// Number of eigenvalues of the tridiagonal T (norm <= 1) below x: sign changes
// of the leading principal minors p_i = (d_i - x) p_(i-1) - e_(i-1)^2 p_(i-2).
// e^2 is at least 2^-60 (e moved by less than fp32's rounding of the matrix),
// so a minor that is exactly zero is followed by one that is not, and four
// steps between two rescalings stay inside the fp32 range.
__device__ __forceinline__ int sturm_count(const float* d, const float* e2, float x) {
  float p0 = 0.0f, p1 = 1.0f;
  int n = 0;
#pragma unroll 1
  for (int j = 0; j < 128; j += 32) {
    uint32_t chg = 0u;   // one bit per step
#pragma unroll 4
    for (int i = j; i < j + 32; i += 4) {
      const float4 dv = *reinterpret_cast<const float4*>(d + i);
      const float4 ev = *reinterpret_cast<const float4*>(e2 + i);   // e2[i] couples i - 1 and i
      const float dd[4] = {dv.x, dv.y, dv.z, dv.w}, ee[4] = {ev.x, ev.y, ev.z, ev.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float p = fmaf(dd[k] - x, p1, -(ee[k] * p0));
        chg = __funnelshift_l(__float_as_uint(p) ^ __float_as_uint(p1), chg, 1);
        p0 = p1;
        p1 = p;
      }
      const uint32_t ex = __float_as_uint(fmaxf(fabsf(p0), fabsf(p1))) >> 23;
      const float sc = __uint_as_float((254u - ex) << 23);   // 2^-exponent of the larger
      p0 *= sc;
      p1 *= sc;
    }
    n += __popc(chg);
  }
  return n;
}

// w from the diagonal of S (Eq. 8) and the leading eigenvectors of M = S /
// count (Eq. 15), one CTA per head: Householder tridiagonalisation with M in
// registers (thread = 4 rows x 8 columns), eigenvalues by multisection on
// Sturm counts, the r leading vectors by inverse iteration from fixed
// pseudo-random vectors (LU with partial pivoting, a thread per vector; two
// steps, and more while a residual is above 2^-17 of the norm), each step
// followed by modified Gram-Schmidt in decreasing order (so equal eigenvalues
// get an orthonormal basis), and the Householder vectors applied back.  A matrix whose off-diagonal entries are all below 2^-20 of its norm
// counts as diagonal.
// Bound by the latency of its serial chain: at 40 heads 126 reduction steps of
// 1.7 K cycles (214 K), multisection 42 K, LU 11 K, inverse iteration and
// Gram-Schmidt 35 K, back-transformation 19 K (r = 16).  With a row and a
// quarter of its columns per thread a step took 2.1 K cycles: every thread then
// read 32 values of v and of p from shared memory, 1 K cycles of its bandwidth.
// Statistics reset, update and basis of the Wan-14B layer: 884 us with cyclic
// Jacobi (7 sweeps of 127 rounds of 2 K cycles), 191 us (189 without the
// residuals).
__global__ void __launch_bounds__(kBThreads, 1) basis_kernel(uint8_t* stats, float* w, __nv_bfloat16* U, float* evals,
                                                             int r, int eig) {
  extern __shared__ __align__(16) float js[];
  float* red = js + Q_RED;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int h = blockIdx.x;
  const unsigned long long cnt = *reinterpret_cast<const unsigned long long*>(stats + 8);
  const float* S = reinterpret_cast<const float*>(stats + kStatsHeader) + (size_t)h * 128 * 128;

  // ---- Eq. 8: w_c = S_cc / mean_c' S_c'c' (the 1/count of M cancels)
  if (tid < 128) {
    const float dg = S[tid * 129];
    float t = dg;
#pragma unroll
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    if (lane == 0) red[warp] = t;
    named_bar_sync(1, 128);
    const float sum = (red[0] + red[1]) + (red[2] + red[3]);
    if (w) w[h * 128 + tid] = (cnt > 0 && sum > 0.0f) ? dg * 128.0f / sum : 1.0f;
  }
  if (!eig) return;
  __syncthreads();

  // ---- M = S / count: thread (g, c) holds rows g + 32 s, columns 4 (c + 16 m)
  // .. + 3 (s < 4, m < 2): as many rows as columns, because every step reads v
  // and p for the columns from shared memory, 128 bytes a cycle for the whole SM
  const int g = tid >> 4, c = tid & 15;
  const float inv = cnt ? (float)(1.0 / (double)cnt) : 0.0f;
  uint64_t a[4][4];
  float top = 0.0f, offmax = 0.0f;
#pragma unroll
  for (int sl = 0; sl < 4; ++sl)
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const int i = g + 32 * sl, j0 = 4 * (c + 16 * m);
      const float4 v = *reinterpret_cast<const float4*>(S + i * 128 + j0);
      const float x[4] = {v.x * inv, v.y * inv, v.z * inv, v.w * inv};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (j0 + e == i) js[Q_D + i] = x[e];
        else offmax = fmaxf(offmax, fabsf(x[e]));
        top = fmaxf(top, fabsf(x[e]));
      }
      a[sl][2 * m] = f2pack(x[0], x[1]);
      a[sl][2 * m + 1] = f2pack(x[2], x[3]);
    }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    offmax = fmaxf(offmax, __shfl_xor_sync(0xFFFFFFFFu, offmax, o));
    top = fmaxf(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
  }
  if (lane == 0) {
    red[warp] = top;
    red[16 + warp] = offmax;
  }
  __syncthreads();
  for (int k = 0; k < 16; ++k) {
    top = fmaxf(top, red[k]);
    offmax = fmaxf(offmax, red[16 + k]);
  }
  // entries scaled (by a power of two) to at most 1
  int ex0 = 0;
  if (top > 0.0f && top < INFINITY) frexpf(top, &ex0);
  ex0 = ex0 < -126 ? -126 : ex0;
  const float sc0 = ldexpf(1.0f, -ex0);
  float ss = 0.0f;
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    float x0, x1;
    a[m >> 2][m & 3] = mul2(a[m >> 2][m & 3], f2pack(sc0, sc0));
    f2unpack(a[m >> 2][m & 3], x0, x1);
    ss = fmaf(x0, x0, fmaf(x1, x1, ss));
  }
  offmax *= sc0;
  ss = warp_sum(ss);
  __syncthreads();
  if (lane == 0) red[warp] = ss;
  __syncthreads();
  float fro2 = 0.0f;
  for (int k = 0; k < 16; ++k) fro2 += red[k];
  // not above the threshold, a norm that is not finite included: diagonal
  if (!(offmax > ldexpf(sqrtf(fro2), -20)) || !(fro2 < INFINITY)) {
    int* order = reinterpret_cast<int*>(js + Q_ORD);
    if (tid < 128) {   // decreasing order (equal values by increasing index; NaN last)
      float ki = js[Q_D + tid];
      if (ki != ki) ki = -INFINITY;
      int rk = 0;
      for (int j = 0; j < 128; ++j) {
        float kj = js[Q_D + j];
        if (kj != kj) kj = -INFINITY;
        rk += (kj > ki) || (kj == ki && j < tid);
      }
      order[rk] = tid;
      if (evals) evals[h * 128 + rk] = js[Q_D + tid];
    }
    if (tid == 0) atomicMax(reinterpret_cast<int*>(stats + 16), 1);
    __syncthreads();
    if (U)
      for (int e = tid; e < 128 * r; e += kBThreads) {
        const int row = e / r, j = e - row * r;
        U[((size_t)h * 128 + row) * r + j] = __float2bfloat16_rn(cnt && order[j] == row ? 1.0f : 0.0f);
      }
    return;
  }

  // ---- T = Q^T M Q: step k takes row k past the diagonal (x, zero up to k) to
  // beta e_(k+1) with H = I - s v v^T, v = x - beta e_(k+1), s = 1 / (beta (beta
  // - x_(k+1))); p = s A v, K = s p.v / 2, A -= v (p - K v)^T + (p - K v) v^T.
  float* xb = js + Q_XB;        // v of the step
  float* pb = xb + 128;
  float* hs = js + Q_RED + 16;  // s of the step
  // row k (slot E = k / 32, threads g = k % 32) of the current matrix: d_k, e_(k+1) = beta, v and s
  auto publish = [&](auto slot, int k) {
    constexpr int E = decltype(slot)::value;
    if (g != (k & 31)) return;
    const uint32_t half = 0xFFFFu << (lane & 16);
    float x[8], sig = 0.0f, alpha = 0.0f;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      f2unpack(a[E][2 * m], x[4 * m], x[4 * m + 1]);
      f2unpack(a[E][2 * m + 1], x[4 * m + 2], x[4 * m + 3]);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = 4 * (c + 16 * m) + e;
        if (j == k) js[Q_D + k] = x[4 * m + e];
        x[4 * m + e] = j > k ? x[4 * m + e] : 0.0f;
        alpha = j == k + 1 ? x[4 * m + e] : alpha;
        sig = fmaf(x[4 * m + e], x[4 * m + e], sig);
      }
    }
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      sig += __shfl_xor_sync(half, sig, o);
      alpha += __shfl_xor_sync(half, alpha, o);
    }
    const bool refl = sig > 1e-30f;   // entries are at most 1: a smaller row counts as zero
    const float beta = -copysignf(sig * rsqrtf(fmaxf(sig, 1e-30f)), alpha);
    const float vk1 = alpha - beta;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const int j0 = 4 * (c + 16 * m);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j0 + e == k + 1) x[4 * m + e] = vk1;
      const float4 o = make_float4(x[4 * m], x[4 * m + 1], x[4 * m + 2], x[4 * m + 3]);
      *reinterpret_cast<float4*>(xb + j0) = o;
      if (k < 126) *reinterpret_cast<float4*>(js + Q_HV + k * 128 + j0) = o;   // for the back-transformation
    }
    if (c == 0) {
      const float s = refl ? __fdividef(1.0f, beta * (beta - alpha)) : 0.0f;
      hs[0] = s;
      js[Q_HC + k] = s;
      if (k < 127) js[Q_E + k + 1] = k == 126 ? alpha : (refl ? beta : 0.0f);
    }
  };
  // steps 32 E .. 32 E + 31: rows of the slots before E and, from E = 2, columns below 64 are done
  auto segment = [&](auto slot) {
    constexpr int E = decltype(slot)::value, M0 = E >> 1;
#pragma unroll 1
    for (int k = 32 * E; k < (E == 3 ? 126 : 32 * E + 32); ++k) {
      const float s = hs[0];
      uint64_t v[4];
#pragma unroll
      for (int m = M0; m < 2; ++m) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(xb + 4 * (c + 16 * m));
        v[2 * m] = t.x;
        v[2 * m + 1] = t.y;
      }
      float p[4] = {0.0f, 0.0f, 0.0f, 0.0f}, vr[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int sl = E; sl < 4; ++sl) {
        vr[sl] = xb[g + 32 * sl];
        uint64_t acc = 0;
#pragma unroll
        for (int q = 2 * M0; q < 4; ++q) acc = fma2(a[sl][q], v[q], acc);
        float y0, y1;
        f2unpack(acc, y0, y1);
        p[sl] = y0 + y1;
      }
      // sums over the 16 threads of a row, a row slot per lane quarter: lane bits 3, 2 = slot
      const bool b3 = lane & 8, b2 = lane & 4;
      float u0 = b3 ? p[2] : p[0], u1 = b3 ? p[3] : p[1];
      u0 += __shfl_xor_sync(0xFFFFFFFFu, b3 ? p[0] : p[2], 8);
      u1 += __shfl_xor_sync(0xFFFFFFFFu, b3 ? p[1] : p[3], 8);
      float pr = b2 ? u1 : u0;
      pr += __shfl_xor_sync(0xFFFFFFFFu, b2 ? u0 : u1, 4);
      pr += __shfl_xor_sync(0xFFFFFFFFu, pr, 2);
      pr += __shfl_xor_sync(0xFFFFFFFFu, pr, 1);
      const int sl_of = (lane >> 2) & 3, i = g + 32 * sl_of;
      pr = i > k ? pr * s : 0.0f;
      if ((lane & 3) == 0) pb[i] = pr;
      float kp = pr * (b3 ? (b2 ? vr[3] : vr[2]) : (b2 ? vr[1] : vr[0]));
      kp += __shfl_xor_sync(0xFFFFFFFFu, kp, 4);
      kp += __shfl_xor_sync(0xFFFFFFFFu, kp, 8);
      kp += __shfl_xor_sync(0xFFFFFFFFu, kp, 16);
      if (lane == 0) red[warp] = kp;
      __syncthreads();
      float K = red[lane & 15];
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) K += __shfl_xor_sync(0xFFFFFFFFu, K, o);
      K *= -0.5f * s;
      const uint64_t nK = f2pack(K, K);
      uint64_t w2[4];
#pragma unroll
      for (int m = M0; m < 2; ++m) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(pb + 4 * (c + 16 * m));
        w2[2 * m] = fma2(nK, v[2 * m], t.x);
        w2[2 * m + 1] = fma2(nK, v[2 * m + 1], t.y);
      }
#pragma unroll
      for (int sl = E; sl < 4; ++sl) {
        const float wi = fmaf(K, vr[sl], pb[g + 32 * sl]);
        const uint64_t nv = f2pack(-vr[sl], -vr[sl]), nw = f2pack(-wi, -wi);
#pragma unroll
        for (int q = 2 * M0; q < 4; ++q) a[sl][q] = fma2(nv, w2[q], fma2(nw, v[q], a[sl][q]));
      }
      if (E < 3 && k == 32 * E + 31) publish(std::integral_constant<int, (E < 3 ? E + 1 : 3)>(), k + 1);
      else publish(slot, k + 1);
      __syncthreads();
    }
  };
  publish(std::integral_constant<int, 0>(), 0);
  __syncthreads();
  segment(std::integral_constant<int, 0>());
  segment(std::integral_constant<int, 1>());
  segment(std::integral_constant<int, 2>());
  segment(std::integral_constant<int, 3>());
  publish(std::integral_constant<int, 3>(), 127);
  if (tid == 0) js[Q_E] = 0.0f;
  __syncthreads();

  // ---- scale T to norm <= 1 (a power of two), Gershgorin bounds
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int j = lane + 32 * q;
    const float rad = fabsf(js[Q_E + j]) + (j < 127 ? fabsf(js[Q_E + j + 1]) : 0.0f);
    lo = fminf(lo, js[Q_D + j] - rad);
    hi = fmaxf(hi, js[Q_D + j] + rad);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xFFFFFFFFu, hi, o));
  }
  int ex;
  frexpf(fmaxf(fabsf(lo), fabsf(hi)), &ex);   // norm < 2^ex
  const float scale = ldexpf(1.0f, -ex), unscale = ldexpf(1.0f, ex + ex0);
  __syncthreads();
  if (tid < 128) {
    const float e = js[Q_E + tid] * scale;
    js[Q_D + tid] *= scale;
    js[Q_E + tid] = e;
    js[Q_E2 + tid] = fmaxf(e * e, 8.6736174e-19f);   // 2^-60 (see sturm_count)
  }
  lo = lo * scale - 1e-6f;
  hi = hi * scale + 1e-6f;
  __syncthreads();

  // ---- eigenvalues: counts at a grid of 128 points, then each one's interval
  // in sections, a point per thread.  The leading ones (r of them at least) by
  // threads 0 .. 127, the others, when they are asked for, by two threads each
  // of the warps after them: the leading ones, which the vectors' solves are
  // shifted by, are the same bits either way.  (A warp per sub-partition for
  // the leading ones: the counts of 16 warps are bound by issue, those of four
  // by latency.)
  {
    const float* d = js + Q_D;
    const float* e2 = js + Q_E2;
    int* gc = reinterpret_cast<int*>(js + Q_CNT);
    constexpr int np = 128;                                  // grid points
    const int lper = r > 16 ? 4 : r > 8 ? 8 : 16;            // threads per leading eigenvalue
    const int nlead = 128 / lper;
    const float st = (hi - lo) / (float)(np + 1);
    if (tid < np) gc[tid] = sturm_count(d, e2, fmaf(st, (float)(tid + 1), lo));
    __syncthreads();
    if (tid < 128 || (evals && warp < 4 + (2 * (128 - nlead) + 31) / 32)) {
      const int per = tid < 128 ? lper : 2;
      const int own = tid < 128 ? tid / lper : nlead + (tid - 128) / 2;
      const int ev = min(own, 127), q = tid & (per - 1);     // past the last one (in whole warps): its copies
      const int idx = 127 - ev;   // eigenvalue ev of the decreasing order is number idx of the increasing one
      int g0 = 0, g1 = np;        // first grid point with more than idx eigenvalues below it
      while (g0 < g1) {
        const int mid = (g0 + g1) >> 1;
        if (gc[mid] > idx) g1 = mid;
        else g0 = mid + 1;
      }
      float l = g0 == 0 ? lo : fmaf(st, (float)g0, lo), u = g0 == np ? hi : fmaf(st, (float)(g0 + 1), lo);
      const float part = 1.0f / (float)(per + 1);
      // until the interval is below 2^-24: 2 / 129 / 3^12, 5^8, 9^6, 17^5
      const int rounds = per == 2 ? 12 : per == 4 ? 8 : per == 8 ? 6 : 5;
#pragma unroll 1
      for (int it = 0; it < rounds; ++it) {
        const float wd = (u - l) * part;
        const float x = fmaf(wd, (float)(q + 1), l);
        const uint32_t above = __ballot_sync(0xFFFFFFFFu, sturm_count(d, e2, x) > idx) >> (lane & ~(per - 1));
        const uint32_t all = (1u << per) - 1u;
        const int first = __ffs((int)((above & all) | (all + 1u))) - 1;   // section that holds the eigenvalue
        const float nl = first == 0 ? l : fmaf(wd, (float)first, l);
        u = first == per ? u : fmaf(wd, (float)(first + 1), l);
        l = nl;
      }
      if (q == 0 && own == ev) js[Q_LAM + ev] = 0.5f * (l + u);
    }
  }
  __syncthreads();
  if (warp == 0) {   // rounding may not put a value above the one before it
    float run = INFINITY;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float x = js[Q_LAM + 32 * q + lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x = fminf(x, y);
      }
      x = fminf(x, run);
      run = __shfl_sync(0xFFFFFFFFu, x, 31);
      js[Q_LAM + 32 * q + lane] = x;
      if (evals) evals[h * 128 + 32 * q + lane] = x * unscale;
    }
  }
  if (!U || r == 0) {
    if (tid == 0) atomicMax(reinterpret_cast<int*>(stats + 16), 1);
    return;
  }
  __syncthreads();

  // ---- LU of T - lambda_j with partial pivoting (lane j of warp 0), pivots of
  // at least 2^-23 in magnitude
  float* fi = js + Q_LU;                 // 1 / pivot
  float* f1 = fi + 128 * kVecs;          // first and second superdiagonal of U
  float* f2 = f1 + 128 * kVecs;
  float* fl = f2 + 128 * kVecs;          // multiplier
  float* X = js + Q_X;
  uint32_t swp[4] = {0u, 0u, 0u, 0u};    // rows swapped
  if (warp == 0 && lane < r) {
    const float lam = js[Q_LAM + lane];
    float D = js[Q_D] - lam, Us = js[Q_E + 1];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll 4
      for (int b = 0; b < 32; ++b) {
        const int n = 32 * q + b;
        if (n == 127) break;
        const float e = js[Q_E + n + 1], dn = js[Q_D + n + 1] - lam, en = n < 126 ? js[Q_E + n + 2] : 0.0f;
        const bool s1 = fabsf(D) < fabsf(e);
        float piv = s1 ? e : D;
        piv = fabsf(piv) < kTinyPivot ? copysignf(kTinyPivot, piv) : piv;
        const float rp = rcp_approx(piv), l = (s1 ? D : e) * rp;
        const float m1 = s1 ? dn : Us, m2 = s1 ? en : 0.0f;
        D = fmaf(-l, m1, s1 ? Us : dn);
        Us = s1 ? -l * en : en;
        swp[q] |= (s1 ? 1u : 0u) << b;
        fi[n * kVecs + lane] = rp;
        f1[n * kVecs + lane] = m1;
        f2[n * kVecs + lane] = m2;
        fl[n * kVecs + lane] = l;
      }
    }
    if (fabsf(D) < kTinyPivot) D = copysignf(kTinyPivot, D);
    fi[127 * kVecs + lane] = __fdividef(1.0f, D);
    f1[127 * kVecs + lane] = 0.0f;
    f2[127 * kVecs + lane] = 0.0f;
  }
  // fixed pseudo-random start, entries of magnitude 2^-20 .. 2^-19 (a solve grows them by up to 2^23 and more)
  for (int e = tid; e < 128 * kVecs; e += kBThreads) {
    uint32_t z = (uint32_t)e * 2654435769u + 12345u;
    z ^= z >> 16;
    z *= 0x85EBCA6Bu;
    z ^= z >> 13;
    z *= 0xC2B2AE35u;
    z ^= z >> 16;
    X[(e / kVecs) * kXs + (e % kVecs)] = __uint_as_float((z & 0x807FFFFFu) | (107u << 23));
  }
  __syncthreads();
  // From here each vector lives in eight lanes (vector tid / 8, entries 4 (p +
  // 8 m) .. + 3, p = tid % 8): three shuffle steps a sum and few warps on the
  // shuffle and shared-memory pipes.
  const int vec = tid >> 3, vp = tid & 7, nact = r * 8;   // nact threads hold vectors (whole warps)
  auto sum8 = [](float x) {
    x += __shfl_xor_sync(0xFFFFFFFFu, x, 1);
    x += __shfl_xor_sync(0xFFFFFFFFu, x, 2);
    x += __shfl_xor_sync(0xFFFFFFFFu, x, 4);
    return x;
  };
  float y[16];
  int it = 0;
  for (;;) {
    if (warp == 0 && lane < r) {
      // eight steps' operands are loaded before the chain runs through them
      float bc = X[lane];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t sw = swp[q];
#pragma unroll 1
        for (int b0 = 32 * q; b0 < 32 * q + 32; b0 += 8) {
          float nx[8], l[8];
#pragma unroll
          for (int b = 0; b < 8; ++b) {
            const int n = min(b0 + b, 126);
            nx[b] = X[(n + 1) * kXs + lane];
            l[b] = fl[n * kVecs + lane];
          }
#pragma unroll
          for (int b = 0; b < 8; ++b) {
            if (b0 + b < 127) {
              const bool s1 = (sw >> b) & 1u;
              const float keep = s1 ? nx[b] : bc, other = s1 ? bc : nx[b];
              X[(b0 + b) * kXs + lane] = keep;
              bc = fmaf(-l[b], keep, other);
            }
          }
          sw >>= 8;
        }
      }
      X[127 * kXs + lane] = bc;
      float x1 = 0.0f, x2 = 0.0f;
#pragma unroll 1
      for (int n0 = 120; n0 >= 0; n0 -= 8) {
        float b[8], u1[8], u2[8], ip[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int n = n0 + k;
          b[k] = X[n * kXs + lane];
          u1[k] = f1[n * kVecs + lane];
          u2[k] = f2[n * kVecs + lane];
          ip[k] = fi[n * kVecs + lane];
        }
#pragma unroll
        for (int k = 7; k >= 0; --k) {
          const float x0 = fmaf(-u1[k], x1, fmaf(-u2[k], x2, b[k])) * ip[k];
          X[(n0 + k) * kXs + lane] = x0;
          x2 = x1;
          x1 = x0;
        }
      }
    }
    __syncthreads();
    bool bad = false;   // a residual above the tolerance, or no vector left
    // modified Gram-Schmidt, largest eigenvalue first
    if (tid < nact) {
      float mx = 0.0f;
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        y[m] = X[(4 * (vp + 8 * (m >> 2)) + (m & 3)) * kXs + vec];
        mx = fmaxf(mx, fabsf(y[m]));
      }
#pragma unroll
      for (int o = 4; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
      const float sc = mx > 0.0f && mx < INFINITY ? __fdividef(1.0f, mx) : 0.0f;
#pragma unroll
      for (int m = 0; m < 16; ++m) y[m] = fabsf(y[m]) < INFINITY ? y[m] * sc : 0.0f;
      // a second pass when a vector lost most of its length in the first (its
      // direction is then no longer orthogonal to fp32)
      float n0 = 0.0f;
#pragma unroll
      for (int m = 0; m < 16; ++m) n0 = fmaf(y[m], y[m], n0);
      n0 = sum8(n0);
      bool lost = false;
#pragma unroll 1
      for (int j = 0; j < r; ++j) {
        float4* vb = reinterpret_cast<float4*>(xb + 128 * (j & 1)) + vp;
        if (warp == (j >> 2)) {   // the vector's eight lanes are in this warp
          float s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
          for (int m = 0; m < 16; ++m) s4[m & 3] = fmaf(y[m], y[m], s4[m & 3]);
          const float n2 = sum8((s4[0] + s4[1]) + (s4[2] + s4[3]));
          if (vec == j) {
            const float sc1 = n2 > 0.0f ? rsqrtf(n2) : 0.0f;
            lost |= n2 < 1e-2f * n0;
            bad |= !(n2 > 0.0f);
#pragma unroll
            for (int m = 0; m < 16; ++m) y[m] *= sc1;
#pragma unroll
            for (int m = 0; m < 4; ++m) vb[8 * m] = make_float4(y[4 * m], y[4 * m + 1], y[4 * m + 2], y[4 * m + 3]);
          }
        }
        named_bar_sync(1, nact);
        if (warp >= (j >> 2)) {
          float b[16], s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const float4 t = vb[8 * m];
            b[4 * m] = t.x; b[4 * m + 1] = t.y; b[4 * m + 2] = t.z; b[4 * m + 3] = t.w;
          }
#pragma unroll
          for (int m = 0; m < 16; ++m) s4[m & 3] = fmaf(b[m], y[m], s4[m & 3]);
          const float dt = sum8((s4[0] + s4[1]) + (s4[2] + s4[3]));
          if (vec > j)
#pragma unroll
            for (int m = 0; m < 16; ++m) y[m] = fmaf(-dt, b[m], y[m]);
        }
        if (j == r - 1 && named_bar_or(1, nact, lost)) {
          j = -1;
          n0 = 0.0f;
          lost = false;
        }
      }
      // T y - lambda y: the neighbouring entries come from the lanes beside
      if (it + 1 >= kIter) {
        const float lam = js[Q_LAM + vec];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int i0 = 4 * (vp + 8 * m), base = lane & 24;
          const float before = vp == 7 ? (m > 0 ? y[4 * m - 1] : 0.0f) : y[4 * m + 3];
          const float after = vp == 0 ? (m < 3 ? y[4 * m + 4] : 0.0f) : y[4 * m];
          const float lf = __shfl_sync(0xFFFFFFFFu, before, base | ((vp + 7) & 7));
          const float rt = __shfl_sync(0xFFFFFFFFu, after, base | ((vp + 1) & 7));
          const float4 dv = *reinterpret_cast<const float4*>(js + Q_D + i0);
          const float4 ev = *reinterpret_cast<const float4*>(js + Q_E + i0);   // e[i] couples i - 1 and i
          const float e4 = i0 + 4 < 128 ? js[Q_E + i0 + 4] : 0.0f;
          const float r0 = fmaf(dv.x - lam, y[4 * m], fmaf(ev.x, lf, ev.y * y[4 * m + 1]));
          const float r1 = fmaf(dv.y - lam, y[4 * m + 1], fmaf(ev.y, y[4 * m], ev.z * y[4 * m + 2]));
          const float r2 = fmaf(dv.z - lam, y[4 * m + 2], fmaf(ev.z, y[4 * m + 1], ev.w * y[4 * m + 3]));
          const float r3 = fmaf(dv.w - lam, y[4 * m + 3], fmaf(ev.w, y[4 * m + 2], e4 * rt));
          bad |= !(fmaxf(fmaxf(fabsf(r0), fabsf(r1)), fmaxf(fabsf(r2), fabsf(r3))) <= kResidual);
        }
      }
    }
    // two steps, and more while a residual is above the tolerance
    ++it;
    if (!__syncthreads_or(it < kIter || bad) || it == kMaxIter) break;
    if (tid < nact)
#pragma unroll
      for (int m = 0; m < 16; ++m) X[(4 * (vp + 8 * (m >> 2)) + (m & 3)) * kXs + vec] = y[m] * 9.5367432e-7f;
    __syncthreads();
  }
  if (tid == 0) atomicMax(reinterpret_cast<int*>(stats + 16), it);
  if (tid >= nact) return;

  // ---- back to M's coordinates: H_0 ... H_125 y, two reflections at a time:
  // H_(k-1) H_k y needs v_k.y, v_(k-1).y and v_(k-1).v_k, whose sums run together
  const float4* hv = reinterpret_cast<const float4*>(js + Q_HV + 125 * 128) + vp;
#pragma unroll 1
  for (int k = 125; k > 0; k -= 2, hv -= 64) {
    float b[16], g[16], d4[4] = {0.0f, 0.0f, 0.0f, 0.0f}, g4[4] = {0.0f, 0.0f, 0.0f, 0.0f}, q4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const float4 t = hv[8 * m], u = hv[8 * m - 32];
      b[4 * m] = t.x; b[4 * m + 1] = t.y; b[4 * m + 2] = t.z; b[4 * m + 3] = t.w;
      g[4 * m] = u.x; g[4 * m + 1] = u.y; g[4 * m + 2] = u.z; g[4 * m + 3] = u.w;
    }
    const float s = -js[Q_HC + k], t = -js[Q_HC + k - 1];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      d4[m & 3] = fmaf(b[m], y[m], d4[m & 3]);
      g4[m & 3] = fmaf(g[m], y[m], g4[m & 3]);
      q4[m & 3] = fmaf(b[m], g[m], q4[m & 3]);
    }
    float d0 = (d4[0] + d4[1]) + (d4[2] + d4[3]), g0 = (g4[0] + g4[1]) + (g4[2] + g4[3]);
    float bg = (q4[0] + q4[1]) + (q4[2] + q4[3]);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      d0 += __shfl_xor_sync(0xFFFFFFFFu, d0, o);
      g0 += __shfl_xor_sync(0xFFFFFFFFu, g0, o);
      bg += __shfl_xor_sync(0xFFFFFFFFu, bg, o);
    }
    d0 *= s;
    g0 = t * fmaf(d0, bg, g0);
#pragma unroll
    for (int m = 0; m < 16; ++m) y[m] = fmaf(g0, g[m], fmaf(d0, b[m], y[m]));
  }
  // the sign rule (the largest |entry|, the first one on ties, is positive) and bf16
  float best = -1.0f, val = 0.0f;
  int bi = 0;
#pragma unroll
  for (int m = 0; m < 16; ++m)   // ascending entries of this lane
    if (fabsf(y[m]) > best) {
      best = fabsf(y[m]);
      val = y[m];
      bi = 4 * (vp + 8 * (m >> 2)) + (m & 3);
    }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const float ob = __shfl_xor_sync(0xFFFFFFFFu, best, o), ov = __shfl_xor_sync(0xFFFFFFFFu, val, o);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
    if (ob > best || (ob == best && oi < bi)) {
      best = ob;
      val = ov;
      bi = oi;
    }
  }
  const float sg = val < 0.0f ? -1.0f : 1.0f;
#pragma unroll
  for (int m = 0; m < 16; ++m)
    U[((size_t)h * 128 + 4 * (vp + 8 * (m >> 2)) + (m & 3)) * r + vec] = __float2bfloat16_rn(sg * y[m]);
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) !=
                                                 cudaSuccess || n < 1)
    return 1;
  return n;
}

bool stats_ok(const qwm_config* cfg, const void* stats) {
  return cfg && stats && config_supported(cfg) && (reinterpret_cast<uintptr_t>(stats) & 255u) == 0;
}

}  // namespace
}  // namespace qwm

extern "C" {

QWM_API size_t qwm_query_stats_bytes(const qwm_config* cfg) {
  if (!cfg || !qwm::config_supported(cfg)) return 0;
  return (size_t)qwm::kStatsHeader + (size_t)cfg->num_heads * 128 * 128 * 4;
}

QWM_API qwm_status qwm_query_stats_reset(const qwm_config* cfg, void* stats, void* stream) {
  if (!cfg || !stats) return QWM_ERR_INVALID_ARG;
  if (!qwm::config_supported(cfg)) return QWM_ERR_UNSUPPORTED;
  if (!qwm::stats_ok(cfg, stats)) return QWM_ERR_INVALID_ARG;
  return cudaMemsetAsync(stats, 0, qwm_query_stats_bytes(cfg), static_cast<cudaStream_t>(stream)) == cudaSuccess
             ? QWM_OK
             : QWM_ERR_CUDA;
}

QWM_API qwm_status qwm_query_stats_update(const qwm_config* cfg, void* stats, const void* q, int64_t N,
                                          void* stream) {
  using namespace qwm;
  if (!cfg || !stats || N < 0) return QWM_ERR_INVALID_ARG;
  if (!config_supported(cfg)) return QWM_ERR_UNSUPPORTED;
  if (!stats_ok(cfg, stats)) return QWM_ERR_INVALID_ARG;
  if (N == 0) return QWM_OK;
  if (!q || (reinterpret_cast<uintptr_t>(q) & 15u)) return QWM_ERR_INVALID_ARG;
  if (N > ((int64_t)1 << 31) - kGTok) return QWM_ERR_UNSUPPORTED;
  const int H = cfg->num_heads;
  CUtensorMap tm;
  if (!make_token_map(&tm, q, N, H, kGTok)) return QWM_ERR_CUDA;
  // S CTAs per head (a power of two <= 8, at most one per token tile), as
  // many as keep the grid within two CTAs per SM
  const int64_t ntile = (N + kGTok - 1) / kGTok;
  const int slots = 2 * sm_count();
  int S = 1;
  while (S < 8 && 2 * S <= ntile && (int64_t)H * 2 * S <= slots) S *= 2;
  if (cudaFuncSetAttribute(gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGSmem) != cudaSuccess)
    return QWM_ERR_CUDA;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3((unsigned)S, (unsigned)H);
  lc.blockDim = dim3(kGThreads);
  lc.dynamicSmemBytes = kGSmem;
  lc.stream = static_cast<cudaStream_t>(stream);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)S;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  uint8_t* st = static_cast<uint8_t*>(stats);
  if (cudaLaunchKernelEx(&lc, gram_kernel, tm, st, N, S) != cudaSuccess) return QWM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? QWM_OK : QWM_ERR_CUDA;
}

QWM_API qwm_status qwm_query_basis(const qwm_config* cfg, const void* stats, float* w, void* U, float* eigenvalues,
                                   void* stream) {
  using namespace qwm;
  if (!cfg || !stats) return QWM_ERR_INVALID_ARG;
  if (!config_supported(cfg)) return QWM_ERR_UNSUPPORTED;
  if (!stats_ok(cfg, stats)) return QWM_ERR_INVALID_ARG;
  if ((w && (reinterpret_cast<uintptr_t>(w) & 3u)) || (eigenvalues && (reinterpret_cast<uintptr_t>(eigenvalues) & 3u)) ||
      (U && (reinterpret_cast<uintptr_t>(U) & 1u)))
    return QWM_ERR_INVALID_ARG;
  const int H = cfg->num_heads, r = cfg->psac_rank;
  __nv_bfloat16* Ub = (U && r > 0) ? static_cast<__nv_bfloat16*>(U) : nullptr;
  const int eig = (Ub || eigenvalues) ? 1 : 0;
  if (!w && !eig) return QWM_OK;
  if (cudaFuncSetAttribute(basis_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBasisSmem) != cudaSuccess)
    return QWM_ERR_CUDA;
  uint8_t* st = static_cast<uint8_t*>(const_cast<void*>(stats));
  basis_kernel<<<H, kBThreads, kBasisSmem, static_cast<cudaStream_t>(stream)>>>(st, w, Ub, eigenvalues, r, eig);
  return cudaGetLastError() == cudaSuccess ? QWM_OK : QWM_ERR_CUDA;
}

QWM_API qwm_status qwm_query_stats_read(void* stats, int32_t* status, int64_t* count, void* stream) {
  if (!stats || !status) return QWM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int64_t hdr[2] = {0, 0};
  if (cudaMemcpyAsync(hdr, stats, sizeof hdr, cudaMemcpyDeviceToHost, s) != cudaSuccess) return QWM_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return QWM_ERR_CUDA;
  const int32_t v = (int32_t)(hdr[0] & 0xFFFFFFFF);
  if (v != 0 && cudaMemsetAsync(stats, 0, sizeof(int32_t), s) != cudaSuccess) return QWM_ERR_CUDA;
  *status = v;
  if (count) *count = hdr[1];
  return QWM_OK;
}

}  // extern "C"
