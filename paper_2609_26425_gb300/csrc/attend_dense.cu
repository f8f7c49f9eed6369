// attend_dense.cu -- attention over the packed cache and the active chunk with
// a caller-owned scratch buffer (qwm_attend_ws): every key is rebuilt once per
// call into binary16 operand images in the scratch, and a dense attention
// kernel streams the images.
//
//   rebuild_kernel  a CTA per (128-token source tile, head, chunk): K_hat =
//                   mu_id + s (q - z) + (C U_r^T) (Sec. 2 Eq. 4, Sec. 4.2 Eq.
//                   17) and V_hat = mu_id + s (q - z), or the active chunk's
//                   rows, rounded once to binary16.  The keys of all chunks are
//                   packed without gaps, so that a 128-key tile of the images
//                   may hold the end of one chunk and the start of the next.
//   dense_kernel    persistent, one CTA per SM: 256 queries of one head (two
//                   128-row Q tiles) against a range of key tiles.
//   dense_combine   joins the partial results of the query blocks whose keys
//                   were split over several CTAs.
//
// Why the keys are rebuilt outside the attention kernel: a head's keys are
// read by ceil(Nq / 256) query blocks (19 at the Wan-14B layer) and inside the
// attention kernel (attend.cu) the rebuild took issue slots and memory pipes
// from the softmax and MMA warps in each of them.  Wan-14B layer (4680 queries,
// 32760 keys, 40 heads), whole call: 3.67 ms there, 2.14-2.24 ms here (rebuild
// 0.18, attention 1.87 ms = 1.67 PFLOP/s of MMA work; the longer figure under
// the power cap of back-to-back calls); 15 x 880 + 880 keys, 880 queries, 12
// heads: 154 -> 109 us; 4 heads, 880 queries, 2640 keys: 42 -> 29 us; 1024
// queries over 66544 keys, 40 heads: 1.62 -> 1.24 ms.
//
// The rebuild writes 512 bytes per token and head; its bulk stores alone take
// 111 us at the Wan-14B layer (6.0 TB/s), the whole kernel 178: it waits for the
// centroid rows (16 warps an SM).  The attention kernel runs at the tensor
// pipe's rate (64 cycles per 128 x 128 x 16 MMA, 32 of them a tile pair) less
// the gaps of the softmax -> MMA chain: 3.0 K cycles per 128 keys against 2.05 K.
// One CTA per 256 queries (cta_group::1) rather than pairs: hand-offs stay
// inside an SM, and the shared-memory reads of its MMAs do not slow them (the
// same 64 cycles with both operands in shared memory).
#include "ptx_sm103.cuh"
#include "qwm_internal.cuh"

namespace qwm {
namespace {

using namespace ptx;

constexpr int kImgTile = 65536;          // one 128-key tile: K image, then V image
constexpr int kImgSide = 32768;          // two blocks of [128 keys][64 channels] f16, 128-byte swizzled

__device__ __forceinline__ uint4 ldg16(const void* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ __half2 u2h(uint32_t u) { return *reinterpret_cast<__half2*>(&u); }

// 32-byte read-only global load (address 32-byte aligned).
__device__ __forceinline__ void ldg32B(const void* p, uint32_t (&r)[8]) {
  asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(p));
}
// Programmatic dependent launch: let the next kernel of the stream start its
// prologue / wait until the kernels before this one have completed.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t ex2_f16x2(uint32_t x) {
  uint32_t y;
  asm("ex2.approx.f16x2 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_f16_sat(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// ------------------------------------------------------------------ rebuild
// D[16 x 8] += A[16 x K] B[K x 8], binary16 operands, fp32 accumulation.  A:
// this thread's rows g = lane / 4 and g + 8, columns 2 t, 2 t + 1 (t = lane %
// 4) and the same + 8; B: rows like A's columns, column g; D: columns 2 t, 2 t + 1.
__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}
// Two PSAC INT8 codes (low half-word) times the row scale, each rounded once to
// binary16: byte t becomes the f16 1024 + (t + 128) (its byte XOR 0x80 under
// exponent bits 0x64), minus 1152 gives t exactly.
__device__ __forceinline__ uint32_t coef_f16x2(uint32_t w, __half2 sg2) {
  const uint32_t x = __byte_perm(w ^ 0x8080u, 0x64646464u, 0x4140u);
  const __half2 y = __hmul2(__hsub2(u2h(x), u2h(0x64806480u)), sg2);
  return *reinterpret_cast<const uint32_t*>(&y);
}
// a * b + c with binary16 a, b and fp32 c (fp32 result; the product is exact).
__device__ __forceinline__ float fma_mixed(unsigned short a, unsigned short b, float c) {
  float d;
  asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(d) : "h"(a), "h"(b), "f"(c));
  return d;
}

constexpr int kRebThreads = 256;
constexpr int kUStride = 20;             // words per U row in shared memory (16 used at r = 32): no bank conflicts

// A warp's 32 rows of one tile and side are staged in shared memory, [2 blocks
// of 64 channels][32 rows][128 B] with the swizzle of their image rows, and
// leave as bulk copies (a contiguous range of each block of the image): written
// from registers, 16 or 32 bytes a lane, the images went out at 3.0 TB/s.
constexpr int kStage = 8192;
constexpr int kRecord = 15360;            // a tile's packed record, at most (15104 bytes at G = 32, r = 32)
constexpr int kRebSmem = kRebThreads / 32 * kStage + 2 * kRecord;
__device__ __forceinline__ void stage_row(uint8_t* stg, int i, int xr, int t, int sl, uint4 lo, uint4 hi) {
  const int sw = ((xr & 7) ^ (2 * t)) << 4;   // chunks 2 t, 2 t + 1 of image row xr
  uint8_t* d = stg + sl * 4096 + i * 128;
  *reinterpret_cast<uint4*>(d + sw) = lo;
  *reinterpret_cast<uint4*>(d + (sw ^ 16)) = hi;
}
// Rows 0 .. n - 1 of the staging buffer to packed keys k, k + 1, ... of a side
// (relative to the image tile `img`, k < 256).  Whole warp.
__device__ __forceinline__ void store_rows(const uint8_t* stg, uint8_t* img, int k, int n, int lane) {
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) {
    const int n0 = max(0, min(n, 128 - k));   // rows in the first image tile
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
      const uint32_t src = smem_u32(stg + blk * 4096);
      uint8_t* d = img + blk * 16384;
      if (n0 > 0) bulk_s2g(d + k * 128, src, (uint32_t)n0 * 128u);
      if (n > n0) bulk_s2g(d + kImgTile + (k + n0 - 128) * 128, src + n0 * 128, (uint32_t)(n - n0) * 128u);
    }
    bulk_commit();
  }
}

// The lane's two binary16 group scales of a row (channels 16 t .. and 64 + 16 t
// ..), format 1's code * secondary scale rounded once to binary16.
template <int SF>
__device__ __forceinline__ void row_scales(const uint8_t* sp, const uint8_t* s2p, int row, int ng, int t, uint32_t& s0,
                                           uint32_t& s1) {
  if constexpr (SF == 0) {
    if (ng == 4) {
      const uint2 x = reinterpret_cast<const uint2*>(sp)[row];
      s0 = (t & 2) ? x.x >> 16 : x.x & 0xFFFFu;
      s1 = (t & 2) ? x.y >> 16 : x.y & 0xFFFFu;
    } else {
      const uint32_t x = reinterpret_cast<const uint32_t*>(sp)[row];
      s0 = x & 0xFFFFu;
      s1 = x >> 16;
    }
  } else {
    const __half s2 = __ushort_as_half(reinterpret_cast<const unsigned short*>(s2p)[row]);
    uint32_t c0, c1;
    if (ng == 4) {
      const uint32_t x = reinterpret_cast<const uint32_t*>(sp)[row];
      c0 = (t & 2) ? (x >> 8) & 0xFFu : x & 0xFFu;
      c1 = (t & 2) ? x >> 24 : (x >> 16) & 0xFFu;
    } else {
      const uint32_t x = reinterpret_cast<const unsigned short*>(sp)[row];
      c0 = x & 0xFFu;
      c1 = x >> 8;
    }
    s0 = __half_as_ushort(__hmul(__uint2half_rn(c0), s2));
    s1 = __half_as_ushort(__hmul(__uint2half_rn(c1), s2));
  }
}

// One 128-token tile's fields of a side, and where its rows go.
struct RebTile {
  const uint8_t *codes, *scales, *s2, *coef, *sigma;   // of the record's copy in shared memory
  const uint8_t* tab;   // centroid table (global), the lane's 32-byte slice
  uint4 pm;             // PSAC keep mask
  uint32_t idz;         // id | zero-points << 8 of this warp's row lane
  int r0, nv, ng;       // first row of the warp, rows of the tile, groups per row
  int key0;             // packed key of the tile's row 0, relative to its image tile
  uint8_t* stg;         // this warp's staging buffer
};

// Rows r0 .. r0 + 31 of a tile, 16 at a time: lane = (row g = lane / 4 and row
// g + 8, quarter t = lane % 4), which holds channels 16 t .. 16 t + 15 and 64 +
// 16 t .. of both rows, so that centroid slices are read as whole 32-byte
// sectors.  RK > 0: Keys with a PSAC correction C U_r^T, added by mma.sync to
// the fp32 value mu + s (q - z): its fragment layout is this lane mapping once
// the columns of U are taken in the order channel(b, n) = 64 (b / 8) + 16 (n /
// 2) + 2 (b % 8) + n % 2 of column n of block b, and its size (2 r of 4 x 128
// operations a token) is no work for tcgen05.  One rounding to binary16.
template <int SF, int RK>
__device__ __forceinline__ void rebuild_rows(const RebTile& x, const uint32_t* sU, int lane) {
  const int t = lane & 3, g = lane >> 2;
  const int gsh = x.ng == 4 ? 5 : 6;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    uint32_t mv[2][2][8], word[2][2], sc[2][2], zb[2];
    uint32_t ca[2][4];   // A fragments of the PSAC coefficients, two k-steps of 16 at most
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int lr = 16 * it + 8 * p + g, row = x.r0 + lr;
      const uint32_t idz = __shfl_sync(0xFFFFFFFFu, x.idz, lr);
      zb[p] = idz >> 8;
      const int rw = row < x.nv ? row : 0;   // rows past the chunk read row 0 (nothing is stored for them)
      const uint8_t* mu = x.tab + (idz & 0xFFu) * 256;
      ldg32B(mu, mv[p][0]);
      ldg32B(mu + 128, mv[p][1]);
      const uint32_t* cw = reinterpret_cast<const uint32_t*>(x.codes + rw * 32) + t;
      word[p][0] = cw[0];
      word[p][1] = cw[4];
      row_scales<SF>(x.scales, x.s2, rw, x.ng, t, sc[p][0], sc[p][1]);
      if constexpr (RK > 0) {
        ca[0][p] = ca[0][2 + p] = ca[1][p] = ca[1][2 + p] = 0u;
        const int e = row < x.nv ? psac_entry(x.pm, row) : -1;
        if (e >= 0) {
          const unsigned short sb = reinterpret_cast<const unsigned short*>(x.sigma)[e];
          const __half2 sg2 = u2h((uint32_t)sb | ((uint32_t)sb << 16));
          const unsigned short* cp = reinterpret_cast<const unsigned short*>(x.coef + e * RK) + t;
          ca[0][p] = coef_f16x2(cp[0], sg2);
          if constexpr (RK > 8) ca[0][2 + p] = coef_f16x2(cp[4], sg2);
          if constexpr (RK > 16) {
            ca[1][p] = coef_f16x2(cp[8], sg2);
            ca[1][2 + p] = coef_f16x2(cp[12], sg2);
          }
        }
      }
    }
#pragma unroll
    for (int sl = 0; sl < 2; ++sl) {
      const int gi = (64 * sl + 16 * t) >> gsh;
      __half2 z2[2];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const uint32_t zz = 0x6400u | ((zb[p] >> (2 * gi)) & 3u);
        z2[p] = u2h(zz | (zz << 16));
      }
      if constexpr (RK > 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {   // channels 64 sl + 16 t + 2 k, + 1
          float d[4];
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const uint32_t qq = ((word[p][sl] >> (2 * k)) & 0x00030003u) | 0x64006400u;
            const __half2 dq = __hsub2(u2h(qq), z2[p]);
            const float2 m = __half22float2(u2h(mv[p][sl][k]));
            d[2 * p] = fma_mixed(__half_as_ushort(__low2half(dq)), (unsigned short)sc[p][sl], m.x);
            d[2 * p + 1] = fma_mixed(__half_as_ushort(__high2half(dq)), (unsigned short)sc[p][sl], m.y);
          }
          const uint32_t* up = sU + (8 * (8 * sl + k) + g) * kUStride + t;
          if constexpr (RK == 8) {
            mma_k8(d, ca[0][0], ca[0][1], up[0]);
          } else {
            mma_k16(d, ca[0], up[0], up[4]);
            if constexpr (RK > 16) mma_k16(d, ca[1], up[8], up[12]);
          }
          mv[0][sl][k] = pack_f16_sat(d[0], d[1]);
          mv[1][sl][k] = pack_f16_sat(d[2], d[3]);
        }
      } else {
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const __half2 s2 = u2h(sc[p][sl] | (sc[p][sl] << 16));
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t qq = ((word[p][sl] >> (2 * k)) & 0x00030003u) | 0x64006400u;
            const __half2 y = __hfma2(__hsub2(u2h(qq), z2[p]), s2, u2h(mv[p][sl][k]));
            mv[p][sl][k] = *reinterpret_cast<const uint32_t*>(&y);
          }
        }
      }
    }
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int row = x.r0 + 16 * it + 8 * p + g;
#pragma unroll
      for (int sl = 0; sl < 2; ++sl)
        stage_row(x.stg, row - x.r0, x.key0 + row, t, sl, make_uint4(mv[p][sl][0], mv[p][sl][1], mv[p][sl][2], mv[p][sl][3]),
                  make_uint4(mv[p][sl][4], mv[p][sl][5], mv[p][sl][6], mv[p][sl][7]));
    }
  }
}

// Warps 0-3 rebuild 32 Key rows of a tile each, warps 4-7 the Value rows; a CTA
// runs `tpc` tiles of one chunk and head.
template <int SF, int R>
__global__ void __launch_bounds__(kRebThreads, 2) rebuild_kernel(const DenseArgs a, const AttendSlots S, int tpc) {
  extern __shared__ __align__(128) uint8_t s_stage[];   // kStage bytes per warp, then two packed records
  uint8_t* s_rec = s_stage + kRebThreads / 32 * kStage;
  __shared__ __align__(8) uint64_t s_bar[2];            // record copied
  __shared__ uint32_t sU[R > 0 ? 128 * kUStride : 1];
  pdl_launch();
  const Layout& L = a.L;
  const int u = blockIdx.z, tl0 = (int)blockIdx.x * tpc, h = a.h0 + (int)blockIdx.y;
  const bool cached = u < S.n;
  const int ntok = cached ? S.tokens[u] : (int)a.Ncur;
  if (tl0 * 128 >= ntok) return;
  const int tl1 = min(tl0 + tpc, (ntok + 127) >> 7);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, t = lane & 3, g = lane >> 2;
  const bool key = warp < 4;
  uint8_t* img = a.img + (size_t)blockIdx.y * a.NT * kImgTile + (key ? 0 : kImgSide);
  const uint8_t* hb = cached ? a.base + head_offset(L, S.slot[u], h) : nullptr;
  const bool psac = R > 0 && cached && S.psac[u];
  bool bad = false;
  // The packed records come by bulk copies, a tile ahead: read from global
  // memory in the warps, their latency (twice a tile) bound the kernel.
  int fetched = 0;   // copies issued (thread 0); none under the test hook's idle role
  auto fetch = [&](int tl) {
    if (a.idle_role == QWM_ROLE_V_REBUILD) return;
    ++fetched;
    const int b = (tl - tl0) & 1;
    mbar_arrive_expect_tx(smem_u32(s_bar + b), (uint32_t)L.tile_bytes);
    bulk_g2s(smem_u32(s_rec + b * kRecord), hb + L.tiles_off + (int64_t)tl * L.tile_bytes, (uint32_t)L.tile_bytes,
             smem_u32(s_bar + b));
  };
  if (cached && tid == 0) {
    mbar_init(smem_u32(s_bar), 1);
    mbar_init(smem_u32(s_bar + 1), 1);
    fence_mbar_init();
    fetch(tl0);
  }
  if constexpr (R > 0) {
    if (psac) {
      // U_r^T [r][128] as binary16 into rows of MMA columns n' = 8 b + n, r values each
      unsigned short* su = reinterpret_cast<unsigned short*>(sU);
      for (int i = tid; i < R * 16; i += kRebThreads) {
        const int k = i >> 4, c = 8 * (i & 15);
        const uint4 f = bf16x8_to_f16x8_sat(ldg16(hb + L.ut + (size_t)i * 16), bad);
        const uint32_t w4[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int np = 8 * ((c >> 6) * 8 + ((c & 15) >> 1) + e) + 2 * ((c >> 4) & 3);
          su[np * (2 * kUStride) + k] = (unsigned short)w4[e];
          su[(np + 1) * (2 * kUStride) + k] = (unsigned short)(w4[e] >> 16);
        }
      }
    }
  }
  const int r0 = (warp & 3) * 32;        // this warp's rows of each tile
  bool late = false;                     // a wait ran out (what follows is not used, but stays in bounds: id 0)
  bool stop = false;                     // some warp's wait ran out: tiles were left
  for (int tl = tl0; tl < tl1; ++tl) {
    const int nv = min(128, ntok - tl * 128);
    const int64_t key0 = a.key0[u] + tl * 128;     // the tile's first key among the packed keys
    RebTile x;
    x.stg = s_stage + warp * kStage;
    x.key0 = (int)(key0 & 127);
    const int n = max(0, min(32, nv - r0));
    if (tl > tl0) {
      if (lane == 0) bulk_wait_read();   // the previous tile's rows have left the buffer
      __syncwarp();
    }
    if (!cached) {
      // the active chunk's rows; values beyond binary16 saturate and are reported
#pragma unroll 2
      for (int it = 0; it < 4; ++it) {
        const int row = r0 + 8 * it + g;
        if (row >= nv) continue;
        const __nv_bfloat16* src = (key ? a.kcur : a.vcur) + ((size_t)(tl * 128 + row) * L.H + h) * 128 + 16 * t;
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) {
          const uint4 x0 = ldg16(src + 64 * sl), x1 = ldg16(src + 64 * sl + 8);
          const uint32_t w8[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
          uint32_t mag = 0u;
#pragma unroll
          for (int e = 0; e < 8; ++e) mag = vmax_u16x2(mag, w8[e] & 0x7FFF7FFFu);
          bad |= bf16x2_out_of_f16(mag);
          stage_row(x.stg, row - r0, x.key0 + row, t, sl, bf16x8_to_f16x8(x0), bf16x8_to_f16x8(x1));
        }
      }
      store_rows(x.stg, img + (size_t)(key0 >> 7) * kImgTile, x.key0 + r0, n, lane);
      continue;
    }
    uint4 pm = make_uint4(0u, 0u, 0u, 0u);
    if (psac && key) pm = ldg16(hb + L.pmask + (int64_t)tl * 16);
    // U_r and the barriers are in place; every warp is done with the record
    // before; nothing more is fetched once a wait has run out
    if (tl == tl0) __syncthreads();
    else if ((stop = __syncthreads_or(late))) break;
    if (tid == 0 && tl + 1 < tl1) fetch(tl + 1);
    if (!__all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(s_bar + ((tl - tl0) & 1)), ((tl - tl0) >> 1) & 1, a.wait_ns))) late = true;
    const uint8_t* tb = s_rec + ((tl - tl0) & 1) * kRecord;
    x.codes = tb + (key ? L.k_codes : L.v_codes);
    x.scales = tb + (key ? L.k_scales : L.v_scales);
    x.s2 = tb + (key ? L.k_s2 : L.v_s2);
    x.tab = hb + (key ? L.ktab : L.vtab) + 32 * t;
    x.coef = tb + L.k_coef;
    x.sigma = tb + L.k_sigma;
    x.r0 = r0;
    x.nv = nv;
    x.ng = L.ng;
    x.idz = 0u;
    if (r0 + lane < nv && !late)
      x.idz = (uint32_t)tb[(key ? L.k_ids : L.v_ids) + r0 + lane] |
              ((uint32_t)tb[(key ? L.k_zeros : L.v_zeros) + (r0 + lane) * L.zb] << 8);
    if (psac && key) {
      x.pm = pm;
      rebuild_rows<SF, R>(x, sU, lane);
    } else {
      rebuild_rows<SF, 0>(x, sU, lane);
    }
    store_rows(x.stg, img + (size_t)(key0 >> 7) * kImgTile, x.key0 + r0, n, lane);
  }
  // the last source tile zeroes the images' rows past the last key (the
  // attention kernel masks their logits; their Values must be finite)
  if (a.key0[u] + ntok == a.Nk && tl1 * 128 >= ntok) {
    for (int64_t kk = a.Nk + r0 / 4 + g; kk < (int64_t)a.NT * 128; kk += 32) {
      uint8_t* d = img + (size_t)(kk >> 7) * kImgTile + (kk & 127) * 128 + 32 * t;
#pragma unroll
      for (int sl = 0; sl < 4; ++sl)
        *reinterpret_cast<uint4*>(d + (sl >> 1) * 16384 + (sl & 1) * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  if (late && lane == 0) atomicCAS(a.status, 0, (int)QWM_ERR_TIMEOUT);
  if (bad) atomicCAS(a.status, 0, (int)QWM_ERR_NONFINITE);
  if (lane == 0) bulk_wait_all();
  // records still under way (a wait ran out) land before the CTA's memory goes away
  if (late || stop)
    for (int k = fetched > 2 ? fetched - 2 : 0; k < fetched; ++k)
      mbar_wait(smem_u32(s_bar + (k & 1)), (k >> 1) & 1, a.wait_ns);
}

// ------------------------------------------------------------------ attention
constexpr int kDWarps = 10;
constexpr int kDThreads = kDWarps * 32;
constexpr int W_MMA = 8;                         // warp 9 streams the images
constexpr float kTauLog2 = 8.0f;
constexpr int kStages = 5;                       // ring of K and V images, alternating
constexpr int D_Q = 0;                           // two Q tiles, 32 KB each
constexpr int D_KV = 65536;
constexpr int D_BAR = D_KV + kStages * kImgSide;
enum { B_FULL = 0, B_EMPTY = kStages, B_Q = 2 * kStages, B_S = B_Q + 2, B_P = B_S + 2, B_O = B_P + 4, B_DRAIN,
       D_NBAR };
constexpr int D_SMEM = D_BAR + 256 + 1024;
static_assert(D_NBAR * 8 + 16 <= 256 && D_SMEM <= 232448, "shared memory of the dense attention kernel");

// 8 f16 of row `row`, chunk `ch` into two 128-byte-swizzled blocks of 128 rows.
__device__ __forceinline__ void st_chunk(uint8_t* base, int row, int ch, uint4 v) {
  *reinterpret_cast<uint4*>(base + (ch >> 3) * 16384 + row * 128 + (((ch & 7) ^ (row & 7)) << 4)) = v;
}

// One item of a CTA: key tiles [lo, hi) of a query block; slot < 0: every key,
// written to the output; otherwise the slot of its partial result.
struct DenseItem {
  int unit, lo, hi, slot;
};
// First of CTA b's key tiles among the tail's flattened tiles: equal parts of
// one query block per CTA (tail_parts > 0), or tail_per tiles each, one more for
// the first tail_more CTAs, whatever block they fall in.
__device__ __forceinline__ int64_t tail_start(const DenseArgs& a, int b) {
  if (a.tail_parts > 0) {
    const int k = b / a.tail_parts;
    return (int64_t)k * a.NT + (int64_t)(b - k * a.tail_parts) * a.NT / a.tail_parts;
  }
  return (int64_t)b * a.tail_per + min(b, a.tail_more);
}
// Items of CTA b in order: one whole query block per full wave, then its share
// of the tail blocks' key tiles (contiguous over the tail's flattened tiles).
struct DenseItems {
  int w, seg;
  int64_t t0, t1;
  __device__ __forceinline__ void init(const DenseArgs& a) {
    w = 0;
    seg = 0;
    const int b = blockIdx.x;
    t0 = b < a.tail_ctas ? tail_start(a, b) : 0;
    t1 = b < a.tail_ctas ? tail_start(a, b + 1) : 0;
  }
  __device__ __forceinline__ bool next(const DenseArgs& a, DenseItem& it) {
    if (w < a.waves) {
      it.unit = w++ * (int)gridDim.x + (int)blockIdx.x;
      it.lo = 0;
      it.hi = a.NT;
      it.slot = -1;
      return true;
    }
    if (t0 >= t1) return false;
    const int k = (int)(t0 / a.NT);
    it.unit = a.waves * (int)gridDim.x + k;
    it.lo = (int)(t0 - (int64_t)k * a.NT);
    it.hi = (int)min((int64_t)a.NT, it.lo + (t1 - t0));
    it.slot = it.hi - it.lo == a.NT ? -1 : 2 * (int)blockIdx.x + seg;
    ++seg;
    t0 += it.hi - it.lo;
    return true;
  }
};

// Warps 0-3, 4-7: softmax of Q tile 0 / 1 (thread = query row); warp 8 issues
// the MMAs; warp 9 streams the K and V images (bulk copies, 5 stages of 32 KB).
// TMEM: S0 | S1 | O0 | O1, 128 fp32 columns each; P_i (f16) overwrites S_i.
// Order per key tile j: P0 V(j), S0(j+1), P1 V(j), S1(j+1).  Each half of P_i
// (64 keys) is handed over on its own, so that its MMAs run under the second
// half's exponentials.
__global__ void __launch_bounds__(kDThreads, 1) dense_kernel(const DenseArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = a.L.H;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + D_BAR);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + D_BAR + D_NBAR * 8);
  volatile int* s_err = reinterpret_cast<volatile int*>(sm + D_BAR + D_NBAR * 8 + 4);
  volatile int* s_bad = reinterpret_cast<volatile int*>(sm + D_BAR + D_NBAR * 8 + 8);  // a query beyond binary16
  const uint32_t bar0 = smem_u32(bars);
  auto bar = [&](int i) { return bar0 + 8 * i; };
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bar(B_FULL + s), 1);
      mbar_init(bar(B_EMPTY + s), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(B_Q + i), 4);
      mbar_init(bar(B_S + i), 1);
      mbar_init(bar(B_P + 2 * i), 4);
      mbar_init(bar(B_P + 2 * i + 1), 4);
    }
    mbar_init(bar(B_O), 1);
    mbar_init(bar(B_DRAIN), 1);
    *s_err = 0;
    *s_bad = 0;
    fence_mbar_init();
  }
  if (warp == W_MMA) {
    tmem_alloc(smem_u32(tslot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *tslot;
  pdl_launch();
  DenseItems items;
  items.init(a);
  DenseItem it;
  bool ok = true;

  if (warp < 8) {
    // ------------------------------------------------------------ softmax
    const int i = warp >> 2, row = tid & 127;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS = tbase + 128 * i + lrow, tO = tbase + 256 + 128 * i + lrow;
    uint8_t* sQi = sm + D_Q + i * kImgSide;
    const float sl2 = a.sm_scale * 1.4426950408889634f;
    const uint64_t SL = f2pack(sl2, sl2);
    uint32_t jt = 0, nit = 0;
    bool more = items.next(a, it);
    // the query row of an item into the operand buffer (free once the last S
    // of the item before has completed)
    auto load_q = [&](const DenseItem& x) {
      const int hl = x.unit / a.bph;
      const int64_t qi = (int64_t)(x.unit - hl * a.bph) * 256 + 128 * i + row;
      if (qi < a.Nq) {
        const __nv_bfloat16* src = a.q + ((size_t)qi * H + a.h0 + hl) * 128;
        bool qbad = false;
#pragma unroll
        for (int ch = 0; ch < 16; ++ch) st_chunk(sQi, row, ch, bf16x8_to_f16x8_sat(ldg16(src + ch * 8), qbad));
        if (qbad) *s_bad = 1;
      } else {
#pragma unroll
        for (int ch = 0; ch < 16; ++ch) st_chunk(sQi, row, ch, make_uint4(0u, 0u, 0u, 0u));
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_Q + i));
    };
    if (more) load_q(it);
    while (more && ok) {
      const int hl = it.unit / a.bph;
      const int64_t q0 = (int64_t)(it.unit - hl * a.bph) * 256;
      const int64_t qi = q0 + 128 * i + row;
      const bool qvalid = qi < a.Nq;
      const bool active = i == 0 || q0 + 128 < a.Nq;   // the second Q tile may hold no query
      float m_run = -INFINITY, l_run = 0.0f;
      if (active) {
        for (int j = it.lo; j < it.hi; ++j, ++jt) {
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar(B_S + i), jt & 1, a.wait_ns));
          if (!ok) break;
          tc_fence_after();
          float v[128];
          float mt = tmem_ld128_max(tS, v);
          const int64_t left = a.Nk - (int64_t)j * 128;
          if (left < 128) {   // the last tile's columns past the last key
            mt = -INFINITY;
#pragma unroll
            for (int e = 0; e < 128; ++e) {
              v[e] = e < (int)left ? v[e] : -INFINITY;
              mt = fmaxf(mt, v[e]);
            }
          }
          // O and l are rescaled only when the running maximum grows by more
          // than 2^8 (every P stays <= 2^8); S_i of this tile complete implies
          // that the P_i V before it is, so O_i can be rescaled here
          const float m_new = fmaxf(m_run, mt);
          const bool need = (m_new - m_run) * sl2 > kTauLog2;
          float alpha = 1.0f;
          if (need) {
            alpha = ex2((m_run - m_new) * sl2);
            m_run = m_new;
            l_run *= alpha;
          }
          if (__any_sync(0xFFFFFFFFu, need) && j > it.lo) {
#pragma unroll 1
            for (int cb = 0; cb < 8; ++cb) {
              uint32_t t[16];
              tmem_ld16(tO + cb * 16, t);
#pragma unroll
              for (int e = 0; e < 16; ++e) t[e] = __float_as_uint(__uint_as_float(t[e]) * alpha);
              tmem_st16(tO + cb * 16, t);
            }
          }
          const float mb = -m_run * sl2;
          const uint64_t MB = f2pack(mb, mb);
          // P = 2^(s scale log2 e - m) as f16 pairs; the row sum adds exactly
          // those f16 values, 32 at a time in a packed f16 tree (each partial
          // <= 32 * 2^8, exact to 2^-11 relative), then in fp32
          float lsum = 0.0f;
          uint32_t pk[64];
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
            for (int e = 0; e < 32; ++e) {
              float x0, x1;
              f2unpack(fma2(f2pack(v[64 * hf + 2 * e], v[64 * hf + 2 * e + 1]), SL, MB), x0, x1);
              pk[32 * hf + e] = ex2_f16x2(pack_f16(x0, x1));
            }
            tmem_st32u(tS + 32 * hf, pk + 32 * hf);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_P + 2 * i + hf));
          }
#pragma unroll
          for (int bq = 0; bq < 4; ++bq) {
            __half2 t8[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) t8[k] = __hadd2(u2h(pk[16 * bq + 2 * k]), u2h(pk[16 * bq + 2 * k + 1]));
#pragma unroll
            for (int k = 0; k < 4; ++k) t8[k] = __hadd2(t8[2 * k], t8[2 * k + 1]);
            t8[0] = __hadd2(t8[0], t8[1]);
            t8[2] = __hadd2(t8[2], t8[3]);
            const float2 f = __half22float2(__hadd2(t8[0], t8[2]));
            lsum += f.x + f.y;
          }
          l_run += lsum;
        }
      }
      if (!ok) break;
      const DenseItem done = it;
      more = items.next(a, it);
      // a group without queries in this item loads its next rows only once the
      // MMA warp is done with the item: B_Q must not run two phases ahead of it
      if (more && active) load_q(it);
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar(B_O), nit & 1, a.wait_ns));
      ++nit;
      if (!ok) break;
      if (more && !active) load_q(it);
      tc_fence_after();
      if (active) {
        const int h = a.h0 + hl;
        if (done.slot < 0) {
          const float inv_l = 1.0f / l_run;
#pragma unroll
          for (int cb = 0; cb < 4; ++cb) {
            float v[32];
            tmem_ld32(tO + cb * 32, v);
            if (qvalid) {
              uint4* dst = reinterpret_cast<uint4*>(a.out + ((size_t)qi * H + h) * 128 + cb * 32);
#pragma unroll
              for (int k = 0; k < 4; ++k)
                dst[k] = make_uint4(pack_bf16(v[8 * k] * inv_l, v[8 * k + 1] * inv_l),
                                    pack_bf16(v[8 * k + 2] * inv_l, v[8 * k + 3] * inv_l),
                                    pack_bf16(v[8 * k + 4] * inv_l, v[8 * k + 5] * inv_l),
                                    pack_bf16(v[8 * k + 6] * inv_l, v[8 * k + 7] * inv_l));
            }
          }
        } else {
          const size_t prow = (size_t)done.slot * 256 + 128 * i + row;
#pragma unroll
          for (int cb = 0; cb < 4; ++cb) {
            float v[32];
            tmem_ld32(tO + cb * 32, v);
            if (qvalid) {
              float4* dst = reinterpret_cast<float4*>(a.part_o + prow * 128 + cb * 32);
#pragma unroll
              for (int k = 0; k < 8; ++k) dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
            }
          }
          if (qvalid) *reinterpret_cast<float2*>(a.part_ml + prow * 2) = make_float2(m_run, l_run);
        }
        tc_fence_before();   // O_i is read before the next item's first P_i hand-off
      }
    }
    if (!ok) *s_err = 1;
  } else if (warp == W_MMA) {
    // ------------------------------------------------------------ MMA issue
    const uint32_t e = elect_one();
    const uint64_t dQ = desc_sw128(smem_u32(sm + D_Q)), dK = desc_sw128(smem_u32(sm + D_KV));
    const uint64_t dV = desc_sw128_mn(smem_u32(sm + D_KV), 16384);
    auto off = [](int bytes) { return (uint64_t)(bytes >> 4); };
    constexpr uint32_t idS = idesc_f16(128, 128, false), idPV = idesc_f16(128, 128, true);
    auto wait_all = [&](int b, uint32_t ph) -> bool {
      return __all_sync(0xFFFFFFFFu, mbar_wait(bar(b), ph, a.wait_ns));
    };
    // ring position of the next image, and the phase of its full barrier
    int ks = 0, vs = 1;                   // stages of the next K and V tile
    uint32_t kph = 0, vph = 0;
    auto step = [](int& s, uint32_t& ph) {
      s += 2;
      if (s >= kStages) {
        s -= kStages;
        ph ^= 1;
      }
    };
    uint32_t pph[2] = {0, 0}, qph = 0;
    while (ok && items.next(a, it)) {
      const int64_t q0 = (int64_t)(it.unit % a.bph) * 256;
      const int nqt = q0 + 128 < a.Nq ? 2 : 1;
      const int n = it.hi - it.lo;
      auto issue_S = [&](int i, bool last_q) {
        tc_fence_after();
#pragma unroll
        for (int kb = 0; kb < 2; ++kb)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            umma_ss_e(tbase + 128 * i, dQ + off(i * kImgSide + kb * 16384 + k * 32),
                      dK + off(ks * kImgSide + kb * 16384 + k * 32), idS, (kb | k) != 0, e);
        umma_commit_e(bar(B_S + i), e);
        if (last_q) {
          umma_commit_e(bar(B_EMPTY + ks), e);
          step(ks, kph);
        }
      };
      ok = wait_all(B_Q, qph) && wait_all(B_Q + 1, qph) && wait_all(B_FULL + ks, kph);
      qph ^= 1;
      if (!ok) break;
      issue_S(0, nqt == 1);
      if (nqt == 2) issue_S(1, true);
      for (int j = 0; j < n && ok; ++j) {
        if (!(ok = wait_all(B_FULL + vs, vph))) break;
        for (int i = 0; i < nqt; ++i) {
          const uint32_t tP = tbase + 128 * i, tO = tbase + 256 + 128 * i;
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            if (!(ok = wait_all(B_P + 2 * i + hf, pph[i]))) break;
            tc_fence_after();
#pragma unroll
            for (int k = 4 * hf; k < 4 * hf + 4; ++k)
              umma_ts_e(tO, tP + 8 * k, dV + off(vs * kImgSide + k * 2048), idPV, (j > 0 || k > 0) ? 1u : 0u, e);
          }
          if (!ok) break;
          pph[i] ^= 1;
          if (i == nqt - 1) {
            umma_commit_e(bar(B_EMPTY + vs), e);
            step(vs, vph);
          }
          if (j + 1 < n) {
            if (i == 0 && !(ok = wait_all(B_FULL + ks, kph))) break;
            issue_S(i, i == nqt - 1);
          }
        }
      }
      if (ok) umma_commit_e(bar(B_O), e);
    }
    if (!ok) {
      // a wait ran out: let the MMAs already issued finish before the TMEM is released
      umma_commit_e(bar(B_DRAIN), e);
      mbar_wait(bar(B_DRAIN), 0, a.wait_ns);
      *s_err = 1;
    }
  } else {
    // ------------------------------------------------------------ image stream
    pdl_wait();   // the rebuild has completed
    if (lane == 0) {
      uint32_t n = 0;   // images issued: image n goes to stage n % kStages
      while (ok && items.next(a, it)) {
        const uint8_t* src = a.img + ((size_t)(it.unit / a.bph) * a.NT + it.lo) * kImgTile;
        for (int j = 0; j < 2 * (it.hi - it.lo); ++j, ++n) {
          if ((j & 1) && a.idle_role == QWM_ROLE_V_REBUILD) {   // test hook: no Value image is published
            ok = false;
            break;
          }
          const int s = (int)(n % kStages);
          if (n >= kStages && !mbar_wait(bar(B_EMPTY + s), ((n / kStages) - 1) & 1, a.wait_ns)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(bar(B_FULL + s), kImgSide);
          bulk_g2s(smem_u32(sm + D_KV + s * kImgSide), src + (size_t)j * kImgSide, kImgSide, bar(B_FULL + s));
        }
      }
      // copies still in flight land before the CTA's memory goes away
      for (uint32_t k = n > kStages ? n - kStages : 0; k < n; ++k)
        mbar_wait(bar(B_FULL + (int)(k % kStages)), (k / kStages) & 1, a.wait_ns);
      if (!ok) *s_err = 1;
    }
    __syncwarp();
  }

  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *s_err) atomicCAS(a.status, 0, (int)QWM_ERR_TIMEOUT);
  if (tid == 0 && *s_bad) atomicCAS(a.status, 0, (int)QWM_ERR_NONFINITE);
  if (warp == W_MMA) {
    tc_fence_after();
    tmem_dealloc(tbase, 512);
  }
}

// The partial results of each tail block combined (m = max_p m_p, l = sum_p l_p
// 2^((m_p - m) c), O = sum_p O_p 2^((m_p - m) c) / l with c = sm_scale
// log2(e)); a warp per query row, four channels per lane, eight rows of one
// block per CTA.  A block that one CTA ran over every key is already in the
// output.
// Bound by the latency of its loads: B parts' rows are fetched ahead of their
// sums, the first B ahead of the maximum.  Four at a time without that, 35
// parts of 128 rows (4 heads, 15 x 880 keys) took 15 us, now 8, the whole call
// 45 and 35 us (38 in the kernel without images).  B = 8 where a block has more
// than four parts, else 4: with few parts and many blocks the registers of eight
// rows cost a wave (1536 CTAs of three parts: 9.3 us with 8, 7.4 with 4).
template <int B>
__global__ void __launch_bounds__(256) dense_combine(const DenseArgs a, int grid) {
  const int lane = threadIdx.x & 31;
  const int k = (int)blockIdx.x >> 5, prow = ((int)blockIdx.x & 31) * 8 + (int)(threadIdx.x >> 5);
  const int unit = a.waves * grid + k, hl = unit / a.bph, h = a.h0 + hl;
  const int64_t qi = (int64_t)(unit - hl * a.bph) * 256 + prow;
  const int64_t x0 = (int64_t)k * a.NT, x1 = x0 + a.NT;
  // parts b0 .. b1 - 1: CTA b's share of this block is its first unless its range starts in the block before
  const int64_t big = (int64_t)a.tail_more * (a.tail_per + 1);
  auto cta_of = [&](int64_t x) {
    return (int)(x < big ? x / (a.tail_per + 1) : a.tail_more + (x - big) / a.tail_per);
  };
  const int b0 = a.tail_parts > 0 ? k * a.tail_parts : cta_of(x0);
  const int b1 = a.tail_parts > 0 ? b0 + a.tail_parts : cta_of(x1 - 1) + 1;
  pdl_wait();
  if (qi >= a.Nq || b1 == b0 + 1) return;
  const size_t base = (size_t)(2 * b0 + (tail_start(a, b0) < x0 ? 1 : 0)) * 256 + prow;   // part b0
  auto at = [&](int p) { return p == 0 ? base : (size_t)(2 * (b0 + p)) * 256 + prow; };   // later parts start here
  const float c = a.sm_scale * 1.4426950408889634f;
  const int np = b1 - b0;
  float4 v[B];
  auto rows = [&](float4 (&x)[B], int p0) {
#pragma unroll
    for (int i = 0; i < B; ++i) {
      x[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (p0 + i < np) x[i] = *reinterpret_cast<const float4*>(a.part_o + at(p0 + i) * 128 + 4 * lane);
    }
  };
  auto ml_of = [&](int p) {
    return p < np ? *reinterpret_cast<const float2*>(a.part_ml + at(p) * 2) : make_float2(-INFINITY, 0.0f);
  };
  float2 ml = ml_of(lane);
  rows(v, 0);
  float m = ml.x;
#pragma unroll 1
  for (int p = lane + 32; p < np; p += 32) m = fmaxf(m, ml_of(p).x);
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  float l = 0.0f, wl = 0.0f;
  float4 o = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 1
  for (int p0 = 0; p0 < np; p0 += B) {
    if ((p0 & 31) == 0) {   // the weights of the next 32 parts, one per lane
      if (p0 > 0) ml = ml_of(p0 + lane);
      wl = exp2f((ml.x - m) * c);
      l = fmaf(ml.y, wl, l);
    }
    float4 u[B];
    rows(u, p0 + B);
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const float wgt = __shfl_sync(0xFFFFFFFFu, wl, (p0 & 31) + i);   // 0 past the last part
      o.x = fmaf(v[i].x, wgt, o.x); o.y = fmaf(v[i].y, wgt, o.y); o.z = fmaf(v[i].z, wgt, o.z); o.w = fmaf(v[i].w, wgt, o.w);
      v[i] = u[i];
    }
  }
#pragma unroll
  for (int s = 16; s; s >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, s);
  const float inv_l = 1.0f / l;
  uint2* dst = reinterpret_cast<uint2*>(a.out + ((size_t)qi * a.L.H + h) * 128 + 4 * lane);
  *dst = make_uint2(pack_bf16(o.x * inv_l, o.y * inv_l), pack_bf16(o.z * inv_l, o.w * inv_l));
}

constexpr int kMinTail = 3;   // key tiles of a CTA's share of the tail, at least
constexpr int kPartCost = 12;  // fixed time of a part (its Queries in, its partial results out and combined), in key tiles
constexpr int kWholeCost = 4;  // of a whole block

}  // namespace

DensePlan plan_dense(int64_t Nq, int heads, int64_t Nk, int nsm) {
  DensePlan p{};
  p.nsm = nsm;
  p.bph = (int)((Nq + 255) / 256);
  p.NT = (int)((Nk + 127) / 128);
  const int64_t units = (int64_t)heads * p.bph;
  p.waves = (int)(units / nsm);
  p.n_tail = (int)(units - (int64_t)p.waves * nsm);
  const int64_t T = (int64_t)p.n_tail * p.NT;
  if (p.n_tail > 0) {
    // Equal parts of each block, one per CTA, or the flattened tiles over every
    // CTA: the latter leaves none idle, but most CTAs then run two parts.  48
    // blocks of 110 tiles: 144 CTAs of 37 tiles 112 us a call, 152 of 35 126 us;
    // 64 of 53: 87 and 93 us; 80 of 32: whole blocks 92, over every CTA 102 us;
    // 80 of 272: 437 and 315 us.
    int64_t s = nsm / p.n_tail, per = (p.NT + s - 1) / s;
    if (per < kMinTail) per = kMinTail;
    s = (p.NT + per - 1) / per;
    int64_t g = (T + kMinTail - 1) / kMinTail;
    if (g < p.n_tail) g = p.n_tail;
    if (g > nsm) g = nsm;
    if (per + (s > 1 ? kPartCost : kWholeCost) <= (T + g - 1) / g + 2 * kPartCost) {
      p.tail_parts = (int)s;
      p.tail_ctas = (int)(s * p.n_tail);
    } else {
      p.tail_ctas = (int)g;
      p.tail_per = T / g;
      p.tail_more = (int)(T % g);
    }
  }
  p.grid = p.waves > 0 ? nsm : p.tail_ctas;
  return p;
}

size_t dense_part_bytes(const DensePlan& p) {
  return p.tail_ctas > p.n_tail ? (size_t)p.tail_ctas * 2 * 256 * (128 + 2) * sizeof(float) : 0;
}
size_t dense_head_bytes(const DensePlan& p) { return (size_t)p.NT * kImgTile; }

cudaError_t launch_dense(const DenseArgs& a0, const AttendSlots& slots, const DensePlan& p, int heads, int max_tiles,
                         cudaStream_t st) {
  DenseArgs a = a0;
  a.bph = p.bph;
  a.NT = p.NT;
  a.waves = p.waves;
  a.n_tail = p.n_tail;
  a.tail_ctas = p.tail_ctas;
  a.tail_parts = p.tail_parts;
  a.tail_per = p.tail_per;
  a.tail_more = p.tail_more;
  auto reb = a.L.sf ? (a.L.r == 0    ? rebuild_kernel<1, 0>
                       : a.L.r == 8  ? rebuild_kernel<1, 8>
                       : a.L.r == 16 ? rebuild_kernel<1, 16>
                                     : rebuild_kernel<1, 32>)
                    : (a.L.r == 0    ? rebuild_kernel<0, 0>
                       : a.L.r == 8  ? rebuild_kernel<0, 8>
                       : a.L.r == 16 ? rebuild_kernel<0, 16>
                                     : rebuild_kernel<0, 32>);
  const int n_units = slots.n + (a.Ncur > 0 ? 1 : 0);
  // Tiles per CTA: U_r is staged once per CTA and each record but the first is
  // copied a tile ahead, so as many as leave two CTAs for every place on the GPU
  // (two per SM), eight at most.  Wan-14B layer, per launch: 205 us with one
  // tile, 184 with two, 178 with four or eight; 84 tiles in all: 6.4 us with one
  // each, 9.7 with two.
  const int64_t all = (int64_t)max_tiles * heads * n_units, per = all / (4 * p.nsm);
  const int tpc = per < 1 ? 1 : per > 8 ? 8 : (int)per;
  cudaError_t e = cudaFuncSetAttribute(reb, cudaFuncAttributeMaxDynamicSharedMemorySize, kRebSmem);
  if (e != cudaSuccess) return e;
  reb<<<dim3((unsigned)((max_tiles + tpc - 1) / tpc), (unsigned)heads, (unsigned)n_units), kRebThreads, kRebSmem, st>>>(
      a, slots, tpc);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(dense_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, D_SMEM)) != cudaSuccess)
    return e;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3((unsigned)p.grid);
  lc.blockDim = dim3(kDThreads);
  lc.dynamicSmemBytes = D_SMEM;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  if ((e = cudaLaunchKernelEx(&lc, dense_kernel, a)) != cudaSuccess) return e;
  if (p.tail_ctas <= p.n_tail) return cudaSuccess;
  lc.gridDim = dim3((unsigned)(p.n_tail * 32));   // 8 rows per CTA
  lc.blockDim = dim3(256);
  lc.dynamicSmemBytes = 0;
  if ((e = cudaLaunchKernelEx(&lc, p.tail_parts > 4 ? dense_combine<8> : dense_combine<4>, a, p.grid)) != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace qwm
