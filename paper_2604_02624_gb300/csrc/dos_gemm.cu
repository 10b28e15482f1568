// dos_gemm.cu - split-BF16 DFT-GEMM form of the propagation (tcgen05, TMEM).
//
// See dos_gemm.cuh for the formulation.  The GEMM kernel is persistent and
// warp-specialised: one CTA per SM walks its share of the output tiles, 128 x
// 256 or, for few tiles, 128 x 128 (narrow_tiles; the figures here are the wide
// tile's).  Warp 0 (one lane) streams the operands: both are kept in global
// memory tile by tile in the tensor core's K-major core-matrix order
// (gemm_tiled), so a K chunk of 64 is two bulk copies (16 KB of A, 32 KB of B,
// cp.async.bulk with completion counted in bytes on the stage's "full"
// mbarrier) into a ring of four.  Warp 1 (one lane) issues the MMAs into
// one of two TMEM accumulators (2 x 256 columns) and frees each stage through
// tcgen05.commit on its "empty" mbarrier; a commit on "acc_full" hands a
// finished accumulator to the sixteen epilogue warps, which drain it (warp w
// reads TMEM lanes 32 (w % 4) .. +31 and a quarter of the columns) while the
// MMAs of the next tile run into the other accumulator, and release it on
// "acc_empty".  Every wait is bounded and watches a shared abort flag: on
// expiry the CTA records the error flag, lets its copies and MMAs in flight
// finish (bounded) and ends cleanly.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "dos_gemm.cuh"
#include "dos_internal.h"
#include "dos_pass.cuh"

namespace dos {

// One tile and MMA: 128 x TN, K steps of 16; TN = 256, or 128 (narrow_tiles).
constexpr int GTM = 128, GTK = 64;
template <int TN>
constexpr int gstages() { return TN == 256 ? 4 : 6; }  // of 48 or 32 KB
constexpr int kEpiWarps = 16;                   // 4 per TMEM lane quarter, a quarter of the columns each
constexpr int kGemmThreads = 32 * (2 + kEpiWarps);
constexpr long kSpinLimit = 1L << 26;           // bounded mbarrier wait (a fraction of a second)

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t kmajor_desc(uint32_t saddr) {
  // start >> 4 | LBO 128 B (next 8 k) | SBO 1024 B (next 8 rows) | descriptor version 1 | no swizzle
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46);
}

// kind::f16 instruction descriptor: D f32, A and B bf16, both K-major, N = TN, M = 128
template <int TN>
constexpr uint32_t idesc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(GTM >> 4) << 24);
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
// bounded wait; gives up early when another role of the CTA raised *abort
// (then returns false without raising it again)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort = nullptr) {
  for (long it = 0; it < kSpinLimit; ++it) {
    if (mbar_try(bar, parity)) return true;
    if (abort && (it & 255) == 255 && *abort) return false;
  }
  if (abort) *abort = 1;
  return false;
}

__device__ __forceinline__ void bar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// one contiguous global -> shared bulk copy, completion counted on `bar`
__device__ __forceinline__ void bulk_tile(void* dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

template <int TN>
struct __align__(1024) GemmSmem {
  static constexpr int GSTAGES = gstages<TN>();
  uint8_t a[GSTAGES][GTM * GTK * 2];  // 16 KB per stage
  uint8_t b[GSTAGES][TN * GTK * 2];   // 32 or 16 KB per stage
  uint64_t full[GSTAGES];             // copies of the stage landed
  uint64_t empty[GSTAGES];            // MMAs reading the stage done
  uint64_t acc_full[2];               // accumulator ready for the epilogue
  uint64_t acc_empty[2];              // accumulator drained (one arrival per epilogue warp)
  uint32_t tmem;
  int abort;
};

// ------------------------------------------------------------ epilogues
// x -> bf16 parts: each the round-to-nearest of what the earlier parts leave
__device__ __forceinline__ void split_store(const Parts& P, size_t i, float v) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  P.p[0][i] = h;
  const float r1 = v - __bfloat162float(h);
  const __nv_bfloat16 m = __float2bfloat16_rn(r1);
  P.p[1][i] = m;
  if (P.k > 2) P.p[2][i] = __float2bfloat16_rn(r1 - __bfloat162float(m));
}

// x -> bf16 parts of 8 consecutive K entries (8-aligned) of one operand row:
// one 16-byte store per part
__device__ __forceinline__ void split_store8(const Parts& P, size_t at, const float* x) {
  uint32_t w0[4], w1[4], w2[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    __nv_bfloat16 h[2], m[2], l[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float v = x[2 * e + q];
      h[q] = __float2bfloat16_rn(v);
      const float r1 = v - __bfloat162float(h[q]);
      m[q] = __float2bfloat16_rn(r1);
      l[q] = __float2bfloat16_rn(r1 - __bfloat162float(m[q]));
    }
    w0[e] = (uint32_t)__bfloat16_as_ushort(h[0]) | ((uint32_t)__bfloat16_as_ushort(h[1]) << 16);
    w1[e] = (uint32_t)__bfloat16_as_ushort(m[0]) | ((uint32_t)__bfloat16_as_ushort(m[1]) << 16);
    w2[e] = (uint32_t)__bfloat16_as_ushort(l[0]) | ((uint32_t)__bfloat16_as_ushort(l[1]) << 16);
  }
  *reinterpret_cast<uint4*>(P.p[0] + at) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
  *reinterpret_cast<uint4*>(P.p[1] + at) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
  if (P.k > 2) *reinterpret_cast<uint4*>(P.p[2] + at) = make_uint4(w2[0], w2[1], w2[2], w2[3]);
}

// Accumulator columns an epilogue warp takes at a time.  The spectrum epilogue
// takes 16, so that the transfer-function values of the next ones can be on
// their way (in registers) while it works on the current ones: with K = 512 a
// tile's MMAs take about as long as its epilogue, which then bounds the launch.
// With the field epilogue's 16-byte stores: 540 -> 498 us per propagation (128
// channels, 256 x 256, two parts).
template <int MODE>
constexpr int epi_cols() { return MODE == GEMM_OUT_SPECTRUM ? 16 : 32; }

// Transfer-function values of accumulator row r = (w, kx), columns cb ..
// cb + 15 = eight ky (spectrum epilogue)
__device__ __forceinline__ void spectrum_h(const GemmArgs& g, int r, int cb, float2 (&hv)[8]) {
  const int m = g.m, w = r / m, kx = r - w * m;
  const int bx = min(kx, m - kx);
  const float2* Hw = g.Hq + (size_t)w * g.hs * g.hs;
  const int ky0 = cb >> 1;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int ky = ky0 + q;
    hv[q] = ky < m ? __ldg(Hw + (size_t)min(ky, m - ky) * g.hs + bx) : make_float2(0.f, 0.f);
  }
}

// accumulator row r, columns cb .. cb + epi_cols - 1 (values v) -> the
// destination of MODE (hv: the spectrum epilogue's transfer-function values)
template <int MODE>
__device__ __forceinline__ void epilogue(const GemmArgs& g, int r, int cb, const float* v, const float2 (&hv)[8]) {
  if constexpr (MODE == GEMM_OUT_ROWS) {
    const int k = r >> 1, p = r & 1;
    if (g.nj % 8 == 0) {
      // 8-aligned groups never straddle a channel: one 16-byte store per part
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = cb + 8 * q;
        if (c >= g.vcols) break;
        const int w = c / g.nj, j = c - w * g.nj;
        split_store8(g.xo, gemm_tiled((size_t)w * g.nk + k, p * g.nj + j, g.kpo), v + 8 * q);
      }
    } else {
      for (int q = 0; q < 32; ++q) {
        const int c = cb + q;
        if (c >= g.vcols) break;
        const int w = c / g.nj, j = c - w * g.nj;
        split_store(g.xo, gemm_tiled((size_t)w * g.nk + k, p * g.nj + j, g.kpo), v[q]);
      }
    }
  } else if constexpr (MODE == GEMM_OUT_SPECTRUM) {
    // row r = (w, kx); columns 2ky + {0, 1}: eight spectrum values
    const int m = g.m, w = r / m, kx = r - w * m;
    const int bx = min(kx, m - kx);
    const float* Sw = g.mis.sq ? g.mis.sq + (size_t)w * g.hs * g.hs : nullptr;
    const int ky0 = cb >> 1;  // multiple of 8
    if (ky0 >= m) return;     // m is a multiple of 8 for every compiled size: whole groups of 8
    float re[8], im[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int ky = ky0 + q;
      float2 h = hv[q];
      if (Sw) h = cmul(h, misalign_factor(g.mis, ky, kx, m, Sw[(size_t)min(ky, m - ky) * g.hs + bx]));
      const float2 b = make_float2(v[2 * q], v[2 * q + 1]);
      const float2 val = g.adj ? cmulc(b, h) : cmul(b, h);
      re[q] = val.x;
      im[q] = val.y;
    }
    split_store8(g.xo, gemm_tiled((size_t)r, ky0, g.kpo), re);
    split_store8(g.xo, gemm_tiled((size_t)r, m + ky0, g.kpo), im);
  } else {
    // row r = (w, y); columns 2x + {0, 1}: sixteen field values
    const int n = g.n, w = r / n, y = r - w * n;
    const int x0 = cb >> 1;
    if (!g.o && n % 2 == 0) {
      float4* row = reinterpret_cast<float4*>(g.fld + (size_t)r * n + x0);  // two values a store
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (x0 + 2 * q < n) row[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      return;
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int x = x0 + q;
      if (x >= n) break;
      const float2 val = make_float2(v[2 * q], v[2 * q + 1]);
      if (g.o) {
        const int fy = y - g.of, fx = x - g.of;
        if (fy >= 0 && fy < g.fov && fx >= 0 && fx < g.fov) {
          const size_t qo = ((size_t)w * g.fov + fy) * g.fov + fx;
          g.o[qo] = val;
          if (g.I) g.I[qo] = fmaf(val.x, val.x, val.y * val.y);
        }
      } else {
        g.fld[((size_t)w * n + y) * n + x] = val;
      }
    }
  }
}

// CW columns of this warp's 32 accumulator rows, one row per lane
template <int CW>
__device__ __forceinline__ void tmem_load(uint32_t addr, uint32_t (&u)[CW]) {
  static_assert(CW == 16 || CW == 32, "compiled widths");
  if constexpr (CW == 32) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
          "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]),
          "=r"(u[16]), "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]),
          "=r"(u[24]), "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
        : "r"(addr));
  } else {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
          "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
        : "r"(addr));
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;");
}

template <int MODE, int TN>
__global__ void __launch_bounds__(kGemmThreads, 1) k_tc_gemm(const __grid_constant__ GemmArgs g) {
  constexpr int GSTAGES = gstages<TN>();
  extern __shared__ __align__(1024) uint8_t gsm_raw[];
  GemmSmem<TN>& sm = *reinterpret_cast<GemmSmem<TN>*>(gsm_raw);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  volatile int* abort = &sm.abort;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&sm.tmem)),
                 "r"(2 * TN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 32) {
    for (int s = 0; s < GSTAGES; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sm.full[s])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sm.empty[s])));
    }
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sm.acc_full[b])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&sm.acc_empty[b])), "r"(kEpiWarps));
    }
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  pdl_wait();
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = sm.tmem;
  const int kchunks = g.K / GTK;
  const int total = g.nseg * kchunks;  // K chunks per tile
  // tiles, the DFT matrix's (few) tiles the fast index: the CTAs that share a
  // data tile run together
  const int tilesA = g.rows / GTM, tilesB = (g.cols + TN - 1) / TN;
  const int ntiles = tilesA * tilesB;
  auto tile_of = [&](int t, int& mt, int& nt) {
    if (g.w_is_b) {
      nt = t % tilesB;
      mt = t / tilesB;
    } else {
      mt = t % tilesA;
      nt = t / tilesA;
    }
  };
  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    if (lane == 0) {
      int c = 0;
      int last[GSTAGES];
      for (int s = 0; s < GSTAGES; ++s) last[s] = -1;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        int mt, nt;
        tile_of(t, mt, nt);
        for (int it = 0; it < total; ++it, ++c) {
          const int st = c % GSTAGES;
          if (c >= GSTAGES &&
              !mbar_wait(smem_addr(&sm.empty[st]), (uint32_t)(((c / GSTAGES) - 1) & 1), abort)) {
            ok = false;
            break;
          }
          const int seg = it / kchunks, kc = it % kchunks;
          const uint32_t fb = smem_addr(&sm.full[st]);
          bar_expect_tx(fb, (GTM + TN) * GTK * 2);
          // 128-row A tile mt: half (mt & 1) of the stored 256-row tile mt / 2, and so B tile nt of TN = 128
          bulk_tile(sm.a[st], g.a[seg] + (((size_t)(mt >> 1) * kchunks + kc) << 14) + ((size_t)(mt & 1) << 13),
                    GTM * GTK * 2, fb);
          const size_t bt = TN == 256 ? (((size_t)nt * kchunks + kc) << 14)
                                      : (((size_t)(nt >> 1) * kchunks + kc) << 14) + ((size_t)(nt & 1) << 13);
          bulk_tile(sm.b[st], g.b[seg] + bt, TN * GTK * 2, fb);
          last[st] = c;
        }
      }
      // no copy may still target shared memory when the CTA ends
      for (int s = 0; s < GSTAGES; ++s)
        if (last[s] >= 0) (void)mbar_wait(smem_addr(&sm.full[s]), (uint32_t)((last[s] / GSTAGES) & 1));
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issue
    if (lane == 0) {
      int c = 0, tc = 0;
      uint32_t last_bar = 0, last_par = 0;  // the latest commit (covers every MMA before it)
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tc) {
        const int b = tc & 1;
        if (tc >= 2 && !mbar_wait(smem_addr(&sm.acc_empty[b]), (uint32_t)(((tc >> 1) - 1) & 1), abort)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t acc0 = tmem + (uint32_t)(b * TN);
        for (int it = 0; it < total; ++it, ++c) {
          const int st = c % GSTAGES;
          if (!mbar_wait(smem_addr(&sm.full[st]), (uint32_t)((c / GSTAGES) & 1), abort)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t sa = smem_addr(sm.a[st]), sb = smem_addr(sm.b[st]);
#pragma unroll
          for (int kk = 0; kk < GTK / 16; ++kk) {
            const uint64_t da = kmajor_desc(sa + kk * 256), db = kmajor_desc(sb + kk * 256);
            const uint32_t acc = (it > 0 || kk > 0) ? 1u : 0u;
            asm volatile(
                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc0),
                "l"(da), "l"(db), "r"(idesc<TN>()), "r"(acc));
          }
          last_bar = smem_addr(&sm.empty[st]);
          last_par = (uint32_t)((c / GSTAGES) & 1);
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(last_bar));
        }
        if (!ok) break;
        last_bar = smem_addr(&sm.acc_full[b]);
        last_par = (uint32_t)((tc >> 1) & 1);
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(last_bar));
      }
      // no MMA may still write tensor memory when it is released
      if (last_bar) (void)mbar_wait(last_bar, last_par);
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- epilogue
    const int q = warp & 3;                 // TMEM lane quarter
    const int part = (warp - 2) >> 2;       // column quarter
    constexpr int CW = epi_cols<MODE>();
    int tc = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++tc) {
      const int b = tc & 1;
      int mt, nt;
      tile_of(t, mt, nt);
      const int r = mt * GTM + q * 32 + lane;  // accumulator row of this thread
      const int cbeg = part * (TN / 4), cend = cbeg + TN / 4;
      float2 hv[8];
      if constexpr (MODE == GEMM_OUT_SPECTRUM) {
        if (r < g.vrows) spectrum_h(g, r, nt * TN + cbeg, hv);  // before the wait for the accumulator
      }
      if (!mbar_wait(smem_addr(&sm.acc_full[b]), (uint32_t)((tc >> 1) & 1), abort)) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll 1
      for (int c0 = cbeg; c0 < cend; c0 += CW) {
        uint32_t u[CW];
        tmem_load<CW>(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * TN + c0), u);
        float2 hn[8];
        if constexpr (MODE == GEMM_OUT_SPECTRUM) {
          if (c0 + CW < cend && r < g.vrows) spectrum_h(g, r, nt * TN + c0 + CW, hn);
        }
        if (r < g.vrows) {
          float v[CW];
#pragma unroll
          for (int j = 0; j < CW; ++j) v[j] = __uint_as_float(u[j]);
          epilogue<MODE>(g, r, nt * TN + c0, v, hv);
        }
        if constexpr (MODE == GEMM_OUT_SPECTRUM) {
#pragma unroll
          for (int j = 0; j < 8; ++j) hv[j] = hn[j];
        }
      }
      // this warp is done with the accumulator
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&sm.acc_empty[b])) : "memory");
    }
  }
  __syncthreads();
  if (tid == 0 && sm.abort) atomicExch(g.err, 1);
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TN));
}

// Column width of the tiles.  A launch runs in waves of one tile per SM.  A
// narrow tile took 0.70 to 0.73 of a wide one's time in launches of many waves
// (each MMA reads the whole A tile for half the columns), so narrow tiles are
// taken where they need less than 1 / kNarrow as many waves: mostly where both
// are one wave, or where the wide tiles leave half the chip idle.  A step of
// three layers, wide / narrow in every launch / by this rule: 4 x 256 551 / 483 /
// 483 us, 24 x 200 (three parts) 965 / 1345 / 960, 128 x 256 3742 / 5453 / 3749.
constexpr double kNarrow = 0.8;
static bool narrow_tiles(const GemmArgs& g, int sms) {
  const long rows = g.rows / GTM;
  const long wide = (rows * ((g.cols + 255) / 256) + sms - 1) / sms;
  const long narrow = (rows * ((g.cols + 127) / 128) + sms - 1) / sms;
  return kNarrow * (double)narrow < (double)wide;
}

template <int MODE, int TN>
static cudaError_t launch_tiles(const GemmArgs& g, int sms, cudaStream_t s) {
  const size_t sm = sizeof(GemmSmem<TN>) + 1024;
  const cudaError_t e = cudaFuncSetAttribute(k_tc_gemm<MODE, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int tiles = (g.rows / GTM) * ((g.cols + TN - 1) / TN);
  return launch_next(k_tc_gemm<MODE, TN>, dim3(std::min(tiles, sms)), kGemmThreads, sm, s, g);
}

template <int MODE>
static cudaError_t launch_mode(const GemmArgs& g, cudaStream_t s) {
  // attribute and SM count of the current device, every launch (contexts may
  // live on different devices of one process; both calls are host-side only)
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  return narrow_tiles(g, sms) ? launch_tiles<MODE, 128>(g, sms, s) : launch_tiles<MODE, 256>(g, sms, s);
}

cudaError_t launch_tc_gemm(const GemmArgs& g, cudaStream_t s) {
  switch (g.mode) {
    case GEMM_OUT_ROWS: return launch_mode<GEMM_OUT_ROWS>(g, s);
    case GEMM_OUT_SPECTRUM: return launch_mode<GEMM_OUT_SPECTRUM>(g, s);
    default: return launch_mode<GEMM_OUT_FIELD>(g, s);
  }
}

// ------------------------------------------------------------ constant matrices

// W rows r: output o = r / 2 (re for even r, im for odd r); K index c: input
// element c (its real part) for c < kin, input c - kin (imaginary part) for
// kin <= c < 2 kin.  Entry exp(sign 2 pi j o x / m) in FP64, split into bf16.
__global__ void k_dft_matrix(Parts W, int rows_pad, int kpad, int nout, int kin, int m, int sign) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)rows_pad * kpad) return;
  const int r = (int)(i / kpad), c = (int)(i % kpad);
  const int o = r / 2;
  const size_t at = gemm_tiled((size_t)r, c, kpad);
  float v = 0.f;
  if (o < nout && c < 2 * kin) {
    const int x = c < kin ? c : c - kin;
    const long e = ((long)o * x) % m;
    double s, co;
    sincospi(2.0 * sign * (double)e / (double)m, &s, &co);
    // row 2o: [Re W, -Im W];  row 2o+1: [Im W, Re W]
    if ((r & 1) == 0) v = (float)(c < kin ? co : -s);
    else v = (float)(c < kin ? s : co);
  }
  split_store(W, at, v);
}

cudaError_t launch_build_dft(GemmPlan& p, cudaStream_t s) {
  const size_t nf = (size_t)p.rp1 * p.kp1, ng = (size_t)p.rp2 * p.kp2;
  k_dft_matrix<<<(unsigned)((nf + 255) / 256), 256, 0, s>>>(p.F, p.rp1, p.kp1, p.m, p.n, p.m, -1);
  k_dft_matrix<<<(unsigned)((ng + 255) / 256), 256, 0, s>>>(p.G, p.rp2, p.kp2, p.n, p.m, p.m, +1);
  return cudaGetLastError();
}

// ------------------------------------------------------------ conversion kernels
// What becomes the operand rows (w, y) = [Re(u), Im(u)] of a propagation.
enum {
  PREP_LAYER = 1,     // checkpoint the field v, u = t(h) v (forward layer)
  PREP_APERTURE = 2,  // u = the square aperture
  PREP_SEED = 3       // u = 2 dL/dI o on the FOV, zero elsewhere (adjoint seed)
};
struct PrepArgs {
  const float2* v;        // [nwc][n][n] (LAYER)
  float2* ckpt;           // [nwc][n][n] (LAYER)
  const float* h;         // [n][n] (LAYER)
  const ChanConst* chan;  // [nwc] (LAYER)
  const float2* o;        // [nwc][fov][fov] (SEED)
  const float* dLdI;      // [nwc][fov][fov] (SEED)
  int a_off, a_w;         // APERTURE: first pixel and side
  int of, fov;            // SEED
};

// value of pixel (y, x) of channel w; LAYER also stores its checkpoint
template <int MODE>
__device__ __forceinline__ float2 prep_value(const PrepArgs& g, int n, int w, int y, int x) {
  if constexpr (MODE == PREP_APERTURE) {
    const bool in = y >= g.a_off && y < g.a_off + g.a_w && x >= g.a_off && x < g.a_off + g.a_w;
    return make_float2(in ? 1.f : 0.f, 0.f);
  } else if constexpr (MODE == PREP_SEED) {
    const int fy = y - g.of, fx = x - g.of;
    if (fy < 0 || fy >= g.fov || fx < 0 || fx >= g.fov) return make_float2(0.f, 0.f);
    const size_t q = ((size_t)w * g.fov + fy) * g.fov + fx;
    return cscale(g.o[q], 2.0f * g.dLdI[q]);
  } else {
    const size_t at = ((size_t)w * n + y) * n + x;
    const float2 vv = g.v[at];
    g.ckpt[at] = vv;
    return cmul(transmission<true>(g.h[(size_t)y * n + x], g.chan[w]), vv);
  }
}

// One thread per pixel (any n).
template <int MODE>
__global__ void k_prep_field(PrepArgs g, Parts X, int n, int kp) {
  pdl_wait();
  const int wy = blockIdx.x, w = wy / n, y = wy % n;
  for (int x = threadIdx.x; x < n; x += blockDim.x) {
    const float2 u = prep_value<MODE>(g, n, w, y, x);
    split_store(X, gemm_tiled((size_t)wy, x, kp), u.x);
    split_store(X, gemm_tiled((size_t)wy, n + x, kp), u.y);
  }
}

// One thread per 8 pixels of a row (n % 8 == 0): 16-byte accesses on every
// array.  A warp takes 8 rows x 4 neighbouring groups, so that an operand store
// covers whole 128-byte core matrices and a field access 256 bytes of each row.
// Bound by memory (24 bytes a pixel with the checkpoint).  All field kernels of
// a 128-channel, 8-layer, 256 x 256 step: 1784 us with one thread per operand
// entry (each value formed twice, 2-byte stores scattered over the tiles, a
// serial channel loop per pixel in the adjoint) -> 813 us.
struct Px8 {
  int wy, w, y, x0;  // operand row, channel, field row, first pixel
};
__device__ __forceinline__ bool px8(size_t i, int n, int rows, Px8& p) {
  const int groups = n / 8;
  const size_t g = i >> 3;
  p.wy = (int)(g / groups) * 8 + (int)(i & 7);
  p.x0 = (int)(g % groups) * 8;
  p.w = p.wy / n;
  p.y = p.wy - p.w * n;
  return p.wy < rows;
}
template <int MODE>
__global__ void __launch_bounds__(256) k_prep_field8(PrepArgs g, Parts X, int n, int kp, int rows) {
  pdl_wait();
  Px8 p;
  if (!px8((size_t)blockIdx.x * blockDim.x + threadIdx.x, n, rows, p)) return;
  float re[8], im[8];
  if constexpr (MODE == PREP_LAYER) {
    const size_t at = (size_t)p.wy * n + p.x0;
    const float4* v4 = reinterpret_cast<const float4*>(g.v + at);
    const float* hp = g.h + (size_t)p.y * n + p.x0;
    float4 v[4];
    float hv[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = v4[q];
#pragma unroll
    for (int e = 0; e < 8; ++e) hv[e] = __ldg(hp + e);  // the caller's array: any 4-byte alignment
    const ChanConst cc = g.chan[p.w];
    float4* c4 = reinterpret_cast<float4*>(g.ckpt + at);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      c4[q] = v[q];
      const float2 u0 = cmul(transmission<true>(hv[2 * q], cc), make_float2(v[q].x, v[q].y));
      const float2 u1 = cmul(transmission<true>(hv[2 * q + 1], cc), make_float2(v[q].z, v[q].w));
      re[2 * q] = u0.x, im[2 * q] = u0.y, re[2 * q + 1] = u1.x, im[2 * q + 1] = u1.y;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float2 u = prep_value<MODE>(g, n, p.w, p.y, p.x0 + e);
      re[e] = u.x, im[e] = u.y;
    }
  }
  split_store8(X, gemm_tiled((size_t)p.wy, p.x0, kp), re);
  split_store8(X, gemm_tiled((size_t)p.wy, n + p.x0, kp), im);
}

// adjoint layer: per pixel, over the chunk's channels in order:
//   partial += Re(conj(grad_u) c t v);  grad_v = conj(t) grad_u -> operand rows
//   (FIRST: not for the first layer, where the adjoint ends)
template <bool FIRST>
__global__ void k_field_adj(const float2* __restrict__ field, const float2* __restrict__ ckpt,
                            const float* __restrict__ h, const ChanConst* __restrict__ chan,
                            float* __restrict__ partial, Parts X, int nwc, int n, int kp) {
  pdl_wait();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const int n2 = n * n;
  if (p >= n2) return;
  const int y = p / n, x = p - y * n;
  const float hv = h[p];
  float acc = 0.f;
  for (int w = 0; w < nwc; ++w) {
    const ChanConst cc = chan[w];
    const float2 u = adjoint_pixel(field[(size_t)w * n2 + p], transmission<true>(hv, cc), ckpt[(size_t)w * n2 + p], cc, acc);
    if constexpr (!FIRST) {
      split_store(X, gemm_tiled((size_t)w * n + y, x, kp), u.x);
      split_store(X, gemm_tiled((size_t)w * n + y, n + x, kp), u.y);
    }
  }
  partial[p] = acc;
}

// The same with one thread per 8 pixels of a row (n % 8 == 0, mapping as
// k_prep_field8) and the chunk's channels in gridDim.y slices, each with a
// partial plane of its own (part_stride apart): enough threads to fill the
// chip, and FP32 sums of fewer terms.
template <bool FIRST>
__global__ void __launch_bounds__(128) k_field_adj8(const float2* __restrict__ field, const float2* __restrict__ ckpt,
                                                    const float* __restrict__ h, const ChanConst* __restrict__ chan,
                                                    float* __restrict__ partial, size_t part_stride, Parts X, int nwc,
                                                    int n, int kp) {
  pdl_wait();
  Px8 p;
  if (!px8((size_t)blockIdx.x * blockDim.x + threadIdx.x, n, n, p)) return;  // rows of one channel: w = 0
  const int per = (nwc + gridDim.y - 1) / gridDim.y;
  const int w0 = blockIdx.y * per, w1 = min(nwc, w0 + per);
  const size_t n2 = (size_t)n * n, at = (size_t)p.y * n + p.x0;
  float hv[8], acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f, hv[e] = __ldg(h + at + e);  // h: the caller's, any 4-byte alignment
  for (int w = w0; w < w1; ++w) {
    const ChanConst cc = chan[w];
    const float4* f4 = reinterpret_cast<const float4*>(field + (size_t)w * n2 + at);
    const float4* c4 = reinterpret_cast<const float4*>(ckpt + (size_t)w * n2 + at);
    float4 f[4], c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) f[q] = f4[q], c[q] = c4[q];
    float re[8], im[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float2 au = (e & 1) ? make_float2(f[e / 2].z, f[e / 2].w) : make_float2(f[e / 2].x, f[e / 2].y);
      const float2 v = (e & 1) ? make_float2(c[e / 2].z, c[e / 2].w) : make_float2(c[e / 2].x, c[e / 2].y);
      const float2 u = adjoint_pixel(au, transmission<true>(hv[e], cc), v, cc, acc[e]);
      re[e] = u.x, im[e] = u.y;
    }
    if constexpr (!FIRST) {
      split_store8(X, gemm_tiled((size_t)w * n + p.y, p.x0, kp), re);
      split_store8(X, gemm_tiled((size_t)w * n + p.y, n + p.x0, kp), im);
    }
  }
  float4* out = reinterpret_cast<float4*>(partial + blockIdx.y * part_stride + at);
  out[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
  out[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
}

// ------------------------------------------------------------ one propagation
// The kept products of the parts: (0,0), (0,1), (1,0) and, with three parts,
// (0,2), (2,0), (1,1).  The tensor core's FP32 accumulation loses a little of
// every partial sum (measured: the relative error grows with the number of
// accumulation steps at the accumulator's magnitude), so the small products go
// first and the large (0,0) product last: the error is then that of the (0,0)
// product alone.
static void set_terms(GemmArgs& g, const Parts& A, const Parts& B) {
  static const int ta2[3] = {0, 1, 0}, tb2[3] = {1, 0, 0};
  static const int ta3[6] = {1, 0, 2, 0, 1, 0}, tb3[6] = {1, 2, 0, 1, 0, 0};
  const bool three = A.k == 3;
  g.nseg = three ? 6 : 3;
  for (int t = 0; t < g.nseg; ++t) {
    g.a[t] = A.p[three ? ta3[t] : ta2[t]];
    g.b[t] = B.p[three ? tb3[t] : tb2[t]];
  }
}

// X1 rows (w, y) of the chunk hold the field; computes the propagated field
// (into fld) or, with o non-null, the output plane.  Operands: X1 (field) -> Y1
// (after the row DFT) -> X2 (after the column DFT and H) -> Y2 (after the
// column IDFT) -> field.  Each has its own buffer, so that the K entries that
// pad its rows to whole 64s, zeroed once at create, stay zero.
cudaError_t gemm_propagate(GemmPlan& p, int nwc, const float2* Hq, int hs, bool adj, float2* o, float* I, int of,
                           int fov, const Misalign& mis, int* launches, cudaStream_t s) {
  const int n = p.n, m = p.m;
  auto pad = [](int v, int q) { return (v + q - 1) / q * q; };
  const int c1 = nwc * n, c2 = nwc * m;
  cudaError_t e;
  GemmArgs g;
  std::memset(&g, 0, sizeof(g));
  g.err = p.err;
  // row DFT: D = F X1^T -> Y1 rows (w, kx), K = p n + y
  set_terms(g, p.F, p.X1);
  g.rows = pad(2 * m, GTM); g.cols = c1; g.K = p.kp1; g.w_is_b = 0;
  g.mode = GEMM_OUT_ROWS; g.vrows = 2 * m; g.vcols = c1; g.nk = m; g.nj = n; g.xo = p.Y1; g.kpo = p.kp1;
  if ((e = launch_tc_gemm(g, s)) != cudaSuccess) return e;
  // column DFT and H: D = Y1 F^T -> X2 rows (w, kx), K = ky | m + ky
  set_terms(g, p.Y1, p.F);
  g.rows = pad(c2, GTM); g.cols = 2 * m; g.K = p.kp1; g.w_is_b = 1;
  g.mode = GEMM_OUT_SPECTRUM; g.vrows = c2; g.vcols = 2 * m; g.xo = p.X2; g.kpo = p.kp2;
  g.Hq = Hq; g.hs = hs; g.m = m; g.adj = adj ? 1 : 0; g.mis = mis;
  if ((e = launch_tc_gemm(g, s)) != cudaSuccess) return e;
  // column IDFT: D = G X2^T -> Y2 rows (w, y), K = p m + kx
  set_terms(g, p.G, p.X2);
  g.rows = pad(2 * n, GTM); g.cols = c2; g.K = p.kp2; g.w_is_b = 0;
  g.mode = GEMM_OUT_ROWS; g.vrows = 2 * n; g.vcols = c2; g.nk = n; g.nj = m; g.xo = p.Y2; g.kpo = p.kp2;
  if ((e = launch_tc_gemm(g, s)) != cudaSuccess) return e;
  // row IDFT: D = Y2 G^T -> field (or the output plane)
  set_terms(g, p.Y2, p.G);
  g.rows = pad(c1, GTM); g.cols = 2 * n; g.K = p.kp2; g.w_is_b = 1;
  g.mode = GEMM_OUT_FIELD; g.vrows = c1; g.vcols = 2 * n; g.fld = p.fld; g.o = o; g.I = I; g.n = n; g.of = of;
  g.fov = fov;
  if ((e = launch_tc_gemm(g, s)) != cudaSuccess) return e;
  *launches += 4;
  return cudaSuccess;
}

template <int MODE>
static cudaError_t launch_prep(GemmPlan& p, int nwc, const PrepArgs& g, cudaStream_t s) {
  if (p.n % 8 == 0) {
    const int rows = nwc * p.n;
    const size_t threads = (size_t)rows * (p.n / 8);
    return launch_next(k_prep_field8<MODE>, dim3((unsigned)((threads + 255) / 256)), 256, 0, s, g, p.X1, p.n, p.kp1,
                       rows);
  }
  return launch_next(k_prep_field<MODE>, dim3(nwc * p.n), 128, 0, s, g, p.X1, p.n, p.kp1);
}

cudaError_t gemm_prep_aperture(GemmPlan& p, int nwc, int a_off, int a_w, cudaStream_t s) {
  PrepArgs g = {};
  g.a_off = a_off;
  g.a_w = a_w;
  return launch_prep<PREP_APERTURE>(p, nwc, g, s);
}

cudaError_t gemm_prep_layer(GemmPlan& p, int nwc, float2* ckpt, const float* h, const ChanConst* chan,
                            cudaStream_t s) {
  PrepArgs g = {};
  g.v = p.fld;
  g.ckpt = ckpt;
  g.h = h;
  g.chan = chan;
  return launch_prep<PREP_LAYER>(p, nwc, g, s);
}

cudaError_t gemm_prep_seed(GemmPlan& p, int nwc, const float2* o, const float* dLdI, int of, int fov, cudaStream_t s) {
  PrepArgs g = {};
  g.o = o;
  g.dLdI = dLdI;
  g.of = of;
  g.fov = fov;
  return launch_prep<PREP_SEED>(p, nwc, g, s);
}

// about 128 K threads, in whole channels
int gemm_adj_slices(const GemmPlan& p) {
  if (p.n % 8 != 0) return 1;
  return std::max(1, std::min(p.nwc, (1 << 20) / (p.n * p.n)));
}

cudaError_t gemm_adj_layer(GemmPlan& p, int nwc, const float2* ckpt, const float* h, const ChanConst* chan,
                           float* partial, size_t part_stride, bool first, cudaStream_t s) {
  const int n2 = p.n * p.n;
  if (p.n % 8 == 0) {
    const dim3 grid((n2 / 8 + 127) / 128, gemm_adj_slices(p));
    return launch_next(first ? k_field_adj8<true> : k_field_adj8<false>, grid, 128, 0, s, p.fld, ckpt, h, chan, partial,
                       part_stride, p.X1, nwc, p.n, p.kp1);
  }
  return launch_next(first ? k_field_adj<true> : k_field_adj<false>, dim3((n2 + 255) / 256), 256, 0, s, p.fld, ckpt, h,
                     chan, partial, p.X1, nwc, p.n, p.kp1);
}

}  // namespace dos

