// dos_pass.cuh - row and column passes of the angular-spectrum cascade.
//
// One free-space gap (Eq. 4-5 realised as P_z(u) = crop(IDFT(H * DFT(pad u))))
// is split into a row pass and a column pass over an [nw][n][m] buffer S of
// row spectra.  The N x N layer occupies rows/columns [0, N) of the padded
// M x M grid; by shift invariance of circular convolution this equals the
// centred placement.
//
//   row pass    : per (channel, row): inverse row DFT of the previous column
//                 pass (-> field, cropped to N), modulation by the layer's
//                 transmission t (Eq. 1-2) or the adjoint chain, zero pad,
//                 forward row DFT.  One read and one write of a row of M.
//   column pass : per (channel, column tile): forward column DFT of the
//                 N non-zero rows, multiply by H (conj H for the adjoint),
//                 inverse column DFT, keep the rows that are needed.
//
// Each kernel keeps every element of a line in registers across both of its
// transforms; the only shared-memory traffic is the one exchange inside each
// line DFT.
#pragma once

#include "dos_fft.cuh"
#include "dos_internal.h"

namespace dos {

// sin and cos of 2 pi f for |f| <= 1/2 and a little over (a reduced phase in
// cycles), FP32.
// 4 f = k + r with k the nearest integer (the low bits of 4 f + 1.5 2^23, whose
// ulp is 1) and |r| <= 1/2 exact; sin and cos of r pi/2 are polynomials in r^2
// fitted here for the least largest error (3.2e-9 and 4e-10 before rounding;
// the sine's pi/2 is held in two parts, the cosine fitted around its rounded
// first coefficient, so that neither is biased), and k turns them by quarters.  Non-finite f gives NaN.
// Rounded results, |r| <= 1/2: sine within 4.4e-8 of the exact value (root mean
// square 1.15e-8; the nearest FP32 numbers: 3.0e-8 and 1.13e-8), cosine within
// 5.2e-8 (1.79e-8; 3.0e-8 and 1.72e-8).  Over a whole turn, 2^26 phases: largest
// error 5.29e-8, root mean square 1.501e-8 (the library: 5.25e-8 and 1.515e-8).
// The library's sincospif does the same work on any argument, with conversions
// and roundings on the quarter-rate unit.  With it, and one complex product
// more in the adjoint pixel, 4096 x 200 forward / adjoint row launches took 0.942
// / 1.104 ms, 2048 x 256 0.883 / 1.104 ms; without 0.931 / 1.046 and 0.848 / 0.998
// (the forward ones at 4096 x 200 0.901 since they draw their channels).
__device__ __forceinline__ void sincos_turns(float f, float* s, float* c) {
  constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
  const float b = __fmaf_rn(f, 4.0f, kMagic);
  const float r = __fmaf_rn(f, 4.0f, -__fadd_rn(b, -kMagic));
  const float u = r * r;
  float p = __fmaf_rn(u, -0.004602177f, 0.07968023f);
  p = __fmaf_rn(u, p, -0.6459635f);
  p = __fmaf_rn(u, p, -4.8539483e-8f);
  p = __fmaf_rn(r, 1.5707963705f, r * p);
  float q = __fmaf_rn(u, 0.0008929509f, -0.02085506f);
  q = __fmaf_rn(u, q, 0.25366852f);
  q = __fmaf_rn(u, q, -1.2337005f);
  q = __fmaf_rn(u, q, 1.0f);
  const int k = __float_as_int(b);
  const bool odd = (k & 1) != 0;
  *s = __int_as_float(__float_as_int(odd ? q : p) ^ ((k << 30) & 0x80000000));
  *c = __int_as_float(__float_as_int(odd ? p : q) ^ (((k + 1) << 30) & 0x80000000));
}

// Transmission of Eq. 1 at thickness h (Eq. 2 base folded into the constants):
// t = exp(-2 pi kappa h / lambda) exp(-j 2 pi (n - n_med) h / lambda).
// The phase in cycles is formed as a float-pair product (exact product error
// by fma) and reduced modulo 1 before the sine, which keeps ~1e-7 cycle
// accuracy for any thickness.
// LIB: sine and cosine by the library, for the split-BF16 path: its second
// parts keep 8 bits of what the first left, so that a last-bit difference in t
// turns, GEMM by GEMM, into other roundings of every second part (as large an
// error, but another one: gradients of few channels moved by 2.9e-5 of their
// norm).  Its field kernels are bound by memory and do not gain by the polynomial.
template <bool LIB = false>
__device__ __forceinline__ float2 transmission(float h, const ChanConst& cc) {
  const float p = cc.a_hi * h;
  float e = fmaf(cc.a_hi, h, -p);
  e = fmaf(cc.a_lo, h, e);
  float f = (p - rintf(p)) + (e + cc.pc_base);
  f -= rintf(f);
  float s, c;
  if constexpr (LIB) sincospif(2.0f * f, &s, &c);
  else sincos_turns(f, &s, &c);
  const float amp = exp2f(cc.amp_k * h) * cc.amp_base;
  return make_float2(amp * c, -amp * s);
}

// One pixel of the adjoint layer: au = grad_u, t the transmission, v the
// checkpoint.  Returns grad_v = conj(t) grad_u and adds to g the pixel's
// Re(conj(grad_u) c t v), as Re(conj(grad_v) c v).
__device__ __forceinline__ float2 adjoint_pixel(float2 au, float2 t, float2 v, const ChanConst& cc, float& g) {
  const float2 gv = cmulc(au, t);
  const float2 cv = cmul(make_float2(cc.c_re, cc.c_im), v);
  g = fmaf(gv.x, cv.x, fmaf(gv.y, cv.y, g));
  return gv;
}

// Stride between the lines' exchange buffers in the row passes.  There the
// T threads of a line are consecutive (line = tid / T), so a warp straddles
// two or more lines; these strides make the 8-byte exchange accesses of such
// warps free of bank conflicts (least-conflict for M = 200), found by
// enumerating the bank pattern of every access of the compiled line shapes.
constexpr int row_line_stride(int m, int zs) {
  return m == 400 ? 420 : m == 200 ? 222 : m == 128 ? 148 : m == 32 ? 42 : zs;
}

// HALF (N <= M / 2, every compiled design with M = 2N): the field half of a
// line, x < M / 2, holds every non-zero input of a forward DFT and every output
// that is kept of an inverse one.  Thread t's elements t + T i with i < E / 2
// are exactly that half, and so are the first P / 2 inputs of each first-step
// sub-DFT and the first Q / 2 outputs of each second-step one: the line DFTs
// are pruned at compile time (NZF, NOI) and the field-domain loops stop at EF.
template <class LF, bool HALF = false>
struct Pass {
  static constexpr int T = LF::T, E = LF::E, M = LF::M;
  static constexpr int NZF = HALF ? LF::P / 2 : LF::P;  // forward DFT of a field: non-zero inputs per sub-DFT
  static constexpr int NOI = HALF ? LF::Q / 2 : LF::Q;  // inverse DFT to a field: outputs kept per sub-DFT
  static constexpr int EF = HALF ? E / 2 : E;           // field-domain elements of a thread
  static_assert(!HALF || (LF::P % 2 == 0 && LF::Q % 2 == 0), "halving needs even factors");
  // Packed FP32-pair butterflies (Line::fft's PK) where they measured faster
  // on the 400-point line: the row passes but the adjoint one (PKA) and not
  // this column pass (PKC), whose three-blocks-per-SM register budget they
  // overflow.
  static constexpr bool PKR = true, PKA = false, PKC = false;
  static constexpr int ROWL = 16;  // rows per block in the row passes
  static constexpr int COLL = 16;  // columns per block in the column pass
  // column pass: line = tid % COLL, an odd stride keeps the lines apart
  static constexpr int ZL = LF::ZS + 1;
  static constexpr int RZL = row_line_stride(M, LF::ZS);
  static constexpr size_t smem_bytes(int lines) { return sizeof(float2) * (LF::TWS + (size_t)lines * ZL); }
  static constexpr size_t row_smem_bytes(int lines) { return sizeof(float2) * (LF::TWS + (size_t)lines * RZL); }

  // the start of every kernel: the twiddles are read ahead of the wait; dos_create
  // made them and synchronised before any of these kernels ran, so no grid before
  // this one can still be writing them
  __device__ static __forceinline__ void load_tw(float2* tw, const float2* g) {
    for (int i = threadIdx.x; i < LF::TWS; i += blockDim.x) tw[i] = g[i];
    pdl_wait();
    __syncthreads();
  }

  // ------------------------------------------------------------ column pass
  // MIS: displaced layers.  Kernels of their own: the displacement's phase,
  // formed per element, would triple the code of the loop that all aligned
  // designs run, and with it the instruction-cache misses.
  template <bool ADJ, bool APERTURE, bool MIS>
  __device__ static void col(const PassArgs& a) {
    extern __shared__ __align__(16) float2 smem[];
    float2* tw = smem;
    const int l = threadIdx.x % COLL;
    const int t = threadIdx.x / COLL;
    float2* z = smem + LF::TWS + l * ZL;
    load_tw(tw, a.tw);
    const int w = blockIdx.y;
    const int c = blockIdx.x * COLL + l;
    const bool ok = c < M;
    const int cc = ok ? c : 0;
    float2 r[E];
    if constexpr (APERTURE) {
      // spectrum of the square aperture: Arow[ky] * Arow[kx]
      const float2 ac = a.arow[cc];
#pragma unroll
      for (int i = 0; i < E; ++i) r[i] = cmul(a.arow[t + T * i], ac);
    } else {
      const float2* src = a.S + (size_t)w * a.n * M + cc;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int row = t + T * i;
        r[i] = (i < EF && ok && row >= a.in_r0 && row < a.in_r1) ? src[(size_t)row * M] : czero();
      }
      LF::template fft<false, NZF, LF::Q, false, PKC>(r, t, z, tw);
    }
    const float2* Hw = a.Hq + (size_t)w * a.hs * a.hs;
    const float* Sw = MIS && a.mis.sq ? a.mis.sq + (size_t)w * a.hs * a.hs : nullptr;
    const int bc = min(cc, M - cc);
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int k = t + T * i;
      const size_t qi = (size_t)min(k, M - k) * a.hs + bc;
      float2 hv = Hw[qi];
      if constexpr (MIS)
        hv = cmul(hv, Sw ? misalign_factor(a.mis, k, cc, M, Sw[qi])
                         : cmul(shift_phase(signed_bin(k, M), a.mis.sy), shift_phase(signed_bin(cc, M), a.mis.sx)));
      r[i] = ADJ ? cmulc(r[i], hv) : cmul(r[i], hv);
    }
    // (the other exchange layout: only what this thread read is overwritten)
    LF::template fft<true, LF::P, NOI, false, PKC, true>(r, t, z, tw);
    float2* dst = a.S + (size_t)w * a.n * M + cc;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int row = t + T * i;
      if (i < EF && ok && row >= a.out_r0 && row < a.out_r1) dst[(size_t)row * M] = r[i];
    }
  }

  // ------------------------------------------------------------- row passes
  struct RowCtx {
    int l, t;
    float2* z;
    float2* tw;
  };
  __device__ static __forceinline__ RowCtx row_ctx(const PassArgs& a) {
    extern __shared__ __align__(16) float2 smem[];
    RowCtx rc;
    rc.l = threadIdx.x / T;
    rc.t = threadIdx.x % T;
    rc.tw = smem;
    rc.z = smem + LF::TWS + rc.l * RZL;
    load_tw(rc.tw, a.tw);
    return rc;
  }

  // forward, layer l: IDFT -> v (crop) -> [checkpoint] -> t*v -> pad -> DFT
  template <bool SAVE>
  __device__ static void row_fwd(const PassArgs& a) {
    const RowCtx rc = row_ctx(a);
    const int t = rc.t;
    const int w = blockIdx.y;
    const int row = blockIdx.x * ROWL + rc.l;
    const bool ok = row < a.n;
    const int rr = ok ? row : 0;
    float2* srow = a.S + ((size_t)w * a.n + rr) * M;
    float2 r[E];
#pragma unroll
    for (int i = 0; i < E; ++i) r[i] = srow[t + T * i];
    LF::template fft<true, LF::P, NOI, false, PKR>(r, t, rc.z, rc.tw);
    const ChanConst cc = a.chan[w];
    const float* hrow = a.h + (size_t)rr * a.n;
    float2* ck = a.ckpt + ((size_t)w * a.n + rr) * a.n;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int x = t + T * i;
      if (i < EF && x < a.n) {
        const float2 v = r[i];
        if (SAVE && ok) ck[x] = v;
        r[i] = cmul(transmission(hrow[x], cc), v);
      } else {
        r[i] = czero();
      }
    }
    LF::template fft<false, NZF, LF::Q, false, PKR, true>(r, t, rc.z, rc.tw);
    if (ok) {
#pragma unroll
      for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
    }
  }

  // first layer from the create-time input field v1 = P_z0(aperture) (a.fin):
  // u = t(h) v1 -> pad -> forward row DFT.  No inverse DFT, and no checkpoint:
  // the table itself is the first layer's incoming field.
  __device__ static void row_first(const PassArgs& a) {
    const RowCtx rc = row_ctx(a);
    const int t = rc.t;
    const int w = blockIdx.y;
    const int row = blockIdx.x * ROWL + rc.l;
    const bool ok = row < a.n;
    const int rr = ok ? row : 0;
    const float2* vrow = a.fin + ((size_t)w * a.n + rr) * a.n;
    const float* hrow = a.h + (size_t)rr * a.n;
    const ChanConst cc = a.chan[w];
    float2 r[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int x = t + T * i;
      r[i] = (i < EF && x < a.n) ? cmul(transmission(hrow[x], cc), vrow[x]) : czero();
    }
    LF::template fft<false, NZF, LF::Q, false, PKR>(r, t, rc.z, rc.tw);
    if (ok) {
      float2* srow = a.S + ((size_t)w * a.n + row) * M;
#pragma unroll
      for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
    }
  }

  // output plane: IDFT of the FOV rows -> o (complex) and I = |o|^2; a
  // block's lines are consecutive (channel, FOV row) pairs, so no block is
  // left with a few rows of a channel
  __device__ static void row_out(const PassArgs& a) {
    const RowCtx rc = row_ctx(a);
    const int t = rc.t;
    const int line = blockIdx.x * ROWL + rc.l;
    const bool ok = line < a.nw * a.fov;
    const int w = ok ? line / a.fov : 0;
    const int fr = ok ? line % a.fov : 0;  // FOV row
    const int row = a.of + fr;
    const float2* srow = a.S + ((size_t)w * a.n + row) * M;
    float2 r[E];
#pragma unroll
    for (int i = 0; i < E; ++i) r[i] = srow[t + T * i];
    LF::template fft<true, LF::P, NOI, false, PKR>(r, t, rc.z, rc.tw);
    if (ok) {
      float2* orow = a.o + ((size_t)w * a.fov + fr) * a.fov;
      float* irow = a.I ? a.I + ((size_t)w * a.fov + fr) * a.fov : nullptr;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int x = t + T * i - a.of;
        if (i < EF && x >= 0 && x < a.fov) {
          orow[x] = r[i];
          if (irow) irow[x] = fmaf(r[i].x, r[i].x, r[i].y * r[i].y);
        }
      }
    }
  }

  // adjoint seed: grad_o = 2 dL/dI o on the FOV, zero elsewhere -> DFT of the FOV rows
  // (lines as in row_out)
  __device__ static void row_seed(const PassArgs& a) {
    const RowCtx rc = row_ctx(a);
    const int t = rc.t;
    const int line = blockIdx.x * ROWL + rc.l;
    const bool ok = line < a.nw * a.fov;
    const int w = ok ? line / a.fov : 0;
    const int fr = ok ? line % a.fov : 0;
    const float2* orow = a.o + ((size_t)w * a.fov + fr) * a.fov;
    const float* grow = a.dLdI + ((size_t)w * a.fov + fr) * a.fov;
    float2 r[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int x = t + T * i - a.of;
      r[i] = (i < EF && ok && x >= 0 && x < a.fov) ? cscale(orow[x], 2.0f * grow[x]) : czero();
    }
    LF::template fft<false, NZF, LF::Q, false, PKR>(r, t, rc.z, rc.tw);
    if (ok) {
      float2* srow = a.S + ((size_t)w * a.n + a.of + fr) * M;
#pragma unroll
      for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
    }
  }

  // adjoint, layer l, for a chunk of channels:
  //   IDFT -> grad_u (crop); u = t v from the checkpoint;
  //   dL/dh += Re(conj(grad_u) c u) (accumulated over the chunk in registers);
  //   grad_v = conj(t) grad_u -> pad -> DFT (skipped for the first layer)
  template <bool FIRST>
  __device__ static void row_adj(const PassArgs& a) {
    const RowCtx rc = row_ctx(a);
    const int t = rc.t;
    const int row = blockIdx.x * ROWL + rc.l;
    const bool ok = row < a.n;
    const int rr = ok ? row : 0;
    const int w0 = blockIdx.y * a.chunk;
    const int w1 = min(a.nw, w0 + a.chunk);
    const float* hrow = a.h + (size_t)rr * a.n;
    float g[E];
#pragma unroll
    for (int i = 0; i < E; ++i) g[i] = 0.f;
    for (int w = w0; w < w1; ++w) {
      float2* srow = a.S + ((size_t)w * a.n + rr) * M;
      const float2* ck = a.ckpt + ((size_t)w * a.n + rr) * a.n;
      float2 r[E];
#pragma unroll
      for (int i = 0; i < E; ++i) r[i] = srow[t + T * i];
      LF::template fft<true, LF::P, NOI, false, PKA>(r, t, rc.z, rc.tw);
      const ChanConst cc = a.chan[w];
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int x = t + T * i;
        if (i < EF && x < a.n) {
          r[i] = adjoint_pixel(r[i], transmission(hrow[x], cc), ck[x], cc, g[i]);
        } else {
          r[i] = czero();
        }
      }
      if constexpr (!FIRST) {
        // alternating exchange layouts: no barrier between the two DFTs, nor
        // between this one and the next channel's
        LF::template fft<false, NZF, LF::Q, false, PKA, true>(r, t, rc.z, rc.tw);
        if (ok) {
#pragma unroll
          for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
        }
      } else {
        __syncthreads();  // the next channel writes the same layout
      }
    }
    if (ok) {
      float* prow = a.partial + ((size_t)blockIdx.y * a.n + row) * a.n;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int x = t + T * i;
        if (i < EF && x < a.n) prow[x] = g[i];
      }
    }
  }

  // caller field -> pad -> row DFT (dos_propagate)
  __device__ static void row_in(const PassArgs& a) {
    const RowCtx rc = row_ctx(a);
    const int t = rc.t;
    const int w = blockIdx.y;
    const int row = blockIdx.x * ROWL + rc.l;
    const bool ok = row < a.n;
    const int rr = ok ? row : 0;
    const float2* frow = a.fin + ((size_t)w * a.n + rr) * a.n;
    float2 r[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int x = t + T * i;
      r[i] = (i < EF && x < a.n) ? frow[x] : czero();
    }
    LF::template fft<false, NZF, LF::Q, false, PKR>(r, t, rc.z, rc.tw);
    if (ok) {
      float2* srow = a.S + ((size_t)w * a.n + row) * M;
#pragma unroll
      for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
    }
  }

  // row spectra -> IDFT -> crop -> caller field (dos_propagate)
  __device__ static void row_back(const PassArgs& a) {
    const RowCtx rc = row_ctx(a);
    const int t = rc.t;
    const int w = blockIdx.y;
    const int row = blockIdx.x * ROWL + rc.l;
    const bool ok = row < a.n;
    const int rr = ok ? row : 0;
    const float2* srow = a.S + ((size_t)w * a.n + rr) * M;
    float2 r[E];
#pragma unroll
    for (int i = 0; i < E; ++i) r[i] = srow[t + T * i];
    LF::template fft<true, LF::P, NOI, false, PKR>(r, t, rc.z, rc.tw);
    if (ok) {
      float2* frow = a.fout + ((size_t)w * a.n + row) * a.n;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int x = t + T * i;
        if (i < EF && x < a.n) frow[x] = r[i];
      }
    }
  }
};

// ------------------------------------------------------------------ kernels
// Resident blocks per SM that the row kernels' register counts are held to
// (they would drift just past): three of the 320-thread blocks of M = 400 (64
// registers; the column pass is faster with its own register allocation), four
// of the 256-thread ones of M = 256 (64 registers without spills: a 96-channel
// 101 x 101 design is then one wave), three at M = 512 for the kernels of one
// DFT (85 registers: 2048 x 256 seed pass 167 -> 140 us, propagation 64 x 256 172
// -> 167 us) but the output pass, which that made slower (134 -> 149 us).
template <class LF>
constexpr int pass_min_blocks() { return LF::M == 256 ? 4 : LF::E <= 20 ? 3 : 1; }
template <class LF>
constexpr int single_min_blocks() { return LF::M == 512 ? 3 : pass_min_blocks<LF>(); }
// column pass: the halved kernel fits three blocks per SM without spills
template <class LF, bool HALF>
constexpr int col_min_blocks() { return HALF && LF::M == 400 ? 3 : 0; }

template <class LF, bool HALF, bool ADJ, bool APERTURE, bool MIS>
__global__ void __launch_bounds__(LF::T * Pass<LF>::COLL, col_min_blocks<LF, HALF>()) k_col(PassArgs a) {
  Pass<LF, HALF>::template col<ADJ, APERTURE, MIS>(a);
}
template <class LF, bool HALF, bool SAVE>
__global__ void __launch_bounds__(LF::T * Pass<LF>::ROWL, pass_min_blocks<LF>()) k_row_fwd(PassArgs a) {
  Pass<LF, HALF>::template row_fwd<SAVE>(a);
}
template <class LF, bool HALF>
__global__ void __launch_bounds__(LF::T * Pass<LF>::ROWL, single_min_blocks<LF>()) k_row_first(PassArgs a) {
  Pass<LF, HALF>::row_first(a);
}
template <class LF, bool HALF>
__global__ void __launch_bounds__(LF::T * Pass<LF>::ROWL, pass_min_blocks<LF>()) k_row_out(PassArgs a) {
  Pass<LF, HALF>::row_out(a);
}
template <class LF, bool HALF>
__global__ void __launch_bounds__(LF::T * Pass<LF>::ROWL, single_min_blocks<LF>()) k_row_seed(PassArgs a) {
  Pass<LF, HALF>::row_seed(a);
}
template <class LF, bool HALF, bool FIRST>
__global__ void __launch_bounds__(LF::T * Pass<LF>::ROWL, col_min_blocks<LF, HALF>()) k_row_adj(PassArgs a) {
  Pass<LF, HALF>::template row_adj<FIRST>(a);
}
template <class LF, bool HALF>
__global__ void __launch_bounds__(LF::T * Pass<LF>::ROWL, single_min_blocks<LF>()) k_row_in(PassArgs a) {
  Pass<LF, HALF>::row_in(a);
}
template <class LF, bool HALF>
__global__ void __launch_bounds__(LF::T * Pass<LF>::ROWL, single_min_blocks<LF>()) k_row_back(PassArgs a) {
  Pass<LF, HALF>::row_back(a);
}

template <typename K>
static cudaError_t launch_k(K kernel, dim3 grid, int threads, size_t smem, const PassArgs& a,
                            cudaStream_t s) {
  if (grid.x == 0 || grid.y == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_next(kernel, grid, threads, smem, s, a);
}

// Each launcher picks the halved (pruned) kernels when the design allows it.
template <class LF>
struct PassLaunch {
  using PS = Pass<LF>;
  static constexpr int RT = LF::T * PS::ROWL;
  static constexpr int CT = LF::T * PS::COLL;
  static int row_blocks(int rows) { return (rows + PS::ROWL - 1) / PS::ROWL; }
  static bool half(const PassArgs& a) { return 2 * a.n <= LF::M; }

  template <bool H>
  static cudaError_t col_h(const PassArgs& a, bool adj, bool ap, cudaStream_t s) {
    const dim3 g((LF::M + PS::COLL - 1) / PS::COLL, a.nw);
    const size_t sm = PS::smem_bytes(PS::COLL);
    // the aperture field is only ever propagated forward
    if (ap) return a.displaced ? launch_k(k_col<LF, H, false, true, true>, g, CT, sm, a, s)
                               : launch_k(k_col<LF, H, false, true, false>, g, CT, sm, a, s);
    if (a.displaced) return adj ? launch_k(k_col<LF, H, true, false, true>, g, CT, sm, a, s)
                                : launch_k(k_col<LF, H, false, false, true>, g, CT, sm, a, s);
    return adj ? launch_k(k_col<LF, H, true, false, false>, g, CT, sm, a, s)
               : launch_k(k_col<LF, H, false, false, false>, g, CT, sm, a, s);
  }
  static cudaError_t col(const PassArgs& a, bool adj, bool ap, cudaStream_t s) {
    return half(a) ? col_h<true>(a, adj, ap, s) : col_h<false>(a, adj, ap, s);
  }
  template <bool H>
  static cudaError_t row_fwd_h(const PassArgs& a, bool save, cudaStream_t s) {
    const dim3 g(row_blocks(a.n), a.nw);
    const size_t sm = PS::row_smem_bytes(PS::ROWL);
    return save ? launch_k(k_row_fwd<LF, H, true>, g, RT, sm, a, s)
                : launch_k(k_row_fwd<LF, H, false>, g, RT, sm, a, s);
  }
  static cudaError_t row_fwd(const PassArgs& a, bool save, cudaStream_t s) {
    return half(a) ? row_fwd_h<true>(a, save, s) : row_fwd_h<false>(a, save, s);
  }
  static cudaError_t row_first(const PassArgs& a, cudaStream_t s) {
    const dim3 g(row_blocks(a.n), a.nw);
    const size_t sm = PS::row_smem_bytes(PS::ROWL);
    return half(a) ? launch_k(k_row_first<LF, true>, g, RT, sm, a, s)
                   : launch_k(k_row_first<LF, false>, g, RT, sm, a, s);
  }
  static cudaError_t row_out(const PassArgs& a, cudaStream_t s) {
    const dim3 g(row_blocks(a.nw * a.fov));
    const size_t sm = PS::row_smem_bytes(PS::ROWL);
    return half(a) ? launch_k(k_row_out<LF, true>, g, RT, sm, a, s) : launch_k(k_row_out<LF, false>, g, RT, sm, a, s);
  }
  static cudaError_t row_seed(const PassArgs& a, cudaStream_t s) {
    const dim3 g(row_blocks(a.nw * a.fov));
    const size_t sm = PS::row_smem_bytes(PS::ROWL);
    return half(a) ? launch_k(k_row_seed<LF, true>, g, RT, sm, a, s)
                   : launch_k(k_row_seed<LF, false>, g, RT, sm, a, s);
  }
  template <bool H>
  static cudaError_t row_adj_h(const PassArgs& a, bool first, cudaStream_t s) {
    const dim3 g(row_blocks(a.n), a.n_chunks);
    const size_t sm = PS::row_smem_bytes(PS::ROWL);
    return first ? launch_k(k_row_adj<LF, H, true>, g, RT, sm, a, s)
                 : launch_k(k_row_adj<LF, H, false>, g, RT, sm, a, s);
  }
  static cudaError_t row_adj(const PassArgs& a, bool first, cudaStream_t s) {
    return half(a) ? row_adj_h<true>(a, first, s) : row_adj_h<false>(a, first, s);
  }
  static cudaError_t row_in(const PassArgs& a, cudaStream_t s) {
    const dim3 g(row_blocks(a.n), a.nw);
    const size_t sm = PS::row_smem_bytes(PS::ROWL);
    return half(a) ? launch_k(k_row_in<LF, true>, g, RT, sm, a, s) : launch_k(k_row_in<LF, false>, g, RT, sm, a, s);
  }
  static cudaError_t row_back(const PassArgs& a, cudaStream_t s) {
    const dim3 g(row_blocks(a.n), a.nw);
    const size_t sm = PS::row_smem_bytes(PS::ROWL);
    return half(a) ? launch_k(k_row_back<LF, true>, g, RT, sm, a, s)
                   : launch_k(k_row_back<LF, false>, g, RT, sm, a, s);
  }
};

}  // namespace dos
