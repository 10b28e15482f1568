// dos_loss.cu - objective, quality metric and the gradient reduction.
//
// Section 2: the design minimises an MSE between the output intensity O_w of
// every channel and its target; reconstruction quality is a PSNR.  The
// detector (Section 4: the FOV divided into output pixels) reads pixel (y, x)
// as the sum of the b x b simulation intensities it covers (b = 1: I itself).
// Per-pixel arithmetic and the 256 strided partial sums of a channel run in FP32 (at
// most a few hundred terms each); partials are added in FP64, two by two as FP32
// pairs first (GB300's FP64 rate is a small fraction of its FP32 rate), and what
// follows is FP64 but for the PSNR's logarithm and the gradient parts' sums (FP32
// pairs).  Every sum has a fixed order, so results are reproducible bit for bit.
#include "dos_decibel.cuh"
#include "dos_internal.h"

#include "../../include/dos.h"

namespace dos {

constexpr int kRedThreads = 256;  // threads of a reducing block (k_loss also has a smaller one)

__device__ __forceinline__ double block_sum(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

__device__ __forceinline__ float intensity(float2 o) { return fmaf(o.x, o.x, o.y * o.y); }

// detector pixel p = (y, x) of a channel's F x F output field: sum over its b x b block
__device__ __forceinline__ float detector(const float2* ow, int fov, int b, int p) {
  if (b == 1) return intensity(ow[p]);
  const int fd = fov / b, y = (p / fd) * b, x = (p % fd) * b;
  float s = 0.f;
  for (int i = 0; i < b; ++i)
    for (int j = 0; j < b; ++j) s += intensity(ow[(size_t)(y + i) * fov + x + j]);
  return s;
}

// (s, e) += x with s + e kept exact up to the rounding of e
__device__ __forceinline__ void pair_add(float& s, float& e, float x) {
  const float t = __fadd_rn(s, x);
  const float z = __fadd_rn(t, -s);
  e = __fadd_rn(e, __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -z)), __fadd_rn(x, -z)));
  s = t;
}

// Fixed-order FP64 total of 256 FP32 partials, by one warp: partials i and i + 128
// are added as an FP32 pair, lane l adds four of the pairs in FP64 and
// their low parts in FP32, a shuffle tree the 32 lanes.  The total is valid in
// lane 0.  (An FP64 addition occupies the SM's FP64 pipe for many cycles: one warp
// issues ten of them here where a block-wide tree in shared memory issues them
// from every warp and takes eight barriers per sum.  With each of the 256 partials
// added in FP64 the launch took 6.1 us for 4 channels, now 5.7.)
__device__ __forceinline__ double warp_total(const float* part, int lane) {
  double v = 0.0;
  float l = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float s = part[lane + 32 * i], e = 0.f;
    pair_add(s, e, part[lane + 32 * i + 128]);
    v += (double)s;
    l += e;
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    v += __shfl_down_sync(0xffffffffu, v, s);
    l += __shfl_down_sync(0xffffffffu, l, s);
  }
  l = __shfl_sync(0xffffffffu, l, 0);
  if (!isnan(l)) return v + (double)l;
  // an infinite partial, or a pair past FP32's range (no low part): all of it in FP64
  v = 0.0;
  for (int i = 0; i < kRedThreads / 32; ++i) v += (double)part[lane + 32 * i];
  for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
  return v;
}

// Detector pixels a channel may have for its values to stay in shared memory
// between the two loops (16 KB: five blocks and more per SM); above it the
// second loop forms them again.
constexpr int kLossKeep = 4096;
// Up to this many detector pixels, and above as many channels as blocks of 256
// threads are resident at once (eight per SM), a channel gets a block of 128
// threads, so that twice as many are in flight: 2048 channels of 32 x 32 on 4 x
// 4-pixel detectors 37 -> 31 us, but 4 channels of 32 x 32 1.3 us more.  A thread
// of it keeps its even and its odd strides apart, as the partials that two threads
// of the larger block have: the sums are the same bit for bit.
constexpr int kLossSmall = 1280, kLossMany = 1024;

// One block per channel: sum (D-T)^2, sigma = sum D T / sum D^2, sum (sigma D
// - T)^2, the PSNR (psnr not null) and (dLdI not null) dL/dI of the channel's
// simulation pixels: dL/dD of the detector pixel covering it, 2 (D - T) / norm,
// or 2 sigma (sigma D - T) / norm for the scaled loss (scale = 2 / norm).  The
// last block to finish adds the channels' terms in a fixed order to the loss.
//
// Bound by latency, not bandwidth, below a few hundred channels: one launch
// instead of two, four barriers per channel instead of about forty, one FP64
// division and one logarithm per channel, each in a block of its own (the
// total kernel took them all in one block), and the detector sums formed once.
// 4096 channels of 50 x 50: 157 -> 64 us; 2048 channels of 32 x 32 on
// 4 x 4-pixel detectors 88 -> 31 us; 4 channels of 32 x 32 20 -> 11 us (with the
// total and the PSNR, both launches before).
template <int NT>
__global__ void __launch_bounds__(NT) k_loss(const float2* __restrict__ o, const float* __restrict__ T,
                                                      LossStats* __restrict__ st, int fov, int b,
                                                      float* __restrict__ dLdI, float scale, double norm, int mode,
                                                      float* __restrict__ psnr, double* __restrict__ d_loss,
                                                      unsigned* __restrict__ ticket) {
  extern __shared__ float dsh[];  // [det2] detector values, when det2 <= kLossKeep
  __shared__ float part[3][kRedThreads];  // chain i: pixels i, i + 256, ...
  __shared__ double tot[3];
  __shared__ float sg_sh;
  __shared__ bool last;
  pdl_wait();
  const int w = blockIdx.x, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int fd = fov / b, det2 = fd * fd;
  const bool keep = det2 <= kLossKeep;
  const float2* ow = o + (size_t)w * fov * fov;
  const float* tw = T + (size_t)w * det2;
#pragma unroll 1
  for (int i = threadIdx.x; i < kRedThreads; i += NT) {
    float fse = 0.f, fit = 0.f, fii = 0.f;
    for (int p = i; p < det2; p += kRedThreads) {
      const float I = detector(ow, fov, b, p);
      const float t = tw[p];
      const float d = I - t;
      if (keep) dsh[p] = I;
      fse = fmaf(d, d, fse);
      fit = fmaf(I, t, fit);
      fii = fmaf(I, I, fii);
    }
    part[0][i] = fse;
    part[1][i] = fit;
    part[2][i] = fii;
  }
  __syncthreads();
  if (warp < 3) {
    const double v = warp_total(part[warp], lane);
    if (lane == 0) tot[warp] = v;
  }
  __syncthreads();
  double sigma = 0.0;
  if (threadIdx.x == 0) {
    if (tot[2] > 0.0) sigma = tot[1] / tot[2];
    sg_sh = (float)sigma;
  }
  __syncthreads();
  const float sg = sg_sh;
  const bool scaled = mode == DOS_LOSS_MSE_SCALED;
  float* gw = dLdI ? dLdI + (size_t)w * fov * fov : nullptr;
#pragma unroll 1
  for (int i = threadIdx.x; i < kRedThreads; i += NT) {
    float fsc = 0.f;
    for (int p = i; p < det2; p += kRedThreads) {
      const float I = keep ? dsh[p] : detector(ow, fov, b, p);
      const float t = tw[p];
      const float d = fmaf(sg, I, -t);
      fsc = fmaf(d, d, fsc);
      if (gw && b == 1) gw[p] = scaled ? scale * sg * d : scale * (I - t);
    }
    part[0][i] = fsc;  // (its last reads were two barriers ago)
  }
  if (gw && b > 1) {
    const int fov2 = fov * fov;
    for (int q = threadIdx.x; q < fov2; q += NT) {
      const int p = ((q / fov) / b) * fd + (q % fov) / b;  // detector pixel covering q
      const float I = keep ? dsh[p] : detector(ow, fov, b, p);
      const float t = tw[p];
      gw[q] = scaled ? scale * sg * fmaf(sg, I, -t) : scale * (I - t);
    }
  }
  __syncthreads();
  if (warp == 0) {
    const double ssc = warp_total(part[0], lane);
    if (lane == 0) {
      LossStats s;
      s.sse = tot[0];
      s.sigma = sigma;
      s.sse_sc = ssc;
      s.pad = 0;
      st[w] = s;
      tot[1] = ssc;
      __threadfence();  // the record is visible before the ticket is taken
      last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
  }
  __syncthreads();
  // the PSNR, off the path that the total waits for
  if (psnr && threadIdx.x == NT - 32) psnr[w] = ten_log10((double)det2 / tot[1]);
  if (!last) return;
  // every channel's record is in place: the total, in a fixed order (each
  // thread a stride of the channels, the threads in order of one tree)
  __shared__ double acc[NT];
  __threadfence();
  double v = 0.0;
  for (int c = threadIdx.x; c < (int)gridDim.x; c += NT)
    v += __ldcg(scaled ? &st[c].sse_sc : &st[c].sse);
  acc[threadIdx.x] = v;
  __syncthreads();
  if (warp == 0) {
    v = 0.0;
#pragma unroll
    for (int i = 0; i < NT / 32; ++i)
      if (32 * i < (int)gridDim.x) v += acc[lane + 32 * i];
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
    if (lane == 0) {
      *d_loss = v / norm;
      *ticket = 0;  // the next launch starts from zero
    }
  }
}

cudaError_t launch_loss(const float2* o, const float* T, LossStats* st, int nw, int fov, int bin, float* dLdI,
                        double norm, int mode, float* psnr, double* d_loss, unsigned* ticket, cudaStream_t s) {
  const float scale = (float)(2.0 / norm);  // dL/dD = 2 (D - T) / norm
  const int det2 = (fov / bin) * (fov / bin);
  const size_t sm = det2 <= kLossKeep ? sizeof(float) * det2 : 0;
  const bool small = det2 <= kLossSmall && nw > kLossMany;
  return launch_next(small ? k_loss<128> : k_loss<kRedThreads>, dim3(nw), small ? 128 : kRedThreads, sm, s, o, T, st,
                     fov, bin, dLdI, scale, norm, mode, psnr, d_loss, ticket);
}

__global__ void __launch_bounds__(kRedThreads) k_loss_final(const LossStats* __restrict__ st, int nw,
                                                            int fov2, double norm, int mode,
                                                            double* __restrict__ d_loss,
                                                            float* __restrict__ psnr) {
  __shared__ double sh[kRedThreads];
  double acc = 0;
  for (int w = threadIdx.x; w < nw; w += kRedThreads) {
    const LossStats s = st[w];
    acc += mode == DOS_LOSS_MSE_SCALED ? s.sse_sc : s.sse;
    if (psnr) psnr[w] = (float)(10.0 * log10((double)fov2 / s.sse_sc));
  }
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) *d_loss = acc / norm;
}

cudaError_t launch_loss_final(const LossStats* st, int nw, int fov2, double norm, int mode,
                              double* d_loss, float* d_psnr, cudaStream_t s) {
  k_loss_final<<<1, kRedThreads, 0, s>>>(st, nw, fov2, norm, mode, d_loss, d_psnr);
  return cudaGetLastError();
}

// grad[g] = sum over the parts c of partial[layer(g)][c][pixel(g)], in a fixed
// order.  Sums of FP32 partials carried as an FP32 pair (a running sum and the
// exact rounding errors of its additions, Knuth's two-sum), about 48 bits, and
// rounded to FP32 once at the end like the FP64 sum before it: GB300 adds and
// converts FP64 at a small fraction of its FP32 rate, which bound the kernel.
// Where the running sum leaves FP32's range the parts are added in FP64 after all:
// they may come back.
// A block's 256 threads take 32 pixels x 8 slices of the parts, eight loads of a
// slice in flight, so that small layers with many parts still fill the chip; or
// 256 pixels each with all of them where the parts are few and the pixels many
// (below 64 parts a slice is shorter than one unrolled step).
// 5 layers of 200 x 200: 92 parts 86 -> 22 us, 86 parts 81 -> 26 us, 18 parts with
// eight slices 18 us, with one 9 us; 3 layers of 64 x 64, 293 parts 57 -> 12 us.
// A step's thickness is copied here too (h not null), which saves the step a
// copy of its own.
constexpr int kGradThreads = 256;

template <int SLICES>
__global__ void __launch_bounds__(kGradThreads) k_grad_reduce(const float* __restrict__ partial,
                                                              float* grad, int n_parts, size_t count, size_t n2,
                                                              const float* h, float* h_keep) {
  constexpr int PX = kGradThreads / SLICES;
  __shared__ float2 sh[SLICES][PX];
  pdl_wait();
  const int lane = threadIdx.x % PX, slice = threadIdx.x / PX;
  const size_t g = (size_t)blockIdx.x * PX + lane;
  const int per = (n_parts + SLICES - 1) / SLICES;
  const int c0 = min(slice * per, n_parts), c1 = min(c0 + per, n_parts);
  float s = 0.f, e = 0.f;
  if (g < count) {
    const size_t layer = g / n2, px = g % n2;
    const float* p = partial + (layer * n_parts + c0) * n2 + px;
    int c = c0;
    for (; c + 8 <= c1; c += 8, p += 8 * n2) {
      float x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = __ldcs(p + i * n2);
#pragma unroll
      for (int i = 0; i < 8; ++i) pair_add(s, e, x[i]);
    }
    for (; c < c1; ++c, p += n2) pair_add(s, e, __ldcs(p));
  }
  if constexpr (SLICES > 1) {
    sh[slice][lane] = make_float2(s, e);
    __syncthreads();
  }
  if (slice != 0 || g >= count) return;
#pragma unroll
  for (int q = 1; q < SLICES; ++q) {
    const float2 v = sh[q][lane];
    pair_add(s, e, v.x);
    e = __fadd_rn(e, v.y);
  }
  if (h) h_keep[g] = h[g];
  float v = s + e;
  if (!isfinite(v)) {
    const float* p = partial + g / n2 * n_parts * n2 + g % n2;
    double acc = 0.0;
    for (int c = 0; c < n_parts; ++c) acc += (double)p[(size_t)c * n2];
    v = (float)acc;
  }
  grad[g] = v;  // (the caller's gradient may lie where its thickness does: h is read first)
}

cudaError_t launch_grad_reduce(const float* partial, float* grad, int n_parts, size_t count, size_t n2, const float* h,
                               float* h_keep, cudaStream_t s) {
  const bool one = n_parts < 64 && count >= (size_t)64 * kGradThreads;
  const size_t px = one ? kGradThreads : kGradThreads / 8;
  return launch_next(one ? k_grad_reduce<1> : k_grad_reduce<8>, dim3((unsigned)((count + px - 1) / px)), kGradThreads, 0,
                     s, partial, grad, n_parts, count, n2, h, h_keep);
}

}  // namespace dos
