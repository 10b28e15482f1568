// dos_pass_bulk.cuh - the multi-pass row and column passes with bulk-async prefetch.
//
// Same arithmetic as dos_pass.cuh; what changes is how the input reaches the
// block.  Blocks loop over several work items and the bulk-copy engine
// (cp.async.bulk global -> shared, completion counted in bytes on an
// mbarrier) fetches the next item while the block computes the current one:
//   column pass : item = a group of 8 columns of one channel (persistent
//                 blocks, items drawn from a counter); tensor copies (TMA) of
//                 the group's input rows and of the transfer-table tile;
//   row passes  : item = the block's RL rows of its next channel (drawn from a
//                 counter in the forward passes, the next of a chunk in the
//                 adjoint ones); one cp.async.bulk per row (rows padded in
//                 shared memory against bank conflicts): spectra rows, the rows
//                 of the input-field table in the first forward pass, and
//                 spectra plus checkpoint rows in the adjoint pass.
// One staging buffer per input suffices: the item is moved from the stage to
// registers and the next copy is issued at the first block barrier after
// that (the one inside the item's first line DFT), so the copy overlaps most
// of the item's DFT / modulation / DFT / store.
// Every wait is bounded (one second of global time).  Each thread times its
// own wait, and the block takes one verdict from them (a block-wide AND at the
// barrier after the wait), so that no thread goes on with an item another
// thread gave up on: when any wait expires the whole block issues no further
// copy, leaves its loop without writing partial results, waits once more
// (bounded) for its copies in flight and sets *err.
// PassArgs::stall (fault injection for tests): 1 makes the blocks announce
// their bytes without copying them, so that the first wait of every block
// expires; 2 lets the copies land but makes the odd threads of every block
// give up their first wait (a split verdict that the block-wide AND resolves).
#pragma once

#include <cuda.h>

#include <algorithm>
#include <cstdint>

#include "dos_pass.cuh"

namespace dos {

constexpr unsigned long long kBulkWaitNs = 1000000000ull;  // bounded wait: one second
constexpr long kBulkSpin = 1L << 30;                        // and an iteration cap behind it

__device__ __forceinline__ uint32_t sh_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// First 16-byte boundary at or after p: the line DFTs read the twiddle table
// in 16-byte pairs (the layouts reserve one extra float2 for the shift).
__device__ __forceinline__ float2* tw_align(float2* p) { return p + ((sh_addr(p) >> 3) & 1u); }

__device__ __forceinline__ void bulk_bar_init(uint64_t* b) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sh_addr(b)));
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void bulk_expect(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sh_addr(b)), "r"(bytes) : "memory");
}
// global -> shared copy of `bytes` (multiple of 16, both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   sh_addr(dst)),
               "l"(src), "r"(bytes), "r"(sh_addr(b))
               : "memory");
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// true once the phase with this parity has completed; false after kBulkWaitNs
// (or at once when `give_up` is set: the injected split verdict of the tests)
__device__ __forceinline__ bool bulk_wait(uint64_t* b, uint32_t parity, bool give_up = false) {
  if (give_up) return false;
  const unsigned long long t0 = global_ns();
  for (long it = 0; it < kBulkSpin; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(sh_addr(b)), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 15) == 15 && global_ns() - t0 > kBulkWaitNs) return false;
  }
  return false;
}

// Injected split verdict (PassArgs::stall == 2, tests only): the odd threads
// of every block give up their first wait although the copy lands.
__device__ __forceinline__ bool split_verdict(const PassArgs& a, int item) {
  return a.stall == 2 && item == 0 && (threadIdx.x & 1);
}

// Items 0 .. items - 1 of a launch, taken in order by whichever of its blocks is
// free: block b has item b, the others' numbers come from a counter that is zero
// between launches.  A block's thread 0 draws ahead; every block draws until its
// first number past the end, items draws in all, and whoever drew the last one
// sets the counter back to zero.  A block that gives up (an expired wait) goes
// on drawing without working (drain), so that this holds for it as well and the
// next launch, which may be queued before the host has seen the error, starts
// from zero.
struct Draws {
  unsigned* work;
  unsigned blocks, items;
  unsigned drawn;  // the counter's latest answer, taken by ahead()
  DOS_HD void ahead() {
#ifdef __CUDA_ARCH__
    drawn = atomicAdd(work, 1u);
#else
    drawn = (*work)++;
#endif
  }
  // the item of the latest number (items: none is left)
  DOS_HD unsigned item() const {
    if (drawn == items - 1u) *work = 0u;
    const unsigned n = drawn + blocks;
    return n < items ? n : items;
  }
  // gives up: n is the item of the latest number
  DOS_HD void drain(unsigned n) {
    while (n < items) {
      ahead();
      n = item();
    }
  }
};

// Row stride of the row passes' staging buffer: a warp reads the rows of two
// or more lines at once, and these strides make those 8-byte reads free of
// bank conflicts (enumerated on the host for the compiled line shapes).
constexpr int row_stage_stride(int m) {
  return m == 400 ? 404 : m == 200 ? 202 : m == 128 ? 132 : m == 64 ? 68 : m == 32 ? 34 : m == 16 ? 18 : m;
}

// HALF: the pruned line DFTs and field-half loops of Pass<LF, true> (N <= M / 2).
template <class LF, int RL, bool HALF = false>
struct PassBulk {
  static constexpr int T = LF::T, E = LF::E, M = LF::M;
  static constexpr int NZF = Pass<LF, HALF>::NZF, NOI = Pass<LF, HALF>::NOI, EF = Pass<LF, HALF>::EF;
  // packed FP32-pair butterflies in every bulk pass (faster than scalar ones
  // in each of them on the 400-point line)
  static constexpr bool PKR = true, PKC = true;
  static constexpr int RZL = Pass<LF>::RZL;
  static constexpr int SR = row_stage_stride(M);  // even: every staged row starts 16-byte aligned
  static_assert(SR % 2 == 0 && SR >= M, "staged rows must be 16-byte aligned and hold M values");
  static_assert(Pass<LF>::RZL >= LF::ZS, "exchange buffers must not overlap");
  static constexpr int RT = T * RL;

  // ------------------------------------------------------------ column pass
  // An item is a group of 8 columns of one channel: c0 .. c0 + 7, c0 = 8 gi.
  // H depends on |kx| only and the quadrant table is symmetric, H(|ky|, |kx|)
  // = H(|kx|, |ky|) (the setup forms q = k^2 - (fx^2 + fy^2), the same in
  // either order), so the 8 table rows h0 .. h0 + 7 that hold the group's
  // |kx| (h0 = c0 below M/2, M - c0 - 7 above) are fetched whole, all M/2 + 2
  // entries each (a row is a 16-byte multiple), and held as tile[|kx| -
  // h0][|ky|]: then the 16 reads of a half-warp (8 lines x 2 element owners)
  // fall on distinct bank pairs.  Items are numbered so that a group and its
  // mirror image, which read the same rows but one, run side by side (L2).
  //
  // A block holds one group, 8 lines of T threads (thread = element owner t,
  // line lc: t = tid / 8, lc = tid % 8), and four such blocks fit an SM: the
  // exchanges inside the line DFTs synchronise 8 lines and nothing else.  (Two
  // groups to a block, tied by a barrier at the top of the item, left the
  // warps of both waiting for the slower one.)  The item takes two barriers,
  // the ones inside its two line DFTs: the exchange layouts alternate
  // (Line::ALT), so every thread overwrites only what it read itself, and each
  // barrier also carries the block's verdict on the wait before it: on the
  // input rows at the first, on the H tile at the second.  A copy into a
  // buffer is issued by thread 0 after the barrier that ends its reads.
  //
  // Bound by FP32 arithmetic and shared-memory accesses (each near 60 % of its
  // rate), by instruction fetch at M = 512.  One group to a block, two barriers
  // instead of three, and a loop without the displaced layers' code (48 -> 24
  // KB, 73 -> 35 KB at M = 512): 4096 channels, M = 400, 1.56 -> 1.50 ms a
  // launch; 2048 channels, M = 512, 1.40 -> 1.19 ms (with one group to a block
  // but that code still in the loop: 1.46 ms).
  static constexpr int GW = Pass<LF>::COLL / 2;       // columns per group
  static constexpr int HW = GW;                       // |kx| values per H tile
  static constexpr int HP = M / 2 + 2;                // quadrant pitch (rows and columns)
  static_assert(GW == 8, "column groups of 8");
  // The H tile is staged in a region of its own where four blocks fit an SM
  // with it and a table row fits one box (M <= 400: 55 KB at N = 200): the
  // next item's tile is fetched after the second barrier of an item.  At M =
  // 512 the tile takes the input rows' stage slot once they are in registers
  // (SLOT_H): fetched at the first barrier, with the next input rows fetched
  // at the second.  A table row of M/2 + 2 > 256 entries is then two boxes of
  // HB entries, at x = 0 and x = HP - HB.
  static constexpr bool STAGE_H = M <= 400;
  static constexpr bool SLOT_H = !STAGE_H;
  static_assert(!STAGE_H || HP <= 256, "a staged H tile row is one box row (at most 256 entries)");
  static constexpr int HTILE = STAGE_H ? HW * HP : 0;  // float2 of the H tile in shared memory
  static constexpr int HB = (HP / 2 + 1) / 2 * 2;         // SLOT_H box width: even (16-byte box rows)
  static constexpr int HSLOT = SLOT_H ? 2 * GW * HB : 0;  // float2 of the H tile: [2 boxes][8][HB]
  static_assert(!SLOT_H || (HB <= 256 && (HP - HB) % 2 == 0 && 2 * HB >= HP),
                "two 16-byte aligned boxes cover a table row");
  // every register's |ky| range (over the T element owners) lies in one box
  static constexpr bool slot_boxes_cover() {
    for (int i = 0; i < E; ++i) {
      const int lo = i < E / 2 ? T * i : M - T * i - T + 1, hi = i < E / 2 ? T * i + T - 1 : M - T * i;
      if (!(hi < HB || lo >= HP - HB)) return false;
    }
    return true;
  }
  static_assert(!SLOT_H || slot_boxes_cover(), "each register's H values come from one box");
  // the stage (float2): whole 128-byte lines for any row count, and room for
  // the H tile under SLOT_H
  __host__ __device__ static int col_stage(int rows) {
    const int s = (rows + 1) / 2 * 2 * GW, h = (HSLOT + 15) / 16 * 16;
    return s > h ? s : h;
  }
  static constexpr int GT = GW * T;                    // threads of a block
  static constexpr bool GROUP_BARS = GT % 32 == 0;     // whole warps, all sizes but M = 200 (host checks of the layout)
  // Exchange matrices of the column lines: even pitch ZX (row entries k1,
  // k1 + 1 are one 16-byte access), stride ZLB between the lines at least
  // Q ZX and 2 mod 16.  A warp holds 8 lines x 4 consecutive element owners;
  // its 8-byte accesses (the column side of either layout) then fall on
  // distinct bank pairs in each half-warp (8 lines x 2 owners) and its
  // 16-byte ones (the row side) on distinct bank quads in each quarter-warp
  // (8 lines, one owner).
  static constexpr int ZX = LF::P + (LF::P & 1), ZSX = LF::Q * ZX;
  static constexpr int ZLB = ZSX + ((2 - ZSX % 16) + 16) % 16;
  static_assert(ZX % 2 == 0 && ZLB % 16 == 2, "16-byte aligned rows, conflict-free line stride");
  static_assert(LF::ALT, "the two line DFTs of an item alternate their exchange layouts");
  // dynamic shared memory (from a 128-byte aligned base):
  //   stage[rows][8] | H tile[8][M/2+2] | exchange[8][ZLB] | tw[TWS] | barrier[2] | next item | ey[M/2+1] (MIS)
  // (the H tile starts on a 128-byte boundary, as tensor copies need)
  static constexpr int HTILE_PAD = (HTILE + 15) / 16 * 16;
  static size_t col_smem(int n, bool mis) {
    return 128 + sizeof(float2) * ((size_t)col_stage(n) + (size_t)HTILE_PAD + (size_t)GW * ZLB + LF::TWS + 1 +
                                   (mis ? M / 2 + 1 : 0)) +
           3 * sizeof(uint64_t);
  }

  // MIS: displaced layers.  The table of the copies already holds the gap's
  // length change; the lateral shift exp(-2 pi j (fx ax + fy ay)) is separable:
  // ey[|ky|] is tabled once per block (its conjugate at negative ky, the bin
  // M/2 counting as negative) and multiplies H, and the line's ex(kx), a
  // constant of its column, multiplies the kept outputs.  Four blocks per SM
  // still fit.
  template <bool ADJ, bool MIS>
  __device__ static void col(const PassArgs& a, const CUtensorMap* smap, const CUtensorMap* hmap) {
    extern __shared__ __align__(16) unsigned char col_raw[];
    // 128-byte aligned start, by pointer arithmetic on the shared array: the
    // compiler keeps seeing shared-memory pointers (an integer round trip
    // would turn every access below into a generic one)
    float2* stage = reinterpret_cast<float2*>(col_raw + ((128u - (sh_addr(col_raw) & 127u)) & 127u));
    float2* htile = SLOT_H ? stage : stage + (size_t)col_stage(a.n);
    float2* zb = stage + (size_t)col_stage(a.n) + HTILE_PAD;
    float2* tw = tw_align(zb + (size_t)GW * ZLB);
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + LF::TWS);  // [0] input rows, [1] H tile
    int* next_item = reinterpret_cast<int*>(bar + 2);           // thread 0's, read after the first barrier
    const int lc = threadIdx.x % GW, t = threadIdx.x / GW;
    const bool leader = threadIdx.x == 0;  // issues the copies
    float2* z = zb + lc * ZLB;
    constexpr int ngroups = M / GW;
    const int items = a.nw * ngroups;
    const uint32_t sbytes = GW * 8u * (uint32_t)(a.in_r1 - a.in_r0);
    constexpr uint32_t hbytes = (uint32_t)(SLOT_H ? HSLOT : HTILE) * 8u;
    // item -> channel and first column: neighbouring items are mirror images
    auto place = [](int it, int& w, int& c0) {
      w = it / ngroups;
      const int q = it - w * ngroups;
      c0 = GW * ((q & 1) ? ngroups - 1 - (q >> 1) : q >> 1);
    };
    auto table_row = [](int c0) { return c0 < M / 2 ? c0 : M - c0 - (GW - 1); };
    if (leader) {
      bulk_bar_init(&bar[0]);
      bulk_bar_init(&bar[1]);
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(smap)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(hmap)) : "memory");
    }
    for (int i = threadIdx.x; i < LF::TWS; i += blockDim.x) tw[i] = a.tw[i];
    float2* ey = reinterpret_cast<float2*>(bar + 3);
    if constexpr (MIS) {
      for (int i = threadIdx.x; i <= M / 2; i += blockDim.x) ey[i] = shift_phase(i, a.mis.sy);
    }
    pdl_wait();
    __syncthreads();
    auto tensor_copy = [](float2* dst, const CUtensorMap* map, int x, int y, int zc, uint64_t* b) {
      asm volatile(
          "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
          "[%5];" ::"r"(sh_addr(dst)),
          "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(zc), "r"(sh_addr(b))
          : "memory");
    };
    // the input rows of item it (thread 0)
    auto fetch_s = [&](int it) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_expect(&bar[0], sbytes);
      if (a.stall == 1) return;  // injected fault: the expected bytes never arrive
      int w, c0;
      place(it, w, c0);
      tensor_copy(stage, smap, c0, a.in_r0, a.tmap_w0 + w, &bar[0]);
    };
    // the H tile of item it (thread 0)
    auto fetch_h = [&](int it) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_expect(&bar[1], hbytes);
      if (a.stall == 1) return;
      int w, c0;
      place(it, w, c0);
      tensor_copy(htile, hmap, 0, table_row(c0), a.hmap_z0 + w, &bar[1]);
      if constexpr (SLOT_H) tensor_copy(htile + GW * HB, hmap, HP - HB, table_row(c0), a.hmap_z0 + w, &bar[1]);
    };
    bool ok = true;
    int k = 0, issued_s = 0, issued_h = 0, done_s = 0, done_h = 0;  // copies per barrier (thread 0's view)
    // Items are drawn (Draws).  (Blocks that stepped through the items by
    // gridDim finished far apart: SMs differ in how far they are
    // from the memory they read, and 16 of 20 warps were resident on average.
    // 4096 x 200 launch 1.50 -> 1.34 ms, 256 x 200 103 -> 94 us, 2048 x 256
    // 1.19 -> 1.10 ms.)
    // Thread 0 draws two items ahead, so that the counter's answer is there
    // when the next copy is issued.
    Draws draws{a.work, gridDim.x, (unsigned)items, 0u};  // thread 0: the item after the current one
    if (leader) {
      fetch_s(blockIdx.x);
      if constexpr (STAGE_H) fetch_h(blockIdx.x);
      draws.ahead();
    }
    issued_s = 1;
    issued_h = STAGE_H ? 1 : 0;
    for (int it = blockIdx.x; it < items; ++k) {
      int w, c0;
      place(it, w, c0);
      const int cc = c0 + lc;  // this line's column
      const int hc = min(cc, M - cc) - table_row(c0);  // |kx|'s row of the H tile
      if (leader) *next_item = (int)draws.item();
      // this item's input rows; a thread whose wait expires goes on to the
      // barrier with what is there, where the whole block stops
      const bool got_s = bulk_wait(&bar[0], (uint32_t)(k & 1), split_verdict(a, k));
      float2 r[E];
      const float2* sg = stage + lc - (ptrdiff_t)a.in_r0 * GW;  // row y at sg[y * GW]
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int row = t + T * i;
        r[i] = (i < EF && row >= a.in_r0 && row < a.in_r1) ? sg[row * GW] : czero();
      }
      LF::template step1<false, NZF, PKC, false, ZX>(r, t, z, tw);
      ok = __syncthreads_and(got_s) != 0;  // one verdict for the whole block, past its stage reads
      if (!ok) break;
      ++done_s;
      const int next = *next_item;
      const bool more = next < items;
      if constexpr (SLOT_H) {
        if (leader) fetch_h(it);
        ++issued_h;
      } else if (more) {
        if (leader) fetch_s(next);
        ++issued_s;
      }
      if (leader && more) draws.ahead();
      LF::template step2<false, LF::Q, PKC, false, ZX>(r, t, z);
      // (injected, tests: the wait of the block's last item gives up)
      const bool got_h = (a.stall == 3 && !more) ? false : bulk_wait(&bar[1], (uint32_t)(k & 1));
      // STAGE_H: tile[hc][|ky|] (pitch HP), |ky| = k below M/2 and M - k above,
      // both affine in i at compile time.  SLOT_H: box b of the tile,
      // [hc][|ky| - b (HP - HB)] (pitch HB); box 0 holds |ky| < HB, box 1
      // |ky| >= HP - HB, and which one a register's |ky| range lies in is
      // known at compile time.
      const float2* hlo = htile + hc * (STAGE_H ? HP : HB) + t;
      const float2* hhi = htile + hc * (STAGE_H ? HP : HB) + (M - t);
#pragma unroll
      for (int i = 0; i < E; ++i) {
        float2 h;
        if constexpr (STAGE_H) {
          h = i < E / 2 ? hlo[T * i] : hhi[-T * i];
        } else {
          // |ky| in [T i, T i + T - 1] (i < E/2) or [M - T i - T + 1, M - T i]
          constexpr int B1 = GW * HB - (HP - HB);  // offset of box 1, less its first |ky|
          if (i < E / 2) h = T * i + T - 1 < HB ? hlo[T * i] : hlo[B1 + T * i];
          else h = M - T * i < HB ? hhi[-T * i] : hhi[B1 - T * i];
        }
        if constexpr (MIS) h = i < E / 2 ? cmul(h, ey[t + T * i]) : cmulc(h, ey[M - t - T * i]);
        r[i] = ADJ ? cmulc(r[i], h) : cmul(r[i], h);
      }
      LF::template step1<true, LF::P, PKC, true, ZX>(r, t, z, tw);
      ok = __syncthreads_and(got_h) != 0;  // the verdict on the tile, past its reads
      if (!ok) break;
      ++done_h;
      if (more) {
        if constexpr (SLOT_H) {
          if (leader) fetch_s(next);
          ++issued_s;
        } else {
          if (leader) fetch_h(next);
          ++issued_h;
        }
      }
      LF::template step2<true, NOI, PKC, true, ZX>(r, t, z);
      if constexpr (MIS) {
        const float2 ex = shift_phase(signed_bin(cc, M), a.mis.sx);
#pragma unroll
        for (int i = 0; i < EF; ++i) r[i] = ADJ ? cmulc(r[i], ex) : cmul(r[i], ex);
      }
      float2* dst = a.S + (size_t)w * a.n * M + cc;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int row = t + T * i;
        if (i < EF && row >= a.out_r0 && row < a.out_r1) dst[(size_t)row * M] = r[i];
      }
      it = next;
    }
    if (!ok && leader) {
      // the number drawn after the first barrier has not been looked at when the block leaves at the second
      const unsigned n = *next_item;
      draws.drain(done_s > done_h && n < draws.items ? draws.item() : n);
      // the copies in flight land (bounded waits) before the block leaves
      if (issued_s > done_s) (void)bulk_wait(&bar[0], (uint32_t)(done_s & 1));
      if (issued_h > done_h) (void)bulk_wait(&bar[1], (uint32_t)(done_h & 1));
      atomicExch(a.err, 1);
    }
  }

  // ------------------------------------------------------------- row passes
  // Block (x, y) of a forward pass holds the rows [x RL, +RL).  With up to 20
  // elements per thread (DRAW) the blocks are persistent and take channel y,
  // then whatever a counter of their row block says (Draws), as the column pass
  // does: thread 0 draws two channels ahead and publishes the next one before the
  // first barrier of the current one.  4096 x 200 launch 0.931 ->
  // 0.901 ms, 1024 x 200 236 -> 225 us, 256 x 200 70.5 -> 67.5 us.  At M = 512 that
  // was slower (2048 x 256 0.848 -> 0.866 ms): there block (x, y) takes the
  // channels of chunk y.  (The adjoint passes sum a fixed chunk of channels per
  // block, so that the gradient is reproducible; persistent blocks drawing such
  // chunks were slower: 4096 x 200 1.05 -> 1.12 ms.)
  static constexpr bool DRAW = LF::E <= 20;
  struct Draw {
    Draws draws;     // thread 0: this row block's counter, the channel after the current one
    int* next_sh;    // published next channel
    int w;           // current channel
    int nw, end;     // channels; end of the chunk (not DRAW)
    __device__ __forceinline__ Draw(const PassArgs& a, int* sh)
        : draws{a.row_work + blockIdx.x, gridDim.y, (unsigned)a.nw, 0u}, next_sh(sh) {
      nw = a.nw;
      if constexpr (DRAW) {
        w = blockIdx.y;
        if (threadIdx.x == 0) draws.ahead();
      } else {
        w = blockIdx.y * a.chunk;
        end = min(nw, w + a.chunk);
      }
    }
    // thread 0, before the first barrier of a channel
    __device__ __forceinline__ void publish() {
      if (!DRAW || threadIdx.x != 0) return;
      *next_sh = (int)draws.item();
    }
    // thread 0, when the block gives up at that barrier
    __device__ __forceinline__ void give_up() {
      if constexpr (DRAW) draws.drain((unsigned)*next_sh);
    }
    // every thread, after that barrier: the channel that follows (nw: none)
    __device__ __forceinline__ int next() {
      if constexpr (!DRAW) return w + 1 < end ? w + 1 : nw;
      const int n = *next_sh;
      if (threadIdx.x == 0 && n < nw) draws.ahead();
      return n;
    }
  };

  // dynamic shared memory: stage[RL][SR] | exchange[RL][RZL] | tw[TWS] | barrier | next channel
  static size_t row_smem() {
    return sizeof(float2) * ((size_t)RL * SR + (size_t)RL * RZL + LF::TWS + 1) + 2 * sizeof(uint64_t);
  }

  // Forward layer pass (as Pass::row_fwd), SAVE = save the checkpoint.
  template <bool SAVE>
  __device__ static void row_fwd(const PassArgs& a) {
    extern __shared__ __align__(16) float2 smem[];
    float2* stage = smem;
    float2* zb = stage + (size_t)RL * SR;
    float2* tw = tw_align(zb + (size_t)RL * RZL);
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + LF::TWS);
    const int l = threadIdx.x / T, t = threadIdx.x % T;
    float2* z = zb + l * RZL;
    const int r0 = blockIdx.x * RL;
    const int nrows = min(RL, a.n - r0);
    const bool ok = l < nrows;
    const int rr = ok ? r0 + l : r0;
    const uint32_t bytes = (uint32_t)nrows * M * 8u;
    if (threadIdx.x == 0) bulk_bar_init(bar);
    for (int i = threadIdx.x; i < LF::TWS; i += blockDim.x) tw[i] = a.tw[i];
    pdl_wait();
    __syncthreads();
    // thread 0 copies the block's rows of channel w, one bulk copy (M * 8 bytes) per row
    auto fetch = [&](int w) {
      if (threadIdx.x != 0) return;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_expect(bar, bytes);
      if (a.stall == 1) return;  // injected fault: the expected bytes never arrive
      const float2* src = a.S + ((size_t)w * a.n + r0) * M;
      for (int q = 0; q < nrows; ++q) bulk_g2s(stage + (size_t)q * SR, src + (size_t)q * M, M * 8u, bar);
    };
    Draw draw(a, reinterpret_cast<int*>(bar + 1));
    fetch(draw.w);
    // the thickness row stays in registers
    const float* hrow = a.h + (size_t)rr * a.n;
    float hv[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int x = t + T * i;
      hv[i] = (i < EF && x < a.n) ? __ldg(hrow + x) : 0.f;
    }
    bool okw = true;
    int k = 0;
    // the next channel's constants are loaded one iteration ahead
    ChanConst cnext = a.chan[draw.w];
    for (; draw.w < a.nw; ++k) {
      const int w = draw.w;
      const ChanConst cc = cnext;
      draw.publish();
      // a thread whose wait expires goes on to the barrier with what is there,
      // where the whole block stops
      const bool got = bulk_wait(bar, (uint32_t)(k & 1), split_verdict(a, k));
      float2 r[E];
#pragma unroll
      for (int i = 0; i < E; ++i) r[i] = stage[(size_t)(ok ? l : 0) * SR + t + T * i];
      LF::template step1<true, LF::P, PKR>(r, t, z, tw);
      // one verdict for the whole block; every thread is past its stage reads:
      // the next channel may land there
      okw = __syncthreads_and(got) != 0;
      if (!okw) break;
      const int wn = draw.next();
      if (wn < a.nw) {
        fetch(wn);
        cnext = a.chan[wn];
      }
      // the forward DFT below writes the exchange matrix in the other layout
      // (only what this thread reads here), and the next channel's inverse
      // DFT again: no barrier between them
      LF::template step2<true, NOI, PKR>(r, t, z);
      float2* srow = a.S + ((size_t)w * a.n + rr) * M;
      float2* ck = a.ckpt + ((size_t)w * a.n + rr) * a.n;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int x = t + T * i;
        if (i < EF && x < a.n) {
          const float2 v = r[i];
          if (SAVE && ok) ck[x] = v;
          r[i] = cmul(transmission(hv[i], cc), v);
        } else {
          r[i] = czero();
        }
      }
      LF::template fft<false, NZF, LF::Q, false, PKR, true>(r, t, z, tw);
      if (ok) {
#pragma unroll
        for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
      }
      draw.w = wn;
    }
    if (!okw && threadIdx.x == 0) {
      draw.give_up();
      (void)bulk_wait(bar, (uint32_t)(k & 1));  // a late copy lands (bounded) before the block leaves
      atomicExch(a.err, 1);
    }
  }

  // Adjoint layer pass (as Pass::row_adj) over the rows [blockIdx.x * RL, +RL)
  // of the channels of chunk blockIdx.y, FIRST = first layer, for odd N (the
  // checkpoint rows are then not 16-byte multiples and are read directly);
  // row_adj_staged otherwise.
  template <bool FIRST>
  __device__ static void row_adj(const PassArgs& a) {
    extern __shared__ __align__(16) float2 smem[];
    float2* stage = smem;
    float2* zb = stage + (size_t)RL * SR;
    float2* tw = tw_align(zb + (size_t)RL * RZL);
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + LF::TWS);
    const int l = threadIdx.x / T, t = threadIdx.x % T;
    float2* z = zb + l * RZL;
    const int r0 = blockIdx.x * RL;
    const int nrows = min(RL, a.n - r0);
    const int row = r0 + l;
    const bool ok = l < nrows;
    const int rr = ok ? row : r0;
    const int w0 = blockIdx.y * a.chunk;
    const int w1 = min(a.nw, w0 + a.chunk);
    const uint32_t bytes = (uint32_t)nrows * M * 8u;
    if (threadIdx.x == 0) bulk_bar_init(bar);
    for (int i = threadIdx.x; i < LF::TWS; i += blockDim.x) tw[i] = a.tw[i];
    pdl_wait();
    __syncthreads();
    // thread 0 copies the block's rows of channel w, one bulk copy (M * 8 bytes) per row
    auto fetch = [&](int w) {
      if (threadIdx.x != 0) return;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_expect(bar, bytes);
      if (a.stall == 1) return;  // injected fault: the expected bytes never arrive
      const float2* src = a.S + ((size_t)w * a.n + r0) * M;
      for (int q = 0; q < nrows; ++q) bulk_g2s(stage + (size_t)q * SR, src + (size_t)q * M, M * 8u, bar);
    };
    // the thickness row is re-read from L1 per channel (beside the gradient
    // sums and the checkpoint)
    const float* hrow = a.h + (size_t)rr * a.n;
    float g[E];
#pragma unroll
    for (int i = 0; i < E; ++i) g[i] = 0.f;
    bool okw = true;
    if (w0 < w1) fetch(w0);
    int k = 0;
    // the next channel's constants are loaded one iteration ahead
    ChanConst cnext = a.chan[w0 < w1 ? w0 : 0];
    for (int w = w0; w < w1; ++w, ++k) {
      const ChanConst cc = cnext;
      if (w + 1 < w1) cnext = a.chan[w + 1];
      // a thread whose wait expires goes on to the barrier with what is there,
      // where the whole block stops
      const bool got = bulk_wait(bar, (uint32_t)(k & 1), split_verdict(a, k));
      float2 r[E];
#pragma unroll
      for (int i = 0; i < E; ++i) r[i] = stage[(size_t)(ok ? l : 0) * SR + t + T * i];
      LF::template step1<true, LF::P, PKR>(r, t, z, tw);
      // one verdict for the whole block; every thread is past its stage reads:
      // the next channel may land there
      okw = __syncthreads_and(got) != 0;
      if (!okw) break;
      if (w + 1 < w1) fetch(w + 1);
      // the forward DFT below writes the exchange matrix in the other layout
      // (only what this thread reads here), and the next channel's inverse
      // DFT again: no barrier between them
      LF::template step2<true, NOI, PKR>(r, t, z);
      float2* srow = a.S + ((size_t)w * a.n + rr) * M;
      const float2* ck = a.ckpt + ((size_t)w * a.n + rr) * a.n;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int x = t + T * i;
        if (i < EF && x < a.n) {
          r[i] = adjoint_pixel(r[i], transmission(__ldg(hrow + x), cc), ck[x], cc, g[i]);
        } else {
          r[i] = czero();
        }
      }
      if constexpr (!FIRST) {
        LF::template fft<false, NZF, LF::Q, false, PKR, true>(r, t, z, tw);
        if (ok) {
#pragma unroll
          for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
        }
      } else {
        __syncthreads();  // the next channel writes the exchange matrix in the same layout
      }
    }
    if (!okw) {
      if (threadIdx.x == 0) {
        (void)bulk_wait(bar, (uint32_t)(k & 1));  // a late copy lands (bounded) before the block leaves
        atomicExch(a.err, 1);
      }
      return;
    }
    {
      if (ok) {
        float* prow = a.partial + ((size_t)blockIdx.y * a.n + row) * a.n;
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const int x = t + T * i;
          if (i < EF && x < a.n) prow[x] = g[i];
        }
      }
    }
  }

  // -------------------------------------------------------- first row pass
  // t(h) * v1 -> pad -> DFT (as Pass::row_first) with the next channel's rows
  // of the input-field table v1 (fin) staged by bulk copies.  Needs N even.
  // dynamic shared memory: stage[RL][cks] | exchange[RL][RZL] | tw[TWS] | barrier | next channel
  static size_t first_smem(int n) {
    return sizeof(float2) * ((size_t)RL * ck_stride(n) + (size_t)RL * RZL + LF::TWS + 1) + 2 * sizeof(uint64_t);
  }

  __device__ static void row_first_staged(const PassArgs& a) {
    extern __shared__ __align__(16) float2 smem[];
    const int cks = ck_stride(a.n);
    float2* stage = smem;
    float2* zb = stage + (size_t)RL * cks;
    float2* tw = tw_align(zb + (size_t)RL * RZL);
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + LF::TWS);
    const int l = threadIdx.x / T, t = threadIdx.x % T;
    float2* z = zb + l * RZL;
    const int r0 = blockIdx.x * RL;
    const int nrows = min(RL, a.n - r0);
    const int row = r0 + l;
    const bool ok = l < nrows;
    const int rr = ok ? row : r0;
    const int lr = ok ? l : 0;
    const uint32_t bytes = (uint32_t)nrows * a.n * 8u;
    if (threadIdx.x == 0) bulk_bar_init(bar);
    for (int i = threadIdx.x; i < LF::TWS; i += blockDim.x) tw[i] = a.tw[i];
    pdl_wait();
    __syncthreads();
    auto fetch = [&](int w) {
      if (threadIdx.x != 0) return;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_expect(bar, bytes);
      if (a.stall == 1) return;  // injected fault: the expected bytes never arrive
      const float2* src = a.fin + ((size_t)w * a.n + r0) * a.n;
      for (int q = 0; q < nrows; ++q) bulk_g2s(stage + (size_t)q * cks, src + (size_t)q * a.n, a.n * 8u, bar);
    };
    Draw draw(a, reinterpret_cast<int*>(bar + 1));
    fetch(draw.w);
    const float* hrow = a.h + (size_t)rr * a.n;
    float hv[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int x = t + T * i;
      hv[i] = (i < EF && x < a.n) ? __ldg(hrow + x) : 0.f;
    }
    bool okw = true;
    int k = 0;
    // the next channel's constants are loaded one iteration ahead
    ChanConst cnext = a.chan[draw.w];
    for (; draw.w < a.nw; ++k) {
      const int w = draw.w;
      const ChanConst cc = cnext;
      draw.publish();
      okw = __syncthreads_and(bulk_wait(bar, (uint32_t)(k & 1), split_verdict(a, k))) != 0;  // one verdict for the whole block
      if (!okw) break;
      const int wn = draw.next();
      if (wn < a.nw) cnext = a.chan[wn];
      float2 r[E];
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int x = t + T * i;
        r[i] = (i < EF && x < a.n) ? cmul(transmission(hv[i], cc), stage[(size_t)lr * cks + x]) : czero();
      }
      LF::template step1<false, NZF, PKR>(r, t, z, tw);
      __syncthreads();  // every thread is past its stage reads: the next channel may land there
      if (wn < a.nw) fetch(wn);
      LF::template step2<false, LF::Q, PKR>(r, t, z);  // next z write follows the loop-top barrier
      if (ok) {
        float2* srow = a.S + ((size_t)w * a.n + rr) * M;
#pragma unroll
        for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
      }
      draw.w = wn;
    }
    if (!okw && threadIdx.x == 0) {
      draw.give_up();
      (void)bulk_wait(bar, (uint32_t)(k & 1));  // a late copy lands (bounded) before the block leaves
      atomicExch(a.err, 1);
    }
  }

  // Row stride in shared memory of staged N-point rows (checkpoint, input
  // field): >= N, and congruent to SR mod 16, so that the rows of consecutive
  // lines fall in different banks the same way as in the staged spectra.
  __host__ __device__ static int ck_stride(int n) { return n + (((SR - n) % 16) + 16) % 16; }

  // ------------------------------------------- adjoint row pass, both inputs staged
  // Both inputs of a channel arrive by bulk copies: its spectra rows (into a
  // stage that is emptied into registers at the top of the iteration, so the
  // next channel's copy overlaps the whole iteration) and its checkpoint rows
  // (read after the inverse DFT; the next channel's copy is issued as soon as
  // every thread is past them, at the barrier inside the forward DFT).  With
  // few rows per block three blocks fit on an SM.  Needs N even.
  // SHARE (32 elements per thread, M = 512): the two inputs take turns in one
  // stage, which leaves room for three blocks per SM: the channel's checkpoint
  // rows are fetched at the barrier inside its inverse DFT (every thread is
  // past its spectra reads) and the next channel's spectra rows at the
  // barrier inside its forward DFT (every thread is past its checkpoint reads).
  static constexpr bool SHARE = LF::E > 20;
  // dynamic shared memory: stage[RL][SR] | ck[RL][cks] (not with SHARE) | exchange[RL][RZL] | tw[TWS] | barrier[2]
  static size_t adj_staged_smem(int n) {
    return sizeof(float2) * ((size_t)RL * SR + (SHARE ? 0 : (size_t)RL * ck_stride(n)) + (size_t)RL * RZL +
                             LF::TWS + 1) +
           2 * sizeof(uint64_t);
  }

  template <bool FIRST>
  __device__ static void row_adj_staged(const PassArgs& a) {
    extern __shared__ __align__(16) float2 smem[];
    const int cks = ck_stride(a.n);
    float2* stage = smem;
    float2* ckb = SHARE ? stage : stage + (size_t)RL * SR;
    float2* zb = SHARE ? stage + (size_t)RL * SR : ckb + (size_t)RL * cks;
    static_assert(!SHARE || SR % 2 == 0, "the checkpoint rows share the 16-byte aligned stage");
    float2* tw = tw_align(zb + (size_t)RL * RZL);
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + LF::TWS);  // [0] spectra rows, [1] checkpoint rows
    const int l = threadIdx.x / T, t = threadIdx.x % T;
    float2* z = zb + l * RZL;
    const int r0 = blockIdx.x * RL;
    const int nrows = min(RL, a.n - r0);
    const int row = r0 + l;
    const bool ok = l < nrows;
    const int rr = ok ? row : r0;
    const int lr = ok ? l : 0;
    const int w0 = blockIdx.y * a.chunk;
    const int w1 = min(a.nw, w0 + a.chunk);
    if (threadIdx.x == 0) {
      bulk_bar_init(&bar[0]);
      bulk_bar_init(&bar[1]);
    }
    for (int i = threadIdx.x; i < LF::TWS; i += blockDim.x) tw[i] = a.tw[i];
    pdl_wait();
    __syncthreads();
    // thread 0 copies the block's rows of channel w: spectra (M * 8 bytes a
    // row) into the stage, checkpoint (N * 8 bytes a row) into ck
    auto fetch_s = [&](int w) {
      if (threadIdx.x != 0) return;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_expect(&bar[0], (uint32_t)nrows * M * 8u);
      if (a.stall == 1) return;  // injected fault: the expected bytes never arrive
      const float2* src = a.S + ((size_t)w * a.n + r0) * M;
      for (int q = 0; q < nrows; ++q) bulk_g2s(stage + (size_t)q * SR, src + (size_t)q * M, M * 8u, &bar[0]);
    };
    auto fetch_c = [&](int w) {
      if (threadIdx.x != 0) return;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_expect(&bar[1], (uint32_t)nrows * a.n * 8u);
      if (a.stall == 1) return;
      const float2* src = a.ckpt + ((size_t)w * a.n + r0) * a.n;
      for (int q = 0; q < nrows; ++q) bulk_g2s(ckb + (size_t)q * cks, src + (size_t)q * a.n, a.n * 8u, &bar[1]);
    };
    // the thickness row stays in registers across the chunk's channels
    const float* hrow = a.h + (size_t)rr * a.n;
    float hv[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int x = t + T * i;
      hv[i] = (i < EF && x < a.n) ? __ldg(hrow + x) : 0.f;
    }
    float g[E];
#pragma unroll
    for (int i = 0; i < E; ++i) g[i] = 0.f;
    bool okw = true;
    int issued_s = 0, issued_c = 0, done_s = 0, done_c = 0;  // copies per barrier (thread 0's view)
    if (w0 < w1) {
      fetch_s(w0);
      issued_s = 1;
      if constexpr (!SHARE) {
        fetch_c(w0);
        issued_c = 1;
      }
    }
    for (int w = w0; w < w1; ++w) {
      // a thread whose wait expires goes on to the barrier with what is there,
      // where the whole block stops
      const bool got_s = bulk_wait(&bar[0], (uint32_t)(done_s & 1), split_verdict(a, done_s));
      float2 r[E];
#pragma unroll
      for (int i = 0; i < E; ++i) r[i] = stage[(size_t)lr * SR + t + T * i];
      LF::template step1<true, LF::P, PKR>(r, t, z, tw);
      // one verdict for the block; every thread is past its stage reads: the
      // next channel (SHARE: this channel's checkpoint) may land there
      okw = __syncthreads_and(got_s) != 0;
      if (!okw) break;
      ++done_s;
      if constexpr (SHARE) {
        fetch_c(w);
        ++issued_c;
      } else if (w + 1 < w1) {
        fetch_s(w + 1);
        ++issued_s;
      }
      // the forward DFT below writes the exchange matrix in the other layout
      // (only what this thread reads here), and the next channel's inverse
      // DFT again: no barrier between them
      LF::template step2<true, NOI, PKR>(r, t, z);
      const bool got_c = bulk_wait(&bar[1], (uint32_t)(done_c & 1));
      // the channel's constants, loaded here rather than held through the
      // inverse DFT (the registers they would take there spill)
      const ChanConst cc = a.chan[w];
      const float2* ck = ckb + (size_t)lr * cks;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int x = t + T * i;
        if (i < EF && x < a.n) {
          r[i] = adjoint_pixel(r[i], transmission(hv[i], cc), ck[x], cc, g[i]);
        } else {
          r[i] = czero();
        }
      }
      if constexpr (!FIRST) {
        LF::template step1<false, NZF, PKR, true>(r, t, z, tw);
        // the verdict on the checkpoint rows, past their reads (the gradient
        // sums of an expired wait are never written)
        okw = __syncthreads_and(got_c) != 0;
        if (!okw) break;
        ++done_c;
        if (w + 1 < w1) {
          if constexpr (SHARE) {
            fetch_s(w + 1);
            ++issued_s;
          } else {
            fetch_c(w + 1);
            ++issued_c;
          }
        }
        LF::template step2<false, LF::Q, PKR, true>(r, t, z);
        if (ok) {
          float2* srow = a.S + ((size_t)w * a.n + rr) * M;
#pragma unroll
          for (int i = 0; i < E; ++i) srow[t + T * i] = r[i];
        }
      } else {
        okw = __syncthreads_and(got_c) != 0;  // as above; also ends the exchange reads
        if (!okw) break;
        ++done_c;
        if (w + 1 < w1) {
          if constexpr (SHARE) {
            fetch_s(w + 1);
            ++issued_s;
          } else {
            fetch_c(w + 1);
            ++issued_c;
          }
        }
      }
    }
    if (!okw) {
      // copies still in flight land (bounded waits) before the block leaves
      if (threadIdx.x == 0) {
        if (issued_s > done_s) (void)bulk_wait(&bar[0], (uint32_t)(done_s & 1));
        if (issued_c > done_c) (void)bulk_wait(&bar[1], (uint32_t)(done_c & 1));
        atomicExch(a.err, 1);
      }
      return;
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
};

// the staged adjoint row pass: three blocks of few rows per SM
template <class LF, int RL, bool HALF, bool FIRST>
__global__ void __launch_bounds__(LF::T * RL, 3) k_row_adj_staged(PassArgs a) {
  PassBulk<LF, RL, HALF>::template row_adj_staged<FIRST>(a);
}
// Column pass: resident blocks of 8 lines per SM that the registers are held to.
// Four where lines have 16 owners and more (M = 400: 20 warps at up to 102
// registers, M = 512: 16 at up to 128), six at M = 256 (85 registers: step of 1024
// channels of 128 x 128 1495 us with four, 1484 with six), eight for shorter lines
// (M = 200, 1024 channels of 100 x 100: 1132 us with four, 1111 with eight; M = 128
// and 64 need no more registers than eight blocks leave: no difference).
template <class LF>
constexpr int col_bulk_min_blocks() { return LF::M == 256 ? 6 : LF::T >= 16 ? 4 : 8; }
template <class LF, int RL, bool HALF, bool ADJ, bool MIS>
__global__ void __launch_bounds__(PassBulk<LF, RL, HALF>::GT, col_bulk_min_blocks<LF>())
    k_col_bulk(PassArgs a, const __grid_constant__ CUtensorMap smap, const __grid_constant__ CUtensorMap hmap) {
  PassBulk<LF, RL, HALF>::template col<ADJ, MIS>(a, &smap, &hmap);
}
// the row passes: as many resident blocks as their shared memory allows
template <class LF, int RL>
constexpr int row_bulk_min_blocks() { return LF::E <= 20 ? (RL <= 8 ? 4 : 2) : 1; }
template <class LF, int RL, bool HALF, bool SAVE>
__global__ void __launch_bounds__(LF::T * RL, row_bulk_min_blocks<LF, RL>()) k_row_bulk(PassArgs a) {
  PassBulk<LF, RL, HALF>::template row_fwd<SAVE>(a);
}
template <class LF, int RL, bool HALF, bool FIRST>
__global__ void __launch_bounds__(LF::T * RL, row_bulk_min_blocks<LF, RL>()) k_row_adj_bulk(PassArgs a) {
  PassBulk<LF, RL, HALF>::template row_adj<FIRST>(a);
}
template <class LF, int RL, bool HALF>
__global__ void __launch_bounds__(LF::T * RL, row_bulk_min_blocks<LF, RL>()) k_row_first_staged(PassArgs a) {
  PassBulk<LF, RL, HALF>::row_first_staged(a);
}

// Channels per block of a row pass in chunks.  A launch of rb row blocks x c chunks runs
// in waves of `slots` resident blocks, each as long as one block's channels
// plus about one channel's time to start (twiddles, thickness row, the first
// copy's latency) and to finish: the split with the smallest waves x (channels
// + 1), and of equals the one with the fewest waves.  (Chunks made for about
// eight blocks per SM whatever the kernel's residency left a last wave with 20
// blocks of 456 at 4096 channels of 200 x 200, and three channels per block at
// 256.)  most: the largest chunk allowed.
inline int balanced_chunk(int nw, int rb, int slots, int most) {
  int best = std::max(1, std::min(nw, most));
  double cost = 1e30;
  for (int waves = 1; waves <= 64; ++waves) {
    const int c = std::max(1, std::min(nw, waves * slots / std::max(1, rb)));
    const int chunk = (nw + c - 1) / c, cc = (nw + chunk - 1) / chunk;
    if (chunk > most) continue;
    const double t = (double)(((long)rb * cc + slots - 1) / slots) * (chunk + 1.0);
    if (t < 0.999 * cost) cost = t, best = chunk;
    if (c == nw) break;
  }
  return best;
}
// Most channels per block, unless the plain pass's chunk is larger: the adjoint row
// pass sums its chunk's channels in FP32 registers, and long chunks spread the
// blocks that run together over the whole spectra buffer.  The sums' terms are lost
// in the fields' own rounding: 256 channels of 200 x 200, gradient error against 64
// bits 4.516e-7 with three channels to a block (the plain pass's chunk there),
// 4.529e-7 with the fifteen that balanced_chunk takes (mean of six designs); row
// launches of 88 us with the first, 83 with the second.
constexpr int kRowChunk = 48;

// Launchers.  The column pass runs one persistent block per resident slot
// (blocks per SM from the occupancy calculator x SMs), the forward row passes
// with DRAW the resident slots shared out over the row blocks; the other row
// passes run (row blocks) x (channel chunks) blocks, each looping over its chunk.
template <class LF, int RL>
struct PassBulkLaunch {
  using PB = PassBulk<LF, RL>;
  template <typename K>
  static cudaError_t slots(K kernel, int threads, size_t smem, int* out) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem)) != cudaSuccess) return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    *out = std::max(1, per_sm) * sms;
    return cudaSuccess;
  }
  // The tensor copy needs a map whose box holds the input rows (at most 256);
  // without one the plain kernel runs.
  static bool half(const PassArgs& a) { return 2 * a.n <= LF::M; }
  template <bool H>
  static cudaError_t col_h(const PassArgs& a, bool adj, size_t sm, cudaStream_t s) {
    const int items = a.nw * (LF::M / PB::GW);
    if (items == 0) return cudaSuccess;
    int n_slots = 0;
    auto kern = a.displaced ? (adj ? k_col_bulk<LF, RL, H, true, true> : k_col_bulk<LF, RL, H, false, true>)
                            : (adj ? k_col_bulk<LF, RL, H, true, false> : k_col_bulk<LF, RL, H, false, false>);
    cudaError_t e = slots(kern, PB::GT, sm, &n_slots);
    if (e != cudaSuccess) return e;
    return launch_next(kern, dim3(std::min(items, n_slots)), PB::GT, sm, s, a,
                       *static_cast<const CUtensorMap*>(a.tmap), *static_cast<const CUtensorMap*>(a.hmap));
  }
  // The tensor copies need maps whose boxes hold the input rows (at most 256)
  // and the H tile, and M a multiple of 8 (whole 8-column groups); otherwise
  // the plain kernel runs.
  static cudaError_t col(const PassArgs& a, bool adj, cudaStream_t s) {
    const size_t sm = PB::col_smem(a.n, a.displaced);
    if (!a.tmap || !a.hmap || a.tmap_rows != a.in_r1 - a.in_r0 || a.tmap_rows > 256 ||
        (a.displaced && a.mis.sq) ||  // the length change is not in the table
        LF::M % PB::GW != 0 || sm > 227 * 1024)
      return PassLaunch<LF>::col(a, adj, false, s);
    return half(a) ? col_h<true>(a, adj, sm, s) : col_h<false>(a, adj, sm, s);
  }
  // Launch of a forward row kernel: persistent blocks (DRAW), as many per row
  // block as are resident at once and at most one per channel, or one per chunk.
  template <typename K>
  static cudaError_t launch_rows(K kernel, size_t sm, const PassArgs& a, cudaStream_t s) {
    int n_slots = 0;
    cudaError_t e = slots(kernel, PB::RT, sm, &n_slots);
    if (e != cudaSuccess) return e;
    PassArgs b = a;
    const int rb = (a.n + RL - 1) / RL;
    b.chunk = balanced_chunk(a.nw, rb, n_slots, kRowChunk);
    const int per = PB::DRAW ? std::min(a.nw, std::max(1, n_slots / rb)) : (a.nw + b.chunk - 1) / b.chunk;
    return launch_next(kernel, dim3(rb, per), PB::RT, sm, s, b);
  }
  template <bool H>
  static cudaError_t row_fwd_h(const PassArgs& a, bool save, cudaStream_t s) {
    const size_t sm = PB::row_smem();
    return save ? launch_rows(k_row_bulk<LF, RL, H, true>, sm, a, s)
                : launch_rows(k_row_bulk<LF, RL, H, false>, sm, a, s);
  }
  static cudaError_t row_fwd(const PassArgs& a, bool save, cudaStream_t s) {
    return half(a) ? row_fwd_h<true>(a, save, s) : row_fwd_h<false>(a, save, s);
  }
  // the first forward row pass (t * v1 -> DFT) with staged input rows; the
  // plain kernel where N is odd or the stage does not fit
  static cudaError_t row_first(const PassArgs& a, cudaStream_t s) {
    const size_t sm = PB::first_smem(a.n);
    if (a.n % 2 != 0 || sm > 227 * 1024) return PassLaunch<LF>::row_first(a, s);
    return half(a) ? launch_rows(k_row_first_staged<LF, RL, true>, sm, a, s)
                   : launch_rows(k_row_first_staged<LF, RL, false>, sm, a, s);
  }
  // rows per block of the staged adjoint row pass
  static constexpr int RLA = RL >= 16 ? RL / 2 : RL;
  using PBA = PassBulk<LF, RLA>;
  template <bool H>
  static cudaError_t row_adj_h(const PassArgs& a, bool first, cudaStream_t s) {
    if (a.n % 2 == 0 && PBA::adj_staged_smem(a.n) <= 227 * 1024) {
      const dim3 g((a.n + RLA - 1) / RLA, a.n_chunks);
      const size_t sm = PBA::adj_staged_smem(a.n);
      return first ? launch_k(k_row_adj_staged<LF, RLA, H, true>, g, PBA::RT, sm, a, s)
                   : launch_k(k_row_adj_staged<LF, RLA, H, false>, g, PBA::RT, sm, a, s);
    }
    // odd N: the spectra rows staged, the checkpoint read directly
    const dim3 g((a.n + RL - 1) / RL, a.n_chunks);
    const size_t sm = PB::row_smem();
    return first ? launch_k(k_row_adj_bulk<LF, RL, H, true>, g, PB::RT, sm, a, s)
                 : launch_k(k_row_adj_bulk<LF, RL, H, false>, g, PB::RT, sm, a, s);
  }
  static cudaError_t row_adj(const PassArgs& a, bool first, cudaStream_t s) {
    return half(a) ? row_adj_h<true>(a, first, s) : row_adj_h<false>(a, first, s);
  }
  // channels per block of row_adj for n x n layers and nw channels, at most
  // kRowChunk or `most` where that is larger (the
  // gradient partials hold one n x n plane per chunk)
  template <bool H>
  static int adj_chunk_h(int n, int nw, int most) {
    int n_slots = 0, rows = RL;
    cudaError_t e;
    if (n % 2 == 0 && PBA::adj_staged_smem(n) <= 227 * 1024) {
      rows = RLA;
      e = slots(k_row_adj_staged<LF, RLA, H, false>, PBA::RT, PBA::adj_staged_smem(n), &n_slots);
    } else {
      e = slots(k_row_adj_bulk<LF, RL, H, false>, PB::RT, PB::row_smem(), &n_slots);
    }
    if (e != cudaSuccess) {
      (void)cudaGetLastError();
      return 0;
    }
    return balanced_chunk(nw, (n + rows - 1) / rows, n_slots, std::max(most, kRowChunk));
  }
  static int adj_chunk(int n, int nw, int most) {
    return 2 * n <= LF::M ? adj_chunk_h<true>(n, nw, most) : adj_chunk_h<false>(n, nw, most);
  }
};

// The launchers of one padded size, plain and bulk-prefetching.
template <class LF, int RL>
const PassOps* pass_ops_table() {
  using PL = PassLaunch<LF>;
  using PBL = PassBulkLaunch<LF, RL>;
  static const PassOps o = {LF::M,       LF::P,          LF::Q,          LF::T,
                            Pass<LF>::ROWL, Pass<LF>::COLL, &PL::col,    &PL::row_fwd,
                            &PL::row_out, &PL::row_seed,  &PL::row_adj,  &PL::row_in,
                            &PL::row_back, &PL::row_first, &PBL::col, &PBL::row_fwd,
                            &PBL::row_adj, &PBL::row_first, &PBL::adj_chunk, PassBulk<LF, RL>::GW,
                            PassBulk<LF, RL>::STAGE_H ? PassBulk<LF, RL>::HP : PassBulk<LF, RL>::HB,
                            PassBulk<LF, RL>::STAGE_H ? PassBulk<LF, RL>::HW : PassBulk<LF, RL>::GW};
  return &o;
}

}  // namespace dos

// One translation unit per padded size: defines dos::pass_ops_<M>() (RL_ rows
// per block in the bulk-prefetching row passes).
#define DOS_DEFINE_PASS_OPS(M_, P_, Q_, T_, RL_)                                              \
  namespace dos {                                                                             \
  const PassOps* pass_ops_##M_() { return pass_ops_table<Line<P_, Q_, T_>, RL_>(); }          \
  }
