// FP64 mode products on the FP16 tensor cores (FP64 form, axes of at most 256
// points).
//
// FP64 arithmetic issues at two lanes per clock and SM here (1.26 TFLOP/s), so
// a mode product done with it is 94 % bound by that pipe however it is tiled
// (k_modeprod_f64).  This kernel computes the same product exactly on slices
// instead: the splitting of Ozaki, Ogita, Oishi and Rump ("Error-free
// transformations of matrix multiplication", Numer. Algorithms 59, 2012).
// Every row of the data and every column of the eigenbasis is scaled by its own
// power of two to a 55-bit integer and written as seven balanced base-256
// digits,
//     x = 2^-sx sum_i X_i 256^(6-i),   w = 2^-sw sum_j W_j 256^(6-j),
// |digit| <= 128, exact in FP16.  The product of two digit matrices over at
// most 256 terms is an integer below 2^22, so the tensor core's FP32 accumulation
// of it is exact, and the digit products of one level s = i + j share an
// accumulator: the four leading levels stay within 2^24 for any input; levels 4
// to 6 could pass it only if nearly every digit of a row and of a column took its
// largest value with matching signs, and each accumulation past it then loses at
// most one unit of its level (level 4: 2^-46 of row max times column max, level 5
// 2^-54).  Levels 7 to 12 are dropped: of row max times column max at worst
// l 2^-53.4, the a-priori bound of the FP64 dot product of l terms; for digits
// without a pattern some sqrt(6 l) 2^-57.6, 2^-52.3 at l = 256.  The operands'
// rounding to 55 bits is at worst l 2^-55.  All of it is relative to the largest
// entries: an entry 2^-k of its row's largest keeps 55 - k bits.
// The seven accumulators are put together in 64-bit integers and rounded to
// FP64 once.
//
// Tile: 32 rows of the data as the B operand, the 7 digits stacked along N, and
// 128 eigenbasis columns as A.  One MMA of eigenbasis digit j against the data
// digits 0 .. 6-j (N = 32 (7 - j)) adds to the levels j .. 6, which are adjacent in
// TMEM: seven MMAs per K step instead of 28, each reading its A tile once.  The
// accumulators of one tile and block take 224 TMEM columns, double-buffered.
// The whole contraction of a row sits in one tile, so a row's scale is found
// while it is loaded: FP64 in, FP64 out, nothing else in memory.
//
// Warps: 0..2 stream the eigenbasis digits (pre-swizzled 16 KB images, a ring of
// ten), 3 issues the MMAs, 4..11 load rows and write their digits (one 64-wide K
// tile of 7 x 32 rows per slot, two slots), 12..27 drain TMEM and store.
//
// Measured at 256 x 256 x 128 (GB300, one application of six passes; k_modeprod_f64: 18.1 ms): 595 us, 108 us per
// pass along a 256-point axis (120 GFLOP of digit products, 63 us at 1.9 PFLOP/s; the MMAs alone 50) and 78-82 along
// the 128-point one, against 898 with MMAs whose descriptors one thread puts together, one producer warp, a ring of
// seven images, eight epilogue warps and a division per point for G.  What is left: with the eigenbasis not
// reloaded 534, without the epilogue's arithmetic 472, without either 412.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "tc_ptx.cuh"

namespace tpcg {

namespace {
using namespace tcx;

constexpr int kDig = 7;                        // base-256 digits of a value
constexpr int kOzRows = 32;                    // data rows per tile
constexpr int kOzImg = 128 * 128;              // one eigenbasis digit: 128 columns x 64 K elements
constexpr int kOzSlot = kDig * kOzRows * 128;  // the data digits of one K tile
constexpr int kOzStages = 10;                  // eigenbasis ring: images in flight or in use
constexpr int kOzSlots = 2;                    // K tiles of data digits
constexpr int kOzProd = 3;                     // producer warps
constexpr int kOzMaxKT = 4;                    // axes of at most 256 points
constexpr int kOzConv = 8, kOzEpi = 16;        // converter and epilogue warps
constexpr int kOzConv0 = kOzProd + 1, kOzEpi0 = kOzConv0 + kOzConv;  // warps: producers, MMA, converters, epilogue
constexpr int kOzThreads = (kOzEpi0 + kOzEpi) * 32;
// Registers: 28 warps launch with 72 a thread (64,512); the producer / MMA warpgroup gives back to 40, the two
// converter warpgroups, which hold a tile's rows, take 88: 128 x 40 + 256 x 88 + 512 x 72 = 64,512.
static_assert(kOzThreads == 896 && 128 * 40 + 256 * 88 + 512 * 72 == kOzThreads * 72, "register split");
// Row-exponent buffers.  The converters write those of tile i when the MMAs of all but the last of its
// predecessors' K tiles but one are done: unit i - 2 at least has begun, so the accumulators of unit i - 4 have been
// read and the epilogue is past unit i - 5.
constexpr int kOzExpBufs = 8;
constexpr int kOzNan = 1 << 20;                // exponent word of a row holding a NaN or an infinity
constexpr unsigned long long kBias = 0x80808080808080ull;

struct OzArgs {
  const double* __restrict__ X;
  double* __restrict__ Y;
  const uint8_t* __restrict__ img;  // eigenbasis digits [MB][KT][7][128 rows][128 B], swizzled
  const int* __restrict__ sw;       // power-of-two scale of each eigenbasis column, MB * 128 entries
  int C, KT, Cout, MB;
  int rows, B, in_pitch;
  long long oa, ob, oc;
  int vec_in, vec_out;  // 16-byte row loads; 32-byte runs of four output rows
  int iters;            // tiles per CTA
  int first;            // the kernel before this one on the stream is not a pass
  int scale;
  const double* __restrict__ G;  // pass with the Hadamard step: G[row][c'], laid out as this pass's output
  const double* __restrict__ R;  // last pass of a solve
  SolveState* st;
  double* partials;
  long long N;
  int* err;
};

// A double of biased exponent field <= E as an integer multiple of 2^(E - 1077): |.| <= 2^55, rounded to
// nearest (E >= 1).
__device__ __forceinline__ long long to_fixed55(double x, int E) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((u >> 52) & 0x7ff);
  unsigned long long m = u & 0xfffffffffffffull;
  m |= (unsigned long long)(e != 0) << 52;
  const int d = min(E - max(e, 1), 60);
  m <<= 2;
  const unsigned long long q = (m + ((1ull << d) >> 1)) >> d;
  return (u >> 63) ? -(long long)q : (long long)q;
}

// Digit i (0 = leading) of two biased values as a pair of FP16 integers in [-128, 128].
__device__ __forceinline__ uint32_t digit_pair(unsigned long long a, unsigned long long b, int i) {
  uint32_t v;
  if (i == 0) {  // the leading digit may be 128: nine bits after the bias
    v = ((uint32_t)(a >> 48) & 0x1ffu) | (((uint32_t)(b >> 48) & 0x1ffu) << 16);
  } else {
    const int byte = 6 - i;
    const uint32_t wa = byte >= 4 ? (uint32_t)(a >> 32) : (uint32_t)a;
    const uint32_t wb = byte >= 4 ? (uint32_t)(b >> 32) : (uint32_t)b;
    const uint32_t s = (uint32_t)(byte & 3);
    v = __byte_perm(wa, wb, s | (s << 4) | ((4u + s) << 8)) & 0x00ff00ffu;
    // bytes: [0] = a's byte, [1] masked, [2] = b's byte
  }
  v |= 0x64006400u;  // 1024 + value, exact in FP16
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&v), __half2half2(__ushort_as_half(0x6480)));  // 1152
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Four columns of the thread's TMEM lane.
__device__ __forceinline__ void tc_ld4_issue(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
// Every load issued before has landed; names the seven destinations so that none is read earlier.
__device__ __forceinline__ void tc_ld4_wait(uint32_t (&t)[kDig][4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int s = 0; s < kDig; ++s) asm volatile("" : "+r"(t[s][0]), "+r"(t[s][1]), "+r"(t[s][2]), "+r"(t[s][3]));
}

// Contiguous global -> shared copy.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// v * 2^e rounded once to FP64 (|v| < 2^63); outside the normal range by the general scaling.
__device__ __forceinline__ double scaled_i64(long long v, int e) {
  if (e > -900 && e < 900) return i64_to_f64_scaled_hw(v, e);
  return ldexp(__ll2double_rn(v), e);
}

template <bool FINAL>
__global__ void __launch_bounds__(kOzThreads, 1) k_modeprod_oz(OzArgs a) {
  if (a.first) asm volatile("griddepcontrol.wait;" ::: "memory");  // the kernel before may set `done`
  if (a.st && paused(a.st)) return;  // (uniform over the grid)
  // Programmatic dependent launch: the next pass sets up on SMs this grid has left and waits
  // (griddepcontrol.wait) before it touches this pass's output.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* sm = smem_raw + (base - raw);
  const uint32_t sW = base;                                       // ring of eigenbasis digits
  const uint32_t sX = sW + (uint32_t)(kOzStages * kOzImg);        // ring of data digits
  uint8_t* tail = sm + kOzStages * kOzImg + kOzSlots * kOzSlot;
  const uint32_t bars = smem_u32(tail);
  auto wfull = [&](int s) { return bars + 8u * s; };
  auto wempty = [&](int s) { return bars + 8u * (kOzStages + s); };
  auto dfull = [&](int s) { return bars + 8u * (2 * kOzStages + s); };
  auto dempty = [&](int s) { return bars + 8u * (2 * kOzStages + kOzSlots + s); };
  auto eready = [&](int s) { return bars + 8u * (2 * kOzStages + 2 * kOzSlots + s); };
  constexpr int kT = 2 * kOzStages + 2 * kOzSlots + kOzExpBufs;
  auto tfull = [&](int b) { return bars + 8u * (kT + b); };
  auto tempty = [&](int b) { return bars + 8u * (kT + 2 + b); };
  const uint32_t drain = bars + 8u * (kT + 4);
  int* sE = reinterpret_cast<int*>(tail + 8 * (kT + 5));  // row exponents [kOzExpBufs][kOzRows]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(sE + kOzExpBufs * kOzRows);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  const Abort ab{abort_flag, a.err, a.st};

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kOzStages; ++s) {
      mbar_init(wfull(s), 1);
      mbar_init(wempty(s), 1);
    }
    for (int s = 0; s < kOzSlots; ++s) {
      mbar_init(dfull(s), kOzConv * 32);
      mbar_init(dempty(s), 1);
    }
    for (int s = 0; s < kOzExpBufs; ++s) mbar_init(eready(s), kOzConv);
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull(b), 1);
      mbar_init(tempty(b), kOzEpi * 32);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kOzProd) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  const int iters = a.iters;
  const int units = iters * a.MB;                  // (tile, 128-column block) accumulations of this CTA
  const bool wres = a.MB * a.KT == 1;              // the whole eigenbasis fits the ring: loaded once
  double red0 = 0.0, red1 = 0.0;

  if (warp <= kOzProd) {  // one warpgroup
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp < kOzProd) {
      // ---------------- eigenbasis digits: warp w loads images w, w + 3, ... of the sequence [tile][mb][kt][digit]
      // into ring stage (image mod 10).  A bulk copy holds its thread for about 0.3 us whatever its size, so one
      // warp alone could not keep the ring full (2.5 us per K tile, whose MMAs take 1 us).
      if (lane == 0) {
        const int per_tile = a.MB * a.KT * kDig;
        const int total = wres ? kDig : iters * per_tile;
        int it = warp, im = warp % per_tile;
        for (; it < total && !*abort_flag; it += kOzProd) {
          const int s = it % kOzStages;
          if (!wait_bounded(wempty(s), (uint32_t)(((it / kOzStages) & 1) ^ 1), ab)) break;
          mbar_expect_tx(wfull(s), (uint32_t)kOzImg);
          bulk_load(sW + (uint32_t)s * kOzImg, a.img + (size_t)im * kOzImg, (uint32_t)kOzImg, wfull(s));
          im += kOzProd;
          if (im >= per_tile) im -= per_tile;
        }
        // Every copy this warp issued has landed (bounded) before the CTA may leave, also where another warp gives up
        // after the last one was issued: of a whole sequence the last ring of images, which no later one overtakes.
        const int from = it < total ? it - kOzProd - kOzStages + 1 : total - kOzStages;
        for (int j = it - kOzProd; j >= 0 && j >= from; j -= kOzProd)
          wait_landed(wfull(j % kOzStages), (uint32_t)((j / kOzStages) & 1));
      }
      __syncwarp();
    } else {
      // ---------------- MMA issuer: the whole warp walks the loop, one elected lane issues.  The digit loop is
      // unrolled and its control flow warp-uniform: descriptors put together per MMA by one thread took 143
      // clocks each, twice what the tensor pipe needs (71 on average, max(N / 2, 32 + N / 4)).
      const bool lead = elect_one();
      const unsigned long long dW = sw128_desc(sW), dX = sw128_desc(sX);
      auto wait_all = [&](uint32_t bar, uint32_t par) { return wait_bounded_warp(bar, par, ab); };
      bool ok = true;
      uint32_t kts = 0;             // K tiles so far
      uint32_t ws = 0, wpar = 0;    // ring stage of the next image and its parity
      for (int u = 0; ok && u < units; ++u) {
        const int b = u & 1;
        if (!(ok = wait_all(tempty(b), (uint32_t)(((u >> 1) & 1) ^ 1)))) break;
        tc_fence_after();
        const uint32_t dacc = tmem + (uint32_t)(b * 256);
        for (int kt = 0; ok && kt < a.KT; ++kt, ++kts) {
          const uint32_t slot = kts % kOzSlots;
          if (!(ok = wait_all(dfull(slot), (kts / kOzSlots) & 1u))) break;
          tc_fence_after();
          const int nk = min(4, (a.C - kt * 64 + 15) >> 4);
          const unsigned long long xd = dX + slot * (uint32_t)(kOzSlot >> 4);
  #pragma unroll
          for (int j = 0; j < kDig; ++j) {
            if (wres) ws = j;
            if (!wres || u == 0) {
              ok = ok && wait_all(wfull(ws), wpar);
              tc_fence_after();
            }
            if (ok && lead) {
              const unsigned long long wd = dW + ws * (uint32_t)(kOzImg >> 4);
  #pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                if (kk < nk)
                  tc_mma(dacc + (uint32_t)(j * kOzRows), wd + 2u * kk, xd + 2u * kk,
                         idesc_f16kind(128, kOzRows * (kDig - j), 0u), (j > 0 || kk > 0) ? 1u : (kt > 0 ? 1u : 0u));
              if (!wres) tc_commit(wempty(ws));
            }
            if (!wres && ++ws == (uint32_t)kOzStages) {
              ws = 0;
              wpar ^= 1u;
            }
          }
          __syncwarp();
          if (ok && lead) tc_commit(dempty(slot));
        }
        if (ok && lead) tc_commit(tfull(b));
        __syncwarp();
      }
      if (lead) {
        tc_commit(drain);  // every MMA this thread issued is complete once `drain` fires
        const unsigned long long t0 = gtimer();
        while (!mbar_try_wait(drain, 0) && gtimer() - t0 < kWaitLimitNs) {
        }
      }
      __syncwarp();
    }
    __syncwarp();
    // The warps of a warpgroup meet between two setmaxnreg, or what each of them holds is undefined: a producer warp with
    // few images could otherwise ask for its registers back while a neighbour still held its own and a converter waited
    // for them, without end.  The MMA warp is the last here: every converter has its registers by then.
    asm volatile("bar.sync 1, 128;" ::: "memory");
    asm volatile("setmaxnreg.inc.sync.aligned.u32 72;");
  } else if (warp < kOzEpi0) {  // two warpgroups
    asm volatile("setmaxnreg.inc.sync.aligned.u32 88;");
    // ---------------- converters: warp w takes rows 4w .. 4w+3 of a tile; a lane holds elements 64 kt + 2 lane
    // and the next one of each row
    const int w = warp - kOzConv0;
    uint32_t kts = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the data are the previous pass's output
    bool ok = true;
    for (int i = 0; ok && i < iters; ++i) {
      const int row0 = ((int)blockIdx.x + i * (int)gridDim.x) * kOzRows + 4 * w;
      double2 v[4][kOzMaxKT];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const bool in = row0 + r < a.rows;
        const double* px = a.X + (long long)(in ? row0 + r : 0) * a.in_pitch;
#pragma unroll
        for (int kt = 0; kt < kOzMaxKT; ++kt) {
          const int k = 64 * kt + 2 * lane;
          v[r][kt] = make_double2(0.0, 0.0);
          if (in && a.vec_in) {
            if (k < a.C) v[r][kt] = __ldcg(reinterpret_cast<const double2*>(px + k));  // C even
          } else if (in) {
            if (k < a.C) v[r][kt].x = __ldcg(px + k);
            if (k + 1 < a.C) v[r][kt].y = __ldcg(px + k + 1);
          }
        }
      }
      int E[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        uint32_t m = 0;
#pragma unroll
        for (int kt = 0; kt < kOzMaxKT; ++kt)
          m = max(m, max((uint32_t)__double2hiint(v[r][kt].x) & 0x7fffffffu,
                         (uint32_t)__double2hiint(v[r][kt].y) & 0x7fffffffu));
        E[r] = max(1, (int)(__reduce_max_sync(0xffffffffu, m) >> 20));
      }
      // one set of K tiles per 128-column block: the digits are formed again for the second one, so that the
      // ring holds two K tiles instead of a whole row (the room goes to the eigenbasis)
#pragma unroll 1
      for (int mb = 0; ok && mb < a.MB; ++mb) {
        // (the rows stay in registers and are not taken for loop constants: the compiler would otherwise form
        // every digit before the loop and spill them)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int kt = 0; kt < kOzMaxKT; ++kt) asm volatile("" : "+d"(v[r][kt].x), "+d"(v[r][kt].y));
#pragma unroll
        for (int kt = 0; kt < kOzMaxKT; ++kt) {
          if (kt >= a.KT) break;
          const uint32_t slot = kts % kOzSlots;
          if (!(ok = __all_sync(0xffffffffu, wait_bounded(dempty(slot), ((kts / kOzSlots) & 1u) ^ 1u, ab)))) break;
          ++kts;
          if (kt == 0 && mb == 0) {  // (the buffer's previous tile has been stored: see kOzExpBufs)
            if (lane < 4) {
              const int e = lane == 0 ? E[0] : (lane == 1 ? E[1] : (lane == 2 ? E[2] : E[3]));
              sE[(i % kOzExpBufs) * kOzRows + 4 * w + lane] = e == 0x7ff ? kOzNan : 1077 - e;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(eready(i % kOzExpBufs));
          }
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const double2 x = v[r][kt];
            const unsigned long long xa = (unsigned long long)to_fixed55(x.x, E[r]) + kBias;
            const unsigned long long xb = (unsigned long long)to_fixed55(x.y, E[r]) + kBias;
            const uint32_t row = (uint32_t)(4 * w + r);
            const uint32_t dst = sX + slot * kOzSlot + row * 128u + ((((uint32_t)lane >> 2) ^ (row & 7u)) << 4) +
                                 ((uint32_t)lane & 3u) * 4u;
#pragma unroll
            for (int d = 0; d < kDig; ++d)
              asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst + (uint32_t)(d * kOzRows * 128)), "r"(digit_pair(xa, xb, d))
                           : "memory");
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // digits -> async-proxy reads of the MMA
          mbar_arrive(dfull(slot));
        }
      }
    }
    __syncwarp();
    asm volatile("bar.sync %0, 128;" ::"r"(2 + ((warp - kOzConv0) >> 2)) : "memory");
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
  } else {
    // ---------------- epilogue: thread = output column of the block; the four warps of a TMEM lane quadrant take
    // eight of the 32 rows each
    const int q = warp & 3, hf = (warp - kOzEpi0) >> 2;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int u = 0; u < units; ++u) {
      const int b = u & 1, tile = u / a.MB, mb = u - tile * a.MB;
      const int row0 = ((int)blockIdx.x + tile * (int)gridDim.x) * kOzRows + 8 * hf;
      const int c = mb * 128 + q * 32 + lane;
      const int sw = __ldg(a.sw + c);
      const bool okc = c < a.Cout;
      bool ok = wait_bounded(eready(tile % kOzExpBufs), (uint32_t)((tile / kOzExpBufs) & 1), ab);
      ok = ok && wait_bounded(tfull(b), (uint32_t)((u >> 1) & 1), ab);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const uint32_t tacc = tmem + (uint32_t)(b * 256 + 8 * hf) + ((uint32_t)(q * 32) << 16);
      const int* eb = sE + (tile % kOzExpBufs) * kOzRows + 8 * hf;
      auto issue = [&](int ch, uint32_t(&t)[kDig][4]) {
        __syncwarp();  // (lanes past Cout skip the stores)
#pragma unroll
        for (int s = 0; s < kDig; ++s) tc_ld4_issue(tacc + (uint32_t)(s * kOzRows + 4 * ch), t[s]);
      };
      // rows r0 .. r0+3 of the block's column c
      auto process = [&](int ch, const uint32_t(&t)[kDig][4]) {
        const int r0 = row0 + 4 * ch;
        if (r0 >= a.rows || !okc) return;
        const int ia = r0 / a.B, ib = r0 - ia * a.B;
        long long at[4];
        double f[4];
        {
          int xa = ia, xb = ib;
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            at[r] = (long long)xa * a.oa + (long long)xb * a.ob + (long long)c * a.oc;
            if (++xb == a.B) {
              xb = 0;
              ++xa;
            }
            f[r] = 0.0;
            if (r0 + r < a.rows) {
              if (a.scale) f[r] = __ldg(a.G + at[r]);
              else if (FINAL) f[r] = __ldg(a.R + at[r]);
            }
          }
        }
        double y[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int ex = eb[4 * ch + r];
          auto lv = [&](int s) { return __float2int_rn(__uint_as_float(t[s][r])); };
          // T = sum_s acc_s 256^(6-s) = hi 2^32 + lo, kept to 2^8 (below the dropped levels)
          const long long hi = (long long)lv(0) * 65536 + (long long)lv(1) * 256 + lv(2);
          const long long lo = (long long)lv(3) * 16777216 + (long long)lv(4) * 65536 + (long long)lv(5) * 256 + lv(6);
          y[r] = ex == kOzNan ? __longlong_as_double(0x7ff8000000000000ll)
                              : scaled_i64((hi << 24) + ((lo + 128) >> 8), 56 - ex - sw);
        }
        if (a.vec_out) {  // four rows of one a, contiguous: a whole sector
          asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(a.Y + at[0]), "d"(y[0]), "d"(y[1]), "d"(y[2]),
                       "d"(y[3])
                       : "memory");
          return;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          if (r0 + r >= a.rows) break;
          double o = y[r];
          if (a.scale) o *= f[r];  // Algorithm 7, Hadamard step
          a.Y[at[r]] = o;
          if (FINAL) {
            red0 = fma(f[r], o, red0);
            red1 += o;
          }
        }
      };
      uint32_t t[kDig][4];
#pragma unroll
      for (int ch = 0; ch < 2; ++ch) {
        issue(ch, t);
        tc_ld4_wait(t);
        if (ch == 1) {  // the accumulators are in registers
          tc_fence_before();
          mbar_arrive(tempty(b));
        }
        process(ch, t);
        __syncwarp();
      }
    }
  }

  __syncthreads();
  if (warp == kOzProd) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
  if constexpr (FINAL) {
    double acc[2] = {red0, red1};
    SolveState* st = a.st;
    const long long N = a.N;
    // (the shared memory of the tiles is free: every copy and MMA has completed)
    grid_reduce_state<2>(acc, a.partials, st, kTkPrec, gridDim.x, blockIdx.x, reinterpret_cast<unsigned*>(sm),
                         [N](SolveState* st, const double(&s)[2]) {
      if (!st->timeout) {
        fin_precond(st, N, s);
      } else {
        st->status = TPCG_ERR_TIMEOUT;
        st->done = 1;
      }
    });
  }
}

// Bytes of one direction's digit images of an axis and its column scales, which follow them.
size_t oz_digits(int l) { return (size_t)((l + 127) / 128) * ((l + 63) / 64) * kDig * kOzImg; }
size_t oz_image_bytes(int l) { return oz_digits(l) + (size_t)((l + 127) / 128) * 128 * sizeof(int); }

// The digit images of an eigenbasis matrix W (l x l, row-major, contraction index first) and the power-of-two
// scale of each column: column c' as seven base-256 digits at every k, 64-wide K tiles of 128 columns under the
// 128-byte swizzle; zero past l.
void digit_image(const std::vector<double>& W, int l, int KT, std::vector<uint8_t>& out) {
  const size_t img = oz_digits(l);
  out.assign(oz_image_bytes(l), 0);
  uint16_t f16[257];  // FP16 of -128 .. 128
  for (int d = -128; d <= 128; ++d) {
    const int v = d < 0 ? -d : d;
    int e = 0;
    while ((v >> e) > 1) ++e;
    f16[d + 128] = v ? (uint16_t)((d < 0 ? 0x8000 : 0) | ((15 + e) << 10) | ((v << (10 - e)) & 0x3ff)) : (uint16_t)0;
  }
  int* sw = reinterpret_cast<int*>(out.data() + img);
  for (int c = 0; c < l; ++c) {
    double mx = 0.0;
    for (int k = 0; k < l; ++k) mx = std::max(mx, std::fabs(W[(size_t)k * l + c]));
    int e = 0;
    std::frexp(mx, &e);  // mx < 2^e
    sw[c] = 55 - e;
    uint8_t* col = out.data() + (size_t)(c >> 7) * KT * kDig * kOzImg + (size_t)(c & 127) * 128;
    for (int k = 0; k < l; ++k) {
      long long x = std::llrint(std::ldexp(W[(size_t)k * l + c], 55 - e));  // |x| <= 2^55
      uint8_t* p = col + (size_t)(k >> 6) * kDig * kOzImg + ((((k & 63) >> 3) ^ (c & 7)) << 4) + (k & 7) * 2;
      for (int d = kDig - 1; d >= 0; --d) {
        const int v = d ? (int)(int8_t)(x & 0xff) : (int)x;
        std::memcpy(p + (size_t)d * kOzImg, &f16[v + 128], 2);
        x = (x - v) >> 8;  // exact
      }
    }
  }
}

// The Hadamard pseudoinverse G = 1 / (lam_a + lam_b + lam_c), zero at the null index, laid out as the output of the
// pass that applies it.  An FP64 division per point costs that pass 120 us at 256 x 256 x 128 (FP64 pipe 72 % used);
// reading 8 bytes per point costs 10.
__global__ void __launch_bounds__(256) k_oz_ghat(double* __restrict__ G, int A, int B, int C, long long oa, long long ob,
                                                 long long oc, const double* la, const double* lb, const double* lc,
                                                 int singular) {
  const long long n = (long long)A * B * C;
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) {
    const long long r = i / C;
    const int c = (int)(i - r * C), ia = (int)(r / B), ib = (int)(r - (long long)ia * B);
    const bool null = singular && ia == 0 && ib == 0 && c == 0;
    G[ia * oa + ib * ob + c * oc] = null ? 0.0 : 1.0 / (la[ia] + lb[ib] + lc[c]);
  }
}

constexpr size_t kOzSmem = 1024 + (size_t)kOzStages * kOzImg + (size_t)kOzSlots * kOzSlot +
                           8 * (2 * kOzStages + 2 * kOzSlots + kOzExpBufs + 5) + 4 * kOzExpBufs * kOzRows + 16;
static_assert(kOzSmem <= (size_t)kMaxSmem && kOzSmem == sole_smem(kOzSmem), "shared memory of k_modeprod_oz");

}  // namespace

// Axes whose products run on the digits (others: k_modeprod_f64).
bool oz_axis_ok(int l) { return l > 1 && l <= 64 * kOzMaxKT; }

// What oz_plan_setup allocates: the images of both directions of an axis, and G where the pass that applies it runs here.
size_t oz_device_bytes(int nx, int ny, int nz) {
  size_t b = 0;
  for (int l : {nx, ny, nz})
    if (oz_axis_ok(l)) b += 2 * oz_image_bytes(l);
  return b + (oz_axis_ok(nz > 1 ? nz : ny) ? (size_t)nx * ny * nz * sizeof(double) : 0);
}

int oz_plan_setup(tpcg_plan* p) {
  const int lens[3] = {p->nx, p->ny, p->nz};
  bool any = false;
  for (int m = 0; m < 3; ++m) {
    const int l = lens[m];
    if (!oz_axis_ok(l)) continue;
    any = true;
    const int KT = (l + 63) / 64;
    std::vector<double> VT((size_t)l * l);
    for (int i = 0; i < l; ++i)
      for (int j = 0; j < l; ++j) VT[(size_t)j * l + i] = p->ax[m].V[(size_t)i * l + j];
    std::vector<uint8_t> img;
    for (int d = 0; d < 2; ++d) {
      digit_image(d ? VT : p->ax[m].V, l, KT, img);
      if (cudaMalloc((void**)&p->d_oz[m][d], img.size()) != cudaSuccess) {
        cudaGetLastError();
        p->d_oz[m][d] = nullptr;
        return TPCG_ERR_OOM;
      }
      p->device_bytes += img.size();
      if (cudaMemcpy(p->d_oz[m][d], img.data(), img.size(), cudaMemcpyHostToDevice) != cudaSuccess) return TPCG_ERR_CUDA;
    }
  }
  if (any && (cudaFuncSetAttribute(k_modeprod_oz<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kOzSmem) != cudaSuccess ||
              cudaFuncSetAttribute(k_modeprod_oz<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kOzSmem) != cudaSuccess))
    return TPCG_ERR_CUDA;
  for (const StageParams& sp : p->stages) {
    if (!sp.scale || !p->d_oz[sp.axis][sp.dir]) continue;
    if (cudaMalloc((void**)&p->d_G, (size_t)p->N * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      p->d_G = nullptr;
      return TPCG_ERR_OOM;
    }
    p->device_bytes += (size_t)p->N * sizeof(double);
    k_oz_ghat<<<(int)std::min<long long>((p->N + 255) / 256, p->num_sms * 8), 256>>>(
        p->d_G, sp.A, sp.B, sp.Cout, sp.oa, sp.ob, sp.oc, p->d_lam64[sp.lamA], p->d_lam64[sp.lamB],
        p->d_lam64[sp.lamC], p->singular ? 1 : 0);
  }
  return cudaGetLastError() == cudaSuccess ? TPCG_OK : TPCG_ERR_CUDA;
}

// One mode-product pass; false when its axis has no digit images.  `after_pass`: the previous kernel on the stream
// is another of these passes.  Every other kernel may be the one that sets the state's `done` word, so the pass
// behind it waits for it before it looks.
bool run_pass_oz(const tpcg_plan* p, const StageParams& sp, const double* X, double* Y, const double* R, SolveState* st,
                 bool after_pass) {
  const uint8_t* img = p->d_oz[sp.axis][sp.dir];
  if (!img) return false;
  OzArgs a{};
  a.X = X;
  a.Y = Y;
  a.img = img;
  a.C = sp.C;
  a.KT = (sp.C + 63) / 64;
  a.Cout = sp.Cout;
  a.MB = (sp.Cout + 127) / 128;
  a.sw = reinterpret_cast<const int*>(img + (size_t)a.MB * a.KT * kDig * kOzImg);
  a.rows = sp.A * sp.B;
  a.B = sp.B;
  a.in_pitch = sp.in_pitch;
  a.oa = sp.oa;
  a.ob = sp.ob;
  a.oc = sp.oc;
  a.vec_in = (sp.C % 2 == 0 && sp.in_pitch % 2 == 0 && ((uintptr_t)X & 15) == 0) ? 1 : 0;
  a.vec_out = (!sp.scale && !sp.final_stage && sp.ob == 1 && sp.B % 4 == 0 && sp.oa % 4 == 0 && sp.oc % 4 == 0 &&
               ((uintptr_t)Y & 31) == 0)
                  ? 1
                  : 0;
  a.first = after_pass ? 0 : 1;
  a.scale = sp.scale;
  a.G = p->d_G;
  a.R = R;
  a.st = st;
  a.partials = p->d_partials;
  a.N = p->N;
  a.err = p->h_err;
  const int ntiles = (a.rows + kOzRows - 1) / kOzRows;
  const int grid = std::min(ntiles, p->num_sms);
  a.iters = (ntiles + grid - 1) / grid;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kOzThreads);
  cfg.dynamicSmemBytes = kOzSmem;
  cfg.stream = p->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  LaunchScope ls(p, kKModeF64);
  if (sp.final_stage && st) cudaLaunchKernelEx(&cfg, k_modeprod_oz<true>, a);
  else cudaLaunchKernelEx(&cfg, k_modeprod_oz<false>, a);
  return true;
}

}  // namespace tpcg
