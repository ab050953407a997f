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
// largest value with matching signs, and then lose one unit of a level, 2^-48 of
// row times column, the size of the FP64 accumulation's own bound.  Levels 7 to
// 12 are dropped: together with the 55-bit rounding of the operands about 2^-54
// of |row| |column|, below the error of the FP64 dot product (some 2^-51 here).
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
// Warps: 0 streams the eigenbasis digits (pre-swizzled 16 KB images, a ring of
// seven), 1 issues the MMAs, 2..9 load rows and write their digits (one 64-wide K
// tile of 7 x 32 rows per slot), 10..17 drain TMEM and store.  (Sharing the
// eigenbasis stream by TMA multicast in clusters of two or four changed nothing:
// 950 against 953 and 1057 us per application at 256 x 256 x 128.)
#include <cuda_fp16.h>

#include <algorithm>

#include "tc_ptx.cuh"

namespace tpcg {

namespace {
using namespace tcx;

constexpr int kDig = 7;                        // base-256 digits of a value
constexpr int kOzRows = 32;                    // data rows per tile
constexpr int kOzImg = 128 * 128;              // one eigenbasis digit: 128 columns x 64 K elements
constexpr int kOzSlot = kDig * kOzRows * 128;  // the data digits of one K tile
constexpr int kOzStages = 7;
constexpr int kOzMaxKT = 4;                    // axes of at most 256 points
constexpr int kOzConv = 8, kOzEpi = 8;         // converter and epilogue warps
constexpr int kOzThreads = (2 + kOzConv + kOzEpi) * 32;
constexpr int kOzExpBufs = 4;                  // row-exponent buffers (tiles in flight + 1)
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
  int vec_in, vec_out;  // 16-byte row loads; 32-byte runs of eight output rows
  int iters;            // tiles per CTA
  int first;            // the kernel before this one on the stream is not a pass
  int scale, singular;
  const double* lamA;
  const double* lamB;
  const double* lamC;
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

__device__ __forceinline__ void tc_ld8_issue(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tc_ld8_wait(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
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
  if (a.st && a.st->done) return;  // (uniform over the grid)
  // Programmatic dependent launch: the next pass sets up on SMs this grid has left and waits
  // (griddepcontrol.wait) before it touches this pass's output.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* sm = smem_raw + (base - raw);
  const uint32_t sW = base;                                       // ring of eigenbasis digits
  const uint32_t sX = sW + (uint32_t)(kOzStages * kOzImg);        // data digits, one slot per K tile
  uint8_t* tail = sm + kOzStages * kOzImg + a.KT * kOzSlot;
  const uint32_t bars = smem_u32(tail);
  auto wfull = [&](int s) { return bars + 8u * s; };
  auto wempty = [&](int s) { return bars + 8u * (kOzStages + s); };
  auto dfull = [&](int s) { return bars + 8u * (2 * kOzStages + s); };
  auto dempty = [&](int s) { return bars + 8u * (2 * kOzStages + kOzMaxKT + s); };
  auto eready = [&](int s) { return bars + 8u * (2 * kOzStages + 2 * kOzMaxKT + s); };
  constexpr int kT = 2 * kOzStages + 2 * kOzMaxKT + kOzExpBufs;
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
    for (int s = 0; s < kOzMaxKT; ++s) {
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
  if (warp == 1) {
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

  if (warp == 0) {
    // ---------------- eigenbasis digits: four lanes issue a quarter of an image each (one thread's issue rate
    // is below what the MMAs consume)
    constexpr uint32_t part = (uint32_t)kOzImg / 4u;
    const uint32_t off = (uint32_t)(lane & 3) * part;
    const int per_unit = a.KT * kDig;
    const int total = wres ? kDig : units * per_unit;
    const int per_tile = a.MB * per_unit;
    int it = 0, im = 0;  // im: image index within the tile's sequence [mb][kt][digit]
    bool ok = true;
    for (; it < total; ++it) {
      const int s = it % kOzStages;
      if (lane == 0) {
        ok = wait_bounded(wempty(s), (uint32_t)(((it / kOzStages) & 1) ^ 1), ab);
        if (ok) mbar_expect_tx(wfull(s), (uint32_t)kOzImg);
      }
      ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
      if (!ok) break;
      if (lane < 4) bulk_load(sW + (uint32_t)s * kOzImg + off, a.img + (size_t)im * kOzImg + off, part, wfull(s));
      if (++im == per_tile) im = 0;
      __syncwarp();
    }
    if (!ok || *abort_flag) {  // every copy this CTA expects has landed (bounded) before it may leave
      if (lane == 0)
        for (int j = (it > kOzStages ? it - kOzStages : 0); j < it; ++j) {
          const unsigned long long t0 = gtimer();
          while (!mbar_try_wait(wfull(j % kOzStages), (uint32_t)((j / kOzStages) & 1)) && gtimer() - t0 < kWaitLimitNs) {
          }
        }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer
      const unsigned long long dW = sw128_desc(sW), dX = sw128_desc(sX);
      bool ok = true;
      int it = 0;
      for (int u = 0; ok && u < units; ++u) {
        const int b = u & 1, tile = u / a.MB, mb = u - tile * a.MB;
        if (!(ok = wait_bounded(tempty(b), (uint32_t)(((u >> 1) & 1) ^ 1), ab))) break;
        tc_fence_after();
        const uint32_t dacc = tmem + (uint32_t)(b * 256);
        for (int kt = 0; ok && kt < a.KT; ++kt) {
          if (mb == 0 && !(ok = wait_bounded(dfull(kt), (uint32_t)(tile & 1), ab))) break;
          tc_fence_after();
          const int nk = min(4, (a.C - kt * 64 + 15) >> 4);
          const unsigned long long xd = dX + (uint32_t)kt * (uint32_t)(kOzSlot >> 4);
          for (int j = 0; j < kDig; ++j, ++it) {
            const int s = wres ? j : it % kOzStages;
            if (!wres || u == 0) {
              if (!(ok = wait_bounded(wfull(s), (uint32_t)((it / kOzStages) & 1), ab))) break;
              tc_fence_after();
            }
            const unsigned long long wd = dW + (uint32_t)s * (uint32_t)(kOzImg >> 4);
            const uint32_t idesc = idesc_f16kind(128, kOzRows * (kDig - j), 0u);
            const uint32_t d = dacc + (uint32_t)(j * kOzRows);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              if (kk < nk) tc_mma(d, wd + 2u * kk, xd + 2u * kk, idesc, (kt > 0 || kk > 0 || j > 0) ? 1u : 0u);
            if (!wres) tc_commit(wempty(s));
          }
          if (ok && mb == a.MB - 1) tc_commit(dempty(kt));
        }
        if (ok) tc_commit(tfull(b));
      }
      tc_commit(drain);  // every MMA this thread issued is complete once `drain` fires
      const unsigned long long t0 = gtimer();
      while (!mbar_try_wait(drain, 0) && gtimer() - t0 < kWaitLimitNs) {
      }
    }
    __syncwarp();
  } else if (warp < 2 + kOzConv) {
    // ---------------- converters: warp w takes rows 4w .. 4w+3 of a tile; a lane holds elements 64 kt + 2 lane
    // and the next one of each row
    const int w = warp - 2;
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
      const uint32_t dpar = (uint32_t)((i & 1) ^ 1);
#pragma unroll
      for (int kt = 0; kt < kOzMaxKT; ++kt) {
        if (kt >= a.KT) break;
        if (!(ok = __all_sync(0xffffffffu, wait_bounded(dempty(kt), dpar, ab)))) break;
        if (kt == 0) {  // (the buffer's previous tile, four tiles ago, has been stored: its accumulators were reused)
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
          const uint32_t dst = sX + (uint32_t)kt * kOzSlot + row * 128u + ((((uint32_t)lane >> 2) ^ (row & 7u)) << 4) +
                               ((uint32_t)lane & 3u) * 4u;
#pragma unroll
          for (int d = 0; d < kDig; ++d)
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst + (uint32_t)(d * kOzRows * 128)), "r"(digit_pair(xa, xb, d))
                         : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // digits -> async-proxy reads of the MMA
        mbar_arrive(dfull(kt));
      }
    }
  } else {
    // ---------------- epilogue: thread = output column of the block; warp half hf takes 16 of the 32 rows
    const int q = warp & 3, hf = (warp - 2 - kOzConv) >> 2;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int u = 0; u < units; ++u) {
      const int b = u & 1, tile = u / a.MB, mb = u - tile * a.MB;
      const int row0 = ((int)blockIdx.x + tile * (int)gridDim.x) * kOzRows + 16 * hf;
      const int c = mb * 128 + q * 32 + lane;
      const int sw = __ldg(a.sw + c);
      const bool okc = c < a.Cout;
      const double lc = (a.scale && okc) ? a.lamC[c] : 0.0;
      bool ok = wait_bounded(eready(tile % kOzExpBufs), (uint32_t)((tile / kOzExpBufs) & 1), ab);
      ok = ok && wait_bounded(tfull(b), (uint32_t)((u >> 1) & 1), ab);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const uint32_t tacc = tmem + (uint32_t)(b * 256 + 16 * hf) + ((uint32_t)(q * 32) << 16);
      const int* eb = sE + (tile % kOzExpBufs) * kOzRows + 16 * hf;
#pragma unroll 1
      for (int ch = 0; ch < 2; ++ch) {
        uint32_t t[kDig][8];
        __syncwarp();  // (lanes past Cout skip the stores)
#pragma unroll
        for (int s = 0; s < kDig; ++s) tc_ld8_issue(tacc + (uint32_t)(s * kOzRows + 8 * ch), t[s]);
#pragma unroll
        for (int s = 0; s < kDig; ++s) tc_ld8_wait(t[s]);
        if (ch == 1) {  // the accumulators are in registers
          tc_fence_before();
          mbar_arrive(tempty(b));
        }
        const int r0 = row0 + 8 * ch;
        if (r0 >= a.rows || !okc) continue;
        int ia = r0 / a.B, ib = r0 - ia * a.B;
        double y[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int ex = eb[8 * ch + r];
          auto lv = [&](int s) { return __float2int_rn(__uint_as_float(t[s][r])); };
          // T = sum_s acc_s 256^(6-s) = hi 2^32 + lo, kept to 2^8 (below the dropped levels)
          const long long hi = (long long)lv(0) * 65536 + (long long)lv(1) * 256 + lv(2);
          const long long lo = (long long)lv(3) * 16777216 + (long long)lv(4) * 65536 + (long long)lv(5) * 256 + lv(6);
          y[r] = ex == kOzNan ? __longlong_as_double(0x7ff8000000000000ll)
                              : scaled_i64((hi << 24) + ((lo + 128) >> 8), 56 - ex - sw);
        }
        if (a.vec_out) {  // eight rows of one a, contiguous: whole sectors
          double* py = a.Y + (long long)ia * a.oa + ib + (long long)c * a.oc;
          asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(py), "d"(y[0]), "d"(y[1]), "d"(y[2]), "d"(y[3])
                       : "memory");
          asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(py + 4), "d"(y[4]), "d"(y[5]), "d"(y[6]),
                       "d"(y[7])
                       : "memory");
          continue;
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          if (r0 + r >= a.rows) break;
          double o = y[r];
          if (a.scale) {  // Algorithm 7, Hadamard step: G = 1 / (lam_a + lam_b + lam_c), zero at the null index
            const bool null = a.singular && ia == 0 && ib == 0 && c == 0;
            o = null ? 0.0 : o * (1.0 / (a.lamA[ia] + a.lamB[ib] + lc));
          }
          const long long at = (long long)ia * a.oa + (long long)ib * a.ob + (long long)c * a.oc;
          a.Y[at] = o;
          if (FINAL) {
            red0 = fma(__ldg(a.R + at), o, red0);
            red1 += o;
          }
          if (++ib == a.B) {
            ib = 0;
            ++ia;
          }
        }
      }
    }
  }

  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
  if constexpr (FINAL) {
    double acc[2] = {red0, red1};
    SolveState* st = a.st;
    const long long N = a.N;
    grid_reduce<2>(acc, a.partials, &st->tickets[kTkPrec], gridDim.x, blockIdx.x, [st, N](const double(&s)[2]) {
      if (!st->timeout) {
        fin_precond(st, N, s);
      } else {
        st->status = TPCG_ERR_TIMEOUT;
        st->done = 1;
      }
    });
  }
}

// The digit images of an eigenbasis matrix W (l x l, row-major, contraction index first): block c' scales
// column c' by its power of two and writes its seven digits at every k, 64-wide K tiles of 128 columns under the
// 128-byte swizzle.
__global__ void __launch_bounds__(256) k_oz_image(const double* __restrict__ W, int l, int KT, uint8_t* img, int* sw) {
  const int c = blockIdx.x, k = threadIdx.x;
  __shared__ unsigned mx;
  if (k == 0) mx = 0;
  __syncthreads();
  const double v = (c < l && k < l) ? W[(long long)k * l + c] : 0.0;
  atomicMax(&mx, (unsigned)__double2hiint(v) & 0x7fffffffu);
  __syncthreads();
  const int E = max(1, (int)(mx >> 20));
  if (k == 0) sw[c] = 1077 - E;
  if (k >= KT * 64) return;
  const unsigned long long x = (unsigned long long)to_fixed55(v, E) + kBias;
  const int mb = c >> 7, r = c & 127, kt = k >> 6, kk = k & 63;
#pragma unroll
  for (int d = 0; d < kDig; ++d) {
    const uint32_t h = digit_pair(x, x, d);
    uint8_t* p = img + (((size_t)mb * KT + kt) * kDig + d) * kOzImg + r * 128 + (((kk >> 3) ^ (r & 7)) << 4) + (kk & 7) * 2;
    *reinterpret_cast<uint16_t*>(p) = (uint16_t)h;
  }
}

size_t oz_smem(int KT) {
  return 1024 + (size_t)kOzStages * kOzImg + (size_t)KT * kOzSlot + 8 * (2 * kOzStages + 2 * kOzMaxKT + kOzExpBufs + 5) +
         4 * kOzExpBufs * kOzRows + 16;
}

}  // namespace

// Axes whose products run on the digits (others: k_modeprod_f64).
bool oz_axis_ok(int l) { return l > 1 && l <= 64 * kOzMaxKT; }

// Bytes of the digit images and scales of one axis (both directions).
size_t oz_axis_bytes(int l) {
  if (!oz_axis_ok(l)) return 0;
  const size_t MB = (l + 127) / 128, KT = (l + 63) / 64;
  return 2 * (MB * KT * kDig * kOzImg + MB * 128 * sizeof(int));
}

int oz_plan_setup(tpcg_plan* p) {
  const int lens[3] = {p->nx, p->ny, p->nz};
  bool any = false;
  for (int m = 0; m < 3; ++m) {
    const int l = lens[m];
    if (!oz_axis_ok(l)) continue;
    any = true;
    const int MB = (l + 127) / 128, KT = (l + 63) / 64;
    for (int d = 0; d < 2; ++d) {
      const size_t img = (size_t)MB * KT * kDig * kOzImg, bytes = img + (size_t)MB * 128 * sizeof(int);
      if (cudaMalloc((void**)&p->d_oz[m][d], bytes) != cudaSuccess) {
        cudaGetLastError();
        p->d_oz[m][d] = nullptr;
        return TPCG_ERR_OOM;
      }
      p->device_bytes += bytes;
      k_oz_image<<<MB * 128, 256>>>(p->d_W64[m][d], l, KT, p->d_oz[m][d], reinterpret_cast<int*>(p->d_oz[m][d] + img));
    }
  }
  if (any && (cudaFuncSetAttribute(k_modeprod_oz<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)oz_smem(kOzMaxKT)) != cudaSuccess ||
              cudaFuncSetAttribute(k_modeprod_oz<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)oz_smem(kOzMaxKT)) != cudaSuccess))
    return TPCG_ERR_CUDA;
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
  a.vec_out = (!sp.scale && !sp.final_stage && sp.ob == 1 && sp.B % 8 == 0 && sp.oa % 4 == 0 && sp.oc % 4 == 0 &&
               ((uintptr_t)Y & 31) == 0)
                  ? 1
                  : 0;
  a.first = after_pass ? 0 : 1;
  a.scale = sp.scale;
  a.singular = p->singular ? 1 : 0;
  a.lamA = p->d_lam64[sp.lamA];
  a.lamB = p->d_lam64[sp.lamB];
  a.lamC = p->d_lam64[sp.lamC];
  a.R = R;
  a.st = st;
  a.partials = p->d_partials;
  a.N = p->N;
  a.err = p->d_err;
  const int ntiles = (a.rows + kOzRows - 1) / kOzRows;
  const int grid = std::min(ntiles, p->num_sms);
  a.iters = (ntiles + grid - 1) / grid;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kOzThreads);
  cfg.dynamicSmemBytes = oz_smem(a.KT);
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
