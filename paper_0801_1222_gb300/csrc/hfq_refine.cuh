// Recompute of the FP32 delayed path by one or two Newton steps from the
// current G, with the residual formed exactly enough on the tensor cores.
//
// The Hirsch-Fye Dyson equation G = [1 + (1 - M)(e^V - 1)]^{-1} M, with
// D = diag(e^{sigma lambda s} - 1), reads G^{-1} = B = M^{-1}(1 + D) - D =
// A (1 + D), A = M^{-1} - diag(1 - e^{-sigma lambda s_j}).  For an FP32 G
// that has drifted by rounding since the last recompute, Newton's iteration
// for the inverse
//     E = 1 - B G',      G_new = G' + G' E,      1 - B G_new = E^2,
// brings G back to the inverse of B for the current field in one step when
// |E| is small (the drift of N_wrap = 64 flips gives |E| ~ 1e-4).  Written
// with H' = (1 + D) G' (rows of G' scaled):
//     E = 1 - A H',      G_new = (1 + D)^{-1} (H' + H' E).
//
// E needs FP64-level accuracy where G' nearly inverts B, which FP32 products
// cannot give; the residual product A H' is therefore formed from integer
// slices (the splitting idea of Ozaki, Ogita, Oishi and Rump, written here
// for FP16 tensor-core operands):
//   * A = 2^ea sum_p a_p 2^{-7(p+1)}, 6 signed 7-bit slices;
//   * H' = the FP32 H = fl32((1 + d_j) G_jn) rounded to the grid 2^{eh-28}
//     (eh: |H| < 2^eh) = 2^eh sum_q h_q 2^{-7(q+1)}, 4 slices.  G' =
//     (1 + D)^{-1} H' differs from G by at most half that grid step; E and
//     the update both use this same G', so Newton's identity holds for it;
//   * a_p, h_q are integers with |.| <= 128 (first slice) or <= 64, exact in
//     FP16.  The products with p + q = l go to one FP32 TMEM accumulator per
//     level l = 0..5 (at most four pairs, each K term <= 6 * 2^12 in all, so
//     every partial sum is an integer below 2^24 for Lambda <= 512: the
//     accumulation is exact, in any order).  Dropped levels and the slices'
//     remainders leave |E - E_exact| ~ 1e-10 of |A||H'|.
//   * The six level sums combine as V = sum_l S_l 2^{7 (5 - l)}, so A H' =
//     V 2^{ea + eh - 49}, and E = delta - V 2^{ea+eh-49} is exact before it is
//     rounded to FP32: the cancellation costs nothing.  Near the inverse the
//     leading levels cancel, so Horner's rule in FP32 is exact while its
//     partial sums stay below 2^24 (checked); else 64-bit integers are used.
//
// The residual product on the tensor cores, E^T = 1 - H'^T A^T tile by tile
// (128 columns n of H' = TMEM lanes, 64 rows i of A):
//   * M^{-1} is a function of i - j only (skew-circulant), so an 8 x 8 core
//     matrix of A depends on the difference of its block row and block column
//     alone: a slice needs one core matrix per block diagonal (2 L / 8, not
//     L^2 / 64 of them), and the whole sliced A (45 KiB at Lambda = 240, 96
//     at 512) stays in shared memory for the refinement.  With the
//     contraction run through the blocks J in descending order the core of
//     (I, J' = NJ - 1 - J) lies at (I + J') * 128 bytes: both descriptor
//     strides are 128 bytes and neighbouring tiles overlap.  The earlier form
//     streamed A's 48 KiB per 32 columns of the contraction from L2.
//   * A_jj depends on the field.  The table carries the value for
//     sigma s_j = +1; rows with sigma s_i = -1 get (A_ii difference) x H'_in
//     added to V in the read-out, from the same slices of H'_in with the same
//     products p + q <= 5 dropped, so V is the one of the sliced product.
//   * H'^T is the other operand, cut from G by 14 warps straight into TMEM
//     (the A operand of tcgen05.mma may live there): the tensor cores then
//     read only A's slices, 2 KiB per MMA, from shared memory, and a 128 x 64
//     x 16 MMA runs at its 32 cycles (measured alone: 32.1; with both operands
//     in shared memory 48).  Four TMEM buffers of one K step of 16 each; the
//     cutting warps and the two issuing warps meet on mbarriers, there is no CTA
//     barrier in the loop.
// The update H' E only needs FP32 accuracy (|E| is small): split FP16
// hi/lo parts with power-of-two scales, three products, FP32 accumulation,
// formed transposed as well (E^T H'^T) so that a warp's lanes are consecutive
// columns of G in both read-outs and every access to G and E is coalesced.
//
// SM cycles per refinement of one spin at Lambda = 240 (phase timers in a copy
// of the kernel), with A's slices streamed from L2 and H' cut into shared
// memory, and as it is here: residual product 180k -> 122k (its MMAs alone
// take 69k; what is above is the hand-over between the cutting and the issuing
// warps), its read-outs 50k -> 35k, update product 46k -> 32k, its read-out
// 31k -> 21k, scale pass 16k -> 10k; at Lambda = 500 in all 2.83M -> 1.81M.
// Measured and not kept for Lambda > 256: H' and E^T written once as FP16
// parts and staged by bulk copies (the chains' working set is beyond L2 there:
// 673k cycles for the update product instead of 495k).
//
// max |E| over the matrix decides: above rc.emax_step (2^-8 by default) the
// step is not taken and the caller recomputes G from scratch (Gauss-Jordan);
// above 2^-13 a second step follows.  The drift reported is the largest
// change of an entry over the steps.
#pragma once
#include <cuda_fp16.h>

#include <type_traits>

#include "hfq_delayed.cuh"
#include "hfq_device.cuh"

namespace hfq {

static_assert(kDelNT == 512, "the refinement's TMEM read-out assumes 16 warps");

// TMEM columns of the residual product: kRfLevels accumulators of kRfN
// columns, then kRfBufs buffers of H' slices (one K step of 16 each:
// kRfSlicesH x 8 columns, two FP16 values of the contraction index per column)
constexpr int kRfBufs = 4;
constexpr int kRfBufCol = kRfLevels * kRfN;
constexpr int kRfBufCols = kRfSlicesH * 8;
static_assert(kRfBufCol + kRfBufs * kRfBufCols <= kTmemCols, "accumulators and H' buffers must fit the TMEM allocation");
// Warps 14 and 15 issue the MMAs (one elected lane each), the others cut H'.
// Two, on two schedulers, because each shares its scheduler with three cutting
// warps: one alone took 50 cycles an MMA, which runs in 32.  The residual
// product's levels are dealt out as 5, 4, 0 and 3, 2, 1 (nine products a K step
// each), so that every accumulator belongs to one of them.
constexpr int kRfIssueWarp = 15, kRfIssuers = 2;
__host__ __device__ constexpr int rf_issuer_of(int level) { return level == 0 || level >= 4 ? 0 : 1; }
constexpr int kRfAhead = 2;       // K steps of the next tile cut before a tile's read-out

// K-major core-matrix layout of the update product's chunks (8 rows x 16
// bytes per core matrix, contiguous along K)
__device__ __forceinline__ uint32_t rf_off2(int r, int k8) {
  return (uint32_t)((r >> 3) * (kRf2KC / 8) * 128 + k8 * 128 + (r & 7) * 16);
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// bulk copy global -> this CTA's shared memory, completion counted on mbar
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   dst),
               "l"(src), "r"(bytes), "r"(mbar)
               : "memory");
}

// 2^k as an FP32 number, -126 <= k <= 127 (scalings by it are exact while
// the result stays normal)
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((127 + k) << 23); }

// 32 lanes x 32 bit, 8 consecutive columns per thread; the values may be
// used after tmem_wait_ld
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld4(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3])::"memory");
}
// the registers pass through the asm, so no use of them moves above the wait
__device__ __forceinline__ void tmem_wait_ld8(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])::"memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(a), "r"(b), "r"(c),
               "r"(d)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// One lane of the (converged) warp, as a predicate for the issuing lane: the
// branch around the MMAs stays warp-uniform, so their descriptors live in
// uniform registers (an issue from a divergent branch costs about 50 cycles).
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r));
  return r;
}
// A warp-uniform value as one the compiler knows to be uniform (a warp
// reduction's result is a uniform register; a shuffle's is not)
__device__ __forceinline__ uint32_t rf_uniform(uint32_t x) { return __reduce_or_sync(0xffffffffu, x); }
// kind::f16 MMA issued by the elected lane (el != 0), A operand in TMEM; the same lane's commit
__device__ __forceinline__ void tc_mma_f16_ts(uint32_t el, uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                              uint32_t idesc, int accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      :
      : "r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(el));
}
__device__ __forceinline__ void tc_commit_el(uint32_t el, uint32_t mbar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "setp.ne.b32 e, %1, 0;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(mbar), "r"(el)
      : "memory");
}
// kind::f16 MMA issued by the elected lane, both operands in shared memory
__device__ __forceinline__ void tc_mma_f16_el(uint32_t el, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                              uint32_t idesc, int accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      :
      : "r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(el));
}

// Block-wide max of non-negative floats, NaN counted as infinity; every
// thread gets the result.  red: kDelNT / 32 floats.  Contains barriers.
__device__ __forceinline__ float rf_block_max(float v, float* red) {
  v = (v == v) ? v : __int_as_float(0x7f800000);
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = 0.f;
#pragma unroll
  for (int w = 0; w < kDelNT / 32; ++w) r = fmaxf(r, red[w]);
  __syncthreads();
  return r;
}

// Eight values y (|y| < 2^7) -> four slices of 7 bits: slice q holds the
// nearest integers (ties to even, as rintf) of the running remainders, which
// then move up 7 bits; w[q]: slice q's eight FP16 values, packed.
// Full-rate FP32 and FP16x2 arithmetic only: adding kC = 1.5 * 2^23 + 0x6600
// rounds to an integer (the FP32 spacing there is 1, and kC is even, so ties
// fall as they would without it) and leaves 0x6600 + v in the low 16 bits,
// the FP16 number 1536 + v (spacing 1 in [1024, 2048)), of which 1536 is
// subtracted exactly.  The remainder times 2^7 is two FMAs, exact as well.
__device__ __forceinline__ void rf_cut8(float* y, uint32_t (*w)[4]) {
  constexpr float kC = 12582912.f + 26112.f;
#pragma unroll
  for (int q = 0; q < kRfSlicesH; ++q) {
#pragma unroll
    for (int t = 0; t < 8; t += 2) {
      const float ta = y[t] + kC, tb = y[t + 1] + kC;
      const uint32_t pk = __byte_perm(__float_as_uint(ta), __float_as_uint(tb), 0x5410);
      const uint32_t c1536 = 0x66006600u;
      __half2 hv, hc;
      memcpy(&hv, &pk, 4);
      memcpy(&hc, &c1536, 4);
      hv = __hsub2(hv, hc);
      memcpy(&w[q][t / 2], &hv, 4);
      if (q + 1 < kRfSlicesH) {
        y[t] = __fmaf_rn(y[t], 128.f, __fmaf_rn(ta, -128.f, 128.f * kC));
        y[t + 1] = __fmaf_rn(y[t + 1], 128.f, __fmaf_rn(tb, -128.f, 128.f * kC));
      }
    }
  }
}

// One element of E = delta - V 2^{-sh} from its six level sums in 64-bit
// integers, for |E| beyond the read-out's FP32 evaluation (see there).
// taddr: the element's level-0 TMEM column; neg: its row has sigma s = -1, y
// then being H'_in 2^{7-eh} and dd the diagonal's slice differences.
__device__ __noinline__ float rf_residual_wide(uint32_t taddr, bool neg, float y, const float* dd, bool diag, int sh) {
  float d[kRfSlicesH];
  for (int q = 0; q < kRfSlicesH; ++q) {
    d[q] = neg ? rintf(y) : 0.f;
    y = (y - d[q]) * (float)(1 << kRfBits);
  }
  long long V = 0;
  for (int lv = 0; lv < kRfLevels; ++lv) {
    uint32_t u;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(u) : "r"(taddr + (uint32_t)(lv * kRfN)));
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(u)::"memory");
    V = V * (1ll << kRfBits) + (long long)__float2int_rn(__uint_as_float(u));
    for (int q = 0; q < kRfSlicesH && q <= lv; ++q) V += (long long)__float2int_rn(dd[lv - q] * d[q]);
  }
  const long long Ei = (diag ? 1ll << sh : 0ll) - V;
  if (Ei > (1ll << 54) || Ei < -(1ll << 54)) return __int_as_float(0x7f800000);  // far beyond the step's range
  const float hi = (float)(int)(Ei >> 24), lo = (float)(int)(Ei & 0xffffffll);
  return fmaf(hi, 16777216.f, lo) * pow2f(-sh);
}

// What one refinement works with, at the start of its shared memory.  Each
// phase takes its own copies of what it needs, so that little is live from
// one phase to the next: with everything live throughout, the compiler spills
// some hundred bytes per thread, which at 512 threads go to L2.
struct RfPar {
  float* G;
  float* wsE;
  const RefineConst* rc;
  const int8_t* s;
  int* status;
  int L, ld, sig;
  uint32_t tmem, cbar;
  RfSync sync;
};
constexpr uint32_t kRfParBytes = 128;
static_assert(sizeof(RfPar) <= kRfParBytes, "the parameters' slot in the refinement's shared memory");
static_assert(kRfParBytes == kRfHead, "rf_smem_need counts the slot");

__host__ __device__ constexpr int rf_lde(int L) { return rf_pad(L, 8); }

// Bounded waits of one thread: after one has given up it waits no more
struct RfWait {
  bool bad = false;
  __device__ __forceinline__ void on(uint32_t bar, uint32_t parity) {
    if (!bad && !mbar_wait_bounded(bar, parity)) bad = true;
  }
};

// The same for a whole (converged) warp, every branch on a vote: control flow
// that the compiler knows to be uniform keeps the MMAs' operands in uniform
// registers
__device__ __forceinline__ bool rf_wait_warp(uint32_t mbar, uint32_t parity) {
  if (__all_sync(0xffffffffu, mbar_try_wait(mbar, parity))) return true;
  const long long t0 = clock64();
  while (!__all_sync(0xffffffffu, mbar_try_wait(mbar, parity)))
    if (__any_sync(0xffffffffu, clock64() - t0 > (1ll << 31))) return false;
  return true;
}

// max |H|, H = fl32((1 + d_j) G_jn); NaN counts as infinity.  All threads.
__device__ __forceinline__ float rf_scale(const RfPar& P, float* red) {
  const int L = P.L, ld = P.ld, sig = P.sig;
  const float* G = P.G;
  const int8_t* s = P.s;
  const float cpl0 = P.rc->cplus[0], cpl1 = P.rc->cplus[1];  // 1 + d_j for sigma s_j = +1, -1
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NW = kDelNT / 32, RB = 4;  // rows per warp in flight, every load before its use
  float hmax = 0.f;
  for (int j0 = warp; j0 < L; j0 += RB * NW) {
    for (int n0 = lane; n0 < L; n0 += 32 * 8) {
      float g[RB][8];
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const float* p = G + (size_t)min(j0 + r * NW, L - 1) * ld;
#pragma unroll
        for (int u = 0; u < 8; ++u) g[r][u] = p[min(n0 + 32 * u, L - 1)];
      }
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const float cp = sig * s[min(j0 + r * NW, L - 1)] > 0 ? cpl0 : cpl1;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float H = fabsf(g[r][u] * cp);
          asm("max.NaN.f32 %0, %0, %1;" : "+f"(hmax) : "f"(H));  // a NaN enters and stays
        }
      }
    }
  }
  return rf_block_max(hmax, red);
}

// E = 1 - A H' -> P.wsE (row stride rf_lde(L)), tile by tile (128 columns n of
// H' = TMEM lanes, kRfN rows i of A); returns this thread's max |E|, sets
// W.bad on a wait that gave up (then every thread returns early, together).
// sm: A's table, then the row factors fs (zero beyond L).
// kAhead4: the read-out's entries of G are loaded four rows ahead instead of all
// 16 before it.  For the two-spin sweep, whose accept loop the compiler spills
// registers of for what is live here: with it, and the other cuts marked in
// k_delayed.cu, 40 two-spin chains at Lambda = 240 without a recompute take 7.9
// ms for 26 sweeps instead of 11.8.  The one-spin kernel is faster without
// (15.7 against 16.8 ms for 160 chains at Lambda = 240, 20 sweeps).
//
// The cutting warps run through the contraction blocks of all tiles as one
// stream (a quarter's blocks dealt round its warps), up to kRfAhead K steps
// into the next tile before they turn to a tile's read-out.
template <bool kAhead4>
__device__ __forceinline__ float rf_product(RfPar& P, const unsigned char* sm, int sh, RfWait& W) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = (int)rf_uniform((uint32_t)tid >> 5);  // see elect_one
  constexpr int NW = kDelNT / 32;
  const int q4 = warp & 3, g4 = warp >> 2;  // TMEM lane quarter; group of rows or contraction blocks
  const int L = P.L;
  const int NJ = rf_nj(L), nib = rf_ni(L) / (kRfN / 8), nmb = (L + 127) / 128;
  const uint32_t cc = P.sync.cc;
  const uint32_t bar_full = P.cbar + 8u, bar_empty = bar_full + 8u * kRfBufs;
  const uint32_t lane_base = P.tmem + ((uint32_t)(32 * q4) << 16);
  const float* fs = reinterpret_cast<const float*>(sm + rf_tab_bytes(L));
  const bool issuer = warp > kRfIssueWarp - kRfIssuers;
  const int stride = q4 > (kRfIssueWarp & 3) - kRfIssuers ? NW / 4 - 1 : NW / 4;
  const int total = nmb * nib * NJ;
  float emax = 0.f;
  int vb = g4, vt = 0, vm = 0;  // the warp's next block: block of its tile, row tile, column block
  int v = g4;                   // ... and its place in the stream
  for (int tile = 0; tile < nmb * nib; ++tile) {
    if (!issuer) {
      // cut in registers, then stored once the buffer is free, so that little
      // is left to do between a buffer's release and its refill; the loads of
      // the warp's next block are issued before the cut.  A block: eight rows
      // (in descending block order: see the table), one column per lane; lanes
      // past the last column repeat it (their results are never read), rows
      // past the last one count zero (fs is 0 there)
      const int ld = P.ld;
      const float* G = P.G;
      float yn[8];  // the next block's values
      auto load = [&]() {
        const int j0 = 8 * (NJ - 1 - vb);
        const float* p = G + min(vm * 128 + 32 * q4 + lane, L - 1);
        if (j0 + 8 <= L) {
          p += (size_t)j0 * ld;
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            yn[t] = *p;
            p += ld;
          }
        } else {
#pragma unroll
          for (int t = 0; t < 8; ++t) yn[t] = p[(size_t)min(j0 + t, L - 1) * ld];
        }
      };
      auto wrap = [&]() {
        while (vb >= NJ) {
          vb -= NJ;
          if (++vt == nib) {
            vt = 0;
            ++vm;
          }
        }
      };
      const int lim = min((tile + 1) * NJ + 2 * kRfAhead, total);
      wrap();
      if (v < lim) load();
#pragma unroll 1
      while (v < lim) {
        float y[8];
        {
          const float4* f4 = reinterpret_cast<const float4*>(fs + 8 * (NJ - 1 - vb));
          const float4 f0 = f4[0], f1 = f4[1];
          y[0] = yn[0] * f0.x, y[1] = yn[1] * f0.y, y[2] = yn[2] * f0.z, y[3] = yn[3] * f0.w;
          y[4] = yn[4] * f1.x, y[5] = yn[5] * f1.y, y[6] = yn[6] * f1.z, y[7] = yn[7] * f1.w;
        }
        const int half = v & 1;  // NJ is even: also the block's half of its K step
        const uint32_t nu = cc + (uint32_t)(v >> 1);
        v += stride;
        vb += stride;
        wrap();
        if (v < lim) load();
        uint32_t w[kRfSlicesH][4];
        rf_cut8(y, w);
        if (nu >= kRfBufs) W.on(bar_empty + 8u * (nu % kRfBufs), (nu / kRfBufs - 1u) & 1u);
        __syncwarp();
        tc_fence_after();
        const uint32_t col = lane_base + (uint32_t)(kRfBufCol + (int)(nu % kRfBufs) * kRfBufCols + half * 4);
#pragma unroll
        for (int q = 0; q < kRfSlicesH; ++q) tmem_st4(col + (uint32_t)(q * 8), w[q][0], w[q][1], w[q][2], w[q][3]);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_full + 8u * (nu % kRfBufs));
      }
    } else {
      // every operand of an MMA warp-uniform in the compiler's eyes
      const uint32_t el = elect_one();
      const uint32_t idesc = make_idesc_f16(kRfN);
      const uint32_t n16 = (uint32_t)NJ / 2u, ib = (uint32_t)tile % (uint32_t)nib;
      const uint32_t tm = rf_uniform(P.tmem), nk = rf_uniform(n16), bar_e = rf_uniform(bar_empty), bar_f = rf_uniform(bar_full);
      const uint32_t c0 = rf_uniform(cc + (uint32_t)tile * n16), slice = rf_uniform((uint32_t)rf_ncore(L) * 8u);
      const uint64_t desc = make_smem_desc(smem_u32(sm) + ib * (kRfN * 16u), 128u, 128u);
      uint32_t bk = rf_uniform((uint32_t)desc);
      bool live = !__any_sync(0xffffffffu, W.bad);
      for (uint32_t k = 0; k < nk; ++k, bk += 16u) {
        const uint32_t nu = c0 + k;
        if (live) live = rf_wait_warp(bar_f + 8u * (nu % kRfBufs), (nu / kRfBufs) & 1u);
        tc_fence_after();
        const uint32_t a0 = tm + kRfBufCol + nu % kRfBufs * kRfBufCols;
        const uint64_t bd = (desc & 0xffffffff00000000ull) | bk;
        auto issue = [&](auto which) {
#pragma unroll
          for (int q = 0; q < kRfSlicesH; ++q)
#pragma unroll
            for (int p = 0; p + q < kRfLevels; ++p)
              if (rf_issuer_of(p + q) == decltype(which)::value)
                tc_mma_f16_ts(el, tm + (uint32_t)((p + q) * kRfN), a0 + (uint32_t)(q * 8),
                              bd + (uint64_t)((uint32_t)p * slice), idesc, q > 0 || k > 0 ? 1 : 0);
        };
        if (live) {
          if (warp == kRfIssueWarp)
            issue(std::integral_constant<int, 0>());
          else
            issue(std::integral_constant<int, 1>());
        }
        tc_commit_el(el, bar_e + 8u * (nu % kRfBufs));
      }
      // the last step's products (the issuers have seen every use before it consumed)
      const uint32_t nl = c0 + nk - 1u;
      if (live) live = rf_wait_warp(bar_e + 8u * (nl % kRfBufs), (nl / kRfBufs) & 1u);
      W.bad = !live;
    }
    // this warp's rows of the tile, ie .. ie + 15: those with sigma s = -1
    // (whose diagonal differs from the table's), and G_in there, loaded while
    // the last MMAs run
    const int ie = tile % nib * kRfN + 16 * g4, n = tile / nib * 128 + 32 * q4 + lane;
    const unsigned neg = __ballot_sync(
        0xffffffffu, lane < 16 && ie + lane < L && P.sig * P.s[ie + lane < L ? ie + lane : 0] < 0);
    float gd[kAhead4 ? 4 : 16];
    auto load_gd = [&](int c0) {  // rows ie + c0 and on
      const float* p = P.G + (size_t)min(ie + c0, L - 1) * P.ld + min(n, L - 1);
      const int ld = P.ld;
#pragma unroll
      for (int c = 0; c < (kAhead4 ? 4 : 16); ++c) {
        if (neg >> (c0 + c) & 1u) gd[c] = *p;  // warp-uniform
        p += ld;
      }
    };
    load_gd(0);
    if (!__syncthreads_and(W.bad ? 0 : 1)) {
      W.bad = true;
      return emax;
    }
    tc_fence_after();
    // Read-out, 4 rows at a time.  Horner's rule from the highest level,
    // x <- 128 x + S_l, with delta subtracted at level 0, in FP32: where |E|
    // is small the level sums cancel, every x up to level 4 is an integer
    // below 2^24, so each FMA is exact and the last one rounds
    // 2^{sh} (A H' - delta) once -- the same E as from 64-bit integers.
    // Checked: an inexact x means |x_4| >= 2^24 (x only grows from there),
    // and the warp evaluates those rows in 64 bits.
    const bool narrow = sh >= 35;  // 2^{sh-35}, delta in units of level 0, is an integer
    const float one0 = pow2f(narrow ? sh - 35 : 0), back = -pow2f(-sh);
    float dd[kRfSlicesA];  // slices of A_jj for sigma s_j = -1 less those for +1
#pragma unroll
    for (int p = 0; p < kRfSlicesA; ++p) dd[p] = P.rc->dd[p];
    float* pe = P.wsE + (size_t)ie * rf_lde(L) + n;
    uint32_t widemask = 0u;  // rows to evaluate in 64 bits (warp-uniform)
#pragma unroll
    for (int h4 = 0; h4 < 4; ++h4) {
      const int i0 = ie + 4 * h4;
      if (i0 < L) {  // warp-uniform
        const uint32_t ta = lane_base + (uint32_t)(16 * g4 + 4 * h4);
        float g4r[4];
        if constexpr (kAhead4) {
#pragma unroll
          for (int c = 0; c < 4; ++c) g4r[c] = gd[c];
          if (h4 < 3) load_gd(4 * h4 + 4);
        }
        uint32_t u[kRfLevels][4];
#pragma unroll
        for (int lv = 0; lv < kRfLevels; ++lv) tmem_ld4_nowait(ta + (uint32_t)(lv * kRfN), u[lv]);
        float x[4];
#pragma unroll
        for (int lv = 0; lv < kRfLevels; ++lv) tmem_wait_ld4(u[lv]);
        bool wide = !narrow;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float S[kRfLevels];
#pragma unroll
          for (int lv = 0; lv < kRfLevels; ++lv) S[lv] = __uint_as_float(u[lv][c]);
          if (neg >> (4 * h4 + c) & 1u) {  // warp-uniform: the other value of A_ii
            float y = (kAhead4 ? g4r[c] : gd[kAhead4 ? 0 : 4 * h4 + c]) * fs[i0 + c];
#pragma unroll
            for (int q = 0; q < kRfSlicesH; ++q) {
              const float d = (y + 12582912.f) - 12582912.f;
#pragma unroll
              for (int p = 0; p + q < kRfLevels; ++p) S[p + q] = __fmaf_rn(dd[p], d, S[p + q]);
              y = __fmaf_rn(y, 128.f, -128.f * d);
            }
          }
          x[c] = S[0] - (i0 + c == n ? one0 : 0.f);
#pragma unroll
          for (int lv = 1; lv < kRfLevels; ++lv) {
            if (lv == kRfLevels - 1) wide = wide || !(fabsf(x[c]) < 16777216.f);
            x[c] = __fmaf_rn(x[c], 128.f, S[lv]);
          }
          x[c] = __fmaf_rn(x[c], back, 0.f);  // E (and +0 for a zero)
        }
        if (__any_sync(0xffffffffu, wide && n < L)) {
          widemask |= 15u << (4 * h4);
        } else if (n < L) {
          // every value before the first store (which would order the loads after it)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (i0 + c < L) {
              pe[(size_t)(4 * h4 + c) * rf_lde(L)] = x[c];
              emax = fmaxf(emax, fabsf(x[c]));
            }
        }
      }
    }
#pragma unroll 1
    for (; widemask; widemask &= widemask - 1u) {  // warp-uniform
      const int c = __ffs(widemask) - 1, i = ie + c;
      if (i >= L) break;
      const bool ng = neg >> c & 1u;
      const float y = ng ? P.G[(size_t)i * P.ld + min(n, L - 1)] * fs[i] : 0.f;
      const float E = rf_residual_wide(lane_base + (uint32_t)(16 * g4 + c), ng, y, P.rc->dd, i == n, sh);
      if (n < L) {
        P.wsE[(size_t)i * rf_lde(L) + n] = E;
        emax = fmaxf(emax, fabsf(E));
      }
    }
    tc_fence_before();
    __syncthreads();
  }
  if (tid == 0) P.sync.cc = rf_uses(cc + (uint32_t)(nmb * nib) * (uint32_t)(NJ / 2), kRfBufs);
  return emax;
}

// G_new^T = (H'^T + E^T H'^T) (1 + D)^{-1}, G replaced; returns this thread's
// largest change of an entry, W.bad as above.  M: columns n of G (E^T), in
// blocks of 128; N: all rows i (H'), up to 256 per MMA; K in chunks of kRf2KC
// through two stage buffers (sm): a chunk is staged while the tensor cores
// multiply the one before.
__device__ __forceinline__ float rf_update(RfPar& P, unsigned char* sm, int eh, int se, RfWait& W) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = (int)rf_uniform((uint32_t)tid >> 5);
  constexpr int NW = kDelNT / 32;
  const int q4 = warp & 3, g4 = warp >> 2;
  const int L = P.L, ld = P.ld, ldE = rf_lde(L), nmb = (L + 127) / 128;
  float* const G = P.G;
  const float* const wsE = P.wsE;
  const int Lp = rf_pad(L, 16), nkc2 = rf_pad(L, kRf2KC) / kRf2KC;
  // two column blocks and at most 256 rows: both blocks' products at once
  // (accumulators at TMEM columns 0 and 256), so each H' chunk is staged once;
  // else one column block at a time, its rows in up to two halves
  const int nr = (nmb == 2 && Lp <= 256) ? 2 : 1;
  const bool direct = nmb <= nr;  // every column block done before G is written
  const bool vec = (ld & 3) == 0;  // rows of G 16-byte aligned
  const uint32_t ebytes = 128u * kRf2KC * 2u;          // one column block's E^T hi (or lo)
  const uint32_t hbytes = (uint32_t)Lp * kRf2KC * 2u;  // H' hi (or lo)
  const uint32_t stage_bytes = rf_stage2_bytes(L), bar_stage = P.cbar + 8u + 16u * kRfBufs;
  uint32_t c2 = P.sync.c2;
  float drift = 0.f;
  // per row: (1 + d_i) 2^{28-eh} (H' = rint(H 2^{28-eh}) 2^{eh-28}) and the FP32 pair of 1 / (1 + d_i)
  float4* const rf = reinterpret_cast<float4*>(sm + 2 * stage_bytes);
  for (int i = tid; i < Lp; i += kDelNT) {
    const int u = i < L && P.sig * P.s[i < L ? i : 0] > 0 ? 0 : 1;
    rf[i] = make_float4(P.rc->cplus[u] * pow2f(28 - eh), P.rc->cminus_hi[u], P.rc->cminus_lo[u], 0.f);
  }
  __syncthreads();
  for (int mb0 = 0; mb0 < nmb; mb0 += nr) {
    {
      // E^T: thread = column n (lanes consecutive: coalesced), 8 rows j.  H':
      // chunk c = row 8 (c / 32) + c % 8, K offset 8 ((c / 8) % 4): a warp
      // covers 8 rows x 32 consecutive columns.  The loads of the next chunk
      // are issued before the barrier of the current one
      const float sE = pow2f(se);
      const int k8e = tid >> 7, re = tid & 127;
      float xe[2][8], xh[2][8];
      auto load_e = [&](int kc) {
        const int j0 = kc * kRf2KC + 8 * k8e;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (u < nr) {
            // columns past the last repeat it (never read back); rows past it are 0
            const float* p = wsE + (size_t)j0 * ldE + min((mb0 + u) * 128 + re, L - 1);
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              xe[u][t] = j0 + t < L ? *p : 0.f;
              p += ldE;
            }
          }
        }
      };
      auto load_h = [&](int kc, int c0) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int c = c0 + u * kDelNT, i = min(((c >> 5) << 3) | (c & 7), L - 1);
          const int k0 = kc * kRf2KC + (((c >> 3) & 3) << 3);
          const float* p = G + (size_t)i * ld + k0;
          if (vec && k0 + 8 <= L) {
            const float4 x0 = *reinterpret_cast<const float4*>(p), x1 = *reinterpret_cast<const float4*>(p + 4);
            xh[u][0] = x0.x, xh[u][1] = x0.y, xh[u][2] = x0.z, xh[u][3] = x0.w;
            xh[u][4] = x1.x, xh[u][5] = x1.y, xh[u][6] = x1.z, xh[u][7] = x1.w;
          } else {
#pragma unroll
            for (int t = 0; t < 8; ++t) xh[u][t] = k0 + t < L ? p[t] : 0.f;
          }
        }
      };
      load_e(0);
      load_h(0, tid);
      for (int kc = 0; kc < nkc2; ++kc, ++c2) {
        if (c2 >= 2u) W.on(bar_stage + 8u * (c2 & 1u), ((c2 >> 1) - 1u) & 1u);
        unsigned char* sb = sm + (c2 & 1u) * stage_bytes;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (u < nr) {
            uint32_t h[4], l[4];
#pragma unroll
            for (int t = 0; t < 8; t += 2) {
              const float xa = xe[u][t] * sE, xb = xe[u][t + 1] * sE;
              h[t / 2] = f32x2_to_f16x2(xa, xb);
              l[t / 2] = f32x2_to_f16x2(xa - f16_lo_to_f32(h[t / 2]), xb - f16_hi_to_f32(h[t / 2]));
            }
            unsigned char* dst = sb + u * 2 * ebytes + rf_off2(re, k8e);
            *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(dst + ebytes) = make_uint4(l[0], l[1], l[2], l[3]);
          }
        }
        if (kc + 1 < nkc2) load_e(kc + 1);
        // H' (x 2^{14-eh}, below 2^14)
        for (int c0 = tid;;) {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int c = c0 + u * kDelNT, i = ((c >> 5) << 3) | (c & 7);
            if (c < Lp * 4) {
              const float cs = rf[i].x;
              uint32_t h[4], l[4];
#pragma unroll
              for (int t = 0; t < 8; t += 2) {
                const float xa = rintf(xh[u][t] * cs) * 0x1p-14f, xb = rintf(xh[u][t + 1] * cs) * 0x1p-14f;
                h[t / 2] = f32x2_to_f16x2(xa, xb);
                l[t / 2] = f32x2_to_f16x2(xa - f16_lo_to_f32(h[t / 2]), xb - f16_hi_to_f32(h[t / 2]));
              }
              unsigned char* dst = sb + nr * 2 * ebytes + rf_off2(i, (c >> 3) & 3);
              *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
              *reinterpret_cast<uint4*>(dst + hbytes) = make_uint4(l[0], l[1], l[2], l[3]);
            }
          }
          c0 += 2 * kDelNT;
          if (c0 >= Lp * 4) break;  // more than 256 rows: a second part, not prefetched
          load_h(kc, c0);
        }
        if (kc + 1 < nkc2) load_h(kc + 1, tid);
        fence_async_smem();
        tc_fence_before();
        if (!__syncthreads_and(W.bad ? 0 : 1)) {
          W.bad = true;
          return drift;
        }
        if (warp == kRfIssueWarp) {
          tc_fence_after();
          const uint32_t el = elect_one();
          const uint32_t tm = rf_uniform(P.tmem), nru = rf_uniform((uint32_t)nr), lpu = rf_uniform((uint32_t)Lp);
          const uint32_t e2 = rf_uniform(smem_u32(sb)), h2 = e2 + nru * 2u * ebytes;
          const uint32_t kcu = rf_uniform((uint32_t)kc);
          const uint64_t lo_e = (uint64_t)(ebytes >> 4), lo_h = (uint64_t)(lpu * (kRf2KC * 2u) >> 4);
          const uint64_t ed = make_smem_desc(e2, 128u, (kRf2KC / 8) * 128u);
          const uint64_t hd = make_smem_desc(h2, 128u, (kRf2KC / 8) * 128u);
          for (uint32_t ur = 0; ur < nru; ++ur)
            for (uint32_t half = 0; half * 256 < lpu; ++half) {
              const uint32_t idesc2 = make_idesc_f16((int)min(lpu - half * 256u, 256u));
              const uint32_t d = tm + (ur + half) * 256u;
#pragma unroll
              for (uint32_t kk = 0; kk < kRf2KC / 16; ++kk) {
                if (kcu * kRf2KC + kk * 16 >= lpu) continue;
                const uint64_t ahi = ed + (uint64_t)(ur * (2u * ebytes >> 4) + kk * 16u);
                const uint64_t bhi = hd + (uint64_t)(half * (32u * (kRf2KC / 8) * 8u) + kk * 16u);
                tc_mma_f16_el(el, d, ahi, bhi, idesc2, (kcu > 0 || kk > 0) ? 1 : 0);
                tc_mma_f16_el(el, d, ahi + lo_e, bhi, idesc2, 1);
                tc_mma_f16_el(el, d, ahi, bhi + lo_h, idesc2, 1);
              }
            }
          if (el) tc_commit(bar_stage + 8u * (c2 & 1u));
          __syncwarp();
        }
      }
    }
    // every product of this group of column blocks
    W.on(bar_stage + 8u * ((c2 - 1u) & 1u), ((c2 - 1u) >> 1) & 1u);
    if (!__syncthreads_and(W.bad ? 0 : 1)) {
      W.bad = true;
      return drift;
    }
    tc_fence_after();
    // read-out: thread = column n, 8 rows i per pass (32 rows of the four
    // groups of warps); the next pass's loads of G are issued before the
    // current pass's arithmetic, the stores come last (a store in between
    // would hold back the loads after it)
    {
      const float sHi = pow2f(eh - 28), sQ = pow2f(eh - 14 - se);
      const uint32_t lane_base = P.tmem + ((uint32_t)(32 * q4) << 16);
      float* const Gn = direct ? G : P.wsE + (size_t)L * ldE;
      const int ldn = direct ? ld : L;
#pragma unroll 1
      for (int ur = 0; ur < nr; ++ur) {
        const int n = (mb0 + ur) * 128 + 32 * q4 + lane;
        float go[8];
        auto load_g = [&](int i0) {
          const float* p = G + (size_t)i0 * ld + min(n, L - 1);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            if (i0 + c < L) go[c] = *p;  // warp-uniform
            p += ld;
          }
        };
        load_g(8 * g4);
#pragma unroll 1
        for (int i0 = 8 * g4; i0 < L; i0 += 32) {
          float g[8];
          uint32_t q[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) g[c] = go[c];
          load_g(i0 + 32);
          tmem_ld8_nowait(lane_base + (uint32_t)(256 * ur + i0), q);
          tmem_wait_ld8(q);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const float4 f = rf[min(i0 + c, Lp - 1)];
            const float Hp = rintf(g[c] * f.x) * sHi;
            const float y = Hp + __uint_as_float(q[c]) * sQ;
            q[c] = __float_as_uint(fmaf(y, f.y, y * f.z));
          }
          if (n < L) {
            float* p = Gn + (size_t)i0 * ldn + n;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              if (i0 + c < L) {  // warp-uniform
                const float gn = __uint_as_float(q[c]);
                drift = fmaxf(drift, fabsf(g[c] - gn));
                *p = gn;
              }
              p += ldn;
            }
          }
        }
      }
    }
    tc_fence_before();
    __syncthreads();
  }
  if (!direct) {
    // every column block has read the old G: the new one moves in
    const float* Gn = wsE + (size_t)L * ldE;
    for (int i0 = warp; i0 < L; i0 += 2 * NW)
      for (int n0 = lane; n0 < L; n0 += 32 * 8) {
        float x[2][8];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int u = 0; u < 8; ++u)
            x[r][u] = (i0 + r * NW < L && n0 + 32 * u < L) ? Gn[(size_t)(i0 + r * NW) * L + n0 + 32 * u] : 0.f;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (i0 + r * NW < L && n0 + 32 * u < L) G[(size_t)(i0 + r * NW) * ld + n0 + 32 * u] = x[r][u];
      }
    __syncthreads();
  }
  if (tid == 0) P.sync.c2 = rf_uses(c2, 2);
  return drift;
}

// One spin: G (L x L, row-major, row stride ld, FP32, in global memory or in
// shared memory outside sm) is replaced by its Newton-refined value.  s: the
// field (shared memory); sig: +1 / -1; ws: the chain's workspace
// (rf_ws_bytes: E, and beyond 256 columns the new G); sm0: rf_smem_need(L) of
// 1024-byte aligned shared memory; tc: the CTA's TMEM allocation and
// mbarriers (tc->cbar: table copy, the H' buffers' "full", their "empty", the
// two update stages' "empty"; sync, in shared memory, counts their uses).
// Returns the largest change of an entry (>= 0), or -1 if the caller must
// recompute from scratch (|E| too large, scale out of range, or a wait gave
// up, which also sets kStatusTimeout).  All threads call it.
template <bool kAhead4>
__device__ __forceinline__ float refine_spin(int L, const RefineConst* rc, const int8_t* s, int sig, float* G, int ld,
                                             float* ws, unsigned char* sm0, TcState* tc, RfSync* sync, float* red,
                                             int* status) {
  RfPar& P = *reinterpret_cast<RfPar*>(sm0);
  unsigned char* sm = sm0 + kRfParBytes;
  // what the region held before was read and written through the generic proxy
  fence_async_smem();
  __syncthreads();
  if (threadIdx.x == 0) P = RfPar{G, ws, rc, s, status, L, ld, sig, tc->tmem, tc->cbar, *sync};
  __syncthreads();
  RfWait W;
  float drift = 0.f, emax = 0.f;
  bool ok = true;
  for (int step = 0; step < 2 && ok; ++step) {
    // A's slice table into shared memory while the scale pass runs
    if (threadIdx.x == 0) {
      const uint32_t bytes = (uint32_t)rf_tab_bytes(P.L);
      mbar_expect_tx(P.cbar, bytes);
      bulk_g2s(smem_u32(sm), P.rc->tab, bytes, P.cbar);
    }
    const float hmax = rf_scale(P, red);
    W.on(P.cbar, P.sync.ct & 1u);
    int eh = 0;
    ok = hmax < 1e30f;
    if (ok && hmax > 0.f) (void)frexpf(hmax, &eh);  // hmax < 2^eh
    const int sh = 49 - P.rc->ea - eh;              // delta in units of the integer sums
    ok = ok && !(sh < 0 || sh > 61 || eh < -60 || eh > 100);  // keeps every scale below normal
    {
      // (1 + d_j) 2^{7-eh}: H 2^{7-eh} is below 2^7 in magnitude
      const int L = P.L;
      const float s7 = pow2f(ok ? kRfBits - eh : 0);
      float* fs = reinterpret_cast<float*>(sm + rf_tab_bytes(L));
      for (int j = threadIdx.x; j < 8 * rf_nj(L); j += kDelNT)
        fs[j] = j < L ? P.rc->cplus[P.sig * P.s[j] > 0 ? 0 : 1] * s7 : 0.f;
    }
    __syncthreads();
    if (threadIdx.x == 0) ++P.sync.ct;
    if (!__syncthreads_and(W.bad ? 0 : 1)) {
      W.bad = true;
      break;
    }
    if (!ok) break;
    emax = rf_product<kAhead4>(P, sm, sh, W);
    if (W.bad) break;
    emax = rf_block_max(emax, red);
    ok = emax <= P.rc->emax_step;  // else too far for Newton steps (default 2^-8)
    if (!ok) break;
    int ee = 0;
    if (emax > 0.f) (void)frexpf(emax, &ee);  // emax < 2^ee
    // E 2^se below 2^15 (FP16 range); for |E| < 2^-25 the scale stops at
    // 2^40, where those corrections are far below G's FP32 rounding anyway
    const int se = emax > 0.f ? min(15 - ee, 40) : 0;
    drift = fmaxf(drift, rf_update(P, sm, eh, se, W));
    if (W.bad || emax <= 0x1p-13f) break;
    fence_async_smem();
    __syncthreads();
  }
  __syncthreads();
  if (threadIdx.x == 0) *sync = P.sync;
  if (W.bad) {  // uniform: every thread has left together
    if (threadIdx.x == 0) atomicOr(status, kStatusTimeout);
    tc->failed = 1;
    return -1.f;
  }
  const float d = rf_block_max(drift, red);
  return ok ? d : -1.f;
}

// G_dn = 1 - G_up^T for a particle-hole symmetric bath (both L x L FP32 at row
// stride ld), through per-warp 32 x 33 shared-memory tiles (tile: 16
// warps x 32 x 33 floats) so that reads and writes are both coalesced.  The
// rows of a tile go in batches of 16 with every load of a batch (G_up, and
// the old G_dn for the drift) issued before its stores.
// Returns max |G_dn(old) - G_dn(new)| (block-wide).  All threads call it.
__device__ inline float ph_mirror(const float* Gu, float* Gd, int L, int ld, float* tile, float* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = kDelNT / 32;
  float* tw = tile + warp * 32 * 33;
  const int nt = (L + 31) / 32;
  float drift = 0.f;
  for (int t = warp; t < nt * nt; t += NW) {
    const int ti = t / nt, tj = t - ti * nt;  // source tile rows ti*32.., columns tj*32..
    const int c = tj * 32 + lane;   // source column
    const int cc = ti * 32 + lane;  // destination column = source row
#pragma unroll
    for (int h = 0; h < 32; h += 16) {
      float v[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int i = ti * 32 + h + r;
        v[r] = (i < L && c < L) ? Gu[(size_t)i * ld + c] : 0.f;
      }
#pragma unroll
      for (int r = 0; r < 16; ++r) tw[(h + r) * 33 + lane] = v[r];
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 32; h += 16) {
      float o[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int i = tj * 32 + h + r;  // destination row = source column
        o[r] = (i < L && cc < L) ? Gd[(size_t)i * ld + cc] : 0.f;
      }
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int i = tj * 32 + h + r;
        if (i < L && cc < L) {
          const float gn = (i == cc ? 1.f : 0.f) - tw[lane * 33 + h + r];
          drift = fmaxf(drift, fabsf(o[r] - gn));
          Gd[(size_t)i * ld + cc] = gn;
        }
      }
    }
    __syncwarp();
  }
  return rf_block_max(drift, red);
}

}  // namespace hfq
