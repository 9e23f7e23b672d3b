// Rank-1 Hirsch-Fye sweep: one CTA per Markov chain, persistent over a
// longest-Lambda-first work queue.  T = double is the plain FP64 baseline
// (decision-for-decision identical to the FP64 oracle); T = float is the
// FP32 rank-1 path.
//
// Per sweep (introduction of the paper: single-slice flips of the binary HS
// field; Hirsch-Fye equations):
//   1. u_l = Philox(l, sweep, chain, grid) for all slices, in parallel.
//   2. Scan l = l0, l0+1, ... a window at a time: R = R^up R^dn from the current
//      diagonals, accept iff u_l < R (or heat bath).  Rejections change
//      nothing, so a warp evaluates a window of consecutive proposals at once
//      and a ballot finds the first accepted one.
//   3. Accepted slice l: u^sigma = G^sigma_{:,l} - e_l, w^sigma = (Delta/R^sigma) G^sigma_{l,:}
//      are staged in shared memory and G^sigma += u w^T (both spins), s_l -> -s_l.
//      Every n_wrap accepted flips: FP64 recompute + drift.
//   4. Measured sweeps: g^sigma(tau_k) and D accumulated per chain in FP64.
// G is staged in shared memory for the whole chain when 2 L (L|1) sizeof(T)
// fits, else it stays in HBM/L2 and is updated there.
//
// What bounds it: an FP64 warp instruction takes 64 cycles of its scheduler
// here (2 DFMA per clock and SM), so per accepted flip T = double cannot take
// less than L^2 cycles for the update and every other FP64 instruction
// counts.  Hence:
//   * one warp scans, 16 slices a window, spin up on its lower and spin down
//     on its upper lanes (half the FP64 instructions of a lane that does both),
//     compares as integers, and the two lanes of the accepted slice divide for
//     the flip factors together.  Before, every thread divided twice: 3000
//     cycles a flip.  It scans for the next slice while the other warps update
//     G with this one: the diagonal is all it needs.
//   * the update has several rows' loads in flight per warp and no condition
//     per element (rank1_rows).
// T = float: the same, with the uniforms rounded once a sweep to the FP32
// thresholds that decide u < R exactly.
// Measured, whole solves before and after: one FP64 chain at Lambda 16, 550
// sweeps, 10.6 -> 6.6 ms; 152 FP64 chains at Lambda 100, 160 and 240, 10 sweeps,
// 122 -> 47 ms; 152 FP32 chains at Lambda 64 and 128, 220 sweeps, 75 -> 34 ms
// (the last two with the recompute's elimination of hfq_gj.cuh).  At Lambda
// 240 a flip takes 66k cycles of which 57.6k are the update's DFMAs.
#include "hfq_device.cuh"
#include "hfq_gj.cuh"
#include "hfq_launch.h"

#include <type_traits>

namespace hfq {

template <typename T>
struct R1Traits;
template <>
struct R1Traits<double> {
  static constexpr int NT = 256;
};
template <>
struct R1Traits<float> {
  static constexpr int NT = 512;
};

__host__ __device__ inline int r1_ld_smem(int L) { return L | 1; }

__host__ __device__ inline size_t r1_align16(size_t x) { return (x + 15) & ~(size_t)15; }

// Dynamic shared-memory layout:
//   head: colk[L] (double, recompute scratch), u[L] (double), perm[L] (int, pivot order of a
//   recompute), s[L] (int8)
//   body: [G^up G^dn (if resident)] diag[2L] col[2L] row[2L]
// During an FP64 recompute with gj_smem the body is overlaid by its workspace.
__host__ __device__ inline size_t r1_head_bytes(int L) {
  return r1_align16((size_t)L * sizeof(double)) * 2 + r1_align16((size_t)L * sizeof(int)) +
         r1_align16((size_t)L);
}
__host__ __device__ inline size_t r1_smem_bytes(int L, bool resident, size_t elem, bool gj_smem) {
  size_t b = 0;
  if (resident) b += r1_align16(2 * (size_t)L * r1_ld_smem(L) * elem);
  b += 3 * r1_align16(2 * (size_t)L * elem);
  if (gj_smem && gj_smem_bytes(L) > b) b = gj_smem_bytes(L);
  return r1_head_bytes(L) + b;
}

template <typename T>
__device__ __forceinline__ T tfma(T a, T b, T c);
template <>
__device__ __forceinline__ double tfma<double>(double a, double b, double c) {
  return __fma_rn(a, b, c);
}
template <>
__device__ __forceinline__ float tfma<float>(float a, float b, float c) {
  return __fmaf_rn(a, b, c);
}

// 1 + (1 - g) Delta, in the written order without contraction (as in the oracle)
__device__ __forceinline__ double flip_ratio(double g, double delta) {
  return __dadd_rn(1.0, __dmul_rn(__dsub_rn(1.0, g), delta));
}
__device__ __forceinline__ float flip_ratio(float g, float delta) {
  return __fadd_rn(1.f, __fmul_rn(__fsub_rn(1.f, g), delta));
}

// The FP32 path's threshold for the uniform u in [0, 1).  Metropolis: the
// smallest float t with u < R  <=>  t <= R for every float R: u rounded up, or
// the next float where u is one itself.  Heat bath: u rounded to nearest.
__device__ __forceinline__ float u_threshold(double u, int rule) {
  if (rule != 0) return (float)u;
  const float t = __double2float_ru(u);
  return (double)t == u ? __int_as_float(__float_as_int(t) + 1) : t;
}

// G += u w^T on the columns c0 .. c0 + 32 NC - 1 of one spin (only the last
// chunk of 32 may reach past L; its lanes there load a clamped column and store
// nothing).  A warp takes R rows a batch, every load before the first store,
// without a condition in between: written with one per element the batch
// compiled to a branch each and took 6000 cycles for a 64 x 64 pair of spins
// in shared memory.
template <typename T, int NC, int R>
__device__ __forceinline__ int rank1_rows(T* G, int ld, int L, const T* cs, const T (&rv)[NC], int j, int jl, int i0,
                                          int NW) {
  for (; i0 + (R - 1) * NW < L; i0 += R * NW) {
    T v[R][NC], ci[R];
    T* g = G + (size_t)i0 * ld;
    const size_t step = (size_t)NW * ld;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      ci[r] = cs[i0 + r * NW];
#pragma unroll
      for (int c = 0; c + 1 < NC; ++c) v[r][c] = g[r * step + j + 32 * c];
      v[r][NC - 1] = g[r * step + jl];
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < NC; ++c) v[r][c] = tfma<T>(ci[r], rv[c], v[r][c]);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c + 1 < NC; ++c) g[r * step + j + 32 * c] = v[r][c];
    if (j + 32 * (NC - 1) < L) {
#pragma unroll
      for (int r = 0; r < R; ++r) g[r * step + jl] = v[r][NC - 1];
    }
  }
  return i0;
}
template <typename T, int NC>
__device__ __forceinline__ void rank1_columns(T* G, int ld, int L, const T* cs, const T* rs, int c0, int w, int nw) {
  const int j = c0 + (threadIdx.x & 31), jl = min(j + 32 * (NC - 1), L - 1);
  T rv[NC];
#pragma unroll
  for (int c = 0; c + 1 < NC; ++c) rv[c] = rs[j + 32 * c];
  rv[NC - 1] = rs[jl];
  const int i0 = rank1_rows<T, NC, 4>(G, ld, L, cs, rv, j, jl, w, nw);
  rank1_rows<T, NC, 1>(G, ld, L, cs, rv, j, jl, i0, nw);
}
// Both spins, by nw warps of which this is number w.
template <typename T>
__device__ __forceinline__ void rank1_update(T* Gu, T* Gd, int ld, int L, const T* col, const T* row, int w, int nw) {
  if (L <= 16) {  // two rows per warp
    for (int i = 2 * w + ((threadIdx.x >> 4) & 1); i < 2 * L; i += 2 * nw) {
      const int j = threadIdx.x & 15, o = i < L ? 0 : L;
      T* g = (i < L ? Gu : Gd) + (size_t)(i - o) * ld + j;
      if (j < L) *g = tfma<T>(col[i], row[o + j], *g);
    }
  } else {
#pragma unroll 1
    for (int sp = 0; sp < 2; ++sp) {
      T* G = sp ? Gd : Gu;
#pragma unroll 1
      for (int c0 = 0; c0 < L; c0 += 128) {
        const int n = L - c0;
        if (n > 96)
          rank1_columns<T, 4>(G, ld, L, col + sp * L, row + sp * L, c0, w, nw);
        else if (n > 64)
          rank1_columns<T, 3>(G, ld, L, col + sp * L, row + sp * L, c0, w, nw);
        else if (n > 32)
          rank1_columns<T, 2>(G, ld, L, col + sp * L, row + sp * L, c0, w, nw);
        else
          rank1_columns<T, 1>(G, ld, L, col + sp * L, row + sp * L, c0, w, nw);
      }
    }
  }
}

// Column and row `first` of both spins: col = G e_first - e_first, row = G^T
// e_first times the flip factors (fu, fd).
template <typename T, int NT>
__device__ __forceinline__ void rank1_fetch(const T* Gu, const T* Gd, int ld, int L, int first, T fu, T fd, T* col,
                                            T* row) {
  for (int i = threadIdx.x; i < L; i += NT) {
    const T cu = Gu[(size_t)i * ld + first], cd = Gd[(size_t)i * ld + first];
    const T ru = Gu[(size_t)first * ld + i], rd = Gd[(size_t)first * ld + i];
    col[i] = i == first ? cu - T(1) : cu;
    col[L + i] = i == first ? cd - T(1) : cd;
    row[i] = ru * fu;
    row[L + i] = rd * fd;
  }
}

__device__ __forceinline__ float signed_by(float x, bool neg) {
  return __int_as_float(__float_as_int(x) ^ (neg ? (int)0x80000000 : 0));
}
__device__ __forceinline__ double signed_by(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000 : 0), __double2loint(x));
}

// The sums of both spins' wrapped diagonal k (sign -1 past the wrap), l = 0 ..
// L - 1 in order, the loads of eight terms before their additions.
template <typename T>
__device__ __forceinline__ void rank1_diagonal(const T* Gu, const T* Gd, int ld, int L, int k, double* su, double* sd) {
  double a = 0.0, b = 0.0;
  for (int l0 = 0; l0 < L; l0 += 8) {
    T x[8], y[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int l = l0 + t, r = l + k < L ? l + k : l + k - L;
      x[t] = l < L ? Gu[(size_t)r * ld + l] : T(0);
      y[t] = l < L ? Gd[(size_t)r * ld + l] : T(0);
    }
    // past the wrap the sign bit is flipped, not the value negated in FP64
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int l = l0 + t;
      if (l < L) {
        a += (double)signed_by(x[t], l + k >= L);
        b += (double)signed_by(y[t], l + k >= L);
      }
    }
  }
  *su = a;
  *sd = b;
}

// kTrace: kTraceRecord sets the bit of every accepted flip in the chain's
// decision trace; kTraceReplay takes the decisions from the trace instead of
// u < R (the flip ratios, flip factors and updates are computed as usual), so
// that an FP64 run follows the trajectory another run recorded.
template <typename T, int kTrace>
__global__ void __launch_bounds__(R1Traits<T>::NT, 1) k_sweep_rank1(SweepArgs a) {
  constexpr int NT = R1Traits<T>::NT;
  constexpr int NW = NT / 32;
  constexpr bool kF64 = std::is_same<T, double>::value;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[NW];
  __shared__ int redi[NW];
  __shared__ double s_inv;
  __shared__ T s_fac[2];  // flip factors of the accepted slice s_first
  __shared__ int s_piv, s_item, s_first;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  for (;;) {
    if (tid == 0) s_item = atomicAdd(a.queue_head, 1);
    __syncthreads();
    const int q = s_item;
    __syncthreads();
    if (q >= a.n_items) break;
    const ItemPtrs ip = a.items[a.order[q]];
    const GridConst gc = a.grids[ip.grid];
    const int L = gc.L;
    const bool resident = gc.resident != 0;

    // carve shared memory
    unsigned char* p = smem;
    double* colk = reinterpret_cast<double*>(p);
    p += r1_align16((size_t)L * sizeof(double));
    double* us = reinterpret_cast<double*>(p);        // this sweep's uniforms (FP64)
    float* uf = reinterpret_cast<float*>(p);          // ... or their FP32 thresholds
    p += r1_align16((size_t)L * sizeof(double));
    int* perm = reinterpret_cast<int*>(p);
    p += r1_align16((size_t)L * sizeof(int));
    int8_t* ss = reinterpret_cast<int8_t*>(p);
    p += r1_align16((size_t)L);
    unsigned char* body = p;
    // G in shared memory or in HBM.  Where it matters the two are told apart in
    // the code as well: through a pointer of unknown address space a shared
    // access costs several times as much
    T* Gu;
    T* Gd;
    const size_t off_G = (size_t)(p - smem);
    int ld;
    T* Ggl = reinterpret_cast<T*>(ip.G);
    if (resident) {
      ld = r1_ld_smem(L);
      Gu = reinterpret_cast<T*>(p);
      Gd = Gu + (size_t)L * ld;
      p += r1_align16(2 * (size_t)L * ld * sizeof(T));
    } else {
      ld = L;
      Gu = Ggl;
      Gd = Ggl + (size_t)L * L;
    }
    T* diag = reinterpret_cast<T*>(p);  // [0,L) up, [L,2L) dn
    p += r1_align16(2 * (size_t)L * sizeof(T));
    T* col = reinterpret_cast<T*>(p);
    p += r1_align16(2 * (size_t)L * sizeof(T));
    T* row = reinterpret_cast<T*>(p);

    if (resident) {
      for (int i = warp; i < 2 * L; i += NW)
        for (int j = lane; j < L; j += 32) Gu[(size_t)i * ld + j] = Ggl[(size_t)i * L + j];
    }
    for (int l = tid; l < L; l += NT) ss[l] = ip.s[l];
    __syncthreads();
    for (int i = tid; i < L; i += NT) {
      diag[i] = Gu[(size_t)i * ld + i];
      diag[L + i] = Gd[(size_t)i * ld + i];
    }
    const ChainCounters c0 = *ip.cnt;
    long long n_acc = c0.accepted;
    // accepted flips until the next recompute (the cumulative count reaches a
    // multiple of n_wrap); counted down so the hot loop needs no 64-bit modulo
    int until_rec = gc.n_wrap > 0 ? (int)(gc.n_wrap - n_acc % gc.n_wrap) : 0;
    long long n_rec = 0, n_bad = 0;
    unsigned long long hash = c0.hash;
    double drift = c0.drift;
    const long long n_sweeps = a.n_warm + a.n_meas;
    __syncthreads();

    // Warp 0: the first accepted slice >= l0 -> s_first (L: none), its flip
    // factors -> s_fac.
    auto scan = [&](long long sw, int l0) {
      int first = L;
      if constexpr (kF64) {
        double Rs = 1.0, dl = 0.0;  // this lane's spin of its slice
        for (int w = l0; w < L; w += 16) {
          const int l = w + (lane & 15);
          const bool in = l < L;
          const bool plus = (ss[in ? l : 0] > 0) == (lane < 16);
          dl = plus ? gc.delta[0] : gc.delta[1];
          Rs = flip_ratio(diag[(lane < 16 ? 0 : L) + (in ? l : 0)], dl);
          const double R = __dmul_rn(Rs, __shfl_xor_sync(0xffffffffu, Rs, 16));
          // R > 0 and finite, and u < R for such an R (u >= 0), on the bit patterns
          const long long rb = __double_as_longlong(R);
          const double u = us[in ? l : 0];
          const bool bad = in && !(rb > 0 && rb < 0x7ff0000000000000ll);
          bool acc;
          if (a.accept_rule == 0)
            acc = rb > __double_as_longlong(u) && rb <= 0x7ff0000000000000ll;
          else
            acc = __dmul_rn(u, __dadd_rn(1.0, R)) < R;
          if constexpr (kTrace == kTraceReplay)
            acc = in && ((ip.trace[(size_t)sw * trace_words(L) + (l >> 5)] >> (l & 31)) & 1u);
          const unsigned b = __ballot_sync(0xffffffffu, in && acc) & 0xffffu;
          const unsigned bb = __ballot_sync(0xffffffffu, bad) & 0xffffu;
          if (b) {
            first = w + __ffs(b) - 1;
            n_bad += __popc(bb & ((2u << (first - w)) - 1u));
            break;
          }
          n_bad += __popc(bb);
        }
        if (first < L) {
          const double f = dl / Rs;  // every lane divides (the same cost); the slice's two lanes count
          if ((lane & 15) == ((first - l0) & 15)) s_fac[lane >> 4] = f;
        }
      } else {
        float Ru = 1.f, Rd = 1.f, du = 0.f, dd = 0.f;
        for (int w = l0; w < L; w += 32) {
          const int l = w + lane;
          bool acc = false, bad = false;
          if (l < L) {
            const bool up = ss[l] > 0;
            du = up ? gc.deltaf[0] : gc.deltaf[1];
            dd = up ? gc.deltaf[1] : gc.deltaf[0];
            Ru = flip_ratio(diag[l], du);
            Rd = flip_ratio(diag[L + l], dd);
            const float R = __fmul_rn(Ru, Rd);
            bad = !(R > 0.f) || !isfinite(R);
            acc = a.accept_rule == 0 ? uf[l] <= R : __fmul_rn(uf[l], __fadd_rn(1.f, R)) < R;
          }
          if constexpr (kTrace == kTraceReplay)
            acc = l < L && ((ip.trace[(size_t)sw * trace_words(L) + (l >> 5)] >> (l & 31)) & 1u);
          const unsigned b = __ballot_sync(0xffffffffu, acc);
          const unsigned bb = __ballot_sync(0xffffffffu, bad);
          if (b) {
            first = w + __ffs(b) - 1;
            const int upto = first - w;  // lanes 0..upto evaluated
            const unsigned valid = upto >= 31 ? 0xffffffffu : ((2u << upto) - 1u);
            n_bad += __popc(bb & valid);
            break;
          }
          n_bad += __popc(bb);
        }
        if (first < L && lane == ((first - l0) & 31)) {
          s_fac[0] = du / Ru;
          s_fac[1] = dd / Rd;
        }
      }
      if (lane == 0) s_first = first;
    };

    for (long long sw = 0; sw < n_sweeps; ++sw) {
      const long long t = c0.t + sw;
      for (int l = tid; l < L; l += NT) {
        const double u = proposal_uniform(l, t, ip.chain, ip.grid, a.seed);
        if constexpr (kF64)
          us[l] = u;
        else
          uf[l] = u_threshold(u, a.accept_rule);
      }
      __syncthreads();
      if (warp == 0) scan(sw, 0);
      __syncthreads();
      int first = s_first;
      while (first < L) {
        if (resident) {
          const T* g = reinterpret_cast<const T*>(smem + off_G);
          rank1_fetch<T, NT>(g, g + (size_t)L * ld, ld, L, first, s_fac[0], s_fac[1], col, row);
        } else {
          rank1_fetch<T, NT>(Ggl, Ggl + (size_t)L * L, L, L, first, s_fac[0], s_fac[1], col, row);
        }
        __syncthreads();
        // Warp 0 advances the diagonal (with the update's own FMA) and scans
        // for the next slice while the other warps update; unless this flip is
        // the one before a recompute, whose diagonal the next slice must see
        const bool rec_now = gc.n_wrap > 0 && until_rec == 1;
        if (warp == 0) {
          for (int i0 = lane; i0 < 2 * L; i0 += 128) {
            T x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int i = min(i0 + 32 * u, 2 * L - 1);
              x[u] = i0 + 32 * u < 2 * L ? tfma<T>(col[i], row[i], diag[i]) : T(0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (i0 + 32 * u < 2 * L) diag[i0 + 32 * u] = x[u];
          }
          if (lane == 0) ss[first] = (int8_t)(-ss[first]);
          __syncwarp();
          if (!rec_now) scan(sw, first + 1);
        }
        // where the scan takes as long as the update, the others do it alone
        const int w0 = (!kF64 || L <= 32) ? 1 : 0;
        if (warp >= w0) {
          if (resident) {
            T* g = reinterpret_cast<T*>(smem + off_G);
            rank1_update<T>(g, g + (size_t)L * ld, ld, L, col, row, warp - w0, NW - w0);
          } else {
            rank1_update<T>(Ggl, Ggl + (size_t)L * L, L, L, col, row, warp - w0, NW - w0);
          }
        }
        hash = (hash ^ (unsigned long long)(t * (long long)L + first)) * kFnvPrime;
        if constexpr (kTrace == kTraceRecord) {
          if (tid == 0) ip.trace[(size_t)sw * trace_words(L) + (first >> 5)] |= 1u << (first & 31);
        }
        ++n_acc;
        __syncthreads();
        if (gc.n_wrap > 0 && --until_rec == 0) {
          until_rec = gc.n_wrap;
          double d;
          if (gc.gj_smem) {
            // the FP64 workspace overlays the body of shared memory: G goes home to HBM first
            if (resident) {
              for (int i = warp; i < 2 * L; i += NW)
                for (int j = lane; j < L; j += 32) Ggl[(size_t)i * L + j] = Gu[(size_t)i * ld + j];
              __syncthreads();
            }
            d = recompute_green_inv<T, NT>(gc, ss, Ggl, Ggl + (size_t)L * L, L,
                                           reinterpret_cast<double*>(body), red, redi, &s_inv, &s_piv,
                                           colk, perm, true, a.status);
            if (resident) {
              for (int i = warp; i < 2 * L; i += NW)
                for (int j = lane; j < L; j += 32) Gu[(size_t)i * ld + j] = Ggl[(size_t)i * L + j];
              __syncthreads();
            }
          } else {
            d = recompute_green_inv<T, NT>(gc, ss, Gu, Gd, ld, ip.ws, red, redi, &s_inv, &s_piv, colk,
                                           perm, true, a.status);
          }
          drift = fmax(drift, d);
          ++n_rec;
          for (int i = tid; i < L; i += NT) {
            diag[i] = Gu[(size_t)i * ld + i];
            diag[L + i] = Gd[(size_t)i * ld + i];
          }
          __syncthreads();
          if (warp == 0) scan(sw, first + 1);
          __syncthreads();
        }
        first = s_first;
      }
      if (sw >= a.n_warm) {
        const long long m = sw - a.n_warm;
        const int b = (int)((kBins * m) / a.n_meas);
        const double invL = 1.0 / (double)L;
        for (int k = tid; k < L; k += NT) {
          double su, sd;
          if (resident) {
            const T* g = reinterpret_cast<const T*>(smem + off_G);
            rank1_diagonal<T>(g, g + (size_t)L * ld, ld, L, k, &su, &sd);
          } else {
            rank1_diagonal<T>(Ggl, Ggl + (size_t)L * L, L, L, k, &su, &sd);
          }
          const double gu = su / (double)L, gd = sd / (double)L;
          ip.acc[k] += gu;
          ip.acc[L + k] += gd;
          ip.bins[(size_t)b * L + k] += 0.5 * (gu + gd);
        }
        double v = 0.0;
        for (int l = tid; l < L; l += NT) v += (1.0 - (double)diag[l]) * (1.0 - (double)diag[L + l]);
        if (L > 32)
          v = block_sum<NT>(v, red);
        else if (warp == 0)  // the other warps hold zeros
          for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (tid == 0) {
          ip.accD[0] += v * invL;
          ip.accD[1 + b] += v * invL;
        }
      }
      __syncthreads();
    }

    // write back the chain state
    if (resident) {
      for (int i = warp; i < 2 * L; i += NW)
        for (int j = lane; j < L; j += 32) Ggl[(size_t)i * L + j] = Gu[(size_t)i * ld + j];
    }
    for (int l = tid; l < L; l += NT) ip.s[l] = ss[l];
    // n_bad is warp-uniform; thread 0 holds warp 0's count, which covers every proposal once
    if (tid == 0) {
      ChainCounters c = c0;
      c.t = c0.t + n_sweeps;
      c.proposals = c0.proposals + n_sweeps * (long long)L;
      c.accepted = n_acc;
      c.recomputes = c0.recomputes + n_rec;
      c.hash = hash;
      c.bad = c0.bad + n_bad;
      c.drift = drift;
      *ip.cnt = c;
    }
    __syncthreads();
  }
}

template <typename T>
static void launch_rank1_t(const SweepArgs& a, int ctas, size_t smem, cudaStream_t st) {
  constexpr int NT = R1Traits<T>::NT;
  if (a.trace_mode == kTraceRecord)
    k_sweep_rank1<T, kTraceRecord><<<ctas, NT, smem, st>>>(a);
  else if (a.trace_mode == kTraceReplay)
    k_sweep_rank1<T, kTraceReplay><<<ctas, NT, smem, st>>>(a);
  else
    k_sweep_rank1<T, kTraceOff><<<ctas, NT, smem, st>>>(a);
}

int launch_sweep_rank1(bool f64, const SweepArgs& a, int ctas, size_t smem, cudaStream_t st) {
  if (f64)
    launch_rank1_t<double>(a, ctas, smem, st);
  else
    launch_rank1_t<float>(a, ctas, smem, st);
  return (int)cudaGetLastError();
}

template <typename T>
static cudaError_t config_rank1_t(size_t smem, int* occ) {
  cudaError_t e = raise_smem_limit(k_sweep_rank1<T, kTraceOff>, smem);
  if (e == cudaSuccess) e = raise_smem_limit(k_sweep_rank1<T, kTraceRecord>, smem);
  if (e == cudaSuccess) e = raise_smem_limit(k_sweep_rank1<T, kTraceReplay>, smem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k_sweep_rank1<T, kTraceOff>, R1Traits<T>::NT,
                                                      smem);
  return e;
}

int rank1_config(bool f64, size_t smem, int* threads, int* ctas_per_sm) {
  int occ = 0;
  const cudaError_t e = f64 ? config_rank1_t<double>(smem, &occ) : config_rank1_t<float>(smem, &occ);
  *threads = f64 ? R1Traits<double>::NT : R1Traits<float>::NT;
  *ctas_per_sm = occ;
  return (int)e;
}

size_t rank1_smem(int L, bool resident, bool f64, bool gj_smem) {
  return r1_smem_bytes(L, resident, f64 ? sizeof(double) : sizeof(float), gj_smem);
}

}  // namespace hfq
