// Set-up and reduction kernels of the sweep library:
//  * bath matrix M of a grid from its G0(tau_k) samples (antiperiodic Toeplitz);
//  * per-chain initial field (Philox) and FP64 Gauss-Jordan Green matrices;
//  * per-call measured-sweep bookkeeping;
//  * per-grid mean over chains and error bars (the paper averages each grid's
//    Green function over 10 to 20 impurity solutions, "Multigrid HF-QMC method").
#include <algorithm>

#include <cuda_fp16.h>

#include "hfq_device.cuh"
#include "hfq_gj.cuh"
#include "hfq_launch.h"

namespace hfq {

__global__ void k_bath_matrix(int L, const double* __restrict__ G0, double* __restrict__ M) {
  const int i = blockIdx.x;
  for (int j = threadIdx.x; j < L; j += blockDim.x)
    M[(size_t)i * L + j] = (i >= j) ? -G0[i - j] : G0[i - j + L];
}

int launch_bath_matrix(int L, const double* G0_tau, double* M, cudaStream_t st) {
  k_bath_matrix<<<L, 128, 0, st>>>(L, G0_tau, M);
  return (int)cudaGetLastError();
}

// colk (L doubles), perm (L ints) and the field (L int8), 16-byte aligned,
// before the workspace
__host__ __device__ inline size_t init_head_bytes(int L) {
  return ((size_t)L * sizeof(double) + (size_t)L * sizeof(int) + (size_t)L + 15) / 16 * 16;
}
// with the workspace in HBM: whether the blocked inversion's panel scratch
// fits after the head
__host__ __device__ inline bool init_blocked(int L) {
  return init_head_bytes(L) + gj_blocked_bytes(L) <= kSmemCap;
}

// M^{-1} of one grid's bath matrix.  M is skew-circulant: M_{ll'} = c(l - l')
// with c(d) = -G0(tau_d) and c(d - L) = -c(d) (the antiperiodic wrap).  The
// plane waves e^{i theta_n l}, theta_n = (2n+1) pi / L (the fermionic
// Matsubara phases of the grid), diagonalise it with eigenvalues
//   mu_n = sum_{d<L} c(d) e^{-i theta_n d},
// so M^{-1} is skew-circulant too, with
//   c'(d) = (1/L) sum_{n<L} Re[e^{i theta_n d} / mu_n]     (real: mu_{L-1-n} = conj mu_n).
// One CTA, O(L^2) FP64 work with a table of e^{i pi m / L}, m < 2L.
__global__ void __launch_bounds__(256) k_bath_inverse(int L, const double* __restrict__ M,
                                                      double* __restrict__ Minv, int* status) {
  extern __shared__ __align__(16) unsigned char dsm[];
  double* twc = reinterpret_cast<double*>(dsm);  // cos(pi m / L), m < 2L
  double* tws = twc + 2 * L;                     // sin(pi m / L)
  double* cc = tws + 2 * L;                      // c(d), d < L
  double* ir = cc + L;                           // Re 1/mu_n
  double* ii = ir + L;                           // Im 1/mu_n
  double* cp = ii + L;                           // c'(d), d < L
  __shared__ int s_bad;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) s_bad = 0;
  for (int m = tid; m < 2 * L; m += nt) sincospi((double)m / (double)L, &tws[m], &twc[m]);
  for (int d = tid; d < L; d += nt) cc[d] = M[(size_t)d * L];  // first column
  __syncthreads();
  for (int n = tid; n < L; n += nt) {
    const int step = 2 * n + 1;  // phase index (2n+1) d mod 2L, advanced per d
    double re = 0.0, im = 0.0;
    int ph = 0;
    for (int d = 0; d < L; ++d) {
      re = fma(cc[d], twc[ph], re);
      im = fma(-cc[d], tws[ph], im);
      ph += step;
      if (ph >= 2 * L) ph -= 2 * L;
    }
    const double den = re * re + im * im;
    if (!(den > 0.0) || !isfinite(den)) atomicOr(&s_bad, 1);
    ir[n] = re / den;
    ii[n] = -im / den;
  }
  __syncthreads();
  if (s_bad) {
    if (tid == 0) atomicOr(status, kStatusSingular);
    return;
  }
  for (int d = tid; d < L; d += nt) {
    const int step = (2 * d) % (2 * L);  // phase index (2n+1) d mod 2L, advanced per n
    double acc = 0.0;
    int ph = d;
    for (int n = 0; n < L; ++n) {
      acc = fma(ir[n], twc[ph], acc);
      acc = fma(-ii[n], tws[ph], acc);
      ph += step;
      if (ph >= 2 * L) ph -= 2 * L;
    }
    cp[d] = acc / (double)L;
  }
  __syncthreads();
  for (int e = tid; e < L * L; e += nt) {
    const int i = e / L, j = e - i * L;
    Minv[e] = i >= j ? cp[i - j] : -cp[i - j + L];
  }
}

int launch_bath_inverse(int L, const double* M, double* Minv, int* status, cudaStream_t st) {
  const size_t smem = 8 * (size_t)L * sizeof(double);
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024)
    e = cudaFuncSetAttribute(k_bath_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return (int)e;
  k_bath_inverse<<<1, 256, smem, st>>>(L, M, Minv, status);
  return (int)cudaGetLastError();
}

// Slices of A = M^{-1} - diag(1 - e^{-sigma lambda s_j}) for the Newton
// refinement (hfq_refine.cuh): every entry x of M^{-1} is written as
//   x = 2^ea sum_{p<6} s_p 2^{-7(p+1)} + (remainder below 2^{ea-43}),
// s_p = rint of the running remainder times 2^7 (|s_0| <= 128, |s_p| <= 64),
// each an integer held exactly in FP16.  M^{-1} is skew-circulant, so one
// 8 x 8 core matrix (rows of A = the MMA's N dimension, columns = K) per
// block diagonal and slice holds it all; entries beyond the matrix's corner
// diagonals are zero.  The table's main diagonal is A_jj for sigma s_j = +1;
// the other value's difference goes into rc->dd; ea covers both.
__device__ __forceinline__ void rf_slice6(double x, int ea, float* q) {
  double y = ldexp(x, kRfBits - ea);
#pragma unroll
  for (int p = 0; p < kRfSlicesA; ++p) {
    const double r = rint(y);
    q[p] = (float)r;
    y = (y - r) * (double)(1 << kRfBits);
  }
}

__global__ void __launch_bounds__(256) k_refine_prep(int L, const double* __restrict__ Minv, double lambda,
                                                     RefineConst* rc, uint16_t* __restrict__ tab) {
  __shared__ double red[8];
  const int tid = threadIdx.x;
  const double a0 = Minv[0] - (1.0 - exp(-lambda)), a1 = Minv[0] - (1.0 - exp(lambda));
  double m = fmax(fabs(a0), fabs(a1));
  for (int d = tid; d < L; d += 256) m = fmax(m, fabs(Minv[(size_t)d * L]));  // c'(d), all d
  m = block_max<256>(m, red);
  int ea = 0;
  if (m > 0.0) (void)frexp(m, &ea);  // m < 2^ea
  if (blockIdx.x == 0 && tid == 0) {
    rc->ea = ea;
    float q0[kRfSlicesA], q1[kRfSlicesA];
    rf_slice6(a0, ea, q0);
    rf_slice6(a1, ea, q1);
    for (int p = 0; p < kRfSlicesA; ++p) rc->dd[p] = q1[p] - q0[p];
  }
  const int ncore = rf_ncore(L), nj = rf_nj(L);
  for (int e = blockIdx.x * 256 + tid; e < ncore * 64; e += gridDim.x * 256) {
    const int d = 8 * (e / 64 - (nj - 1)) + ((e >> 3) & 7) - (e & 7);  // i - j
    double x = 0.0;
    if (d == 0)
      x = a0;
    else if (d > 0 && d < L)
      x = Minv[(size_t)d * L];
    else if (d < 0 && d > -L)
      x = Minv[-d];
    float q[kRfSlicesA];
    rf_slice6(x, ea, q);
    for (int p = 0; p < kRfSlicesA; ++p)
      tab[(size_t)p * ncore * 64 + e] = __half_as_ushort(__float2half_rn(q[p]));
  }
}

int launch_refine_prep(int L, const double* Minv, double lambda, RefineConst* rc, uint16_t* tab, cudaStream_t st) {
  k_refine_prep<<<(rf_ncore(L) * 64 + 255) / 256, 256, 0, st>>>(L, Minv, lambda, rc, tab);
  return (int)cudaGetLastError();
}

// The chain's accumulators zeroed; its counters too on the first bath.
template <int NT>
__device__ __forceinline__ void reset_chain(const ItemPtrs& ip, int L, int first_time) {
  const int tid = threadIdx.x;
  for (int k = tid; k < 2 * L; k += NT) ip.acc[k] = 0.0;
  for (int k = tid; k < kBins * L; k += NT) ip.bins[k] = 0.0;
  for (int k = tid; k < 1 + kBins; k += NT) ip.accD[k] = 0.0;
  if (tid == 0) {
    ChainCounters c;
    if (first_time) {
      c.t = 0;
      c.proposals = 0;
      c.accepted = 0;
      c.recomputes = 0;
      c.hash = kFnvOffset;
      c.bad = 0;
      c.status = 0;
      c.fallbacks = 0;
    } else {
      c = *ip.cnt;
    }
    c.drift = 0.0;
    *ip.cnt = c;
  }
}

// Initial (or, after a new bath, rebuilt) Green matrices of every chain of a
// grid: block (chain, spin), so the two spins of a chain are inverted by two
// CTAs at once.  The spin-up block also resets the chain's accumulators.
// kCtas: CTAs per SM that the registers are bounded for. Three (80 registers)
// where as many are needed and fit: 200 chains at L = 170, both spins, are 400
// CTAs on 152 SMs and take 4.3 ms, with two per SM in two waves 6.0. Otherwise
// unbounded, which is 1 % faster per CTA.
template <typename T, int kCtas>
__global__ void __launch_bounds__(256, kCtas) k_init_chains(SweepArgs a, const GridConst* gptr, int item0,
                                                     int first_time) {
  constexpr int NT = 256;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double red[NT / 32];
  __shared__ int redi[NT / 32];
  __shared__ double s_inv;
  __shared__ int s_piv;
  const int tid = threadIdx.x, sp = blockIdx.y;
  const ItemPtrs ip = a.items[item0 + blockIdx.x];
  const GridConst gc = *gptr;
  const int L = gc.L;
  double* colk = reinterpret_cast<double*>(dsm);
  int* perm = reinterpret_cast<int*>(colk + L);
  int8_t* sf = reinterpret_cast<int8_t*>(perm + L);
  double* W = gc.gj_smem ? reinterpret_cast<double*>(dsm + init_head_bytes(L)) : ip.ws + (size_t)sp * L * L;
  // workspace in HBM: inverted by panels when their scratch fits after the head
  double* pan = !gc.gj_smem && init_blocked(L) ? reinterpret_cast<double*>(dsm + init_head_bytes(L)) : nullptr;
  // the field: drawn afresh (both blocks draw the same values; the spin-up
  // block stores it) or the chain's current one
  for (int l = tid; l < L; l += NT) {
    const int8_t v = first_time ? initial_spin(l, ip.chain, ip.grid, a.seed) : ip.s[l];
    sf[l] = v;
    if (first_time && sp == 0) ip.s[l] = v;
  }
  __syncthreads();
  T* G = reinterpret_cast<T*>(ip.G);
  if (pan)
    recompute_green_inv<T, NT, true>(gc, sf, G, G + (size_t)L * L, L, W, red, redi, &s_inv, &s_piv, colk,
                                     perm, false, a.status, sp, sp + 1, pan);
  else
    recompute_green_inv<T, NT>(gc, sf, G, G + (size_t)L * L, L, W, red, redi, &s_inv, &s_piv, colk, perm,
                               false, a.status, sp, sp + 1);
  if (sp != 0) return;
  reset_chain<NT>(ip, L, first_time);
}

// The same with the workspace in HBM, inverted by panels, np CTAs (a cluster)
// per matrix with a share of the columns each.  Bound by the FP64 pipe (L^3
// DFMA) of the SMs that have a CTA: 128 chains at L = 500 are 256 inversions on
// 152 SMs, two waves of 37 ms, and 16 chains at L = 200 leave 120 SMs idle.  For
// a particle-hole symmetric bath only spin up is inverted and G_dn = 1 - G_up^T
// taken from the FP64 inverse before it is rounded (gridDim.y = 1): half the
// work, and room for twice the CTAs per matrix.  hfqmc_set_G0 (the whole call):
// L = 500, 128 chains 74.9 -> 37.8 ms; L = 240, 64 chains 4.4 -> 2.9; L = 200,
// 16 chains 2.7 -> 1.4; L = 100, 256 chains 1.7 -> 0.95.  Every CTA reduces all
// panels (the serial part), so np CTAs gain less than np times.
template <typename T>
__global__ void __launch_bounds__(256) k_init_chains_cluster(SweepArgs a, const GridConst* gptr, int item0,
                                                             int first_time, int np) {
  constexpr int NT = 256, NW = NT / 32;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double red[NW];
  __shared__ int redi[NW];
  __shared__ double s_inv;
  __shared__ int s_piv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sp = blockIdx.y;
  const int part = blockIdx.x % np;
  const ItemPtrs ip = a.items[item0 + blockIdx.x / np];
  const GridConst gc = *gptr;
  const int L = gc.L;
  const bool mirror = gridDim.y == 1;
  double* colk = reinterpret_cast<double*>(dsm);
  int* perm = reinterpret_cast<int*>(colk + L);
  int* pos = reinterpret_cast<int*>(colk);
  int8_t* sf = reinterpret_cast<int8_t*>(perm + L);
  double* W = ip.ws + (size_t)sp * L * L;
  double* pan = reinterpret_cast<double*>(dsm + init_head_bytes(L));
  for (int l = tid; l < L; l += NT) sf[l] = first_time ? initial_spin(l, ip.chain, ip.grid, a.seed) : ip.s[l];
  __syncthreads();
  // B = M^{-1} (1 + D) - D, a share of the rows each
  const int sig = sp ? -1 : 1;
  for (int i = part * NW + warp; i < L; i += np * NW) {
    const double* Mi = gc.Minv + (size_t)i * L;
    double* Wi = W + (size_t)i * L;
    for (int j = lane; j < L; j += 32) {
      const double d = (sig * (int)sf[j] > 0) ? gc.dV[0] : gc.dV[1];
      __stcg(Wi + j, Mi[j] * (1.0 + d) - ((i == j) ? d : 0.0));
    }
  }
  cluster_barrier();  // also: every CTA of the cluster has read the field
  if (gj_invert_blocked<NT, true>(W, L, red, redi, &s_inv, &s_piv, perm, pos, pan, part, np) != 0) {
    if (tid == 0 && part == 0) atomicOr(a.status, kStatusSingular);
  } else {
    T* G = reinterpret_cast<T*>(ip.G) + (size_t)sp * L * L;
    T* Gd = reinterpret_cast<T*>(ip.G) + (size_t)L * L;
    bool finite = true;
    for (int i = part * NW + warp; i < L; i += np * NW) {
      const double* Si = W + (size_t)perm[i] * L;
      for (int j = lane; j < L; j += 32) {
        const double gn = __ldcg(Si + pos[j]);
        finite = finite && isfinite(gn);
        G[(size_t)i * L + j] = (T)gn;
        if (mirror) Gd[(size_t)j * L + i] = (T)((i == j ? 1.0 : 0.0) - gn);
      }
    }
    if (!finite) atomicOr(a.status, kStatusNonFinite);
  }
  if (sp != 0 || part != 0) return;
  if (first_time)
    for (int l = tid; l < L; l += NT) ip.s[l] = sf[l];
  reset_chain<NT>(ip, L, first_time);
}

size_t init_smem(int L, bool gj_smem) {
  return init_head_bytes(L) + (gj_smem ? gj_smem_bytes(L) : (init_blocked(L) ? gj_blocked_bytes(L) : 0));
}

int launch_init_chains(const SweepArgs& a, const GridConst* d_grid_ptr, int item0, int n_chains,
                       int L, bool f64, bool first_time, bool gj_smem, bool has_U, bool mirror, int n_sm,
                       cudaStream_t st) {
  const size_t sm = init_smem(L, gj_smem);
  if (!gj_smem && init_blocked(L) && has_U) {
    const int spins = mirror ? 1 : 2;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    // The most CTAs per matrix (a portable cluster) for which each has an SM to
    // itself and all matrices are worked on at once.  CTAs that share an SM
    // share its FP64 pipe and repeat each other's panel reductions (64 chains
    // at L = 120, one spin: 0.87 ms with three per matrix, 0.65 with two; 100
    // matrices at L = 240: 4.7 ms with two, 4.3 by k_init_chains, which np = 1
    // without the mirror therefore leaves it to).  Not only powers of two: 24
    // grids of 42 to 46 chains, L = 80 .. 320, take 84 ms with one CTA per
    // matrix and both spins inverted, 59 with powers of two, 47 with this.
    // A cluster lies within one GPC, whose SMs need not divide by np: how many
    // fit is asked for CTAs that take more than half an SM's shared memory, so
    // that no two count as fitting on one.  With the number of SMs alone as the
    // limit, the left-over clusters doubled up: 50 matrices at L = 100 took 0.69
    // ms with three CTAs each, 0.54 with two (0.62 by k_init_chains); 30 at
    // L = 256 3.1 with five, 1.9 with four.
    const size_t alone = std::max(sm, (size_t)116 * 1024);
    auto go = [&](auto* f) {
      cudaError_t r = raise_smem_limit(f, alone);
      if (r != cudaSuccess) return (int)r;
      int np = 8;
      cfg.dynamicSmemBytes = alone;
      for (; np > 1; --np) {
        if (L < 32 * np || np * n_chains * spins > n_sm) continue;
        at[0].val.clusterDim.x = np;
        cfg.gridDim = dim3(n_chains * np, spins);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, f, &cfg) != cudaSuccess) (void)cudaGetLastError();
        if (n >= n_chains * spins) break;
      }
      cfg.dynamicSmemBytes = sm;
      if (np == 1 && !mirror) return -1;
      at[0].val.clusterDim.x = np;
      cfg.gridDim = dim3(n_chains * np, spins);
      return (int)cudaLaunchKernelEx(&cfg, f, a, d_grid_ptr, item0, first_time ? 1 : 0, np);
    };
    const int r = f64 ? go(k_init_chains_cluster<double>) : go(k_init_chains_cluster<float>);
    if (r >= 0) return r;
  }
  const auto go1 = [&](auto* f) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return (int)e;
    f<<<dim3(n_chains, 2), 256, sm, st>>>(a, d_grid_ptr, item0, first_time ? 1 : 0);
    return (int)cudaGetLastError();
  };
  // three per SM: 228 KB of shared memory, 1 KB of it reserved per CTA
  const bool three = n_chains > n_sm && 3 * (sm + 1024) <= 228 * 1024;
  if (f64) return three ? go1(k_init_chains<double, 3>) : go1(k_init_chains<double, 1>);
  return three ? go1(k_init_chains<float, 3>) : go1(k_init_chains<float, 1>);
}

// Measured sweep m (0-based within one call of n_meas) goes to bin floor(32 m / n_meas);
// bin b therefore receives ceil((b+1) n / 32) - ceil(b n / 32) sweeps.
__global__ void k_account(GridAccount* acc, int n_grids, long long n_meas) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n_grids || n_meas <= 0) return;
  acc[g].n_meas += n_meas;
  for (int b = 0; b < kBins; ++b) {
    const long long lo = ((long long)b * n_meas + kBins - 1) / kBins;
    const long long hi = ((long long)(b + 1) * n_meas + kBins - 1) / kBins;
    acc[g].bin_count[b] += hi - lo;
  }
}

int launch_account(GridAccount* acc, int n_grids, long long n_meas, cudaStream_t st) {
  k_account<<<(n_grids + 127) / 128, 128, 0, st>>>(acc, n_grids, n_meas);
  return (int)cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_reduce(const GridConst* grids, const ItemPtrs* items,
                                                const GridAccount* acc, GridOut* gout,
                                                double* outG, double* outErr,
                                                const long long* out_off) {
  const int g = blockIdx.x, tid = threadIdx.x;
  const GridConst gc = grids[g];
  const int L = gc.L, nc = gc.chains, i0 = gc.item0;
  const GridAccount& A = acc[g];
  const double N = (double)A.n_meas;
  double* oG = outG + out_off[g];
  double* oE = outErr + out_off[g];
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  for (int k = tid; k < L; k += blockDim.x) {
    double mean = nan, err = nan;
    if (A.n_meas > 0) {
      if (nc >= 2) {
        double s = 0.0;
        for (int c = 0; c < nc; ++c) {
          const double* ac = items[i0 + c].acc;
          s += -(ac[k] + ac[L + k]) / (2.0 * N);
        }
        mean = s / nc;
        double v = 0.0;
        for (int c = 0; c < nc; ++c) {
          const double* ac = items[i0 + c].acc;
          const double d = -(ac[k] + ac[L + k]) / (2.0 * N) - mean;
          v += d * d;
        }
        err = sqrt(v / (nc - 1) / nc);
      } else {
        const ItemPtrs ip = items[i0];
        mean = -(ip.acc[k] + ip.acc[L + k]) / (2.0 * N);
        int nb = 0;
        double s = 0.0;
        for (int b = 0; b < kBins; ++b)
          if (A.bin_count[b] > 0) {
            s += -ip.bins[(size_t)b * L + k] / (double)A.bin_count[b];
            ++nb;
          }
        if (nb >= 2) {
          const double bm = s / nb;
          double v = 0.0;
          for (int b = 0; b < kBins; ++b)
            if (A.bin_count[b] > 0) {
              const double d = -ip.bins[(size_t)b * L + k] / (double)A.bin_count[b] - bm;
              v += d * d;
            }
          err = sqrt(v / (nb - 1) / nb);
        }
      }
    }
    oG[k] = mean;
    oE[k] = err;
  }
  __syncthreads();
  if (tid == 0) {
    oG[L] = -1.0 - oG[0];
    oE[L] = oE[0];
    GridOut o;
    o.proposals = o.accepted = o.recomputes = o.bad = o.fallbacks = 0;
    o.drift = 0.0;
    for (int c = 0; c < nc; ++c) {
      const ChainCounters cc = *items[i0 + c].cnt;
      o.proposals += cc.proposals;
      o.accepted += cc.accepted;
      o.recomputes += cc.recomputes;
      o.bad += cc.bad;
      o.fallbacks += cc.fallbacks;
      o.drift = fmax(o.drift, cc.drift);
    }
    o.D = nan;
    o.D_err = nan;
    if (A.n_meas > 0) {
      if (nc >= 2) {
        double s = 0.0, v = 0.0;
        for (int c = 0; c < nc; ++c) s += items[i0 + c].accD[0] / N;
        const double m = s / nc;
        for (int c = 0; c < nc; ++c) {
          const double d = items[i0 + c].accD[0] / N - m;
          v += d * d;
        }
        o.D = m;
        o.D_err = sqrt(v / (nc - 1) / nc);
      } else {
        o.D = items[i0].accD[0] / N;
        int nb = 0;
        double s = 0.0, v = 0.0;
        for (int b = 0; b < kBins; ++b)
          if (A.bin_count[b] > 0) {
            s += items[i0].accD[1 + b] / (double)A.bin_count[b];
            ++nb;
          }
        if (nb >= 2) {
          const double m = s / nb;
          for (int b = 0; b < kBins; ++b)
            if (A.bin_count[b] > 0) {
              const double d = items[i0].accD[1 + b] / (double)A.bin_count[b] - m;
              v += d * d;
            }
          o.D_err = sqrt(v / (nb - 1) / nb);
        }
      }
    }
    gout[g] = o;
  }
}

int launch_reduce(const GridConst* grids, const ItemPtrs* items, const GridAccount* acc,
                  GridOut* gout, double* outG, double* outErr, const long long* out_off,
                  int n_grids, cudaStream_t st) {
  k_reduce<<<n_grids, 256, 0, st>>>(grids, items, acc, gout, outG, outErr, out_off);
  return (int)cudaGetLastError();
}

}  // namespace hfq
