// Green-function entry point that allocates no device memory.
//
// hfqmc_green_noalloc() computes, for one HS field s, the FP64 Green matrices
// of both spins, G^sigma = [1 + (1 - M)(e^{sigma lambda s} - 1)]^{-1} M, with
// M the antiperiodic bath matrix built from G0(tau_k) -- the same arithmetic
// that hfqmc_set_G0 runs for every chain of a context -- for callers that
// cannot allocate device memory (a host runtime that owns every device
// buffer through its own pool, a plugin that is not allowed to touch the
// CUDA allocator, code that runs where cudaMalloc is forbidden).  They pass
// their own device buffers for the inputs and outputs; the bath matrix and
// the Gauss-Jordan workspace live in shared memory or in the file-scope array below.
#include <cmath>
#include <cstdint>

#include <cuda_runtime.h>

#include "../../include/hfqmc.h"
#include "hfq_device.cuh"
#include "hfq_gj.cuh"
#include "hfq_launch.h"

namespace hfq {

// Scratch of the entry point: M (L x L) then [A | M] (L x 2L), FP64, for
// L <= HFQMC_NOALLOC_MAX_L; 1.5 MiB held by every GPU that loads the library
// until the process exits.  Followed by the status words.
constexpr int kNoAllocMaxL = HFQMC_NOALLOC_MAX_L;
constexpr size_t kNoAllocScratchDoubles = 3 * (size_t)kNoAllocMaxL * kNoAllocMaxL + 32;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratchDoubles];

constexpr int kNoAllocNT = 256;

// The elimination of [A | M] updates every column from the pivot columns of A
// alone, so the columns of M may be dealt out: kNoAllocShares CTAs per spin,
// each with its own copy of A and L / kNoAllocShares columns of M in shared
// memory, none waiting for another.  The same operations per entry as by one
// CTA over all of [A | M] (1.5 L^3 DFMA per spin, one spin after the other,
// the workspace in L2), (0.5 + 1 / kNoAllocShares) L^3 of them on the critical
// path.  L = 100: 2.17 ms -> 0.39 ms.
constexpr int kNoAllocShares = 8;

__host__ __device__ inline int noalloc_cols(int L) { return (L + kNoAllocShares - 1) / kNoAllocShares; }
__host__ __device__ inline int noalloc_pitch(int L) { return (L + noalloc_cols(L)) | 1; }
__host__ __device__ inline size_t noalloc_smem(int L) {
  return ((size_t)L * noalloc_pitch(L) + L) * sizeof(double);
}
// whether a share's [A | M] fits in shared memory (L <= 159); else the
// workspace is the scratch array and one CTA does both spins
inline bool noalloc_shared(int L) { return noalloc_smem(L) <= kSmemCap; }

__global__ void __launch_bounds__(kNoAllocNT) k_green_noalloc_shares(GridConst gc, const double* G0_tau,
                                                                     const int8_t* s, double* Gup, double* Gdn,
                                                                     int* status) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double red[kNoAllocNT / 32];
  __shared__ int redi[kNoAllocNT / 32];
  __shared__ double s_inv;
  __shared__ int s_piv;
  const int L = gc.L, ld = noalloc_pitch(L), tid = threadIdx.x;
  const int sig = blockIdx.y ? -1 : 1;
  const int r0 = blockIdx.x * noalloc_cols(L), nr = min(noalloc_cols(L), L - r0);
  int* st = status + blockIdx.y * kNoAllocShares + blockIdx.x;  // this CTA's own word
  double* W = reinterpret_cast<double*>(dsm);
  double* colk = W + (size_t)L * ld;
  if (nr <= 0) {
    if (tid == 0) *st = 0;
    return;
  }
  auto bath = [&](int i, int j) { return i >= j ? -G0_tau[i - j] : G0_tau[i - j + L]; };
  for (int e = tid; e < L * (L + nr); e += kNoAllocNT) {
    const int i = e / (L + nr), c = e - i * (L + nr);
    if (c < L) {
      const double d = (sig * (int)s[c] > 0) ? gc.dV[0] : gc.dV[1];
      const double one = (i == c) ? 1.0 : 0.0;
      W[(size_t)i * ld + c] = one + (one - bath(i, c)) * d;
    } else {
      W[(size_t)i * ld + c] = bath(i, r0 + c - L);
    }
  }
  __syncthreads();
  if (gj_eliminate<kNoAllocNT>(W, L, L + nr, ld, red, redi, &s_inv, &s_piv, colk) != 0) {
    if (tid == 0) *st = kStatusSingular;
    return;
  }
  double* G = blockIdx.y ? Gdn : Gup;
  int bad = 0;
  for (int e = tid; e < L * nr; e += kNoAllocNT) {
    const int i = e / nr, c = e - i * nr;
    const double g = W[(size_t)i * ld + L + c];
    bad |= isfinite(g) ? 0 : 1;
    G[(size_t)i * L + r0 + c] = g;
  }
  bad = __syncthreads_or(bad);
  if (tid == 0) *st = bad ? kStatusNonFinite : 0;
}

// The workspace in the scratch array (M, then [A | M]), one CTA, both spins in
// turn: G0_tau is read before G_up is written, s before G_dn, G_dn last.
__global__ void __launch_bounds__(kNoAllocNT) k_green_noalloc(GridConst gc, const double* G0_tau,
                                                              const int8_t* s, double* Gup,
                                                              double* Gdn, double* scratch) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double red[kNoAllocNT / 32];
  __shared__ int redi[kNoAllocNT / 32];
  __shared__ double s_inv;
  __shared__ int s_piv;
  const int L = gc.L;
  double* M = scratch;
  double* W = scratch + (size_t)L * L;
  int* status = reinterpret_cast<int*>(scratch + 3 * (size_t)kNoAllocMaxL * kNoAllocMaxL);
  double* colk = reinterpret_cast<double*>(dsm);
  if (threadIdx.x == 0) *status = 0;  // the array keeps the previous call's word
  for (int e = threadIdx.x; e < L * L; e += kNoAllocNT) {
    const int i = e / L, j = e - i * L;
    M[e] = (i >= j) ? -G0_tau[i - j] : G0_tau[i - j + L];
  }
  __syncthreads();
  gc.M = M;
  recompute_green<double, kNoAllocNT>(gc, s, Gup, Gdn, L, W, red, redi, &s_inv, &s_piv, colk,
                                      false, status);
}

}  // namespace hfq

extern "C" int hfqmc_green_noalloc(const double* G0_tau, const int8_t* s, int L, double dtau,
                                   double U, double* G_up, double* G_dn, void* cuda_stream,
                                   int* status_out) {
  using namespace hfq;
  if (L < 1 || L > kNoAllocMaxL) return HFQMC_EINVAL;
  if (!G0_tau || !s || !G_up || !G_dn) return HFQMC_EINVAL;
  if (!(dtau > 0.0) || !(U >= 0.0)) return HFQMC_EINVAL;
  // The host-side name of the array is not a device address: ask the runtime
  // for the array's address on the current device, on every call (a cached
  // address would outlive the context it belongs to after a device reset;
  // the lookup costs little next to the L^3 elimination).
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
    (void)cudaGetLastError();
    return HFQMC_ECUDA;
  }
  double* scratch = static_cast<double*>(p);
  GridConst gc = {};
  gc.L = L;
  gc.lambda = std::acosh(std::exp(0.5 * dtau * U));
  gc.dV[0] = std::exp(gc.lambda) - 1.0;
  gc.dV[1] = std::exp(-gc.lambda) - 1.0;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  double* status_addr = scratch + 3 * (size_t)kNoAllocMaxL * kNoAllocMaxL;
  // The shares read G0_tau and s while others already write, in no order: where
  // a buffer overlaps another, one CTA takes the call, in the order stated there
  const size_t gbytes = sizeof(double) * (size_t)L * L;
  const auto overlap = [](const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + nb && y < x + na;
  };
  bool apart = !overlap(G_up, gbytes, G_dn, gbytes);
  for (const double* G : {G_up, G_dn})
    apart = apart && !overlap(G, gbytes, G0_tau, sizeof(double) * L) && !overlap(G, gbytes, s, L);
  int n_words = 1;
  if (apart && noalloc_shared(L)) {
    if (raise_smem_limit(k_green_noalloc_shares, noalloc_smem(L)) != cudaSuccess) return HFQMC_ECUDA;
    n_words = 2 * kNoAllocShares;
    k_green_noalloc_shares<<<dim3(kNoAllocShares, 2), kNoAllocNT, noalloc_smem(L), st>>>(
        gc, G0_tau, s, G_up, G_dn, reinterpret_cast<int*>(status_addr));
  } else {
    k_green_noalloc<<<1, kNoAllocNT, (size_t)L * sizeof(double), st>>>(gc, G0_tau, s, G_up, G_dn, scratch);
  }
  if (cudaGetLastError() != cudaSuccess) return HFQMC_ECUDA;
  int words[2 * kNoAllocShares] = {0};
  if (cudaMemcpyAsync(words, status_addr, n_words * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return HFQMC_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return HFQMC_ECUDA;
  int word = 0;
  for (int i = 0; i < n_words; ++i) word |= words[i];
  if (status_out) *status_out = word;
  return (word & (kStatusSingular | kStatusNonFinite)) ? HFQMC_ENUMERIC : HFQMC_OK;
}
