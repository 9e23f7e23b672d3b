// Delayed (rank-k) FP32 Hirsch-Fye sweep: one CTA per Markov chain,
// persistent over the longest-Lambda-first work queue.
//
// The accepted flips of a chain are not applied one by one.  After j accepted
// flips since the last flush the current Green matrix is
//     G_cur = G + U W^T,   U, W: L x j panels (per spin),
// and an accepted flip at slice l appends
//     u = G_cur[:, l] - e_l,           w = (Delta / R) G_cur[l, :],
// whose entries cost O(j) each (the base column / row entry plus a length-j
// dot product with the panels).  Every k accepted flips the panels are
// flushed, G += U W^T -- a dense L x L x k contraction per spin (tcgen05
// tensor cores with scaled split FP16, or FP32 FMA).  In exact arithmetic this is
// the Hirsch-Fye rank-1 update applied k times; only the rounding differs.
// The panels are also flushed before every measurement and every FP64
// recompute (every n_wrap accepted flips).
//
// Work split (16 warps): thread t owns spin (t & 1) of rows r = t/2 + 256 q.  For its
// rows it appends the panel entries, keeps the current diagonal G_cur[r][r]
// in registers, swaps it with its partner thread (the other spin) by one
// shuffle, and right away evaluates slice r as the next proposal (flip ratio
// from the new diagonals, Philox uniform drawn at the start of the sweep).
// Rejections change nothing, so the next accepted slice is the lowest r > l
// that accepts: every warp leaves the lowest of its rows, with its diagonal, in
// a slot of its own, and after one barrier per accepted flip each warp takes
// the minimum of the slots and each thread divides for its flip factor while
// G's column and row are on their way.  (With one atomicMin for all warps, the
// division before the barrier and a branch around every load, 256 chains at
// Lambda = 100 took 86 ms for 550 sweeps; they take 69.)
#include "hfq_delayed.cuh"
#include "hfq_device.cuh"
#include "hfq_gj.cuh"
#include "hfq_launch.h"
#include "hfq_refine.cuh"

namespace hfq {

static_assert(kTileN == kDelayedTile, "tensor-map box and flush tile must agree");

constexpr int kRowsPerThread = 2;  // rows t/2 + 256 q, q < 2: L <= 512
constexpr int kRowStride = kDelNT / 2;
constexpr int kNoSlice = 0x7fffffff;

// Where a chain stands between two stretches of its sweeps (see the kernel)
struct SweepPos {
  long long n_acc;
  unsigned long long hash;  // kept up to date by one thread, for the chain's decision hash
  long long t0;             // global index of the call's first sweep
  uint32_t sw;
  int l, par;
  float f[2];               // flip factors of slice l (threads of spin up, of spin down)
};
// What its recomputes have added up to
struct RecTotals {
  double drift;
  long long n_rec;
  int n_fb;  // handed to Gauss-Jordan by the refinement
};

// A chain's constants, in shared memory, and what follows from them.  Each
// scope of the kernel takes its own copy, so that only what it uses is in
// registers there.
struct ChainConst {
  GridConst gc;
  ItemPtrs ip;
  DelLayout lay;
};
constexpr int kChainOff = kRowsPerThread * kRowStride;  // the field takes L <= 512 bytes
static_assert(kChainOff + sizeof(ChainConst) <= 1024, "the head ends at off_body = 1024");
struct ChainView {
  GridConst gc;
  ItemPtrs ip;
  DelLayout lay;
  int L, ld;
  bool resident;
  float *Ggl, *Gu, *Gd;  // G in HBM; the G the sweep works on (row pitch ld)
  int8_t* ss;            // the field, in shared memory
  __device__ __forceinline__ ChainView(const ChainConst& c, unsigned char* smem) : gc(c.gc), ip(c.ip), lay(c.lay) {
    L = gc.L;
    resident = gc.resident != 0;
    ld = resident ? lay.ldS : L;
    Ggl = reinterpret_cast<float*>(ip.G);
    Gu = resident ? reinterpret_cast<float*>(smem + lay.off_G) : Ggl;
    Gd = Gu + (size_t)L * ld;
    ss = reinterpret_cast<int8_t*>(smem + lay.off_s);
  }
};

// The fallback and the contexts that do not refine: out of line, it is rare or
// long, and its FP64 registers are not the sweep's.
__device__ __noinline__ double recompute_from_scratch(unsigned char* smem, float* Gu, float* Gd, int ld, int n_spins,
                                                      double* red, int* redi, double* s_inv, int* s_piv, int* status) {
  const ChainConst& c = *reinterpret_cast<const ChainConst*>(smem + kChainOff);
  // FP64 workspace in HBM, inverted by panels whose scratch overlays the idle
  // part of shared memory (never G)
  return recompute_green_inv<float, kDelNT, true>(
      c.gc, reinterpret_cast<const int8_t*>(smem + c.lay.off_s), Gu, Gd, ld, c.ip.ws, red, redi, s_inv, s_piv,
      reinterpret_cast<double*>(smem + c.lay.off_colk), reinterpret_cast<int*>(smem + c.lay.off_perm), true, status, 0,
      n_spins, reinterpret_cast<double*>(smem + c.lay.off_gjb));
}

// A chain runs as stretches of sweeping between recomputes.  Everything a
// stretch needs is re-derived at its start -- the field from shared memory,
// the uniforms from Philox, the diagonal from G, the rest from SweepPos -- so
// that no sweep state is live across the recompute: its code, which needs
// every register itself, leaves the accept loop's registers alone (with the
// refinement inside the loop the compiler spilled 300 bytes of both).
//
// kRecord: every accepted flip also sets its bit in the chain's decision
// trace (a.trace_mode == kTraceRecord), for replay by an FP64 run.
// kRefine: the recompute tries the Newton refinement (grids with a
// RefineConst) before Gauss-Jordan; without it the kernel carries only the
// Gauss-Jordan recompute (the refinement's code costs the accept loop some
// registers, so contexts that never refine launch the variant without it).
// kMirror (every grid's bath particle-hole symmetric, so G_dn = 1 - G_up^T
// for every field): the sweep keeps G_up only.  A thread pair owns a row of
// G_up: the even thread appends its column entry u_i, the odd one its row
// entry w_i, and they swap them by one shuffle; G_dn's diagonal is 1 minus
// G_up's, its measured sums follow from G_up's (diagonal L - k for k > 0),
// and the chain's G_dn is written as 1 - G_up^T when the chain ends.
template <bool kRecord, bool kRefine, bool kMirror = false>
__global__ void __launch_bounds__(kDelNT, 1) k_sweep_delayed(SweepArgs a) {
  constexpr int NT = kDelNT;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ double red[NW];
  __shared__ int redi[NW];
  __shared__ double s_inv;
  __shared__ int s_piv, s_item;
  __shared__ int s_bad;
  __shared__ uint32_t s_tmem_base;
  __shared__ __align__(8) unsigned long long s_mbar[12];
  __shared__ RfSync s_rf;
  __shared__ SweepPos s_pos;
  __shared__ RecTotals s_rec;
  // in the head of dynamic shared memory, behind the field (static shared memory is kept to
  // the 512 bytes that kSmemCap leaves)
  ChainConst& s_chain = *reinterpret_cast<ChainConst*>(smem + kChainOff);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool use_tc = a.flush != 2;
  TcState tc;
  if (use_tc) tc_setup(&tc, &s_tmem_base, s_mbar, a.status);
  if (tid == 0) s_rf = RfSync{0u, 0u, 0u};

  for (;;) {
    if (tid == 0) s_item = atomicAdd(a.queue_head, 1);
    __syncthreads();
    const int q = s_item;
    __syncthreads();
    if (q >= a.n_items) break;
    if (tid == 0) {
      s_chain.ip = a.items[a.order[q]];
      s_chain.gc = a.grids[s_chain.ip.grid];
      const GridConst& gc = s_chain.gc;
      s_chain.lay = del_layout(gc.L, gc.k, gc.resident != 0, gc.gj_smem != 0, gc.gtile != 0, gc.ub, gc.rc != nullptr,
                               kMirror ? 1 : 2);
    }
    __syncthreads();
    {
    const ChainView v(s_chain, smem);
    const ItemPtrs& ip = v.ip;
    const int L = v.L, ld = v.ld;
    const bool resident = v.resident;
    float *const Ggl = v.Ggl, *const Gu = v.Gu;
    int8_t* const ss = v.ss;
    if (resident) {
      for (int i = warp; i < (kMirror ? 1 : 2) * L; i += NW)
        for (int jj = lane; jj < L; jj += 32) Gu[(size_t)i * ld + jj] = Ggl[(size_t)i * L + jj];
    }
    for (int l = tid; l < L; l += NT) ss[l] = ip.s[l];
    if (tid == 0) {
      s_bad = 0;
      s_pos = SweepPos{ip.cnt->accepted, ip.cnt->hash, ip.cnt->t, 0u, -1, 0, {0.f, 0.f}};
      s_rec = RecTotals{ip.cnt->drift, 0, 0};
    }
    __syncthreads();
    }

    for (;;) {
    bool done, recompute;
    {  // a stretch of sweeping
    const ChainView v(s_chain, smem);
    const GridConst& gc = v.gc;
    const ItemPtrs& ip = v.ip;
    const DelLayout& lay = v.lay;
    const int L = v.L, ld = v.ld;
    const bool resident = v.resident;
    float *const Ggl = v.Ggl, *const Gu = v.Gu, *const Gd = v.Gd;
    int8_t* const ss = v.ss;
    const int K = gc.k;
    // product tile buffer of the TMA reduce flush (G in HBM, tensor map set)
    float* dtile = gc.gtile ? reinterpret_cast<float*>(smem + lay.off_gtile) : nullptr;
    float* Pu = reinterpret_cast<float*>(smem + lay.off_U);  // [2][L][KP] (spin stride padded): U panels
    float* Pw = reinterpret_cast<float*>(smem + lay.off_W);  // [2][L][KP]: W panels
    // [2][warps that own rows]: each warp's lowest accepting slice, G_up's and
    // G_dn's diagonal there and its field, by rounds of two
    int4* slots = reinterpret_cast<int4*>(smem + lay.off_diag);
    const int nwa = min(NW, (L + 15) >> 4);
    const bool active = warp < nwa;  // this warp owns rows (warp-uniform)
    unsigned char* stage = smem + lay.off_stage;
    const int KP = lay.KP;
    const int panel_floats4 = del_panel_floats(L, KP, kMirror ? 1 : 2) / 4;  // one panel, the kept spins
    auto zero_panels = [&]() {
      for (int e = tid; e < 2 * panel_floats4; e += NT)
        reinterpret_cast<float4*>(e < panel_floats4 ? Pu : Pw)[e < panel_floats4 ? e : e - panel_floats4] =
            make_float4(0.f, 0.f, 0.f, 0.f);
    };
    const float d0 = gc.deltaf[0], d1 = gc.deltaf[1];
    const int rule = a.accept_rule;
    const uint32_t n_sweeps = (uint32_t)(a.n_warm + a.n_meas), n_warm = (uint32_t)a.n_warm;  // at most 2^31 a call
    // per-thread row state: this spin's current diagonal, field, this sweep's uniform
    const int sp = tid & 1;
    const int row0 = tid >> 1;
    float dg[kRowsPerThread], uv[kRowsPerThread];
    int sv[kRowsPerThread];
    bool lastbad[kRowsPerThread];
    float* Gs = (sp && !kMirror) ? Gd : Gu;
    // G_up only: W starts 16 floats into its region (sized one spin plus 16
    // floats), so row r of U and row r of W lie in different shared-memory
    // banks (see the append)
    float* const Pw1 = kMirror ? Pw + 16 : Pw;
    float* Us = Pu + (size_t)(kMirror ? 0 : sp) * del_spin_stride(L, KP);
    float* Ws = Pw1 + (size_t)(kMirror ? 0 : sp) * del_spin_stride(L, KP);
    auto load_diag = [&]() {
#pragma unroll
      for (int qq = 0; qq < kRowsPerThread; ++qq) {
        if (qq * kRowStride >= L) break;  // uniform: rows beyond the grid
        const int r = row0 + qq * kRowStride;
        if (r < L) dg[qq] = Gs[(size_t)r * ld + r];
      }
    };
    uint32_t sw = s_pos.sw;
    int l = s_pos.l;  // next accepted slice; -1: the sweep begins
    int par = s_pos.par;  // slots of the current round
    float f = s_pos.f[tid & 1];  // its flip factor, of this thread's spin
    auto draw_uniforms = [&](long long t) {
#pragma unroll
      for (int qq = 0; qq < kRowsPerThread; ++qq) {
        if (qq * kRowStride >= L) break;  // uniform: rows beyond the grid
        const int r = row0 + qq * kRowStride;
        if (r < L) uv[qq] = proposal_uniform_f32(r, t, ip.chain, ip.grid, a.seed);
      }
    };
#pragma unroll
    for (int qq = 0; qq < kRowsPerThread; ++qq) {
      if (qq * kRowStride >= L) break;  // uniform: rows beyond the grid
      const int r = row0 + qq * kRowStride;
      sv[qq] = r < L ? ss[r] : 1;
      uv[qq] = 0.f;
      lastbad[qq] = false;
      dg[qq] = 0.f;
    }
    if (l >= 0) draw_uniforms(s_pos.t0 + sw);  // mid-sweep: this sweep's uniforms again
    load_diag();
    zero_panels();  // also after a recompute, whose workspace may have overlaid them
    // accepted flips until the next recompute (the cumulative count reaches a
    // multiple of n_wrap), or the longest stretch when there is none; counted
    // down so the hot loop needs no 64-bit count
    const int stretch = gc.n_wrap > 0 ? (int)(gc.n_wrap - s_pos.n_acc % gc.n_wrap) : 0x7fffffff;
    int left = stretch;
    int n_bad = 0;
    int j = 0;     // pending flips in the panels
    uint32_t exq = 0u;  // biased exponents of this thread's largest appended |u| (byte 0), |w| (byte 1)
    __syncthreads();

    // G += U W^T for both spins, then the diagonals are re-read from G.
    auto flush = [&]() {
      if (j == 0) return;
      if (use_tc)
        flush_tcgen05<kMirror ? 1 : 2>(&tc, Gu, Gd, ld, Pu, Pw1, KP, L, j, stage, lay, a.status,
                                       reinterpret_cast<uint32_t*>(red), exq, dtile, gc.tmapG, ip.chain);
      else
        flush_ffma<kMirror ? 1 : 2>(Gu, Gd, ld, Pu, Pw1, KP, L, j);
      __syncthreads();
      load_diag();
      j = 0;
      exq = 0u;
      // the panels restart from zeros, so the dot products may run over whole
      // 16-byte chunks past column j
      zero_panels();
      __syncthreads();
    };

    // Evaluates the owned slices r >= lo as proposals with the current
    // diagonals of both spins (partner threads swap theirs); the warp's lowest
    // accepting slice goes to its slot of this round (read after the next
    // barrier; written again only after the barrier that follows).
    auto propose = [&](int lo) {
      if (!active) return;
      int cand = kNoSlice, own = 0, cs = 0;
      float cgu = 0.f, cgd = 0.f;
#pragma unroll
      for (int qq = 0; qq < kRowsPerThread; ++qq) {
        if (qq * kRowStride >= L) break;  // uniform: rows beyond the grid
        const int r = row0 + qq * kRowStride;
        float gu, gd;
        if constexpr (kMirror) {
          gu = dg[qq];  // both threads of the pair hold G_up's diagonal
          gd = 1.f - gu;
        } else {
          const float other = __shfl_xor_sync(0xffffffffu, dg[qq], 1);
          gu = sp ? other : dg[qq];
          gd = sp ? dg[qq] : other;
        }
        bool bad;
        const bool in = r < L && r >= lo;
        const bool acc = del_decide(d0, d1, gu, gd, sv[qq], uv[qq], rule, &bad) && in;
        lastbad[qq] = bad && in && sp == 0;
        const unsigned b = __ballot_sync(0xffffffffu, acc) & 0x55555555u;
        if (b && cand == kNoSlice) {  // warp-uniform
          own = __ffs(b) - 1;
          cand = qq * kRowStride + warp * 16 + (own >> 1);
          cgu = gu;
          cgd = gd;
          cs = sv[qq];
        }
      }
      if (lane == own) slots[par * nwa + warp] = make_int4(cand, __float_as_int(cgu), __float_as_int(cgd), cs);
    };

    // After the barrier of a round: the lowest of the slots, and this thread's
    // flip factor Delta / R (its spin's; spin up's for a mirrored sweep).  Also
    // counts the bad ratios among the proposals this round decided, i.e. the
    // owned slices in [lo, next].
    auto take_next = [&](int lo) -> int {
      const int4* round = slots + par * nwa;
      const int nxt = __reduce_min_sync(0xffffffffu, round[min(lane, nwa - 1)].x);
      const int4 w = round[nxt < L ? (nxt >> 4) & (NW - 1) : 0];
      par ^= 1;
      const bool plus = (w.w > 0) == (kMirror || sp == 0);
      const float del = plus ? d0 : d1, g = __int_as_float(kMirror || sp == 0 ? w.y : w.z);
      f = del / __fadd_rn(1.f, __fmul_rn(__fsub_rn(1.f, g), del));
      const int hi = nxt < L ? nxt : L - 1;
#pragma unroll
      for (int qq = 0; qq < kRowsPerThread; ++qq) {
        if (qq * kRowStride >= L) break;  // uniform: rows beyond the grid
        const int r = row0 + qq * kRowStride;
        if (r >= lo && r <= hi && lastbad[qq]) ++n_bad;
      }
      return nxt;
    };

    for (; sw < n_sweeps; ++sw) {
      if (l < 0) {
        draw_uniforms(s_pos.t0 + sw);
        propose(0);
        __syncthreads();
        l = take_next(0);
      }
      while (l < L) {
        if (active) {
          // base G entries of every owned row first (before any panel store), so
          // their latency -- L2 when G lives in HBM -- overlaps the dot products.
          // Rows beyond the grid repeat the last one and store nothing; no load
          // sits behind a branch.
          float gc_q[kRowsPerThread], gr_q[kRowsPerThread];  // column / row entry (mirrored: the thread's one of them)
          auto base_entries = [&](const float* g, int gld) {
#pragma unroll
            for (int qq = 0; qq < kRowsPerThread; ++qq) {
              if (qq * kRowStride >= L) break;  // uniform: rows beyond the grid
              const int i = min(row0 + qq * kRowStride, L - 1);
              if constexpr (kMirror) {
                gc_q[qq] = g[sp ? l * gld + i : i * gld + l];
              } else {
                gc_q[qq] = g[i * gld + l];  // 2 L^2 < 2^31: 32-bit offsets
                gr_q[qq] = g[l * gld + i];
              }
            }
          };
          // one spin: G in shared memory and in HBM told apart in the code; two:
          // one copy through the general pointer, their kernel spills more with two
          if constexpr (!kMirror)
            base_entries(Gs, ld);
          else if (resident)
            base_entries(reinterpret_cast<const float*>(smem + lay.off_G), ld);
          else
            base_entries(Ggl, L);
#pragma unroll
          for (int qq = 0; qq < kRowsPerThread; ++qq) {
            if (qq * kRowStride >= L) break;  // uniform: rows beyond the grid
            const int i0 = row0 + qq * kRowStride, i = min(i0, L - 1);
            const int oi = i * KP, ol = l * KP;  // 32-bit shared-memory offsets
            float c4[4] = {0.f, 0.f, 0.f, 0.f};
            if constexpr (kMirror) {
              // the panels are zero past column j: whole groups of eight columns
              const int j8 = (j + 7) >> 3;
              auto dot = [&](const float4* x, const float4* y, float* acc) {
#pragma unroll 1
                for (int m = 0; m < j8; ++m) {
                  const float4 a1 = x[2 * m], b1 = y[2 * m], a2 = x[2 * m + 1], b2 = y[2 * m + 1];
                  acc[0] = __fmaf_rn(a1.x, b1.x, acc[0]);
                  acc[1] = __fmaf_rn(a1.y, b1.y, acc[1]);
                  acc[2] = __fmaf_rn(a1.z, b1.z, acc[2]);
                  acc[3] = __fmaf_rn(a1.w, b1.w, acc[3]);
                  acc[0] = __fmaf_rn(a2.x, b2.x, acc[0]);
                  acc[1] = __fmaf_rn(a2.y, b2.y, acc[1]);
                  acc[2] = __fmaf_rn(a2.z, b2.z, acc[2]);
                  acc[3] = __fmaf_rn(a2.w, b2.w, acc[3]);
                }
              };
              // spin up only: the even thread of a pair appends u_i (column l),
              // the odd one w_i (row l); one shuffle gives both the pair's values.
              // Even lane: U row i . W row l; odd lane: W row i . U row l.  The
              // first operand reads a distinct row in every lane (U or W, whose
              // rows of one index sit 16 banks apart), the second the pair's two
              // shared rows: both conflict-free
              float* mine_p = sp ? Ws : Us;
              dot(reinterpret_cast<const float4*>(mine_p + oi), reinterpret_cast<const float4*>((sp ? Us : Ws) + ol), c4);
              const float v = gc_q[qq] + ((c4[0] + c4[1]) + (c4[2] + c4[3]));
              const float mine = sp ? v * f : v - ((i == l) ? 1.f : 0.f);
              const float theirs = __shfl_xor_sync(0xffffffffu, mine, 1);
              if (i0 < L) {
                exq = __vmaxu4(exq, ((__float_as_uint(mine) << 1) >> 24) << (sp ? 8 : 0));
                mine_p[oi + j] = mine;
                dg[qq] = __fmaf_rn(mine, theirs, dg[qq]);
              }
            } else {
              // append column j of the panels for the owned rows of this thread's spin
              // (both dot products in one loop, four columns a pass: eight
              // accumulators hide the latency that two loops in turn wait for)
              float r4[4] = {0.f, 0.f, 0.f, 0.f};
              const float4 *Ui = reinterpret_cast<const float4*>(Us + oi), *Wl = reinterpret_cast<const float4*>(Ws + ol);
              const float4 *Ul = reinterpret_cast<const float4*>(Us + ol), *Wi = reinterpret_cast<const float4*>(Ws + oi);
              const int j4 = (j + 3) >> 2;
#pragma unroll 1
              for (int m = 0; m < j4; ++m) {
                const float4 a1 = Ui[m], b1 = Wl[m], a2 = Ul[m], b2 = Wi[m];
                c4[0] = __fmaf_rn(a1.x, b1.x, c4[0]);
                c4[1] = __fmaf_rn(a1.y, b1.y, c4[1]);
                c4[2] = __fmaf_rn(a1.z, b1.z, c4[2]);
                c4[3] = __fmaf_rn(a1.w, b1.w, c4[3]);
                r4[0] = __fmaf_rn(a2.x, b2.x, r4[0]);
                r4[1] = __fmaf_rn(a2.y, b2.y, r4[1]);
                r4[2] = __fmaf_rn(a2.z, b2.z, r4[2]);
                r4[3] = __fmaf_rn(a2.w, b2.w, r4[3]);
              }
              const float uu = gc_q[qq] + ((c4[0] + c4[1]) + (c4[2] + c4[3])) - ((i == l) ? 1.f : 0.f);
              const float ww = (gr_q[qq] + ((r4[0] + r4[1]) + (r4[2] + r4[3]))) * f;
              if (i0 < L) {
                exq = __vmaxu4(exq, ((__float_as_uint(uu) << 1) >> 24) | (((__float_as_uint(ww) << 1) >> 24) << 8));
                Us[oi + j] = uu;
                Ws[oi + j] = ww;
                dg[qq] = __fmaf_rn(uu, ww, dg[qq]);
              }
            }
            if (i0 == l) {
              sv[qq] = -sv[qq];
              if (sp == 0) ss[i0] = (int8_t)sv[qq];
            }
          }
        }
        // the decision hash by the last thread (which owns no row for L <= 255)
        if (tid == NT - 1)
          s_pos.hash = (s_pos.hash ^ (unsigned long long)((s_pos.t0 + sw) * (long long)L + l)) * kFnvPrime;
        if constexpr (kRecord) {
          if (tid == 0) ip.trace[(size_t)sw * trace_words(L) + (l >> 5)] |= 1u << (l & 31);
        }
        ++j;
        propose(l + 1);
        __syncthreads();
        l = take_next(l + 1);
        if (j == K) flush();
        if (--left == 0) break;
      }
      // before a recompute, a measurement or the end: one flush in the code for
      // the three (with one each the kernels spill about twice as much; 40
      // half-filled chains at Lambda = 500, 15 sweeps, take 18.0 ms instead of 14.3)
      if (left == 0 || sw >= n_warm || sw + 1 == n_sweeps) flush();
      if (left == 0) break;
      if (sw >= n_warm) {
        const long long m = sw - n_warm;
        const int b = (int)((kBins * m) / a.n_meas);
        // partial sums in the (idle) staging area, totals in the panels' space
        float* part = reinterpret_cast<float*>(smem + lay.off_stage);
        float* gsum = reinterpret_cast<float*>(smem + lay.off_U);
        if (resident)
          measure_diagonals<kMirror ? 1 : 2>(Gu, Gd, ld, L, gsum);
        else
          measure_rows<kMirror ? 1 : 2>(Gu, Gd, ld, L, part, gsum);
        for (int k = tid; k < L; k += NT) {
          const double gu = (double)gsum[k] / (double)L;
          // G_dn = 1 - G_up^T: its sum of diagonal k > 0 is G_up's sum of
          // diagonal L - k, of diagonal 0 it is L minus G_up's
          const double gd = kMirror ? (k == 0 ? (double)L - (double)gsum[0] : (double)gsum[L - k]) / (double)L
                                    : (double)gsum[L + k] / (double)L;
          // the three accumulators loaded before any is stored: one L2 round trip
          double* bk = ip.bins + (size_t)b * L;
          const double a0 = ip.acc[k], a1 = ip.acc[L + k], b0 = bk[k];
          ip.acc[k] = a0 + gu;
          ip.acc[L + k] = a1 + gd;
          bk[k] = b0 + 0.5 * (gu + gd);
        }
        float v = 0.f;
#pragma unroll
        for (int qq = 0; qq < kRowsPerThread; ++qq) {
          if (qq * kRowStride >= L) break;  // uniform: rows beyond the grid
          const float other = __shfl_xor_sync(0xffffffffu, dg[qq], 1);
          const float dn = kMirror ? dg[qq] : 1.f - other;  // 1 - G_dn,ii
          if (sp == 0 && row0 + qq * kRowStride < L) v += (1.f - dg[qq]) * dn;
        }
        __syncthreads();  // every thread has read its totals
        for (int e = tid; e < 2 * L; e += NT) gsum[e] = 0.f;
        v = block_sum_f(v, reinterpret_cast<float*>(red));
        if (tid == 0) {
          const double d0 = ip.accD[0], d1 = ip.accD[1 + b];
          ip.accD[0] = d0 + (double)v / (double)L;
          ip.accD[1 + b] = d1 + (double)v / (double)L;
        }
      }
      l = -1;
      __syncthreads();
    }
    // bad ratios were counted per owned row: sum over the CTA
    {
      const int nb = __reduce_add_sync(0xffffffffu, n_bad);
      if (lane == 0 && nb) atomicAdd(&s_bad, nb);
    }
    if (tid == 0) {
      s_pos.n_acc += stretch - left;
      s_pos.sw = sw;
      s_pos.l = l;
      s_pos.par = par;
    }
    if (tid < 2) s_pos.f[tid] = f;
    done = left != 0;
    recompute = left == 0 && gc.n_wrap > 0;
    }
    __syncthreads();
    if (done) break;
    if (!recompute) continue;

    {  // a recompute
    const ChainView v(s_chain, smem);
    const GridConst& gc = v.gc;
    const ItemPtrs& ip = v.ip;
    const DelLayout& lay = v.lay;
    const int L = v.L, ld = v.ld;
    const bool resident = v.resident;
    float *const Ggl = v.Ggl, *const Gu = v.Gu, *const Gd = v.Gd;
    int8_t* const ss = v.ss;
    double d = -1.0;
    // G in HBM while the refinement runs, where its staging overlays a
    // resident G (else it works on G where it lies)
    constexpr int kSpins = kMirror ? 1 : 2;
    bool in_hbm = false;
    if (kRefine && gc.rc && use_tc && !tc.failed && gc.lambda != 0.0) {
      if (resident && !lay.rf_keeps_G) {
        for (int i = warp; i < kSpins * L; i += NW)
          for (int jj = lane; jj < L; jj += 32) Ggl[(size_t)i * L + jj] = Gu[(size_t)i * ld + jj];
        __syncthreads();
        in_hbm = true;
      }
      float* rws = reinterpret_cast<float*>(ip.ws);
      float* rred = reinterpret_cast<float*>(red);
      float* Ru = in_hbm ? Ggl : Gu;
      float* Rd = in_hbm ? Ggl + (size_t)L * L : Gd;
      const int rld = in_hbm ? L : ld;
      // spin down: not kept during a mirrored sweep; mirrored for a
      // particle-hole symmetric bath, else refined too
      const int n_ref = kMirror || gc.ph ? 1 : 2;
      float dmax = 0.f;
#pragma unroll 1
      for (int r = 0; r < n_ref && dmax >= 0.f; ++r) {
        const float dr = refine_spin<!kMirror>(L, gc.rc, ss, r ? -1 : 1, r ? Rd : Ru, rld, rws, smem + lay.off_rf, &tc,
                                               &s_rf, rred, a.status);
        dmax = dr < 0.f ? -1.f : fmaxf(dmax, dr);
      }
      if (!kMirror && gc.ph && dmax >= 0.f)
        dmax = fmaxf(dmax, ph_mirror(Ru, Rd, L, rld, reinterpret_cast<float*>(smem + lay.off_rf), rred));
      if (dmax >= 0.f)
        d = (double)dmax;
      else if (tid == 0)
        ++s_rec.n_fb;
    }
    if (d < 0.0) {
      d = recompute_from_scratch(smem, in_hbm ? Ggl : Gu, in_hbm ? Ggl + (size_t)L * L : Gd, in_hbm ? L : ld, kSpins, red,
                                 redi, &s_inv, &s_piv, a.status);
    }
    if (in_hbm) {
      for (int i = warp; i < kSpins * L; i += NW)
        for (int jj = lane; jj < L; jj += 32) Gu[(size_t)i * ld + jj] = Ggl[(size_t)i * L + jj];
      __syncthreads();
    }
    if (tid == 0) {
      s_rec.drift = fmax(s_rec.drift, d);
      ++s_rec.n_rec;
    }
    }
    __syncthreads();
    }

    const ChainView v(s_chain, smem);
    const ItemPtrs& ip = v.ip;
    const DelLayout& lay = v.lay;
    const int L = v.L, ld = v.ld;
    const bool resident = v.resident;
    float *const Ggl = v.Ggl, *const Gu = v.Gu;
    int8_t* const ss = v.ss;
    if (resident) {
      for (int i = warp; i < (kMirror ? 1 : 2) * L; i += NW)
        for (int jj = lane; jj < L; jj += 32) Ggl[(size_t)i * L + jj] = Gu[(size_t)i * ld + jj];
    }
    if constexpr (kMirror) {
      // the chain's G_dn for the host and the next call: 1 - G_up^T
      __syncthreads();
      (void)ph_mirror(Ggl, Ggl + (size_t)L * L, L, L, reinterpret_cast<float*>(smem + lay.off_rf),
                      reinterpret_cast<float*>(red));
    }
    for (int l = tid; l < L; l += NT) ip.s[l] = ss[l];
    if (tid == 0) {
      ChainCounters c = *ip.cnt;
      c.t += a.n_warm + a.n_meas;
      c.proposals += (a.n_warm + a.n_meas) * (long long)L;
      c.accepted = s_pos.n_acc;
      c.recomputes += s_rec.n_rec;
      c.hash = s_pos.hash;
      c.bad += s_bad;
      c.drift = s_rec.drift;
      c.fallbacks += s_rec.n_fb;
      *ip.cnt = c;
    }
    __syncthreads();
  }
  if (use_tc) tc_teardown(&tc);
}

size_t delayed_smem(int L, int k, bool resident, bool gj_smem, bool gtile, int ub, bool refine, int ns) {
  return del_layout(L, k, resident, gj_smem, gtile, ub, refine, ns).bytes;
}

int delayed_config(size_t smem, int* threads, int* ctas_per_sm) {
  cudaError_t e = cudaSuccess;
  for (auto* f : {k_sweep_delayed<false, false>, k_sweep_delayed<true, false>, k_sweep_delayed<false, true>,
                  k_sweep_delayed<true, true>, k_sweep_delayed<false, true, true>, k_sweep_delayed<true, true, true>})
    if (e == cudaSuccess) e = raise_smem_limit(f, smem);
  int occ = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sweep_delayed<false, true>, kDelNT, smem);
  *threads = kDelNT;
  // each CTA holds kTmemCols of the SM's 512 TMEM columns for its lifetime
  *ctas_per_sm = occ < 512 / kTmemCols ? occ : 512 / kTmemCols;
  return (int)e;
}

int launch_sweep_delayed(const SweepArgs& a, int ctas, size_t smem, cudaStream_t st) {
  const bool rec = a.trace_mode == kTraceRecord;
  if (a.refine && a.mirror)
    (rec ? k_sweep_delayed<true, true, true> : k_sweep_delayed<false, true, true>)<<<ctas, kDelNT, smem, st>>>(a);
  else if (a.refine)
    (rec ? k_sweep_delayed<true, true> : k_sweep_delayed<false, true>)<<<ctas, kDelNT, smem, st>>>(a);
  else
    (rec ? k_sweep_delayed<true, false> : k_sweep_delayed<false, false>)<<<ctas, kDelNT, smem, st>>>(a);
  return (int)cudaGetLastError();
}

}  // namespace hfq
