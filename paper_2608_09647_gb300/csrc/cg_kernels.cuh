// Kernels of the CG hot path (one GPU, everything resident in HBM):
//   a1  CSR SpMV q = A p fused with the p.q partial sum     (Alg. 1; Sec. 3.3 fused SpMV + dot)
//   a2  alpha, r -= alpha q, r.z and r.r partials, x += alpha p
//                                                          (Alg. 1; Sec. 3.3 fused update + r.r)
//   a3  beta, p = z + beta p                               (Alg. 1)
//   a4  convergence test on the device                     (Alg. 1, relative form)
//   a5  true residual ||b - A x|| / ||b|| in fp64         (Sec. 3.1, recomputed residual)
//
// The loop runs as one persistent cooperative launch.  Phases are separated by
// bounded grid barriers; every CTA forms the scalars redundantly from
// fixed-order sums of per-CTA partials, so there is no host round trip per
// iteration and reruns give identical results.
//
// GB300 design of one iteration:
//  * Jacobi is applied as the symmetric scaling A^ = D^-1/2 A D^-1/2, which
//    is algebraically the same iteration (x = D^-1/2 x^, r = D^1/2 r^,
//    r.z = r^.r^, r.r = r^.D r^) and leaves A^ with a unit diagonal, so the
//    loop streams no D^-1 vector and stores no diagonal entries.
//  * Three streaming phases: [q = A^ p, p.q] | [r^ -= alpha q, r.z, r.r] |
//    [x^ += alpha p, p = r^ + beta p]; the x update rides in the p pass, and
//    on the last iteration that pass writes the caller's x directly.
//    (Forming p on the fly inside the SpMV saves one pass and one barrier
//    but doubles the gathered vectors; measured on GB300 that halves the
//    SpMV's bandwidth, so the p update stays a pass of its own.)
//  * The loop matrix is stored as SELL-32 (sliced ELLPACK, slice height 32 =
//    one warp): the off-diagonal entries of 32 consecutive rows are laid out
//    column-major per slice, so lane l of a warp owns row 32 s + l, every
//    matrix load and most gathers are coalesced, the row sum stays in one
//    register, and warps run with no shared memory and no CTA barrier.  The
//    matrix is streamed with evict-first loads so the L2 keeps the vectors
//    that the gathers reuse.  Rows longer than kLongRow entries leave the
//    slices and are summed by a warp each from a compact CSR.
#pragma once

#include "cg_csr.cuh"

namespace cg {

constexpr int kLongRow = 128;              // off-diagonal entries above which a row leaves SELL
constexpr int kUnroll = 8;                 // slice columns whose loads are issued together
constexpr int kUnrollG = 4;                // the same in the generic (variable-width) slice loop
constexpr double kIrTolInner = 1e-4;       // default inner tolerance: refinement (restarting)
constexpr double kRuTolInner = 1e-1;       // default update threshold: reliable updates
constexpr int kMaxDiag = 32;               // most distinct offsets of the diagonal (DIA) layout
constexpr int kSellSigma = 256;            // rows sorted by length within windows of this many
constexpr double kCsrPadLimit = 1.3;       // slices padding the entries by more: the CSR loop layout

// --------------------------------------------------------------------------
// Persistent solver launch
// --------------------------------------------------------------------------

// Off-diagonal part of the loop matrix (A^ with Jacobi, A without) in
// SELL-32 form, or in its sliced-diagonal special case (dia != 0): when every
// off-diagonal entry lies on one of ndiag <= kMaxDiag diagonals j - i = delta[m]
// and few slots are empty, slice column m holds diagonal m, the column index
// of row i is i + delta[m] (clamped into range for the zero-valued slots) and
// no column array is stored.  Otherwise:  Slice s holds rows [32 s, 32 s + 32); its entries occupy
// [soff[s], soff[s+1]) in units of 32 (column m of the slice is the 32
// consecutive elements at (soff[s] + m) * 32; lane l = row 32 s + l).  Short
// rows are padded to the slice width with (column = own row, value = 0).
// Rows with more than kLongRow off-diagonal entries are marked in lmask and
// kept in a compact CSR (lrow / lptr / lcol / lval) instead.
template <typename T>
struct Sell {
  int64_t n;
  int32_t nslices;
  int32_t uw;  // >= 0: every slice has width uw and no row is long (soff, lmask unread)
  int32_t dia;                // 1: sliced-diagonal layout, width uw = number of diagonals
  int32_t delta[kMaxDiag];    // diagonal offsets (dia only)
  int32_t ring;               // kStaged: the allocated length of the vectors
  int32_t sym;                // 1: dia, and slot m of row i is slot uw-1-m of row i + delta[m], bit for bit (kMirrored)
  const int32_t* __restrict__ soff;
  const uint32_t* __restrict__ lmask;
  const int32_t* __restrict__ col;
  const T* __restrict__ val;
  int32_t nlong;
  const int32_t* __restrict__ lrow;
  const int32_t* __restrict__ lptr;
  const int32_t* __restrict__ lcol;
  const T* __restrict__ lval;
  const int32_t* __restrict__ perm;  // row at each slice position (SELL-C-sigma; n = none), or null
  int32_t csr;                 // 1: the loop matrix is a CSR of the off-diagonal entries (col / val),
  int32_t nrb;                 //    cut into nrb row blocks rb[] over the row pointers rptr[]
  const int32_t* __restrict__ rptr;
  const int32_t* __restrict__ rb;
  const T* __restrict__ dg;    // diagonal of the loop matrix (unused with Jacobi: unit diagonal)
  const T* __restrict__ dn;    // A_ii weights of the true residual norm (Jacobi)
  const T* __restrict__ disq;  // 1/sqrt(A_ii) mapping x^ back to x (Jacobi)
  double dmin, dmax;           // range of A_ii (Jacobi): dmin r^.r^ <= r.r <= dmax r^.r^
};

// With Jacobi the stopping test needs r.r = r^.D r^, two more fp64 operations
// and one more vector per row.  Since dmin rho <= r.r <= dmax rho, the test is
// decided by rho alone except in the band stop^2 / dmax < rho <= stop^2 / dmin
// (empty when the diagonal is constant).  The r update computes r.r only once
// dmin rho comes within kRrMargin of stop^2; if rho jumps into the band before
// that, one extra pass computes r.r, so the test stays exact.
constexpr double kRrMargin = 64.0;

template <typename T>
__device__ __forceinline__ bool rr_wanted(const Sell<T>& S, double rho, double stop2) {
  return S.dmin != S.dmax && S.dmin * rho <= kRrMargin * stop2;
}

// Decide sqrt(r.r) <= stop from rho: 1 converged, 0 not converged, -1 unknown.
// *rr gets dmax rho (exact for a constant diagonal).
template <typename T>
__device__ __forceinline__ int rr_bound_test(const Sell<T>& S, double rho, double stop2, double* rr) {
  *rr = S.dmax * rho;
  if (S.dmax * rho <= stop2) return 1;
  if (S.dmin * rho > stop2) return 0;
  return -1;
}

// Work vectors of the loop on type T.
template <typename T>
struct LoopVecs {
  T* r;       // r^ (scaled residual)
  T* p;       // search direction
  T* q;       // A^ p
  T* xh;      // x^ (scaled iterate; the inner correction d^ when refining)
};

struct SolveParams {
  Csr<double> A;          // caller's fp64 matrix (true residual)
  Sell<double> S64;       // fp64 loop matrix
  Sell<float> S32;        // fp32 loop matrix (refinement)
  LoopVecs<double> V64;
  LoopVecs<float> V32;
  const double* b;
  double* x;
  const double* dsq;      // sqrt(A_ii) (Jacobi)
  const double* disq;     // 1/sqrt(A_ii) (Jacobi)
  double* part;           // per-CTA partials: kParts slots of pstride doubles
  int pstride;            // slot stride (>= the grid of every loop kernel)
  DevState* st;
  XWord* xs;              // words of the grid exchanges
  double tol;             // outer relative tolerance
  double tol_in;          // inner tolerance (refinement)
  int maxit;              // SpMV cap (total inner iterations when refining)
  int max_restarts;       // residual replacements (fp64) / refinement steps
  uint64_t timeout_ns;
  unsigned skip_seq;
  int timers;             // accumulate CTA 0 phase times into st->tphase
};

// Partial-sum slots (each G doubles): 0 = p.q, 1 = r.r fallback, 2/3 = the
// update phase, 4..7 = the residual phase.  Disjoint slots mean a CTA never overwrites a
// partial that a slower CTA still has to read.
constexpr int kParts = 8;
constexpr int kSlotPQ = 0, kSlotRr = 1, kSlotUpd = 2, kSlotRes = 4, kSlotStart = kSlotRes + 3;

// Kinds of the exchanged sums (their scales are kept apart: two quantities of one kind would
// find the other's scale, and a sum that does not suit the scale is formed anew, in two
// more rounds).  The residual phase has three.
constexpr int kKindPQ = 0, kKindUpd = 1, kKindRr = 3, kKindRes = 4;

// Grid coordinates and the barriers of one persistent launch.
struct Grid {
  unsigned G, cta;
  int64_t gtid, gstride;
  DevState* st;
  uint64_t timeout_ns;
  unsigned seq, skip_seq;
  unsigned fills;  // this warp's ring chunks so far (spmv_phase_ring)
  __device__ Grid() : G(gridDim.x), cta(blockIdx.x), gtid((int64_t)blockIdx.x * kBlock + threadIdx.x),
        gstride((int64_t)gridDim.x * kBlock), st(nullptr), timeout_ns(0), seq(0), skip_seq(0), fills(0) {}
  __device__ Grid(DevState* s, uint64_t to, unsigned skip) : Grid() {
    st = s;
    timeout_ns = to;
    skip_seq = skip;
  }
  // a barrier; false: a wait gave up, leave the kernel
  template <class F = Nothing>
  __device__ __forceinline__ bool sync(F meanwhile = F()) {
    return grid_barrier(st, G, timeout_ns, ++seq, skip_seq, meanwhile);
  }
  // a barrier after which every thread has the grid's sums of v, through per-CTA partials
  // part[j G + cta] that every CTA adds up.  (grid_exchange, one round trip instead of
  // two, serves the one-CTA-an-SM forms.  Here phases end more unevenly, and CTAs that poll
  // an exchange's words slow the ones still at work: refinement on 27 points, 160^3 rows,
  // 304 CTAs, 148.7 us an iteration by exchanges, 146.5 so; fp64 on a power-law graph of
  // 20,000 rows 18.3 and 16.4.)  A slot of part is written again only after another
  // barrier: a slower CTA may still be reading it until then.
  template <int NV, class F = Nothing>
  __device__ __forceinline__ bool sum_parts(double (&v)[NV], double* part, F meanwhile = F());
};

// Write this CTA's block sums of v[0..NV) into part[j*G + cta] (v is
// consumed: afterwards it holds the sums in thread 0 only).
template <int NV>
__device__ __forceinline__ void publish(double (&v)[NV], double* part, const Grid& g) {
  cta_sum0<NV>(v);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) part[(size_t)j * g.G + g.cta] = v[j];
  }
}

template <int NV, class F>
__device__ __forceinline__ bool Grid::sum_parts(double (&v)[NV], double* part, F meanwhile) {
  publish<NV>(v, part, *this);
  if (!sync(meanwhile)) return false;
  grid_sum<NV>(part, G, v);
  return true;
}

// publish, then elect the last CTA of the launch to arrive (counter *ctr):
// it sums the G partials once (thread t takes partials t, t + kBlock, ...;
// then cta_sum0), leaves the totals in thread 0's tot, resets the counter and
// returns true in every one of its threads.  Consumers then read finished
// scalars instead of re-summing G partials in every CTA.  Writer: partial,
// fence, counter; reader: counter, fence, L2 loads (no stale L1 lines).
template <int NV>
__device__ __forceinline__ bool publish_last(double (&v)[NV], double* part, const Grid& g, unsigned* ctr,
                                             double (&tot)[NV]) {
  __shared__ int s_last;
  publish<NV>(v, part, g);
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(ctr, 1u) == g.G - 1;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    double t = 0.0;
    for (unsigned c = threadIdx.x; c < g.G; c += kBlock) t += __ldcg(part + (size_t)j * g.G + c);
    tot[j] = t;
  }
  cta_sum0<NV>(tot);
  if (threadIdx.x == 0) *ctr = 0;
  return true;
}

template <typename T> struct Vec;
template <> struct Vec<double> { using type = double2; static constexpr int N = 2; };
template <> struct Vec<float> { using type = float4; static constexpr int N = 4; };

template <typename T, typename VT>
__device__ __forceinline__ T& lane(VT& v, int j) {
  return reinterpret_cast<T*>(&v)[j];
}
template <typename T, typename VT>
__device__ __forceinline__ T lane_c(const VT& v, int j) {
  return reinterpret_cast<const T*>(&v)[j];
}

// Per-thread dot-product accumulator.  fp64: fused multiply-add.  fp32 (the
// refinement's inner solve): fp32 products summed with Kahan compensation, so
// the per-thread partial is accurate to about one fp32 rounding without any
// fp64 instruction (GB300 issues 64 fp32 FMAs per fp64 FMA); partials are
// combined in fp64 across threads and CTAs.
template <typename T> struct Acc;
template <> struct Acc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ double get() const { return s; }
};
template <> struct Acc<float> {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float a, float b) {
    const float y = __fmul_rn(a, b) - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double get() const { return (double)s - (double)c; }
};

// Status codes shared with the host API (values of cg_status).
constexpr int kOk = 0, kNotConverged = 1, kBreakdown = -2, kNumeric = -3, kTimeout = -4;

// CTA-local phase timer (CTA 0, thread 0, when enabled).
struct PhaseClock {
  bool on;
  uint64_t t;
  __device__ PhaseClock(bool enabled) : on(enabled && blockIdx.x == 0 && threadIdx.x == 0), t(0) {
    if (on) t = global_timer_ns();
  }
  __device__ __forceinline__ void lap(DevState* st, int slot) {
    if (on) {
      const uint64_t now = global_timer_ns();
      st->tphase[slot] += now - t;
      t = now;
    }
  }
};

// Streaming (evict-first) loads for the matrix, read once per iteration.
__device__ __forceinline__ int ld_stream(const int* p) { return __ldcs(p); }
__device__ __forceinline__ double ld_stream(const double* p) { return __ldcs(p); }
__device__ __forceinline__ float ld_stream(const float* p) { return __ldcs(p); }

// How spmv_phase_w finds a slot's column and value: in the slice; the column from
// delta[]; or (kSym, matrices equal to their transpose bit for bit) the value of a slot
// left of the diagonal from the row it mirrors, so that only the right half of the
// slices comes from memory and the left half is found in cache a band of rows later.
constexpr int kCols = 0, kDia = 1, kSym = 2;

template <typename T, int W, int DIA>
__device__ __forceinline__ T dia_val(const Sell<T>& S, const T* __restrict__ vp, int i, int m) {
  if constexpr (DIA == kSym) {
    if (m >= W / 2) return __ldg(vp + m * 32);
    const int j = i + S.delta[m];
    const T* u = S.val + (W - 1 - m) * 32;
    return j >= 0 ? __ldg(u + ((int64_t)(j >> 5) * ((W - 1) * 32) + j)) : T(0);
  } else {
    return ld_stream(vp + m * 32);
  }
}

// a1 over the grid for uniform slices of compile-time width W (no long rows):
// every load of a slice is issued at once and the register footprint is
// exactly what W needs, which keeps occupancy high.  DIA: the column of slot m
// is computed from delta[m] instead of loaded.  The diagonal term starts the
// fused multiply-add chain, so each row costs W + 1 fp64 FMAs with the p.q term.
// One slice's off-diagonal sum for uniform width W: loads of a chunk of CH
// columns are issued together, then the multiply-adds.  DIA: the column of
// slot m is i + delta[m], clamped into [0, n) with two 32-bit min/max (only
// zero-valued slots of the first and last slices ever need the clamp).
template <typename T, int W, int DIA>
__device__ __forceinline__ T slice_sum(const Sell<T>& S, const T* __restrict__ p, int64_t s,
                                       int i32, int lane, T acc) {
  constexpr int CH = W > 16 ? (W + 1) / 2 : W;
  const T* vp = S.val + s * (W * 32) + lane;
  const int nm1 = (int)S.n - 1;
#pragma unroll
  for (int m0 = 0; m0 < W; m0 += CH) {
    T v[CH], pc[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      const int m = m0 + u;
      if (m < W) {
        v[u] = dia_val<T, W, DIA>(S, vp, i32, m);
        const int c = DIA ? min(max(i32 + S.delta[m], 0), nm1)
                          : ld_stream(S.col + s * (W * 32) + lane + m * 32);
        pc[u] = p[c];
      }
    }
#pragma unroll
    for (int u = 0; u < CH; ++u)
      if (m0 + u < W) acc = fma(v[u], pc[u], acc);
  }
  return acc;
}

// a1 over the grid for uniform slices of compile-time width W (no long rows).
// Warps take slices round-robin, so at any moment the grid works on one
// contiguous band of rows and the neighbours' lines are shared through L2.
// The diagonal term starts the fused multiply-add chain: W + 1 FMAs per row
// with the p.q term.
template <typename T, bool JAC, int W, int DIA>
__device__ __forceinline__ double spmv_phase_w(const Sell<T>& S, const T* __restrict__ p,
                                               T* __restrict__ q, const Grid& g) {
  const int lane = threadIdx.x & 31;
  const int gw = (int)g.cta * kWarps + (int)(threadIdx.x >> 5);
  const int Wt = (int)g.G * kWarps;
  const int n = (int)S.n;
  Acc<T> dot;
  int s = gw;
  if constexpr (sizeof(T) == 4 && W <= 8) {
    // fp32 loops at 2 CTAs per SM: a warp's slices cost one L2 round trip each, so
    // two slices go together, every load of both issued before the first product
    // (the same arithmetic and order as one slice at a time)
    const int nm1 = n - 1;
    for (; s + Wt < S.nslices; s += 2 * Wt) {
      T v[2][W], pc[2][W], pi[2], acc[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int sh = s + h * Wt, i = sh * 32 + lane;
        const bool live = i < n;
        pi[h] = T(0);
        T dgi = T(1);
        if (live) {
          pi[h] = p[i];
          if (!JAC) dgi = __ldg(S.dg + i);
        }
        acc[h] = JAC ? pi[h] : dgi * pi[h];
        const T* vp = S.val + (int64_t)sh * (W * 32) + lane;
#pragma unroll
        for (int m = 0; m < W; ++m) {
          v[h][m] = dia_val<T, W, DIA>(S, vp, i, m);
          const int c = DIA ? min(max(i + S.delta[m], 0), nm1) : ld_stream(S.col + (int64_t)sh * (W * 32) + lane + m * 32);
          pc[h][m] = p[c];
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int m = 0; m < W; ++m) acc[h] = fma(v[h][m], pc[h][m], acc[h]);
        const int i = (s + h * Wt) * 32 + lane;
        if (i < n) {
          q[i] = acc[h];
          dot.add(pi[h], acc[h]);
        }
      }
    }
  }
  for (; s < S.nslices; s += Wt) {
    const int i = s * 32 + lane;
    const bool live = i < n;
    T pi = T(0), dgi = T(1);
    if (live) {
      pi = p[i];
      if (!JAC) dgi = __ldg(S.dg + i);
    }
    T acc = JAC ? pi : dgi * pi;
    acc = slice_sum<T, W, DIA>(S, p, s, i, lane, acc);
    if (live) {
      q[i] = acc;
      dot.add(pi, acc);
    }
  }
  return dot.get();
}

// Refinement on 27-point stencils (any grid at least four points wide): the SpMV of the
// persistent loop with its operands brought into shared memory ahead of the products.
// With two CTAs per SM the loop holds only 16 warps, and 27 + 26 loads into registers
// per slice left memory waiting: half of the warps' time was a wait for a load.  Here a
// warp has a ring of half slices of values (13 columns, one bulk copy each by one lane,
// an mbarrier per stage) and two windows of p, filled a slice ahead: the columns of a
// slice are 9 runs of 34 neighbouring entries of p, 90 16-byte copies, three a lane,
// where the gathers took 26 loads and their clamps.  160^3 rows, 304 CTAs: the SpMV in the
// loop 111 -> 95 us (426 MB of values: 63 us at the memory's rate), a solve to 1e-12
// 44.9 -> 43.5 ms.
constexpr int kRingW = 26, kRingChunk = kRingW / 2, kRingDepth = 3;
constexpr int kRingChunkBytes = kRingChunk * 32 * (int)sizeof(float);
constexpr int kRingBars = 128 * ((kWarps * kRingDepth * 8 + 127) / 128);
constexpr int kRuns = 9, kRunPieces = 10;         // 16-byte pieces of a run: 3 + 34 entries at most
constexpr int kWinDepth = 2, kWinBytes = kRuns * kRunPieces * 16;
constexpr unsigned kSkipCopy = 1u << 30;          // skip_seq beyond every barrier's number: a ring's copy
constexpr int kRingBytes = kRingBars + kWarps * (kRingDepth * kRingChunkBytes + kWinDepth * kWinBytes);

struct Ring {
  unsigned bar, buf;  // shared addresses of this warp's mbarriers and chunks
  const float* mem;   // the same chunks
  unsigned win;       // and of its windows of p
  const float* wmem;
  __device__ __forceinline__ Ring() {
    extern __shared__ __align__(128) unsigned char ring_smem[];
    const int warp = threadIdx.x >> 5;
    mem = reinterpret_cast<const float*>(ring_smem + kRingBars + warp * kRingDepth * kRingChunkBytes);
    bar = (unsigned)__cvta_generic_to_shared(ring_smem) + warp * kRingDepth * 8;
    buf = (unsigned)__cvta_generic_to_shared(mem);
    wmem = reinterpret_cast<const float*>(ring_smem + kRingBars + kWarps * kRingDepth * kRingChunkBytes +
                                          warp * kWinDepth * kWinBytes);
    win = (unsigned)__cvta_generic_to_shared(wmem);
  }
  // once per launch, by every warp
  __device__ __forceinline__ void init() const {
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
      for (int d = 0; d < kRingDepth; ++d) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar + 8 * d) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
  }
  // one lane: chunk number f of this warp's stream comes from src
  __device__ __forceinline__ void fill(unsigned f, const float* src) const {
    const unsigned d = f % kRingDepth, b = bar + 8 * d;
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(kRingChunkBytes) : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            buf + d * kRingChunkBytes),
        "l"(src), "r"(kRingChunkBytes), "r"(b), "l"(policy)
        : "memory");
  }
  // all lanes: whether chunk f has arrived (false: not within timeout_ns)
  __device__ __forceinline__ bool wait(unsigned f, uint64_t timeout_ns) const {
    const unsigned b = bar + 8 * (f % kRingDepth), parity = (f / kRingDepth) & 1u;
    uint64_t t0 = 0;
    unsigned ok;
    for (unsigned spins = 0;; ++spins) {
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
          : "=r"(ok)
          : "r"(b), "r"(parity)
          : "memory");
      if (ok) break;
      if (spins == 0) t0 = global_timer_ns();
      else if ((spins & 15u) == 0u && global_timer_ns() - t0 > timeout_ns) break;
    }
    return __all_sync(0xffffffffu, ok != 0u);
  }
  // the warp's wait for chunk f gave up: the launch is marked aborted and the copies still
  // under way (chunks f to end - 1, the windows) are waited for, with the same limit each,
  // since the CTA must not leave while they write its shared memory.  The NaN makes the
  // phase's sum NaN, which ends the loop in every CTA.
  __device__ __noinline__ double gave_up(DevState* st, unsigned barrier, uint64_t timeout_ns, unsigned f,
                                         unsigned end) const {
    if ((threadIdx.x & 31) == 0 && atomicCAS(&st->abort, 0, 1) == 0) {
      st->err_cta = (int)blockIdx.x;
      st->err_barrier = (int)barrier;
    }
    for (; f != end; ++f) wait(f, timeout_ns);
    asm volatile("cp.async.wait_all;" ::: "memory");
    return __longlong_as_double(0x7FF8000000000000ll);
  }
  __device__ __forceinline__ const float* chunk(unsigned f) const { return mem + (f % kRingDepth) * (kRingChunkBytes / 4); }
};

// a1 over the grid by the ring, one slice a warp at a time.  Slot m reads position m' = m
// (m < 13) or m + 1 of the 27 ordered offsets, the diagonal's among them: run m' / 3, its
// entry m' % 3 + lane.
// (S.ring is the allocated length of p, whose entries past n are 0.)  Fault injection:
// with skip_seq = kSkipCopy + k, CTA 0's first warp does not start its k-th chunk.
template <bool JAC>
__device__ __forceinline__ double spmv_phase_ring(const Sell<float>& S, const float* __restrict__ p,
                                                  float* __restrict__ q, Grid& g) {
  const Ring R;
  const int lane = threadIdx.x & 31;
  const int s0 = (int)g.cta * kWarps + (int)(threadIdx.x >> 5);
  const int Wt = (int)g.G * kWarps;
  const int n = (int)S.n, last = S.ring - 4;  // start of p's last piece
  const int slices = s0 < S.nslices ? (S.nslices - s0 + Wt - 1) / Wt : 0;  // of this warp
  const unsigned f0 = g.fills;
  const auto source = [&](int c) {  // chunk c of this warp's slices
    return S.val + (int64_t)(s0 + (c >> 1) * Wt) * (kRingW * 32) + (c & 1) * (kRingChunk * 32);
  };
  const auto fill = [&](int c) {
    if (threadIdx.x != 0 || g.cta != 0 || g.skip_seq != kSkipCopy + 1u + f0 + c) R.fill(f0 + c, source(c));
  };
  if (lane == 0)
    for (int c = 0; c < kRingDepth && c < 2 * slices; ++c) fill(c);
  constexpr int kPer = (kRuns * kRunPieces + 31) / 32;
  int off[kPer];  // this lane's pieces: their place in p from the slice's first row
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const int e = min(lane + 32 * u, kRuns * kRunPieces - 1), r = e / kRunPieces;
    off[u] = (S.delta[r <= 4 ? 3 * r : 3 * r - 1] & ~3) + 4 * (e - r * kRunPieces);
  }
  const auto windows = [&](int k) {  // of this warp's slice k
    const int i0 = (s0 + k * Wt) * 32;
    const unsigned dst = R.win + (k & 1) * kWinBytes + lane * 16;
#pragma unroll
    for (int u = 0; u < kPer; ++u)
      if (lane + 32 * u < kRuns * kRunPieces)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + u * 512),
                     "l"(p + min(max(i0 + off[u], 0), last))
                     : "memory");
  };
  const auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
  if (slices > 0) windows(0);
  commit();
  Acc<float> dot;
  for (int k = 0; k < slices; ++k) {
    const int i = (s0 + k * Wt) * 32 + lane;
    if (k + 1 < slices) windows(k + 1);
    commit();
    const float di = JAC ? 1.0f : __ldg(S.dg + min(i, n - 1));
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();  // slice k's windows have arrived
    const float* w = R.wmem + (k & 1) * (kWinBytes / 4) + lane;
    const float pi = w[4 * kRunPieces * 4 + (S.delta[12] & 3) + 1];  // run 4 starts left of the diagonal
    float acc = JAC ? pi : di * pi;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned f = f0 + 2 * k + h;
      if (!R.wait(f, g.timeout_ns))
        return R.gave_up(g.st, g.seq + 1, g.timeout_ns, f, f0 + min(2 * slices, 2 * k + h + kRingDepth));
      const float* v = R.chunk(f) + lane;
#pragma unroll
      for (int u = 0; u < kRingChunk; ++u) {
        const int m = h * kRingChunk + u, mm = m < 13 ? m : m + 1, r = mm / 3, d0 = r <= 4 ? 3 * r : 3 * r - 1;
        acc = fmaf(v[u * 32], w[r * kRunPieces * 4 + (S.delta[d0] & 3) + mm % 3], acc);
      }
      __syncwarp();  // the chunk (and with h = 1 the windows) have been read
      const int c = 2 * k + h + kRingDepth;
      if (lane == 0 && c < 2 * slices) fill(c);
    }
    if (i < n) {
      q[i] = acc;
      dot.add(pi, acc);
    }
  }
  g.fills = f0 + 2 * slices;
  return dot.get();
}

// Sliced-diagonal layout of any width up to kMaxDiag (loads in groups of kUnroll).
template <typename T, bool JAC>
__device__ __forceinline__ double spmv_phase_dia(const Sell<T>& S, const T* __restrict__ p,
                                                 T* __restrict__ q, const Grid& g) {
  const int lane = threadIdx.x & 31;
  const int gw = (int)g.cta * kWarps + (int)(threadIdx.x >> 5);
  const int Wt = (int)g.G * kWarps;
  const int64_t n = S.n;
  const int w = S.uw;
  Acc<T> dot;
  for (int s = gw; s < S.nslices; s += Wt) {
    const int64_t i = (int64_t)s * 32 + lane;
    const bool live = i < n;
    T pi = T(0), dgi = T(1);
    if (live) {
      pi = p[i];
      if (!JAC) dgi = __ldg(S.dg + i);
    }
    const T* vp = S.val + (int64_t)s * w * 32 + lane;
    const int64_t r0 = (int64_t)s * 32;
    const bool inner = r0 + S.delta[0] >= 0 && r0 + 31 + S.delta[w - 1] < n;
    const T* pb = p + i;
    T acc = JAC ? pi : dgi * pi;
    for (int m0 = 0; m0 < w; m0 += kUnroll) {
      T v[kUnroll], pc[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        if (m0 + u < w) {
          v[u] = ld_stream(vp + (m0 + u) * 32);
          if (inner) {
            pc[u] = pb[S.delta[m0 + u]];
          } else {
            const int64_t cc = i + S.delta[m0 + u];
            pc[u] = p[cc < 0 ? 0 : (cc >= n ? n - 1 : cc)];
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        if (m0 + u < w) acc = fma(v[u], pc[u], acc);
    }
    if (live) {
      q[i] = acc;
      dot.add(pi, acc);
    }
  }
  return dot.get();
}

// The CSR loop layout (matrices whose rows are too uneven for slices): one row
// block of q = A^ p, staged as the caller-CSR SpMV stages it (16-byte loads of
// columns and values into shared memory), rows of at most kThreadRow entries by
// a thread, longer ones by eight lanes, a row beyond the block cap by the CTA; the
// diagonal term starts each row's sum; the row's p_i q_i goes to dot.
template <typename T> struct Quad;
template <> struct Quad<double> {
  __device__ static void load(const double* v, double (&o)[4]) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(v));
    const double2 b = __ldg(reinterpret_cast<const double2*>(v + 2));
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
  }
  __device__ static void store(double* s, const double (&o)[4]) {
    reinterpret_cast<double2*>(s)[0] = make_double2(o[0], o[1]);
    reinterpret_cast<double2*>(s)[1] = make_double2(o[2], o[3]);
  }
};
template <> struct Quad<float> {
  __device__ static void load(const float* v, float (&o)[4]) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(v));
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
  }
  __device__ static void store(float* s, const float (&o)[4]) {
    reinterpret_cast<float4*>(s)[0] = make_float4(o[0], o[1], o[2], o[3]);
  }
};

constexpr int kRowStep = 4;  // a row's gathers in flight together in the CSR loop layout

// `next` gets the bounds of block bn (if below S.nrb), read while this block is summed.
template <typename T, bool JAC>
__device__ __forceinline__ void loop_rowblock(const Sell<T>& S, const T* __restrict__ p, T* __restrict__ q,
                                              const BlockSpan& B, int bn, BlockSpan& next, int* s_col, T* s_val,
                                              int2* s_row, Acc<T>& dot) {
  // positions [r0, r1) of the block; position ps holds row S.perm[ps] (the rows of a
  // block sorted by descending length) with entries at [rptr[ps], rptr[ps+1])
  const int r0 = B.r0, r1 = B.r1, k0 = B.k0, k1 = B.k1;
  const int t = threadIdx.x;
  if (k1 - k0 > kCapV) {  // one long row: strided FMA, fixed tree
    double acc = 0.0;
    for (int k = k0 + t; k < k1; k += kBlock) acc = fma((double)__ldg(S.val + k), (double)p[__ldg(S.col + k)], acc);
    double v[1] = {acc};
    block_sum<1>(v);
    if (t == 0) {
      const int i = __ldg(S.perm + r0);
      const T pi = p[i];
      const T qi = (JAC ? pi : __ldg(S.dg + i) * pi) + (T)v[0];
      q[i] = qi;
      dot.add(pi, qi);
    }
    if (bn < S.nrb) next = block_span(S.rb, S.rptr, bn);
    return;
  }
  const int a0 = k0 & ~3;  // the loop arrays start on 256-byte boundaries
  const int nq = (k1 - a0 + 3) >> 2;
  const int ps = r0 + t;
  int len = 0;
  if (ps < r1) {
    const int a = __ldg(S.rptr + ps) - a0;
    len = __ldg(S.rptr + ps + 1) - a0 - a;
    s_row[t] = make_int2((a << 12) | len, __ldg(S.perm + ps));  // a, len < 2^12
  }
#pragma unroll
  for (int j = 0; j < kQuadPasses; ++j) {
    const int qd = t + j * kBlock;
    if (qd >= nq) continue;
    const int k = a0 + 4 * qd;
    int c[4] = {0, 0, 0, 0};
    T v[4] = {T(0), T(0), T(0), T(0)};
    if (k + 4 <= k1) {
      const int4 c4 = __ldg(reinterpret_cast<const int4*>(S.col + k));
      c[0] = c4.x; c[1] = c4.y; c[2] = c4.z; c[3] = c4.w;
      Quad<T>::load(S.val + k, v);
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u < k1) {
          c[u] = __ldg(S.col + k + u);
          v[u] = __ldg(S.val + k + u);
        }
    }
    *reinterpret_cast<int4*>(s_col + 4 * qd) = make_int4(c[0], c[1], c[2], c[3]);
    Quad<T>::store(s_val + 4 * qd, v);
  }
  // (the barrier after the staging also counts the long rows, the block's first)
  const int nmed = __syncthreads_count(len > kThreadRow);
  if (bn < S.nrb) next = block_span(S.rb, S.rptr, bn);
  // long rows by eight lanes each (long_row_sum), 32 rows at a time: a warp per row held
  // the block for a chain of loads and a 5-level fp64 tree per row.  fp64 takes one chain a
  // lane: a predicated fp64 FMA issues in full (2 M rows: 114 us an iteration, 118 with four)
  for (int m = t >> 3; m < (nmed + 3) / 4 * 4; m += kBlock / 8) {
    const int2 e = m < nmed ? s_row[m] : make_int2(0, 0);
    const int am = (unsigned)e.x >> 12, lm = e.x & 0xFFF;
    const T acc = long_row_sum<sizeof(T) == 4 ? 4 : 1, T>(
        lm, [&](int k, T s) { return fma(s_val[am + k], p[s_col[am + k]], s); });
    if ((t & 7) == 0 && m < nmed) {
      const T pi = p[e.y];
      const T qi = (JAC ? pi : __ldg(S.dg + e.y) * pi) + acc;
      q[e.y] = qi;
      dot.add(pi, qi);
    }
  }
  // a warp's other rows, one a thread: the FMA chain runs to the warp's longest row
  // (one fp64 warp instruction per step), each lane keeping its sum past its own
  // row's end
  const bool mine = nmed + t < r1 - r0;
  const int2 e = mine ? s_row[nmed + t] : make_int2(0, 0);
  const int a = (unsigned)e.x >> 12, i = e.y;
  len = e.x & 0xFFF;
  const int wlen = __reduce_max_sync(0xffffffffu, len);
  if (mine) {
    const T pi = p[i];
    T acc = JAC ? pi : __ldg(S.dg + i) * pi;
    int k = 0;
    for (; k + kRowStep <= wlen; k += kRowStep) {  // kRowStep gathers in flight together
      T xv[kRowStep], vv[kRowStep];
#pragma unroll
      for (int u = 0; u < kRowStep; ++u) {
        const bool in = k + u < len;
        vv[u] = in ? s_val[a + k + u] : T(0);
        xv[u] = in ? p[s_col[a + k + u]] : T(0);
      }
#pragma unroll
      for (int u = 0; u < kRowStep; ++u) {
        const T nx = fma(vv[u], xv[u], acc);
        acc = k + u < len ? nx : acc;
      }
    }
    for (; k < wlen; ++k) {  // the warp's last steps, one at a time
      const bool in = k < len;
      const T nx = fma(in ? s_val[a + k] : T(0), in ? p[s_col[a + k]] : T(0), acc);
      acc = in ? nx : acc;
    }
    q[i] = acc;
    dot.add(pi, acc);
  }
  __syncthreads();  // the staging buffers are reused by the next row block
}

template <typename T, bool JAC>
__device__ __forceinline__ double spmv_phase_csr(const Sell<T>& S, const T* __restrict__ p, T* __restrict__ q,
                                                 const Grid& g) {
  __shared__ __align__(16) int s_col[kCap];
  __shared__ __align__(16) T s_val[kCap];
  __shared__ int2 s_row[kBlock];
  Acc<T> dot;
  BlockSpan B{0, 0, 0, 0}, next{0, 0, 0, 0};
  if ((int)g.cta < S.nrb) B = block_span(S.rb, S.rptr, (int)g.cta);
  for (int b = (int)g.cta; b < S.nrb; b += (int)g.G) {
    loop_rowblock<T, JAC>(S, p, q, B, b + (int)g.G, next, s_col, s_val, s_row, dot);
    B = next;
  }
  return dot.get();
}

// The product of a persistent fp32 kernel: from shared memory (spmv_phase_ring), from half
// of a symmetric matrix's slices (kSym), or any layout as it lies.  A kernel each: with the
// first two in the kernel of the third, not taken, every refinement that takes neither was
// 3 to 4 % slower (33^3 rows, 7 points: 11.9 against 11.4 us an iteration, 80^3: 16.9
// against 16.3), and the kernels that take them gain as much.
constexpr int kAsStored = 0, kStaged = 1, kMirrored = 2;

// a1 over the grid: q = A^ p and this thread's share of p.q.  Warps take
// slices round-robin; long rows are summed by a warp each.  Uniform slices of
// width 4, 6 or 8 go to the specialised loop.
template <typename T, bool JAC, int PRODUCT = kAsStored>
__device__ __forceinline__ double spmv_phase(const Sell<T>& S, const T* __restrict__ p,
                                             T* __restrict__ q, Grid& g) {
  static_assert(PRODUCT == kAsStored || sizeof(T) == 4, "fp32 forms");
  if constexpr (PRODUCT == kStaged) return spmv_phase_ring<JAC>(S, p, q, g);
  if constexpr (PRODUCT == kMirrored) {
    if (S.uw == 4) return spmv_phase_w<T, JAC, 4, kSym>(S, p, q, g);
    if (S.uw == 6) return spmv_phase_w<T, JAC, 6, kSym>(S, p, q, g);
    return spmv_phase_w<T, JAC, 8, kSym>(S, p, q, g);
  }
  if (S.csr) return spmv_phase_csr<T, JAC>(S, p, q, g);
  if (S.dia) {
    if (S.uw == 4) return spmv_phase_w<T, JAC, 4, kDia>(S, p, q, g);
    if (S.uw == 6) return spmv_phase_w<T, JAC, 6, kDia>(S, p, q, g);
    if (S.uw == 8) return spmv_phase_w<T, JAC, 8, kDia>(S, p, q, g);
    if (S.uw == 26) return spmv_phase_w<T, JAC, 26, kDia>(S, p, q, g);
    return spmv_phase_dia<T, JAC>(S, p, q, g);
  }
  if (S.uw == 4) return spmv_phase_w<T, JAC, 4, kCols>(S, p, q, g);
  if (S.uw == 6) return spmv_phase_w<T, JAC, 6, kCols>(S, p, q, g);
  if (S.uw == 8) return spmv_phase_w<T, JAC, 8, kCols>(S, p, q, g);
  const int lane = threadIdx.x & 31;
  const int gw = (int)g.cta * kWarps + (int)(threadIdx.x >> 5);
  const int W = (int)g.G * kWarps;
  const int64_t n = S.n;
  Acc<T> dot;
  for (int s = gw; s < S.nslices; s += W) {
    // slice position -> row: with SELL-C-sigma the rows of a window are sorted
    // by length, so one slice holds rows of similar length (little padding)
    const int64_t pos = (int64_t)s * 32 + lane;
    const int64_t i = S.perm ? (int64_t)__ldg(S.perm + pos) : pos;
    int o0, w;
    uint32_t lm;
    if (S.uw >= 0) {  // uniform slices: offsets are arithmetic, no metadata loads
      o0 = s * S.uw;
      w = S.uw;
      lm = 0u;
    } else {
      o0 = __ldg(S.soff + s);
      w = __ldg(S.soff + s + 1) - o0;
      lm = __ldg(S.lmask + s);
    }
    T pi = T(0), dgi = T(1);
    if (i < n) {
      pi = p[i];
      if (!JAC) dgi = __ldg(S.dg + i);
    }
    const int32_t* cp = S.col + (int64_t)o0 * 32 + lane;
    const T* vp = S.val + (int64_t)o0 * 32 + lane;
    T acc = JAC ? pi : dgi * pi;
    for (int m0 = 0; m0 < w; m0 += kUnrollG) {
      int c[kUnrollG];
      T v[kUnrollG], pc[kUnrollG];
#pragma unroll
      for (int u = 0; u < kUnrollG; ++u) {
        if (m0 + u < w) {
          c[u] = ld_stream(cp + (m0 + u) * 32);
          v[u] = ld_stream(vp + (m0 + u) * 32);
        }
      }
#pragma unroll
      for (int u = 0; u < kUnrollG; ++u)
        if (m0 + u < w) pc[u] = p[c[u]];
#pragma unroll
      for (int u = 0; u < kUnrollG; ++u)
        if (m0 + u < w) acc = fma(v[u], pc[u], acc);
    }
    if (i < n && !((lm >> lane) & 1u)) {
      q[i] = acc;
      dot.add(pi, acc);
    }
  }
  // long rows: one warp per row, lanes stride, fixed xor tree
  for (int l = gw; l < S.nlong; l += W) {
    const int i = __ldg(S.lrow + l);
    const int a = __ldg(S.lptr + l), e = __ldg(S.lptr + l + 1);
    T acc = T(0);
    for (int k = a + lane; k < e; k += 32) acc = fma(__ldg(S.lval + k), p[__ldg(S.lcol + k)], acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
      const T pi = p[i];
      const T qi = (JAC ? pi : __ldg(S.dg + i) * pi) + acc;
      q[i] = qi;
      dot.add(pi, qi);
    }
  }
  return dot.get();
}

// a2 over the grid: r^ -= alpha q; rho = r^.r^ (= r.z); rr = r^.D r^ (= r.r,
// Jacobi) or rho.  Two 16-byte vectors per thread per trip, loads first.
template <typename T, bool JAC>
__device__ __forceinline__ void update_r_phase(const Sell<T>& S, const LoopVecs<T>& V, T alpha,
                                               bool want_rr, double& rho, double& rr,
                                               const Grid& g) {
  using VT = typename Vec<T>::type;
  constexpr int VN = Vec<T>::N;
  const int64_t n = S.n;
  const int64_t nv = n / VN;
  VT* r = reinterpret_cast<VT*>(V.r);
  const VT* q = reinterpret_cast<const VT*>(V.q);
  const VT* dn = reinterpret_cast<const VT*>(S.dn);
  const bool with_rr = JAC && want_rr;
  Acc<T> a_rho, a_rr;
  for (int64_t i0 = g.gtid; i0 < nv; i0 += 2 * g.gstride) {
    const int64_t i1 = i0 + g.gstride;
    const bool two = i1 < nv;
    VT rv[2], qv[2], dv[2];
    rv[0] = r[i0];
    qv[0] = q[i0];
    if (with_rr) dv[0] = __ldg(dn + i0);
    if (two) {
      rv[1] = r[i1];
      qv[1] = q[i1];
      if (with_rr) dv[1] = __ldg(dn + i1);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (h == 1 && !two) break;
#pragma unroll
      for (int j = 0; j < VN; ++j) {
        const T ri = fma(-alpha, lane_c<T>(qv[h], j), lane<T>(rv[h], j));
        lane<T>(rv[h], j) = ri;
        a_rho.add(ri, ri);
        if (with_rr) a_rr.add(lane<T>(dv[h], j) * ri, ri);
      }
    }
    r[i0] = rv[0];
    if (two) r[i1] = rv[1];
  }
  for (int64_t i = nv * VN + g.gtid; i < n; i += g.gstride) {
    const T ri = fma(-alpha, V.q[i], V.r[i]);
    V.r[i] = ri;
    a_rho.add(ri, ri);
    if (with_rr) a_rr.add(__ldg(S.dn + i) * ri, ri);
  }
  rho += a_rho.get();
  rr += a_rr.get();
  if (!JAC) rr = rho;
}

// r.r = r^.D r^ from the current r^ (the exact-test fallback).
template <typename T>
__device__ __forceinline__ double rr_phase(const Sell<T>& S, const LoopVecs<T>& V, const Grid& g) {
  Acc<T> rr;
  for (int64_t i = g.gtid; i < S.n; i += g.gstride) {
    const T ri = V.r[i];
    rr.add(__ldg(S.dn + i) * ri, ri);
  }
  return rr.get();
}

// a3 over the grid: x^ += alpha p; p = r^ + beta p.  On the last iteration
// (FINAL) the p update is skipped and the caller's x is written instead:
// out = scale (x^ + alpha p), or out += fl64(scale (x^ + alpha p)) (OUT_ADD).
template <typename T, bool JAC, bool FINAL, bool OUT_ADD>
__device__ __forceinline__ void update_xp_phase(const Sell<T>& S, const LoopVecs<T>& V, T alpha,
                                                T beta, double* out, const Grid& g) {
  using VT = typename Vec<T>::type;
  constexpr int VN = Vec<T>::N;
  const int64_t n = S.n;
  const int64_t nv = n / VN;
  VT* x = reinterpret_cast<VT*>(V.xh);
  VT* p = reinterpret_cast<VT*>(V.p);
  const VT* r = reinterpret_cast<const VT*>(V.r);
  const VT* sc = reinterpret_cast<const VT*>(S.disq);
  for (int64_t iv = g.gtid; iv < nv; iv += g.gstride) {
    VT xv = x[iv], pv = p[iv], rv, dv;
    if (!FINAL) rv = r[iv];
    if (FINAL && JAC) dv = __ldg(sc + iv);
#pragma unroll
    for (int j = 0; j < VN; ++j) {
      const T pj = lane<T>(pv, j);
      const T xj = fma(alpha, pj, lane<T>(xv, j));
      if (FINAL) {
        const T xo = JAC ? xj * lane<T>(dv, j) : xj;
        if (OUT_ADD) out[iv * VN + j] += (double)xo;
        else out[iv * VN + j] = (double)xo;
      } else {
        lane<T>(xv, j) = xj;
        lane<T>(pv, j) = fma(beta, pj, lane_c<T>(rv, j));
      }
    }
    if (!FINAL) {
      x[iv] = xv;
      p[iv] = pv;
    }
  }
  for (int64_t i = nv * VN + g.gtid; i < n; i += g.gstride) {
    const T pj = V.p[i];
    const T xj = fma(alpha, pj, V.xh[i]);
    if (FINAL) {
      const T xo = JAC ? xj * __ldg(S.disq + i) : xj;
      if (OUT_ADD) out[i] += (double)xo;
      else out[i] = (double)xo;
    } else {
      V.xh[i] = xj;
      V.p[i] = fma(beta, pj, V.r[i]);
    }
  }
}

// The CG loop of Alg. 1 on the loop matrix from a (re)start state: r^ set,
// p = r^, x^ set, rho = r^.r^, rr = the true-norm r.r.  Iterates until
// sqrt(rr) <= stop_abs (kOk), maxit SpMVs (kNotConverged), breakdown /
// non-finite (kBreakdown / kNumeric) or a barrier timeout (kTimeout); *iters
// advances by the SpMVs done.  When an iteration ran, the caller's x is
// written (out = scale x^, or out += fl64(scale x^) with OUT_ADD) before the
// final grid barrier; otherwise out keeps its exact value.
template <typename T, bool JAC, bool OUT_ADD, int PRODUCT = kAsStored>
__device__ int cg_loop(const Sell<T>& S, const LoopVecs<T>& V, double rho, double rr,
                       double stop_abs, int maxit, int* iters, double* rr_out, double* out,
                       double* part, int pstride, Grid& g, PhaseClock& clk, double* rho_last = nullptr) {
  if (rho_last) *rho_last = rho;  // r.z before the last step taken (reliable updates)
  int k = *iters;
  int status = kNotConverged;
  const double stop2_hi = stop2_high(stop_abs);
  bool done = sqrt(rr) <= stop_abs || k >= maxit;  // a4: tested before every SpMV
  if (sqrt(rr) <= stop_abs) status = kOk;
  // scalars once per CTA in thread 0, shared (fp64 divisions and tests in every
  // thread would load GB300's narrow fp64 pipe)
  __shared__ double s_alpha, s_beta, s_rho, s_rr, s_inv_rho;
  __shared__ int s_st, s_want, s_exact, s_conv;
  while (!done) {
    // a1: q = A^ p; p.q
    double v1[1] = {spmv_phase<T, JAC, PRODUCT>(S, V.p, V.q, g)};
    clk.lap(g.st, 0);
    const bool ok1 = g.sum_parts(v1, part + kSlotPQ * (size_t)pstride);
    clk.lap(g.st, 1);
    if (threadIdx.x == 0) {
      s_st = !ok1 ? kTimeout
                  : ((!isfinite(v1[0]) || !isfinite(rho)) ? kNumeric : (v1[0] <= 0.0 ? kBreakdown : 0));
      s_alpha = rho / v1[0];
      s_want = JAC && rr_wanted(S, rho, stop_abs * stop_abs);
    }
    __syncthreads();
    if (s_st) { status = s_st; break; }
    const T alpha = (T)s_alpha;
    // a2: r^ -= alpha q; r.z, r.r (r.r only when the test needs it).  1 / rho for
    // this iteration's beta (beta_of) is formed while thread 0 waits at the barrier
    const bool want_rr = s_want != 0;
    const auto reciprocal = [&] { s_inv_rho = 1.0 / rho; };
    double v2[2] = {0.0, 0.0};
    update_r_phase<T, JAC>(S, V, alpha, want_rr, v2[0], v2[1], g);
    clk.lap(g.st, 2);
    bool ok;
    if (JAC) {  // one form with r.r and without: a second costs more than it saves
      ok = g.sum_parts(v2, part + kSlotUpd * (size_t)pstride, reciprocal);
    } else {
      double w[1] = {v2[0]};
      ok = g.sum_parts(w, part + kSlotUpd * (size_t)pstride, reciprocal);
      v2[0] = v2[1] = w[0];  // plain CG: r.z is r.r
    }
    clk.lap(g.st, 3);
    if (threadIdx.x == 0) {
      double rr_ = v2[1];
      if (!ok) s_st = kTimeout;
      s_exact = JAC && !want_rr && rr_bound_test(S, v2[0], stop_abs * stop_abs, &rr_) < 0;
      s_beta = beta_of(v2[0], rho, s_inv_rho);
      s_rho = v2[0];
      s_rr = rr_;
      s_conv = below_stop(rr_, stop_abs, stop2_hi);
    }
    __syncthreads();
    if (s_st) { status = s_st; break; }
    const T beta = (T)s_beta;
    if (rho_last) *rho_last = rho;
    rho = s_rho;
    if (s_exact) {
      double v3[1] = {rr_phase<T>(S, V, g)};  // rho fell into the band early: exact r.r
      const bool ok3 = g.sum_parts(v3, part + kSlotRr * (size_t)pstride);
      if (threadIdx.x == 0) {
        if (!ok3) s_st = kTimeout;
        s_rr = v3[0];
        s_conv = below_stop(v3[0], stop_abs, stop2_hi);
      }
      __syncthreads();
      if (s_st) { status = s_st; break; }
    }
    rr = s_rr;
    ++k;
    const bool conv = s_conv != 0;
    done = conv || k >= maxit;
    if (conv) status = kOk;
    // a3: x^ += alpha p; p = r^ + beta p (last iteration: write the caller's x)
    if (done) update_xp_phase<T, JAC, true, OUT_ADD>(S, V, alpha, beta, out, g);
    else update_xp_phase<T, JAC, false, OUT_ADD>(S, V, alpha, beta, out, g);
    clk.lap(g.st, 4);
    if (!g.sync()) { status = kTimeout; break; }
    clk.lap(g.st, 5);
  }
  *iters = k;
  *rr_out = rr;
  if (status == kNumeric || status == kBreakdown) {
    // the caller's x gets the last iterate
    for (int64_t i = g.gtid; i < S.n; i += g.gstride) {
      const T xo = JAC ? V.xh[i] * __ldg(S.disq + i) : V.xh[i];
      if (OUT_ADD) out[i] += (double)xo;
      else out[i] = (double)xo;
    }
    if (!g.sync()) return kTimeout;
  }
  return status;
}

// Caller's-matrix SpMV q = A x over the original row blocks (a5, restarts,
// the refinement's fp64 residual): the row-block kernel of cg_spmv (one fused
// multiply-add per nonzero in storage order, half the fp64 instructions of a
// separate multiply and add on GB300's narrow fp64 pipe).
__device__ __forceinline__ void spmv_orig(const Csr<double>& A, const double* x, double* q, const Grid& g) {
  __shared__ __align__(16) int s_col[kCap];
  __shared__ __align__(16) double s_val[kCap];
  __shared__ int s_med[kBlock];
  __shared__ int s_sort[32];
  spmv_rowblocks<true>(A, x, q, (int)g.cta, (int)g.G, s_col, s_val, s_med, s_sort);
}

// fp64 (Jacobi-)PCG with true-residual check and residual-replacement
// restarts (readings R1-R5 of the method, see the oracle's header).
template <bool JAC>
__global__ void __launch_bounds__(kBlock, 2) pcg64_kernel(SolveParams P) {
  Grid g(P.st, P.timeout_ns, P.skip_seq);
  PhaseClock clk(P.timers != 0);
  const int64_t n = P.A.n;
  const LoopVecs<double>& V = P.V64;
  int status = kNotConverged, k = 0, restarts = 0;
  double relres_true = 0.0, rr = 0.0, bb = 0.0;
  bool first = true;
  for (;;) {
    // a5 / (re)start: r = b - A x; r^ = D^-1/2 r; x^ = D^1/2 x
    spmv_orig(P.A, P.x, V.q, g);
    if (!g.sync()) { status = kTimeout; break; }
    double v[3] = {0.0, 0.0, 0.0};
    for (int64_t i = g.gtid; i < n; i += g.gstride) {
      const double bi = P.b[i];
      const double ri = bi - V.q[i];
      const double rh = JAC ? ri * __ldg(P.disq + i) : ri;
      V.r[i] = rh;
      V.p[i] = rh;
      V.xh[i] = JAC ? P.x[i] * __ldg(P.dsq + i) : P.x[i];
      v[0] += rh * rh;
      v[1] += ri * ri;
      v[2] += bi * bi;
    }
    if (!g.sum_parts(v, P.part + kSlotRes * (size_t)P.pstride)) { status = kTimeout; break; }
    const double(&s3)[3] = v;
    if (first) {
      bb = s3[2];
      if (bb == 0.0) {  // b = 0: x = 0 solves it
        for (int64_t i = g.gtid; i < n; i += g.gstride) P.x[i] = 0.0;
        status = kOk;
        break;
      }
    } else {
      relres_true = sqrt(s3[1]) / sqrt(bb);
      if (!isfinite(relres_true)) { status = kNumeric; break; }
      if (relres_true <= P.tol) { status = kOk; break; }
      if (k >= P.maxit || restarts >= P.max_restarts) { status = kNotConverged; break; }
      ++restarts;
    }
    const bool was_first = first;
    first = false;
    rr = s3[1];
    const int k_before = k;
    const int st = cg_loop<double, JAC, false>(P.S64, V, s3[0], rr, P.tol * sqrt(bb), P.maxit,
                                               &k, &rr, P.x, P.part, P.pstride, g, clk);
    if (st == kTimeout) { status = kTimeout; break; }
    if (st == kNumeric || st == kBreakdown) {
      status = st;
      spmv_orig(P.A, P.x, V.q, g);  // report the true residual of the last iterate
      if (!g.sync()) { status = kTimeout; break; }
      double w[1] = {0.0};
      for (int64_t i = g.gtid; i < n; i += g.gstride) {
        const double ri = P.b[i] - V.q[i];
        w[0] += ri * ri;
      }
      if (!g.sum_parts(w, P.part + kSlotRes * (size_t)P.pstride)) { status = kTimeout; break; }
      relres_true = sqrt(w[0]) / sqrt(bb);
      break;
    }
    if (was_first && k == k_before && st == kOk) {  // x0 met tol: its true residual is s3[1]
      relres_true = sqrt(s3[1]) / sqrt(bb);
      status = kOk;
      break;
    }
    // kOk or kNotConverged: loop back to recompute the true residual
  }
  // CTA 0 reports; a timeout anywhere is visible to the host through st->abort
  if (g.cta == 0 && threadIdx.x == 0) {
    P.st->status = status;
    P.st->iters = k;
    P.st->restarts = restarts;
    P.st->relres_true = relres_true;
    P.st->relres_rec = bb > 0.0 ? sqrt(rr) / sqrt(bb) : 0.0;
  }
}

// fp32-inner / fp64-outer iterative refinement (reading R6): the outer fp64
// residual, solution update and convergence test, the inner fp32 (scaled
// Jacobi) CG with fp64-accumulated dot products, all in one launch.  CARRY
// (reliable updates, R8): after each fp64 update the inner CG continues from
// the replaced residual with its last search direction, p = r^' + (r^'.r^' /
// rho_k) p_k, instead of restarting from p = r^'.
template <bool JAC, bool CARRY, int PRODUCT>
__global__ void __launch_bounds__(kBlock, 2) pcg_ir_kernel(SolveParams P) {
  Grid g(P.st, P.timeout_ns, P.skip_seq);
  PhaseClock clk(P.timers != 0);
  if constexpr (PRODUCT == kStaged) Ring().init();
  const int64_t n = P.A.n;
  const LoopVecs<float>& V = P.V32;
  int status = kNotConverged, inner = 0, outer = 0;
  double relres = 0.0, bb = 0.0, rr32 = 0.0, rho_k = 0.0;
  for (;;) {
    // outer fp64 residual r = b - A x fused with the inner start:
    // r^32 = fl32(D^-1/2 r), d^ = 0
    spmv_orig(P.A, P.x, P.V64.q, g);
    if (!g.sync()) { status = kTimeout; break; }
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t i = g.gtid; i < n; i += g.gstride) {
      const double bi = P.b[i];
      const double ri = bi - P.V64.q[i];
      const float rh = (float)(JAC ? ri * __ldg(P.disq + i) : ri);
      V.r[i] = rh;
      if (!CARRY || outer == 0) V.p[i] = rh;
      V.xh[i] = 0.0f;
      const double rh2 = (double)rh * (double)rh;
      v[0] += ri * ri;
      v[1] += bi * bi;
      v[2] += rh2;
      v[3] += JAC ? (double)__ldg(P.S32.dn + i) * rh2 : rh2;
    }
    if (!g.sum_parts(v, P.part + kSlotRes * (size_t)P.pstride)) { status = kTimeout; break; }
    const double(&s4)[4] = v;
    if (outer == 0) {
      bb = s4[1];
      if (bb == 0.0) {
        for (int64_t i = g.gtid; i < n; i += g.gstride) P.x[i] = 0.0;
        status = kOk;
        break;
      }
    }
    relres = sqrt(s4[0]) / sqrt(bb);
    if (!isfinite(relres)) { status = kNumeric; break; }
    if (relres <= P.tol) { status = kOk; break; }
    if (outer >= P.max_restarts || inner >= P.maxit) { status = kNotConverged; break; }
    if (CARRY && outer > 0 && rho_k > 0.0) {  // p = r^' + beta p_k
      const float beta = (float)(s4[2] / rho_k);
      for (int64_t i = g.gtid; i < n; i += g.gstride) V.p[i] = fma(beta, V.p[i], V.r[i]);
      if (!g.sync()) { status = kTimeout; break; }
    }
    const int st = cg_loop<float, JAC, true, PRODUCT>(P.S32, V, s4[2], s4[3], P.tol_in * sqrt(s4[3]),
                                             P.maxit, &inner, &rr32, P.x, P.part, P.pstride, g, clk, &rho_k);
    if (st == kTimeout || st == kNumeric || st == kBreakdown) { status = st; break; }
    ++outer;
  }
  if (g.cta == 0 && threadIdx.x == 0) {
    P.st->status = status;
    P.st->iters = inner;
    P.st->restarts = outer;
    P.st->relres_true = relres;
    P.st->relres_rec = relres;
  }
}

}  // namespace cg
