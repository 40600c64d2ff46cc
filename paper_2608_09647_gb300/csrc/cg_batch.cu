// Batched solves: up to CG_BATCH_MAX_SYSTEMS independent SPD systems of
// uneven size in one persistent cooperative launch, captured in a CUDA graph.
// Each system follows the single-system method of cg_solve (CG / Jacobi-PCG
// of Sec. 3 with its stopping rule, true-residual check and restarts); only
// the schedule is shared.
//
// Layout.  The systems are concatenated into one block-diagonal loop matrix
// of 32-row slices stored column-major (the diagonal held apart as a vector;
// with Jacobi the matrix is the scaled D^-1/2 A D^-1/2 of unit diagonal): a
// system whose off-diagonal entries lie on at most kBatchDiag offsets is
// stored by diagonal (a slot per offset, the gather index clamped into the
// system's own rows, no column array), the others as SELL-32 with global
// columns.  Every system is padded to whole 256-row tiles (padding rows are
// identity rows with b = x = 0), so no tile spans two systems; 1, 2 or 8 tiles,
// by the system's size, form a reduction unit.
//
// Schedule.  The grid's CTAs form teams, contiguous runs of CTAs that the hardware
// spreads over the SMs, so the CTAs of one SM belong to different teams.  A team
// solves one system at a time, split over its CTAs by units, with a barrier of its own
// (bounded, a counter in L2) after each phase:
//   R  r = b - A x: the fp64 true-residual test and the (re)start of a loop;
//   A  q = A p and p.q, alpha;
//   B  r -= alpha q, r.r and r.D r, beta and the recursive stopping test;
//   C  x += alpha p, p = r + beta p;
// then it takes the next system of the queue (descending work).  While one team waits
// at its barrier or sums, the SM's other CTAs work on other systems, in other phases:
// the waits are hidden, and phases bound by the fp64 pipe (R, A, B) run beside phases
// bound by memory (C).  (One schedule for all systems, four phases with a barrier of
// the whole grid after each, left both bounds and all waits in sequence, and its work
// lists and system sums cost ~17 us a phase however small the systems: 26.3 ms for 24
// systems of 33^2 to 200^2 rows to 1e-12 with reliable updates, 127.2 ms for 96 fp64
// systems of 32^2 to 512^2; now 10.3 ms and 116 ms.)
// A system's sums are formed from (unit, warp) partials, which depend on the system
// alone, by every CTA of its team in the same fixed order: results depend neither on
// the schedule nor on the other systems.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "cg_handle.cuh"

using namespace cg;

namespace {

constexpr int kTile = kBlock;        // rows per tile (kWarps slices, one per warp)
constexpr int kMaxBatch = CG_BATCH_MAX_SYSTEMS;
constexpr int kNP = 4;               // partial sums per (unit, warp)
constexpr int kBatchDiag = 8;        // offsets of a system in the diagonal layout, at most
constexpr int kStRunning = 100;      // status of a system still being solved
constexpr int kMaxCand = 8;          // autotuner candidates
constexpr double kRrMarginB = 64.0;  // r.D r is computed while dmin r^.r^ <= 64 stop^2
constexpr int kTeamWords = kXAll;      // exchange words of a team

// Tiles per reduction unit: up to 128 units to 262,144 rows (a team's CTAs then sum up
// to 1024 partials, four a thread), so that a team of ~20 CTAs is evenly loaded (64
// units on 19 CTAs left them idle 16 % of a phase), and as many units as there are
// tiles where the system is small, so that it can be spread over as many CTAs.
inline int unit_tiles(int ntile) { return ntile <= 64 ? 1 : (ntile <= 256 ? 2 : 8); }

struct BatchParams {
  int nsys;
  const int32_t* __restrict__ tstart;  // first tile of each system
  const int32_t* __restrict__ ntile;   // tiles of each system
  const int32_t* __restrict__ ustart;  // first reduction unit of each system
  const int32_t* __restrict__ nunit;   // reduction units of each system
  const int32_t* __restrict__ utiles;  // tiles per unit of each system
  const int32_t* __restrict__ sdia;    // offsets of each system in the diagonal layout (0: sliced ELL)
  const int32_t* __restrict__ sdelta;  // those offsets, kBatchDiag per system
  const double* __restrict__ dmin;     // smallest A_ii of each system
  const int32_t* __restrict__ soff;    // slice offsets (units of 32 entries)
  const int32_t* __restrict__ col;     // global (concatenated) column of each entry
  const double* __restrict__ val;
  const double* __restrict__ dg;       // A_ii, 1 on padding rows
  double *r, *p, *q, *xh;
  const double* __restrict__ bh;
  double* relres;
  int *k, *restarts, *status, *zero;
  double* tpart;                       // two banks of kNP partials per (unit, warp)
  int64_t bank;                        // doubles of a bank
  const int32_t* __restrict__ order;   // the queue: systems by descending work
  const int32_t* __restrict__ team0;   // first CTA of each team (nteams + 1)
  int nteams;
  unsigned* queue;                     // systems taken beyond the teams' first
  int* next;                           // each team's next place in the queue
  XWord* words;                        // kTeamWords exchange words per team
  double tol;
  int maxit, max_restarts;
  DevState* st;
  uint64_t timeout_ns;
  unsigned skip_seq;
  // fp32 inner solves with fp64 refinement (batch_ir_kernel only)
  const float* __restrict__ val32;     // the loop matrix values rounded to fp32
  float *r32, *p32, *q32, *d32;        // inner residual, direction, A p, correction d
  double tol_in;
  int max_outer, carry;
};

// acc + off-diagonal part of one row of slice sl: the sum over the slice
// width of val * v[col], all loads of a slice issued together (widths 4 and
// 8, those of the 5- and 9-point stencils, unrolled exactly).
template <int W>
__device__ __forceinline__ double slice_row(const int32_t* __restrict__ cp, const double* __restrict__ vp,
                                            const double* __restrict__ v, double acc) {
  int c[W];
  double a[W];
#pragma unroll
  for (int m = 0; m < W; ++m) {
    c[m] = ld_stream(cp + m * 32);
    a[m] = ld_stream(vp + m * 32);
  }
#pragma unroll
  for (int m = 0; m < W; ++m) acc = fma(a[m], v[c[m]], acc);
  return acc;
}

// The system a team is solving (shared memory) and this CTA's units of it.
struct SegInfo {
  int nd;              // offsets of the diagonal layout (0: sliced ELL)
  int lo, hi;          // the system's first and last concatenated rows
  int delta[kBatchDiag];
  int t0, tend;        // its first tile, the tile after its last
  int ut, un0, nunit;  // tiles per unit, its first unit, its units
  int u0, u1;          // this CTA's units
};

// Diagonal layout: column i + delta[m], clamped into the system's own rows
// (the value is 0 there, and no other system's vector is read).
template <int W>
__device__ __forceinline__ double slice_row_dia(const double* __restrict__ vp, const double* __restrict__ v,
                                                int i, const SegInfo& sg, double acc) {
  double a[W], x[W];
#pragma unroll
  for (int m = 0; m < W; ++m) {
    a[m] = ld_stream(vp + m * 32);
    x[m] = v[min(max(i + sg.delta[m], sg.lo), sg.hi)];
  }
#pragma unroll
  for (int m = 0; m < W; ++m) acc = fma(a[m], x[m], acc);
  return acc;
}

__device__ __forceinline__ double row_spmv(const BatchParams& P, const double* __restrict__ v, int i,
                                           double acc, const SegInfo& sg) {
  const int sl = i >> 5, lane = i & 31;
  const int o0 = __ldg(P.soff + sl);
  const int w = __ldg(P.soff + sl + 1) - o0;
  if (sg.nd) {
    const double* vp = P.val + (int64_t)o0 * 32 + lane;
    if (w == 8) return slice_row_dia<8>(vp, v, i, sg, acc);
    if (w == 4) return slice_row_dia<4>(vp, v, i, sg, acc);
    for (int m = 0; m < w; ++m) acc = fma(ld_stream(vp + m * 32), v[min(max(i + sg.delta[m], sg.lo), sg.hi)], acc);
    return acc;
  }
  const int32_t* cp = P.col + (int64_t)o0 * 32 + lane;
  const double* vp = P.val + (int64_t)o0 * 32 + lane;
  if (w == 8) return slice_row<8>(cp, vp, v, acc);
  if (w == 4) return slice_row<4>(cp, vp, v, acc);
  for (int m0 = 0; m0 < w; m0 += 4) {
    if (m0 + 4 <= w) {
      acc = slice_row<4>(cp + m0 * 32, vp + m0 * 32, v, acc);
    } else {
      for (int m = m0; m < w; ++m) acc = fma(ld_stream(vp + m * 32), v[ld_stream(cp + m * 32)], acc);
    }
  }
  return acc;
}

// The same row sum for any value type TV, accumulator TA and gathered vector:
// gx(j) gives the vector's entry j (the fp32 inner solves gather r + beta0 p on
// the first iteration of an inner solve without storing that vector first).
template <int W, typename TV, typename TA, class Gx>
__device__ __forceinline__ TA slice_row_g(const int32_t* __restrict__ cp, const TV* __restrict__ vp, Gx gx,
                                          TA acc) {
  int c[W];
  TV a[W];
#pragma unroll
  for (int m = 0; m < W; ++m) {
    c[m] = ld_stream(cp + m * 32);
    a[m] = ld_stream(vp + m * 32);
  }
  TA x[W];
#pragma unroll
  for (int m = 0; m < W; ++m) x[m] = gx(c[m]);
#pragma unroll
  for (int m = 0; m < W; ++m) acc = fma((TA)a[m], x[m], acc);
  return acc;
}

template <int W, typename TV, typename TA, class Gx>
__device__ __forceinline__ TA slice_row_dia_g(const TV* __restrict__ vp, Gx gx, int i, const SegInfo& sg, TA acc) {
  TV a[W];
  TA x[W];
#pragma unroll
  for (int m = 0; m < W; ++m) {
    a[m] = ld_stream(vp + m * 32);
    x[m] = gx(min(max(i + sg.delta[m], sg.lo), sg.hi));
  }
#pragma unroll
  for (int m = 0; m < W; ++m) acc = fma((TA)a[m], x[m], acc);
  return acc;
}

template <typename TV, typename TA, class Gx>
__device__ __forceinline__ TA row_spmv_g(const BatchParams& P, const TV* __restrict__ val, int i, TA acc,
                                         const SegInfo& sg, Gx gx) {
  const int sl = i >> 5, lane = i & 31;
  const int o0 = __ldg(P.soff + sl);
  const int w = __ldg(P.soff + sl + 1) - o0;
  const TV* vp = val + (int64_t)o0 * 32 + lane;
  if (sg.nd) {
    if (w == 8) return slice_row_dia_g<8, TV, TA>(vp, gx, i, sg, acc);
    if (w == 4) return slice_row_dia_g<4, TV, TA>(vp, gx, i, sg, acc);
    for (int m = 0; m < w; ++m) acc = fma((TA)ld_stream(vp + m * 32), gx(min(max(i + sg.delta[m], sg.lo), sg.hi)), acc);
    return acc;
  }
  const int32_t* cp = P.col + (int64_t)o0 * 32 + lane;
  if (w == 8) return slice_row_g<8, TV, TA>(cp, vp, gx, acc);
  if (w == 4) return slice_row_g<4, TV, TA>(cp, vp, gx, acc);
  for (int m0 = 0; m0 < w; m0 += 4) {
    if (m0 + 4 <= w) {
      acc = slice_row_g<4, TV, TA>(cp + m0 * 32, vp + m0 * 32, gx, acc);
    } else {
      for (int m = m0; m < w; ++m) acc = fma((TA)ld_stream(vp + m * 32), gx(ld_stream(cp + m * 32)), acc);
    }
  }
  return acc;
}

// One CTA of a team: the team's barrier, the system in hand, the partials' bank.
struct Team {
  const BatchParams& P;
  SegInfo& seg;
  XState* x;
  int id, rank, size;
  int flip;  // reductions so far: the bank the next one writes
  __device__ __forceinline__ bool sync() {
    return __syncthreads_and(grid_exchange<0>(x, 0, 0.0, 0.0).ok) != 0;
  }
  __device__ __forceinline__ double* bank() const { return P.tpart + (flip & 1) * P.bank; }
};

// The team's place in the grid and its barrier; false: a CTA without a team.
__device__ __forceinline__ bool team_init(const BatchParams& P, XState* x, int* id, int* rank, int* size) {
  const int c = (int)blockIdx.x;
  int lo = 0, hi = P.nteams;  // the last team with team0 <= c
  while (lo + 1 < hi) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(P.team0 + mid) <= c) lo = mid;
    else hi = mid;
  }
  const int a = __ldg(P.team0 + lo), e = __ldg(P.team0 + lo + 1);
  *id = lo;
  *rank = c - a;
  *size = e - a;
  if (c >= e) return false;
  x_init(x, P.st, P.words + (size_t)lo * kTeamWords, (unsigned)(e - a), (unsigned)(c - a), c == 0 ? P.skip_seq : 0u,
         P.timeout_ns);
  return true;
}

// The team's next system (-1: the queue is empty, -2: a wait gave up).  Its first one
// is fixed, so that a team sized for a system gets that one.
__device__ __forceinline__ int next_system(Team& T, bool first) {
  const BatchParams& P = T.P;
  int j = T.id;
  if (!first) {
    if (T.rank == 0 && threadIdx.x == 0) P.next[T.id] = P.nteams + (int)atomicAdd(P.queue, 1u);
    if (!T.sync()) return -2;
    j = __ldcg(P.next + T.id);
  }
  if (j >= P.nsys) return -1;
  const int s = __ldg(P.order + j);
  __syncthreads();  // seg may still be read for the system before
  if (threadIdx.x == 0) {
    SegInfo& g = T.seg;
    g.nd = P.sdia[s];
    g.t0 = P.tstart[s];
    g.tend = g.t0 + P.ntile[s];
    g.lo = g.t0 * kTile;
    g.hi = g.tend * kTile - 1;
    g.ut = P.utiles[s];
    g.un0 = P.ustart[s];
    g.nunit = P.nunit[s];
    g.u0 = (int)((int64_t)g.nunit * T.rank / T.size);
    g.u1 = (int)((int64_t)g.nunit * (T.rank + 1) / T.size);
#pragma unroll
    for (int m = 0; m < kBatchDiag; ++m) g.delta[m] = P.sdelta[s * kBatchDiag + m];
  }
  __syncthreads();
  return s;
}

// One phase over this CTA's units.  For every row i of a unit, row(i) does the row's
// loads and arithmetic and returns its commit, which stores the results and adds the
// row's NV contributions to the thread's accumulators.  A thread's rows go in groups
// of ROWS (8, 4, 2 or 1, by the variant's register budget), every row's loads in
// flight before the first commit (a store ahead of the next row's loads would
// serialise them); the accumulation order stays the row order.  The unit's sums are
// then formed per warp and stored; sums NREQ .. NV-1 only with `all`.
template <int NV, int ROWS, int NREQ = NV, class Row>
__device__ __forceinline__ void run_phase(const Team& T, Row row, bool all = true) {
  const SegInfo& seg = T.seg;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int u = seg.u0; u < seg.u1; ++u) {
    const int t0 = seg.t0 + u * seg.ut, t1 = min(t0 + seg.ut, seg.tend);
    double acc[NV > 0 ? NV : 1];
#pragma unroll
    for (int k = 0; k < (NV > 0 ? NV : 1); ++k) acc[k] = 0.0;
    int gt = t0;
    if constexpr (ROWS >= 8) {
      for (; gt + 7 < t1; gt += 8) {
        const auto c0 = row(gt * kTile + t);
        const auto c1 = row((gt + 1) * kTile + t);
        const auto c2 = row((gt + 2) * kTile + t);
        const auto c3 = row((gt + 3) * kTile + t);
        const auto c4 = row((gt + 4) * kTile + t);
        const auto c5 = row((gt + 5) * kTile + t);
        const auto c6 = row((gt + 6) * kTile + t);
        const auto c7 = row((gt + 7) * kTile + t);
        c0(acc);
        c1(acc);
        c2(acc);
        c3(acc);
        c4(acc);
        c5(acc);
        c6(acc);
        c7(acc);
      }
    }
    if constexpr (ROWS >= 4) {
      for (; gt + 3 < t1; gt += 4) {
        const auto c0 = row(gt * kTile + t);
        const auto c1 = row((gt + 1) * kTile + t);
        const auto c2 = row((gt + 2) * kTile + t);
        const auto c3 = row((gt + 3) * kTile + t);
        c0(acc);
        c1(acc);
        c2(acc);
        c3(acc);
      }
    }
    if constexpr (ROWS >= 2) {
      for (; gt + 1 < t1; gt += 2) {
        const auto c0 = row(gt * kTile + t);
        const auto c1 = row((gt + 1) * kTile + t);
        c0(acc);
        c1(acc);
      }
    }
    for (; gt < t1; ++gt) row(gt * kTile + t)(acc);
    if (NV > 0) {
      // the warp's sum of each value, exact and rounded once on the integer pipes: an
      // fp64 xor tree would take 5 warp instructions of the fp64 pipe (one per ~64
      // clocks per SM sub-partition) that the rows' FMAs need
#pragma unroll
      for (int k = 0; k < NV; ++k)
        if (k < NREQ || all) acc[k] = warp_sum_exact(acc[k]);
      if (lane == 0) {
        double* dst = T.bank() + ((size_t)(seg.un0 + u) * kWarps + warp) * kNP;
#pragma unroll
        for (int k = 0; k < NV; ++k)
          if (k < NREQ || all) dst[k] = acc[k];
      }
    }
  }
}

// The team's barrier after a phase that formed sums, then the system's sums of values
// 0 .. NV-1 in warp 0, the same bits in every CTA: thread t adds partials t,
// t + kBlock, ... in order (its loads in flight together), then cta_sum0.  The next
// reduction writes the other bank: a slower CTA may still be reading this one.
template <int NV>
__device__ __forceinline__ bool reduce(Team& T, double (&out)[NV]) {
  constexpr int kSumBatch = 4;
  const double* bank = T.bank();
  T.flip += 1;
  if (!T.sync()) return false;
  const size_t p0 = (size_t)T.seg.un0 * kWarps;
  const int np = T.seg.nunit * kWarps;
#pragma unroll
  for (int j = 0; j < NV; ++j) out[j] = 0.0;
  for (int t0 = threadIdx.x; t0 < np; t0 += kBlock * kSumBatch) {
    double v[kSumBatch][NV];
#pragma unroll
    for (int u = 0; u < kSumBatch; ++u) {
      const int t = t0 + kBlock * u;
#pragma unroll
      for (int j = 0; j < NV; ++j) v[u][j] = t < np ? __ldcg(bank + (p0 + t) * kNP + j) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kSumBatch; ++u) {
      if (t0 + kBlock * u < np) {
#pragma unroll
        for (int j = 0; j < NV; ++j) out[j] += v[u][j];
      }
    }
  }
  cta_sum0<NV>(out);
  return true;
}

// What thread 0 of a CTA decides from a system's sums, for all its threads.
struct Control {
  double alpha, beta, rho, inv_rho, bb, relres, stop, stop2_hi, rho_k, beta0;
  int k, restarts, status, zero;
  int act;   // after R: 1 = iterate, 0 = the system is done; after A: 0 = failed
  int wrr;   // r.D r is formed with the r update
  int last;  // this iteration ends the (inner) loop
  int exact; // r.D r must be formed before the test
};

__device__ __forceinline__ void control_init(Control& c) {
  if (threadIdx.x == 0) {
    c.bb = -1.0;  // "not yet known": the first residual phase records b.b
    c.relres = 0.0;
    c.k = c.restarts = c.zero = 0;
    c.status = kStRunning;
    c.rho_k = 0.0;
  }
  __syncthreads();
}

__device__ __forceinline__ void report(const Team& T, const Control& c, int s) {
  if (T.rank == 0 && threadIdx.x == 0) {
    T.P.relres[s] = c.relres;
    T.P.k[s] = c.k;
    T.P.restarts[s] = c.restarts;
    T.P.status[s] = c.status;
    T.P.zero[s] = c.zero;
  }
}

// The r update's scalars and test (thread 0): rho' = sums[0], r.D r = sums[1] if it was
// formed.  above: r.D r >= dmin rho' > stop^2, so the test fails for sure.
template <bool JAC>
__device__ __forceinline__ void after_update(Control& c, double rho1, double rr, double dmin, double stop2,
                                             int maxit) {
  c.beta = beta_of(rho1, c.rho, c.inv_rho);
  c.rho_k = c.rho;  // r.z of the step just taken (the carry's denominator)
  c.rho = rho1;
  c.k += 1;
  c.exact = 0;
  bool conv = false;
  if (!JAC || c.wrr) conv = below_stop(JAC ? rr : rho1, c.stop, c.stop2_hi);
  else c.exact = dmin * rho1 <= stop2;
  if (JAC) c.wrr = c.exact || dmin * rho1 <= kRrMarginB * stop2;
  c.last = conv || c.k >= maxit;
}

// MINB: resident CTAs per SM the registers are budgeted for (an autotuner choice).
template <bool JAC, int MINB>
__global__ void __launch_bounds__(kBlock, MINB) batch_pcg_kernel(BatchParams P) {
  // rows in flight per thread within the register budget of MINB CTAs per SM
  constexpr int kRows = MINB <= 3 ? 4 : 2;
  // phase B streams only q and r (two loads a row): twice the rows in flight
  constexpr int kRowsB = 2 * kRows;
  __shared__ SegInfo s_seg;
  __shared__ XState s_x;
  __shared__ Control c;
  const int t = threadIdx.x;
  int id, rank, size;
  if (!team_init(P, &s_x, &id, &rank, &size)) return;
  Team T{P, s_seg, &s_x, id, rank, size, 0};
  double* __restrict__ r = P.r;
  double* __restrict__ p = P.p;
  double* __restrict__ q = P.q;
  double* __restrict__ xh = P.xh;
  const double* __restrict__ bh = P.bh;
  const double* __restrict__ dg = P.dg;
  for (bool first_system = true;; first_system = false) {
    const int sys = next_system(T, first_system);
    if (sys < 0) return;
    control_init(c);
    const double dmin = P.dmin[sys];
    for (;;) {
      // ---- R: residual, true-residual test, (re)start
      run_phase<3, kRows>(T, [&](int i) {
        const double xi = xh[i];
        const double ri_ax = row_spmv(P, xh, i, JAC ? xi : __ldg(dg + i) * xi, s_seg);
        const double bi = bh[i];
        const double ri = bi - ri_ax;
        const double d = JAC ? __ldg(dg + i) : 1.0;
        return [=](double* acc) {
          r[i] = ri;
          p[i] = ri;
          acc[0] = fma(ri, ri, acc[0]);      // r^.r^ = r.z
          acc[1] = fma(d * ri, ri, acc[1]);  // r.r
          acc[2] = fma(d * bi, bi, acc[2]);  // b.b
        };
      });
      double s3[3];
      if (!reduce<3>(T, s3)) return;
      if (t == 0) {
        const bool first = c.bb < 0.0;
        if (first) {
          c.bb = s3[2];
          c.stop = P.tol * sqrt(c.bb);
          c.stop2_hi = stop2_high(c.stop);
        }
        const double rel = c.bb > 0.0 ? sqrt(s3[1]) / sqrt(c.bb) : 0.0;
        c.relres = rel;
        c.rho = s3[0];
        c.wrr = JAC && dmin * s3[0] <= kRrMarginB * P.tol * P.tol * c.bb;
        c.act = 0;
        if (c.bb == 0.0) {
          c.status = kOk;
          c.zero = 1;
        } else if (c.status == kBreakdown || c.status == kNumeric) {
          // keep: the residual was only wanted for the report
        } else if (!isfinite(rel)) {
          c.status = kNumeric;
        } else if (rel <= P.tol) {
          c.status = kOk;
        } else if (c.k >= P.maxit || (!first && c.restarts >= P.max_restarts)) {
          c.status = kNotConverged;
        } else {
          if (!first) c.restarts += 1;
          c.act = 1;
        }
      }
      __syncthreads();
      if (!c.act) break;
      for (;;) {
        // ---- A: q = A p, alpha
        run_phase<1, kRows>(T, [&](int i) {
          const double pi = p[i];
          const double qi = row_spmv(P, p, i, JAC ? pi : __ldg(dg + i) * pi, s_seg);
          return [=](double* acc) {
            q[i] = qi;
            acc[0] = fma(pi, qi, acc[0]);
          };
        });
        double s1[1];
        if (!reduce<1>(T, s1)) return;
        if (t == 0) {
          c.act = 1;
          if (!isfinite(s1[0]) || !isfinite(c.rho)) c.status = kNumeric, c.act = 0;
          else if (s1[0] <= 0.0) c.status = kBreakdown, c.act = 0;
          else c.alpha = c.rho / s1[0];
        }
        __syncthreads();
        if (!c.act) break;  // the residual of the current x, then stop
        // ---- B: r -= alpha q, rho' = r^.r^, r.r near the stopping band, beta, test
        const double alpha = c.alpha;
        const bool flag = JAC && c.wrr;
        if (t == 32) c.inv_rho = 1.0 / c.rho;
        run_phase<2, kRowsB, 1>(T, [&](int i) {
          const double ri = fma(-alpha, q[i], r[i]);
          const double di = flag ? __ldg(dg + i) : 0.0;
          return [=](double* acc) {
            r[i] = ri;
            acc[0] = fma(ri, ri, acc[0]);
            if (flag) acc[1] = fma(di * ri, ri, acc[1]);
          };
        }, flag);
        double s2[2] = {0.0, 0.0};
        if (flag) {
          if (!reduce<2>(T, s2)) return;
        } else {
          double w[1];
          if (!reduce<1>(T, w)) return;
          s2[0] = w[0];
        }
        if (t == 0) after_update<JAC>(c, s2[0], s2[1], dmin, P.tol * P.tol * c.bb, P.maxit);
        __syncthreads();
        if (c.exact) {
          run_phase<1, kRows>(T, [&](int i) {
            const double ri = r[i], di = __ldg(dg + i);
            return [=](double* acc) { acc[0] = fma(di * ri, ri, acc[0]); };
          });
          if (!reduce<1>(T, s1)) return;
          if (t == 0) c.last = below_stop(s1[0], c.stop, c.stop2_hi) || c.k >= P.maxit;
          __syncthreads();
        }
        // ---- C: x += alpha p; p = r + beta p unless the loop ends
        const double beta = c.beta;
        const bool last = c.last != 0;
        run_phase<0, kRows>(T, [&](int i) {
          const double pi = p[i];
          const double xn = fma(alpha, pi, xh[i]);
          const double pn = last ? pi : fma(beta, pi, r[i]);
          return [=](double*) {
            xh[i] = xn;
            if (!last) p[i] = pn;
          };
        });
        if (!T.sync()) return;
        if (last) break;
      }
    }
    report(T, c, sys);
  }
}

// fp32 inner solves with fp64 refinement (readings R6 and R8 per system), each as the
// single-system refinement does it: R forms the fp64 residual r = b^ - A^ x^ with the
// fp64 loop matrix, takes the true-residual test and starts an inner solve on
// r32 = fl32(r) (d = 0; with reliable updates, P.carry, the search direction carries
// over: p = r32 + (r32.r32 / rho_k) p_k); A, B, C are the inner fp32 PCG on the fp32
// loop matrix, sums in fp64, until the inner residual has dropped by tol_in; the inner
// solve's last C phase adds fl64(d + alpha p) to x^.  The carried direction is never
// stored before its first use: A gathers r + beta0 p at neighbouring rows, and B
// writes p = r + beta0 p for its own rows before it updates r.
template <bool JAC, int MINB>
__global__ void __launch_bounds__(kBlock, MINB) batch_ir_kernel(BatchParams P) {
  constexpr int kRows = MINB <= 3 ? 4 : 2;
  __shared__ SegInfo s_seg;
  __shared__ XState s_x;
  __shared__ Control c;
  const int t = threadIdx.x;
  int id, rank, size;
  if (!team_init(P, &s_x, &id, &rank, &size)) return;
  Team T{P, s_seg, &s_x, id, rank, size, 0};
  float* __restrict__ r = P.r32;
  float* __restrict__ p = P.p32;
  float* __restrict__ q = P.q32;
  float* __restrict__ d = P.d32;
  double* __restrict__ xh = P.xh;
  const double* __restrict__ bh = P.bh;
  const double* __restrict__ dg = P.dg;
  for (bool first_system = true;; first_system = false) {
    const int sys = next_system(T, first_system);
    if (sys < 0) return;
    control_init(c);
    const double dmin = P.dmin[sys];
    for (;;) {
      // ---- R: fp64 residual, true-residual test, start of an inner solve
      run_phase<4, kRows>(T, [&](int i) {
        const double xi = xh[i];
        const double ax = row_spmv(P, xh, i, JAC ? xi : __ldg(dg + i) * xi, s_seg);
        const double bi = bh[i];
        const double ri = bi - ax;
        const float r32 = (float)ri;
        const double dd = JAC ? __ldg(dg + i) : 1.0;
        return [=](double* acc) {
          r[i] = r32;
          d[i] = 0.0f;
          const double rs = (double)r32;
          acc[0] = fma(rs, rs, acc[0]);       // r32.r32: the inner rho
          acc[1] = fma(dd * rs, rs, acc[1]);  // r32.D r32: the inner solve's reference norm
          acc[2] = fma(dd * ri, ri, acc[2]);  // fp64 r.r
          acc[3] = fma(dd * bi, bi, acc[3]);  // b.b
        };
      });
      double s4[4];
      if (!reduce<4>(T, s4)) return;
      if (t == 0) {
        if (c.bb < 0.0) c.bb = s4[3];
        const double rel = c.bb > 0.0 ? sqrt(s4[2]) / sqrt(c.bb) : 0.0;
        c.relres = rel;
        c.act = 0;
        if (c.bb == 0.0) {
          c.status = kOk;
          c.zero = 1;
        } else if (c.status == kBreakdown || c.status == kNumeric) {
          // keep: the residual was only wanted for the report
        } else if (!isfinite(rel)) {
          c.status = kNumeric;
        } else if (rel <= P.tol) {
          c.status = kOk;
        } else if (c.k >= P.maxit || c.restarts >= P.max_outer || !(s4[0] > 0.0)) {
          c.status = kNotConverged;  // out of iterations or updates (or r32 underflowed to 0)
        } else {
          c.beta0 = (P.carry && c.rho_k > 0.0) ? s4[0] / c.rho_k : 0.0;
          c.rho = s4[0];
          c.stop = P.tol_in * sqrt(s4[1]);
          c.stop2_hi = stop2_high(c.stop);
          c.wrr = JAC && dmin * s4[0] <= kRrMarginB * c.stop * c.stop;
          c.restarts += 1;  // inner solves started (refinement steps / updates)
          c.act = 1;
        }
      }
      __syncthreads();
      if (!c.act) break;
      const float b0 = (float)c.beta0;
      for (bool start = true;; start = false) {
        // ---- A: q = A p (the first step of an inner solve: p = r + beta0 p gathered), alpha
        auto rows_a = [&](auto gx) {
          run_phase<1, kRows>(T, [&, gx](int i) {
            const float pi = gx(i);
            const float dgi = JAC ? 1.0f : (float)__ldg(dg + i);
            const float qi = row_spmv_g<float, float>(P, P.val32, i, dgi * pi, s_seg, gx);
            return [=](double* acc) {
              q[i] = qi;
              acc[0] = fma((double)pi, (double)qi, acc[0]);
            };
          });
        };
        if (!start) rows_a([=](int j) { return p[j]; });
        else if (b0 != 0.0f) rows_a([=](int j) { return fmaf(b0, p[j], r[j]); });
        else rows_a([=](int j) { return r[j]; });
        double s1[1];
        if (!reduce<1>(T, s1)) return;
        if (t == 0) {
          c.act = 1;
          if (!isfinite(s1[0]) || !isfinite(c.rho) || s1[0] <= 0.0) {
            // x^ gets the inner iterate so far (d), then R reports its true residual
            c.status = (!isfinite(s1[0]) || !isfinite(c.rho)) ? kNumeric : kBreakdown;
            c.alpha = 0.0;
            c.act = 0;
            c.last = 1;
          } else {
            c.alpha = c.rho / s1[0];
          }
        }
        __syncthreads();
        const float alpha = (float)c.alpha;
        if (c.act) {
          // ---- B: p = r + beta0 p at the start of an inner solve; r -= alpha q, rho', r.D r
          //      near the band, beta, the inner test
          const bool flag = JAC && c.wrr;
          if (t == 32) c.inv_rho = 1.0 / c.rho;
          run_phase<2, kRows, 1>(T, [&](int i) {
            const float r0 = r[i];
            const float ri = fmaf(-alpha, q[i], r0);
            const float pn = start ? (b0 != 0.0f ? fmaf(b0, p[i], r0) : r0) : 0.0f;
            const double di = flag ? __ldg(dg + i) : 0.0;
            return [=](double* acc) {
              r[i] = ri;
              if (start) p[i] = pn;
              const double rd = (double)ri;
              acc[0] = fma(rd, rd, acc[0]);
              if (flag) acc[1] = fma(di * rd, rd, acc[1]);
            };
          }, flag);
          double s2[2] = {0.0, 0.0};
          if (flag) {
            if (!reduce<2>(T, s2)) return;
          } else {
            double w[1];
            if (!reduce<1>(T, w)) return;
            s2[0] = w[0];
          }
          if (t == 0) after_update<JAC>(c, s2[0], s2[1], dmin, c.stop * c.stop, P.maxit);
          __syncthreads();
          if (c.exact) {
            run_phase<1, kRows>(T, [&](int i) {
              const double rd = (double)r[i], di = __ldg(dg + i);
              return [=](double* acc) { acc[0] = fma(di * rd, rd, acc[0]); };
            });
            if (!reduce<1>(T, s1)) return;
            if (t == 0) c.last = below_stop(s1[0], c.stop, c.stop2_hi) || c.k >= P.maxit;
            __syncthreads();
          }
        }
        // ---- C: d += alpha p, p = r + beta p; the inner solve's last update x^ += fl64(d + alpha p)
        //      (p stays the last direction)
        const bool last = c.last != 0;
        const float beta = (float)c.beta;
        if (last) {
          run_phase<0, kRows>(T, [&](int i) {
            // alpha = 0 (a breakdown at an inner solve's first step): p is not read
            const float pi = alpha != 0.0f ? p[i] : 0.0f;
            const double xn = xh[i] + (double)fmaf(alpha, pi, d[i]);
            return [=](double*) { xh[i] = xn; };
          });
        } else {
          run_phase<0, kRows>(T, [&](int i) {
            const float pi = p[i];
            const float dn = fmaf(alpha, pi, d[i]), pn = fmaf(beta, pi, r[i]);
            return [=](double*) {
              d[i] = dn;
              p[i] = pn;
            };
          });
        }
        if (!T.sync()) return;
        if (last) break;
      }
    }
    report(T, c, sys);
  }
}

// Per-system copies into the concatenated vectors: b^ = D^-1/2 b, x^ = D^1/2 x
// with Jacobi (b, x unchanged without); zeros on padding rows.
__global__ void batch_gather_kernel(const double* const* b, const double* const* x, const int64_t* n,
                                    const int64_t* r0, const int32_t* ntile, const double* disq,
                                    const double* dsq, int jac, double* bh, double* xh) {
  const int s = blockIdx.y;
  const int64_t ns = n[s], base = r0[s], npad = (int64_t)ntile[s] * kTile;
  const double* bs = b[s];
  const double* xs = x[s];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npad;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t gi = base + i;
    if (i < ns) {
      bh[gi] = jac ? bs[i] * disq[gi] : bs[i];
      xh[gi] = jac ? xs[i] * dsq[gi] : xs[i];
    } else {
      bh[gi] = 0.0;
      xh[gi] = 0.0;
    }
  }
}

// x = D^-1/2 x^ (x^ without Jacobi) back into the caller's vectors; x = 0 for b = 0.
__global__ void batch_scatter_kernel(double* const* x, const int64_t* n, const int64_t* r0,
                                     const double* disq, int jac, const double* xh, const int* zero) {
  const int s = blockIdx.y;
  const int64_t ns = n[s], base = r0[s];
  double* xs = x[s];
  const bool z = zero[s] != 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ns;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t gi = base + i;
    xs[i] = z ? 0.0 : (jac ? xh[gi] * disq[gi] : xh[gi]);
  }
}

// Result words of every system and the queue at the start of a solve.
__global__ void batch_init_kernel(int nsys, int* k, int* restarts, int* status, int* zero, unsigned* queue) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < nsys; s += gridDim.x * blockDim.x) {
    k[s] = 0;
    restarts[s] = 0;
    status[s] = kStRunning;
    zero[s] = 0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *queue = 0u;
}

// One system's rows into the concatenated slices (thread per padded row):
// off-diagonal entries of row i in storage order, then padding (column = the
// row itself, value 0) up to the slice width.  With SCALE the values are
// A_ij / sqrt(A_ii A_jj), the two scales multiplied first so the scaled
// matrix stays bitwise symmetric when A is.  col may be null (written with
// the other value variant).
template <bool SCALE>
__global__ void batch_fill_kernel(int64_t n, int64_t npad, int64_t r0, int64_t sl0,
                                  const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                                  const double* __restrict__ vals, const double* __restrict__ ldisq,
                                  const int32_t* __restrict__ soff, int32_t* col, double* val) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npad;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t sl = sl0 + (i >> 5), l = i & 31;
    const int64_t base = (int64_t)soff[sl] * 32 + l;
    const int w = soff[sl + 1] - soff[sl];
    int m = 0;
    if (i < n) {
      const double si = SCALE ? ldisq[i] : 1.0;
      for (int k = rowptr[i]; k < rowptr[i + 1] && m < w; ++k) {
        const int c = colind[k];
        if ((int64_t)c == i) continue;
        if (col) col[base + (int64_t)m * 32] = (int32_t)(r0 + c);
        val[base + (int64_t)m * 32] = SCALE ? vals[k] * (si * ldisq[c]) : vals[k];
        ++m;
      }
    }
    for (; m < w; ++m) {
      if (col) col[base + (int64_t)m * 32] = (int32_t)(r0 + i);
      val[base + (int64_t)m * 32] = 0.0;
    }
  }
}

// The diagonal layout of one system (thread per padded row): slot m of row i
// holds the sum of the row's entries in column i + delta[m] (0 where there is
// none, and on padding rows), scaled as batch_fill_kernel does.
struct BatchDelta {
  int nd;
  int d[kBatchDiag];
};
template <bool SCALE>
__global__ void batch_fill_dia_kernel(int64_t n, int64_t npad, int64_t sl0, const int32_t* __restrict__ rowptr,
                                      const int32_t* __restrict__ colind, const double* __restrict__ vals,
                                      const double* __restrict__ ldisq, const int32_t* __restrict__ soff,
                                      BatchDelta bd, double* val) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npad;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t base = (int64_t)soff[sl0 + (i >> 5)] * 32 + (i & 31);
    double v[kBatchDiag];
#pragma unroll
    for (int m = 0; m < kBatchDiag; ++m) v[m] = 0.0;
    if (i < n) {
      const double si = SCALE ? ldisq[i] : 1.0;
      for (int k = rowptr[i]; k < rowptr[i + 1]; ++k) {
        const int c = colind[k];
        if ((int64_t)c == i) continue;
        const int o = (int)(c - i);
#pragma unroll
        for (int m = 0; m < kBatchDiag; ++m)
          if (m < bd.nd && bd.d[m] == o) v[m] += SCALE ? vals[k] * (si * ldisq[c]) : vals[k];
      }
    }
#pragma unroll
    for (int m = 0; m < kBatchDiag; ++m)
      if (m < bd.nd) val[base + (int64_t)m * 32] = v[m];
  }
}

// Diagonal vectors of one system at its rows of the concatenation: A_ii,
// sqrt(A_ii), 1/sqrt(A_ii) (1 on padding rows and where A_ii <= 0, which
// only the unpreconditioned solve accepts).
__global__ void batch_diag_kernel(int64_t n, int64_t npad, int64_t r0, const double* __restrict__ diag,
                                  double* gd, double* gdsq, double* gdisq) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npad;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double d = i < n ? diag[i] : 1.0;
    const bool pos = d > 0.0;
    const double s = pos ? sqrt(d) : 1.0;
    gd[r0 + i] = d;
    gdsq[r0 + i] = s;
    gdisq[r0 + i] = pos ? 1.0 / s : 1.0;
  }
}

// Kernel variants the autotuner chooses from: registers budgeted for 3 or 4 resident
// CTAs per SM (more CTAs hide more latency; more registers keep more rows in flight).
constexpr int kVariants = 2;
constexpr int kVariantMinBlocks[kVariants] = {3, 4};

const void* batch_kernel(bool jac, int variant, bool f32) {
  if (f32) {
    if (variant == 0) return jac ? (const void*)batch_ir_kernel<true, 3> : (const void*)batch_ir_kernel<false, 3>;
    return jac ? (const void*)batch_ir_kernel<true, 4> : (const void*)batch_ir_kernel<false, 4>;
  }
  if (variant == 0) return jac ? (const void*)batch_pcg_kernel<true, 3> : (const void*)batch_pcg_kernel<false, 3>;
  return jac ? (const void*)batch_pcg_kernel<true, 4> : (const void*)batch_pcg_kernel<false, 4>;
}

// fp32 copy of the loop matrix values (the same rounding as the single-system
// loop: the scaled fp64 value rounded once).
__global__ void batch_to_f32_kernel(int64_t count, const double* __restrict__ v, float* __restrict__ w) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count; k += (int64_t)gridDim.x * blockDim.x)
    w[k] = (float)v[k];
}

// The autotuner's records and the kernels: one slot per (preconditioner, precision kind).
inline int tune_slot(bool jac, bool f32) { return (jac ? 1 : 0) + (f32 ? 2 : 0); }

unsigned blocks_for(int64_t items) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((items + 255) / 256, 4096));
}

}  // namespace

// Device memory of a batch (owned by its cg_handle).
struct BatchData {
  int nsys = 0;
  std::vector<cg_handle*> sys;     // per-system handles (validation, diagonal)
  std::vector<int64_t> n, r0;      // rows and first concatenated row of each system
  std::vector<int32_t> tstart, ntile;
  int64_t rows = 0;                // padded rows in all
  int ntiles = 0, nslices = 0;
  int64_t entries = 0;             // slice entries (multiple of 32)
  int32_t *d_tstart = nullptr, *d_ntile = nullptr, *soff = nullptr, *col = nullptr;
  int32_t *d_ustart = nullptr, *d_nunit = nullptr, *d_utiles = nullptr, *d_order = nullptr, *d_team0 = nullptr;
  std::vector<int32_t> nunit, order;  // reduction units; the queue (systems by descending work)
  std::vector<double> cost;           // work of an iteration of each system (relative)
  std::vector<int32_t> sdia, sdelta;  // diagonal layout of each system and its offsets (kBatchDiag each)
  int32_t *d_sdia = nullptr, *d_sdelta = nullptr;
  int nunits = 0;                  // reduction units in all
  double* d_dmin = nullptr;        // smallest A_ii per system
  int64_t *d_n = nullptr, *d_r0 = nullptr;
  double* val[2] = {nullptr, nullptr};  // [precond]: unscaled / Jacobi-scaled
  float* val32[2] = {nullptr, nullptr}; // fp32 copies (fp32 precisions)
  float *r32 = nullptr, *p32 = nullptr, *q32 = nullptr, *d32 = nullptr;  // inner fp32 vectors
  double *dg = nullptr, *dsq = nullptr, *disq = nullptr;
  double *r = nullptr, *p = nullptr, *q = nullptr, *xh = nullptr, *bh = nullptr;
  double* relres = nullptr;
  int *k = nullptr, *restarts = nullptr, *status = nullptr, *zero = nullptr, *next = nullptr;
  unsigned* queue = nullptr;
  XWord* words = nullptr;          // the teams' exchange words
  int max_teams = 0;               // teams that words, next and d_team0 hold
  std::vector<int32_t> team0;      // the teams on the device (d_team0)
  double* tpart = nullptr;
  const double** d_b = nullptr;    // the caller's vector pointers, on the device
  double** d_x = nullptr;
  void** host_ptrs = nullptr;      // pinned staging of those pointers (2 nsys)
  int grid_max = 0;                // co-resident CTAs of the most occupant variant
  int vmax[kVariants] = {};        // co-resident CTAs of each kernel variant
  int grid_tuned[4] = {};          // chosen CTAs per tune_slot (0: not yet)
  int var_tuned[4] = {};           // chosen kernel variant per tune_slot
  int teams_tuned[4] = {};         // and most teams
  int tune_chosen[4] = {-1, -1, -1, -1};  // index of the chosen candidate
  float tune_ms[4][kMaxCand] = {}; // autotuner timings of the candidates
  int tune_grid[4][kMaxCand] = {};
  int tune_minb[4][kMaxCand] = {};
  int tune_count[4] = {};
  // graph of one solve: status clear, gather, init, the persistent kernel, scatter
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  int gkey_jac = -1, gkey_grid = -1, gkey_var = -1, gkey_maxit = -1, gkey_restarts = -1;
  int gkey_f32 = -1, gkey_carry = -1, gkey_outer = -1, gkey_teams = -1;
  double gkey_tol = -1.0, gkey_timeout = -1.0, gkey_tol_in = -1.0;
  unsigned gkey_skip = 0;
  std::string graph_refused;       // why graph capture failed (then: direct launches)
  cudaStream_t cap_stream = nullptr;  // private stream the graph is captured on
  bool ran_graph = false;          // form of the last solve
  std::vector<int> host_status, host_iters, host_restarts;
  std::vector<double> host_relres;
};

void cgi::batch_free(BatchData* b) {
  if (!b) return;
  for (cg_handle* h : b->sys) cg_destroy(h);
  void* dev[] = {b->d_tstart, b->d_ntile, b->soff,     b->col,    b->d_n,  b->d_r0,   b->val[0],
                 b->val[1],   b->dg,      b->dsq,      b->disq,   b->r,    b->p,      b->q,
                 b->xh,       b->bh,      b->relres,   b->k,        b->restarts, b->status, b->zero,
                 b->tpart,    (void*)b->d_b, (void*)b->d_x, b->d_ustart, b->d_nunit, b->d_utiles, b->d_order,
                 b->d_team0,  b->next,    b->queue,    b->words,    b->d_dmin,
                 b->d_sdia,   b->d_sdelta, b->val32[0], b->val32[1], b->r32, b->p32, b->q32, b->d32};
  for (void* p : dev)
    if (p) cudaFree(p);
  if (b->host_ptrs) cudaFreeHost(b->host_ptrs);
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
  delete b;
}

namespace {

cg_status bfail(cg_handle* h, cg_status s, const std::string& msg) {
  h->err = msg;
  return s;
}

#define CGB_CUDA(h, call)                                                                    \
  do {                                                                                       \
    cudaError_t e_ = (call);                                                                 \
    if (e_ != cudaSuccess)                                                                   \
      return bfail((h), e_ == cudaErrorMemoryAllocation ? CG_ERR_OOM : CG_ERR_CUDA,          \
                   std::string(#call) + ": " + cudaGetErrorString(e_));                      \
  } while (0)

// The concatenated values for one preconditioner (columns written with the first).
cg_status ensure_batch_vals(cg_handle* h, bool jac) {
  BatchData* B = h->batch;
  if (B->val[jac]) return CG_OK;
  const bool write_col = !B->val[0] && !B->val[1];
  CGB_CUDA(h, cudaMalloc(&B->val[jac], sizeof(double) * (size_t)std::max<int64_t>(B->entries, 32)));
  for (int s = 0; s < B->nsys; ++s) {
    const cg_handle* hs = B->sys[(size_t)s];
    const int64_t npad = (int64_t)B->ntile[(size_t)s] * kTile;
    const int64_t r0 = B->r0[(size_t)s];
    const int64_t sl0 = (int64_t)B->tstart[(size_t)s] * kWarps;
    int32_t* col = write_col ? B->col : nullptr;
    if (B->sdia[(size_t)s]) {
      BatchDelta bd{};
      bd.nd = B->sdia[(size_t)s];
      for (int m = 0; m < kBatchDiag; ++m) bd.d[m] = B->sdelta[(size_t)s * kBatchDiag + m];
      if (jac)
        batch_fill_dia_kernel<true><<<blocks_for(npad), 256, 0, h->stream>>>(
            hs->n, npad, sl0, hs->rowptr, hs->colind, hs->vals, B->disq + r0, B->soff, bd, B->val[jac]);
      else
        batch_fill_dia_kernel<false><<<blocks_for(npad), 256, 0, h->stream>>>(
            hs->n, npad, sl0, hs->rowptr, hs->colind, hs->vals, B->disq + r0, B->soff, bd, B->val[jac]);
      continue;
    }
    if (jac)
      batch_fill_kernel<true><<<blocks_for(npad), 256, 0, h->stream>>>(
          hs->n, npad, r0, sl0, hs->rowptr, hs->colind, hs->vals, B->disq + r0, B->soff, col, B->val[jac]);
    else
      batch_fill_kernel<false><<<blocks_for(npad), 256, 0, h->stream>>>(
          hs->n, npad, r0, sl0, hs->rowptr, hs->colind, hs->vals, B->disq + r0, B->soff, col, B->val[jac]);
  }
  CGB_CUDA(h, cudaGetLastError());
  CGB_CUDA(h, cudaStreamSynchronize(h->stream));
  return CG_OK;
}

// fp32 copies of the loop matrix, the inner vectors and the per-system inner state.
cg_status ensure_batch_f32(cg_handle* h, bool jac) {
  BatchData* B = h->batch;
  if (B->val32[jac]) return CG_OK;
  const cg_status vs = ensure_batch_vals(h, jac);
  if (vs != CG_OK) return vs;
  const size_t ent = (size_t)std::max<int64_t>(B->entries, 32);
  CGB_CUDA(h, cudaMalloc(&B->val32[jac], sizeof(float) * ent));
  batch_to_f32_kernel<<<blocks_for((int64_t)ent), 256, 0, h->stream>>>((int64_t)ent, B->val[jac], B->val32[jac]);
  CGB_CUDA(h, cudaGetLastError());
  if (!B->r32) {
    const size_t nv = (size_t)B->rows;
    for (float** v : {&B->r32, &B->p32, &B->q32, &B->d32}) {
      CGB_CUDA(h, cudaMalloc(v, sizeof(float) * nv));
      CGB_CUDA(h, cudaMemsetAsync(*v, 0, sizeof(float) * nv, h->stream));
    }
  }
  CGB_CUDA(h, cudaStreamSynchronize(h->stream));
  return CG_OK;
}

BatchParams make_params(cg_handle* h, bool jac, double tol, int maxit) {
  BatchData* B = h->batch;
  BatchParams P{};
  P.nsys = B->nsys;
  P.tstart = B->d_tstart;
  P.ntile = B->d_ntile;
  P.ustart = B->d_ustart;
  P.nunit = B->d_nunit;
  P.utiles = B->d_utiles;
  P.sdia = B->d_sdia;
  P.sdelta = B->d_sdelta;
  P.dmin = B->d_dmin;
  P.soff = B->soff;
  P.col = B->col;
  P.val = B->val[jac];
  P.dg = B->dg;
  P.r = B->r;
  P.p = B->p;
  P.q = B->q;
  P.xh = B->xh;
  P.bh = B->bh;
  P.relres = B->relres;
  P.k = B->k;
  P.restarts = B->restarts;
  P.status = B->status;
  P.zero = B->zero;
  P.tpart = B->tpart;
  P.bank = (int64_t)B->nunits * kWarps * kNP;
  P.order = B->d_order;
  P.team0 = B->d_team0;
  P.nteams = (int)B->team0.size() - 1;
  P.queue = B->queue;
  P.next = B->next;
  P.words = B->words;
  P.tol = tol;
  P.maxit = maxit;
  P.max_restarts = h->max_restarts;
  P.st = h->st;
  P.timeout_ns = (uint64_t)(h->timeout_ms * 1e6);
  P.skip_seq = h->skip_seq;
  P.val32 = B->val32[jac];
  P.r32 = B->r32;
  P.p32 = B->p32;
  P.q32 = B->q32;
  P.d32 = B->d32;
  P.max_outer = h->max_outer;
  return P;
}

// The teams of a grid of G CTAs, at most `most` of them: with a team for every system,
// CTAs by the systems' work (no more than units); else equal teams that take the
// systems one after the other.  The fault injection gets one team of all CTAs.
std::vector<int32_t> plan_teams(const BatchData* B, int G, int most, bool one) {
  const int ns = B->nsys;
  const int nt = one ? 1 : std::max(1, std::min({ns, G, most, B->max_teams}));
  std::vector<int32_t> size((size_t)nt, 1);
  if (nt == ns && !one) {
    double total = 0.0;
    for (double w : B->cost) total += w;
    int left = G;
    // in descending work, each its share of what is left (rounded down, one at least)
    for (int t = 0; t < nt; ++t) {
      const int s = B->order[(size_t)t];
      const int share = total > 0.0 ? (int)((double)left * B->cost[(size_t)s] / total) : 1;
      size[(size_t)t] = std::max(1, std::min({share, (int)B->nunit[(size_t)s], left - (nt - 1 - t)}));
      left -= size[(size_t)t];
      total -= B->cost[(size_t)s];
    }
  } else {
    for (int t = 0; t < nt; ++t) size[(size_t)t] = G / nt + (t < G % nt ? 1 : 0);
  }
  std::vector<int32_t> team0(1, 0);
  for (int c : size) team0.push_back(team0.back() + c);
  return team0;
}

// Makes those teams the handle's (an upload ordered on its stream when they change).
cudaError_t set_teams(cg_handle* h, int G, int most) {
  BatchData* B = h->batch;
  std::vector<int32_t> t = plan_teams(B, G, most, h->skip_seq != 0);
  if (t == B->team0) return cudaSuccess;
  const cudaError_t e = cudaMemcpyAsync(B->d_team0, t.data(), sizeof(int32_t) * t.size(), cudaMemcpyHostToDevice,
                                        h->stream);
  if (e == cudaSuccess) B->team0 = std::move(t);
  return e == cudaSuccess ? cudaStreamSynchronize(h->stream) : e;  // t is pageable host memory
}

// The work of one solve on h->stream: clear the status words, gather b and
// x, reset the systems, the persistent kernel on G CTAs and (unless this is
// an autotuner trial, which must leave x alone) the scatter of x.
cudaError_t enqueue_solve(cg_handle* h, cudaStream_t s, bool jac, int var, int G, double tol, int maxit,
                          bool scatter, bool f32, bool carry, double tol_in) {
  BatchData* B = h->batch;
  BatchParams P = make_params(h, jac, tol, maxit);
  P.carry = carry ? 1 : 0;
  P.tol_in = tol_in;
  const dim3 gg(64, (unsigned)B->nsys);
  cudaError_t e = cudaMemsetAsync(h->st, 0, sizeof(DevState), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(B->words, 0, sizeof(XWord) * kTeamWords * (size_t)P.nteams, s);
  if (e != cudaSuccess) return e;
  batch_gather_kernel<<<gg, 256, 0, s>>>(B->d_b, B->d_x, B->d_n, B->d_r0, B->d_ntile, B->disq, B->dsq,
                                          jac ? 1 : 0, B->bh, B->xh);
  batch_init_kernel<<<blocks_for(B->nsys), 256, 0, s>>>(B->nsys, B->k, B->restarts, B->status, B->zero, B->queue);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  void* args[] = {&P};
  e = cudaLaunchCooperativeKernel(batch_kernel(jac, var, f32), dim3((unsigned)G), dim3(kBlock), args, 0, s);
  if (e != cudaSuccess || !scatter) return e;
  batch_scatter_kernel<<<gg, 256, 0, s>>>(B->d_x, B->d_n, B->d_r0, B->disq, jac ? 1 : 0, B->xh, B->zero);
  return cudaGetLastError();
}

// Run one solve (through the cached graph when use_graph) between the
// handle's events; the device time goes to *ms.
cg_status run_solve(cg_handle* h, bool jac, int var, int G, int teams, double tol, int maxit, bool use_graph,
                    bool scatter, float* ms, bool f32, bool carry, double tol_in) {
  BatchData* B = h->batch;
  CGB_CUDA(h, set_teams(h, G, teams));
  const int nteams = (int)B->team0.size() - 1;
  if (use_graph && B->graph_refused.empty()) {
    const bool same = B->gexec && B->gkey_jac == (int)jac && B->gkey_grid == G && B->gkey_var == var &&
                      B->gkey_tol == tol && B->gkey_f32 == (int)f32 && B->gkey_carry == (int)carry &&
                      B->gkey_tol_in == tol_in && B->gkey_outer == h->max_outer && B->gkey_teams == nteams &&
                      B->gkey_maxit == maxit && B->gkey_restarts == h->max_restarts &&
                      B->gkey_timeout == h->timeout_ms && B->gkey_skip == h->skip_seq;
    if (!same) {
      if (B->gexec) cudaGraphExecDestroy(B->gexec);
      if (B->graph) cudaGraphDestroy(B->graph);
      B->gexec = nullptr;
      B->graph = nullptr;
      B->gkey_jac = -1;
      // captured on a private stream (the caller's may be the legacy stream, which
      // cannot capture); the graph is then launched on the caller's stream
      if (!B->cap_stream) CGB_CUDA(h, cudaStreamCreateWithFlags(&B->cap_stream, cudaStreamNonBlocking));
      CGB_CUDA(h, cudaStreamBeginCapture(B->cap_stream, cudaStreamCaptureModeThreadLocal));
      const cudaError_t e = enqueue_solve(h, B->cap_stream, jac, var, G, tol, maxit, true, f32, carry, tol_in);
      cudaGraph_t graph = nullptr;
      const cudaError_t e2 = cudaStreamEndCapture(B->cap_stream, &graph);
      cudaError_t e3 = cudaSuccess;
      if (e == cudaSuccess && e2 == cudaSuccess) e3 = cudaGraphInstantiate(&B->gexec, graph, 0);
      if (e != cudaSuccess || e2 != cudaSuccess || e3 != cudaSuccess) {
        // a runtime that cannot capture or instantiate the cooperative launch:
        // run the same kernels as direct launches from now on
        if (graph) cudaGraphDestroy(graph);
        B->gexec = nullptr;
        cudaGetLastError();
        B->graph_refused = cudaGetErrorString(e != cudaSuccess ? e : (e2 != cudaSuccess ? e2 : e3));
        return run_solve(h, jac, var, G, teams, tol, maxit, false, scatter, ms, f32, carry, tol_in);
      }
      B->graph = graph;
      B->gkey_jac = jac;
      B->gkey_grid = G;
      B->gkey_var = var;
      B->gkey_tol = tol;
      B->gkey_maxit = maxit;
      B->gkey_restarts = h->max_restarts;
      B->gkey_timeout = h->timeout_ms;
      B->gkey_skip = h->skip_seq;
      B->gkey_f32 = f32;
      B->gkey_carry = carry;
      B->gkey_tol_in = tol_in;
      B->gkey_outer = h->max_outer;
      B->gkey_teams = nteams;
    }
    CGB_CUDA(h, cudaEventRecord(h->ev0, h->stream));
    CGB_CUDA(h, cudaGraphLaunch(B->gexec, h->stream));
    CGB_CUDA(h, cudaEventRecord(h->ev1, h->stream));
    B->ran_graph = true;
  } else {
    B->ran_graph = false;
    CGB_CUDA(h, cudaEventRecord(h->ev0, h->stream));
    const cudaError_t e = enqueue_solve(h, h->stream, jac, var, G, tol, maxit, scatter, f32, carry, tol_in);
    if (e != cudaSuccess)
      return bfail(h, e == cudaErrorMemoryAllocation ? CG_ERR_OOM : CG_ERR_CUDA,
                   std::string("cg_solve_batch: launch: ") + cudaGetErrorString(e));
    CGB_CUDA(h, cudaEventRecord(h->ev1, h->stream));
  }
  CGB_CUDA(h, cudaMemcpyAsync(h->host_st, h->st, sizeof(DevState), cudaMemcpyDeviceToHost, h->stream));
  CGB_CUDA(h, cudaStreamSynchronize(h->stream));
  CGB_CUDA(h, cudaEventElapsedTime(ms, h->ev0, h->ev1));
  if (h->host_st->abort)
    return bfail(h, CG_ERR_TIMEOUT, "cg_solve_batch: grid barrier " + std::to_string(h->host_st->err_barrier) +
                                        " timed out in CTA " + std::to_string(h->host_st->err_cta));
  return CG_OK;
}

// Autotuner: the kernel variant (registers budgeted for 3 or 4 CTAs per SM, at full
// residency) and the most teams for this handle and preconditioner, picked by timing
// short trial solves (at most kTrialIters iterations each, x left untouched) of the
// caller's own systems; the choice is kept in the handle.  Few large teams keep few
// systems in flight (L2 holds them); many small ones wait less at their barriers.
constexpr int kTrialIters = 40;
constexpr int kManyTeams = 128, kSomeTeams = 32, kFewTeams = 20;

cg_status autotune(cg_handle* h, bool jac, double tol, int maxit, bool f32, bool carry, double tol_in) {
  const int sl = tune_slot(jac, f32);
  BatchData* B = h->batch;
  struct Cand {
    int var, teams;
  };
  const Cand cand[] = {{1, kManyTeams}, {1, kSomeTeams}, {1, kFewTeams}, {0, kSomeTeams}};
  float best = 3.0e38f;
  int best_i = 0, nt = 0;
  for (const Cand& c : cand) {
    float ms = 0.0f;
    const cg_status ts = run_solve(h, jac, c.var, B->vmax[c.var], c.teams, tol, std::min<int32_t>(maxit, kTrialIters),
                                   false, false, &ms, f32, carry, tol_in);
    if (ts != CG_OK) return ts;
    B->tune_ms[sl][nt] = ms;
    B->tune_grid[sl][nt] = B->vmax[c.var];
    B->tune_minb[sl][nt] = kVariantMinBlocks[c.var];
    if (ms < best) {
      best = ms;
      best_i = nt;
    }
    ++nt;
  }
  B->tune_count[sl] = nt;
  B->tune_chosen[sl] = best_i;
  B->var_tuned[sl] = cand[best_i].var;
  B->grid_tuned[sl] = B->vmax[cand[best_i].var];
  B->teams_tuned[sl] = cand[best_i].teams;
  return CG_OK;
}

}  // namespace

extern "C" {

cg_status cg_batch_create(int32_t nsys, const int64_t* n, const int32_t* const* rowptr,
                          const int32_t* const* colind, const double* const* vals, cg_handle** out) {
  if (!out) {
    cgi::set_create_error("cg_batch_create: out is NULL");
    return CG_ERR_INVALID;
  }
  *out = nullptr;
  if (nsys <= 0 || nsys > kMaxBatch) {
    cgi::set_create_error("cg_batch_create: nsys must be in [1, " + std::to_string(kMaxBatch) + "]");
    return CG_ERR_INVALID;
  }
  if (!n || !rowptr || !colind || !vals) {
    cgi::set_create_error("cg_batch_create: NULL array");
    return CG_ERR_INVALID;
  }
  for (int s = 0; s < nsys; ++s)
    if (n[s] <= 0 || n[s] >= INT32_MAX) {
      cgi::set_create_error("cg_batch_create: system " + std::to_string(s) + " has n outside [1, 2^31-1)");
      return CG_ERR_INVALID;
    }
  cg_handle* h = new cg_handle();
  BatchData* B = new BatchData();
  h->batch = B;
  auto bail = [&](cg_status s) {
    cgi::set_create_error(h->err);
    cg_destroy(h);
    return s;
  };
#define CGB_CREATE(call)                                                                   \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess)                                                                 \
      return bail(bfail(h, e_ == cudaErrorMemoryAllocation ? CG_ERR_OOM : CG_ERR_CUDA,     \
                        std::string(#call) + ": " + cudaGetErrorString(e_)));              \
  } while (0)
  int dev = 0;
  CGB_CREATE(cudaGetDevice(&dev));
  CGB_CREATE(cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, dev));
  CGB_CREATE(cudaMalloc(&h->st, sizeof(DevState)));
  CGB_CREATE(cudaMallocHost(&h->host_st, sizeof(DevState)));
  CGB_CREATE(cudaEventCreate(&h->ev0));
  CGB_CREATE(cudaEventCreate(&h->ev1));
  B->nsys = nsys;
  B->n.assign(n, n + nsys);
  B->r0.resize((size_t)nsys);
  B->tstart.resize((size_t)nsys);
  B->ntile.resize((size_t)nsys);
  int64_t rows = 0, tiles = 0, nnz = 0;
  for (int s = 0; s < nsys; ++s) {
    cg_handle* hs = nullptr;
    const cg_status st = cg_create(n[s], rowptr[s], colind[s], vals[s], &hs);
    if (st != CG_OK)
      return bail(bfail(h, st, "cg_batch_create: system " + std::to_string(s) + ": " + cg_last_error(nullptr)));
    B->sys.push_back(hs);
    B->r0[(size_t)s] = rows;
    B->tstart[(size_t)s] = (int32_t)tiles;
    const int64_t nt = (n[s] + kTile - 1) / kTile;
    B->ntile[(size_t)s] = (int32_t)nt;
    rows += nt * kTile;
    tiles += nt;
    nnz += hs->nnz;
    if (rows >= INT32_MAX) return bail(bfail(h, CG_ERR_INVALID, "cg_batch_create: 2^31 rows or more in all"));
  }
  B->rows = rows;
  B->ntiles = (int)tiles;
  B->nslices = (int)(tiles * kWarps);
  h->n = rows;
  h->nnz = nnz;
  // layout of each system: diagonal (stencils: every off-diagonal entry on one
  // of at most kBatchDiag offsets; a slot per offset, no column array read)
  // or sliced ELL; slice widths: the offsets, or the longest off-diagonal row
  // of each 32-row slice
  B->sdia.assign((size_t)nsys, 0);
  B->sdelta.assign((size_t)nsys * kBatchDiag, 0);
  std::vector<int32_t> soff((size_t)B->nslices + 1, 0);
  int64_t off = 0;
  for (int s = 0; s < nsys; ++s) {
    cg_handle* hs = B->sys[(size_t)s];
    const cg_status so = cgi::ensure_offsets(hs);
    if (so != CG_OK) return bail(bfail(h, so, "cg_batch_create: system " + std::to_string(s) + ": " + hs->err));
    if (hs->noffs_all >= 1 && hs->noffs_all <= kBatchDiag) {
      B->sdia[(size_t)s] = hs->noffs_all;
      for (int m = 0; m < hs->noffs_all; ++m) B->sdelta[(size_t)s * kBatchDiag + m] = hs->offs_all[m];
      const int nsl = B->ntile[(size_t)s] * kWarps;
      for (int j = 0; j < nsl; ++j) {
        off += hs->noffs_all;
        soff[(size_t)B->tstart[(size_t)s] * kWarps + j + 1] = (int32_t)off;
      }
      if (off * 32 >= INT32_MAX) return bail(bfail(h, CG_ERR_INVALID, "cg_batch_create: matrices too large"));
      continue;
    }
    std::vector<int32_t> nd((size_t)hs->n);
    CGB_CREATE(cudaMemcpy(nd.data(), hs->ndiag, sizeof(int32_t) * (size_t)hs->n, cudaMemcpyDeviceToHost));
    const cg_status hr = cgi::ensure_host_rowptr(hs);
    if (hr != CG_OK) return bail(bfail(h, hr, "cg_batch_create: system " + std::to_string(s) + ": " + hs->err));
    const std::vector<int32_t>& rp = hs->host_rowptr;
    const int nsl = B->ntile[(size_t)s] * kWarps;
    for (int j = 0; j < nsl; ++j) {
      int w = 0;
      const int64_t i1 = std::min<int64_t>(hs->n, (int64_t)j * 32 + 32);
      for (int64_t i = (int64_t)j * 32; i < i1; ++i)
        w = std::max(w, rp[(size_t)i + 1] - rp[(size_t)i] - nd[(size_t)i]);
      off += w;
      soff[(size_t)B->tstart[(size_t)s] * kWarps + j + 1] = (int32_t)off;
    }
    if (off * 32 >= INT32_MAX) return bail(bfail(h, CG_ERR_INVALID, "cg_batch_create: matrices too large"));
  }
  B->entries = off * 32;
  const size_t nv = (size_t)rows, ns = (size_t)nsys;
  CGB_CREATE(cudaMalloc(&B->soff, sizeof(int32_t) * soff.size()));
  CGB_CREATE(cudaMemcpy(B->soff, soff.data(), sizeof(int32_t) * soff.size(), cudaMemcpyHostToDevice));
  const bool any_ell = std::count(B->sdia.begin(), B->sdia.end(), 0) > 0;
  CGB_CREATE(cudaMalloc(&B->col, sizeof(int32_t) * (size_t)std::max<int64_t>(any_ell ? B->entries : 0, 32)));
  CGB_CREATE(cudaMalloc(&B->d_tstart, sizeof(int32_t) * ns));
  CGB_CREATE(cudaMalloc(&B->d_ntile, sizeof(int32_t) * ns));
  CGB_CREATE(cudaMalloc(&B->d_n, sizeof(int64_t) * ns));
  CGB_CREATE(cudaMalloc(&B->d_r0, sizeof(int64_t) * ns));
  CGB_CREATE(cudaMemcpy(B->d_tstart, B->tstart.data(), sizeof(int32_t) * ns, cudaMemcpyHostToDevice));
  CGB_CREATE(cudaMemcpy(B->d_ntile, B->ntile.data(), sizeof(int32_t) * ns, cudaMemcpyHostToDevice));
  CGB_CREATE(cudaMemcpy(B->d_n, B->n.data(), sizeof(int64_t) * ns, cudaMemcpyHostToDevice));
  CGB_CREATE(cudaMemcpy(B->d_r0, B->r0.data(), sizeof(int64_t) * ns, cudaMemcpyHostToDevice));
  for (double** v : {&B->dg, &B->dsq, &B->disq, &B->r, &B->p, &B->q, &B->xh, &B->bh})
    CGB_CREATE(cudaMalloc(v, sizeof(double) * nv));
  CGB_CREATE(cudaMalloc(&B->relres, sizeof(double) * ns));
  for (int** v : {&B->k, &B->restarts, &B->status, &B->zero}) CGB_CREATE(cudaMalloc(v, sizeof(int) * ns));
  {
    std::vector<int32_t> ust(ns), ut(ns);
    std::vector<double> dmin(ns);
    B->nunit.resize(ns);
    B->cost.resize(ns);
    B->order.resize(ns);
    int units = 0;
    for (size_t s = 0; s < ns; ++s) {
      ut[s] = unit_tiles(B->ntile[s]);
      ust[s] = units;
      B->nunit[s] = (B->ntile[s] + ut[s] - 1) / ut[s];
      units += B->nunit[s];
      dmin[s] = B->sys[s]->jacobi_ok ? B->sys[s]->dmin : 1.0;
      // work of an iteration: fp64 instructions a row, W + 5 for W stored entries
      const int64_t sl0 = (int64_t)B->tstart[s] * kWarps, sl1 = sl0 + (int64_t)B->ntile[s] * kWarps;
      B->cost[s] = 32.0 * (double)(soff[(size_t)sl1] - soff[(size_t)sl0]) + 5.0 * kTile * (double)B->ntile[s];
      B->order[s] = (int32_t)s;
    }
    std::stable_sort(B->order.begin(), B->order.end(),
                     [&](int32_t x, int32_t y) { return B->cost[(size_t)x] > B->cost[(size_t)y]; });
    B->nunits = units;
    B->max_teams = (int)std::min<int64_t>(nsys, 1024);
    auto upload = [&](int32_t** d, const std::vector<int32_t>& v) {
      cudaError_t e = cudaMalloc(d, sizeof(int32_t) * v.size());
      if (e == cudaSuccess) e = cudaMemcpy(*d, v.data(), sizeof(int32_t) * v.size(), cudaMemcpyHostToDevice);
      return e;
    };
    CGB_CREATE(upload(&B->d_ustart, ust));
    CGB_CREATE(upload(&B->d_nunit, B->nunit));
    CGB_CREATE(upload(&B->d_utiles, ut));
    CGB_CREATE(upload(&B->d_order, B->order));
    CGB_CREATE(cudaMalloc(&B->d_dmin, sizeof(double) * ns));
    CGB_CREATE(cudaMemcpy(B->d_dmin, dmin.data(), sizeof(double) * ns, cudaMemcpyHostToDevice));
    CGB_CREATE(cudaMalloc(&B->d_sdia, sizeof(int32_t) * ns));
    CGB_CREATE(cudaMemcpy(B->d_sdia, B->sdia.data(), sizeof(int32_t) * ns, cudaMemcpyHostToDevice));
    CGB_CREATE(cudaMalloc(&B->d_sdelta, sizeof(int32_t) * ns * kBatchDiag));
    CGB_CREATE(cudaMemcpy(B->d_sdelta, B->sdelta.data(), sizeof(int32_t) * ns * kBatchDiag,
                          cudaMemcpyHostToDevice));
  }
  CGB_CREATE(cudaMalloc(&B->d_team0, sizeof(int32_t) * ((size_t)B->max_teams + 1)));
  CGB_CREATE(cudaMalloc(&B->next, sizeof(int) * (size_t)B->max_teams));
  CGB_CREATE(cudaMalloc(&B->queue, sizeof(unsigned)));
  CGB_CREATE(cudaMalloc(&B->words, sizeof(XWord) * kTeamWords * (size_t)B->max_teams));
  CGB_CREATE(cudaMalloc(&B->tpart, sizeof(double) * 2 * (size_t)B->nunits * kWarps * kNP));
  CGB_CREATE(cudaMalloc((void**)&B->d_b, sizeof(double*) * ns));
  CGB_CREATE(cudaMalloc((void**)&B->d_x, sizeof(double*) * ns));
  CGB_CREATE(cudaMallocHost((void**)&B->host_ptrs, sizeof(void*) * 2 * ns));
  for (int s = 0; s < nsys; ++s) {
    const cg_handle* hs = B->sys[(size_t)s];
    const int64_t npad = (int64_t)B->ntile[(size_t)s] * kTile;
    batch_diag_kernel<<<blocks_for(npad), 256>>>(hs->n, npad, B->r0[(size_t)s], hs->diag, B->dg, B->dsq,
                                                 B->disq);
  }
  CGB_CREATE(cudaGetLastError());
  CGB_CREATE(cudaDeviceSynchronize());
  for (int v = 0; v < kVariants; ++v) {
    int per_sm = 1 << 20;
    for (int kind = 0; kind < 4; ++kind) {
      int ps = 0;
      CGB_CREATE(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, batch_kernel(kind & 1, v, kind >= 2), kBlock, 0));
      per_sm = std::min(per_sm, ps);
    }
    B->vmax[v] = per_sm * h->sm_count;
    B->grid_max = std::max(B->grid_max, B->vmax[v]);
  }
#undef CGB_CREATE
  if (B->grid_max <= 0) return bail(bfail(h, CG_ERR_CUDA, "cg_batch_create: occupancy query failed"));
  h->grid_max = B->grid_max;
  B->host_status.assign(ns, 0);
  B->host_iters.assign(ns, 0);
  B->host_restarts.assign(ns, 0);
  B->host_relres.assign(ns, 0.0);
  *out = h;
  return CG_OK;
}

cg_status cg_solve_batch(cg_handle* h, const double* const* b, double* const* x, double tol, int32_t maxit,
                         int32_t precond, int32_t precision, int32_t* iters, double* relres) {
  if (!h) return CG_ERR_INVALID;
  BatchData* B = h->batch;
  if (!B) return bfail(h, CG_ERR_INVALID, "cg_solve_batch: not a batch handle (made by cg_create)");
  h->last = cg_solve_info{};
  if (!b || !x || !(tol >= 0.0) || maxit < 0)
    return bfail(h, CG_ERR_INVALID, "cg_solve_batch: NULL vector array, tol < 0 or maxit < 0");
  if (precond != CG_PRECOND_NONE && precond != CG_PRECOND_JACOBI)
    return bfail(h, CG_ERR_INVALID, "cg_solve_batch: unknown preconditioner");
  if (precision != CG_PREC_FP64 && precision != CG_PREC_FP32_IR && precision != CG_PREC_FP32_RU)
    return bfail(h, CG_ERR_INVALID, "cg_solve_batch: unknown precision");
  if (h->loop_mode == 3)
    return bfail(h, CG_ERR_INVALID, "cg_solve_batch: CG_OPT_LOOP_MODE 3 (unrolled) has no batch form");
  const bool jac = precond == CG_PRECOND_JACOBI;
  for (int s = 0; s < B->nsys; ++s) {
    if (!b[s] || !x[s]) return bfail(h, CG_ERR_INVALID, "cg_solve_batch: NULL vector of system " + std::to_string(s));
    if (jac && !B->sys[(size_t)s]->jacobi_ok)
      return bfail(h, CG_ERR_INVALID,
                   "cg_solve_batch: Jacobi needs a positive diagonal (system " + std::to_string(s) + ")");
  }
  const bool f32 = precision != CG_PREC_FP64;
  const bool carry = precision == CG_PREC_FP32_RU;
  const double tol_in = h->tol_in_set ? h->tol_in : (carry ? 0.1 : 1e-4);
  cg_status vs = f32 ? ensure_batch_f32(h, jac) : ensure_batch_vals(h, jac);
  if (vs != CG_OK) return vs;
  const size_t ns = (size_t)B->nsys;
  const int sl = tune_slot(jac, f32);
  // the previous solve's copies out of host_ptrs have completed (it synchronised)
  std::memcpy(B->host_ptrs, b, sizeof(void*) * ns);
  std::memcpy(B->host_ptrs + ns, x, sizeof(void*) * ns);
  CGB_CUDA(h, cudaMemcpyAsync(B->d_b, B->host_ptrs, sizeof(void*) * ns, cudaMemcpyHostToDevice, h->stream));
  CGB_CUDA(h, cudaMemcpyAsync(B->d_x, B->host_ptrs + ns, sizeof(void*) * ns, cudaMemcpyHostToDevice, h->stream));
  int G = 0, var = 0, teams = kSomeTeams;
  if (h->grid_opt > 0) {
    // a forced grid runs on the variant with the most registers that can hold it; with CTAs
    // enough every system gets a team of its own, sized by its work (64 systems of up to
    // 512^2 rows on 608 CTAs: 234 ms with 32 teams that take them in turn, 196 so)
    G = std::min(h->grid_opt, B->grid_max);
    while (var + 1 < kVariants && B->vmax[var] < G) ++var;
    if (B->nsys <= kManyTeams && G >= 4 * B->nsys) teams = kManyTeams;
  } else {
    if (B->grid_tuned[sl] == 0) {
      const cg_status ts = autotune(h, jac, tol, maxit, f32, carry, tol_in);
      if (ts != CG_OK) return ts;
    }
    G = B->grid_tuned[sl];
    var = B->var_tuned[sl];
    teams = B->teams_tuned[sl];
  }
  const bool use_graph = h->loop_mode != 1;
  float ms = 0.0f;
  const cg_status rs = run_solve(h, jac, var, G, teams, tol, maxit, use_graph, true, &ms, f32, carry, tol_in);
  if (rs != CG_OK) return rs;
  CGB_CUDA(h, cudaMemcpyAsync(B->host_iters.data(), B->k, sizeof(int) * ns, cudaMemcpyDeviceToHost, h->stream));
  CGB_CUDA(h, cudaMemcpyAsync(B->host_restarts.data(), B->restarts, sizeof(int) * ns, cudaMemcpyDeviceToHost, h->stream));
  CGB_CUDA(h, cudaMemcpyAsync(B->host_relres.data(), B->relres, sizeof(double) * ns, cudaMemcpyDeviceToHost, h->stream));
  CGB_CUDA(h, cudaMemcpyAsync(B->host_status.data(), B->status, sizeof(int) * ns, cudaMemcpyDeviceToHost, h->stream));
  CGB_CUDA(h, cudaStreamSynchronize(h->stream));
  int worst_err = 0, nconv = 0, maxk = 0, rmax = 0;
  int64_t bytes = 0;
  double relmax = 0.0;
  for (size_t s = 0; s < ns; ++s) {
    const int st = B->host_status[s], k = B->host_iters[s];
    if (iters) iters[s] = k;
    if (relres) relres[s] = B->host_relres[s];
    if (st < 0 && (worst_err == 0 || st < worst_err)) worst_err = st;
    if (st == CG_NOT_CONVERGED) ++nconv;
    maxk = std::max(maxk, k);
    rmax = std::max(rmax, B->host_restarts[s]);
    relmax = std::max(relmax, B->host_relres[s]);
    const cg_handle* hs = B->sys[s];
    // the single-system traffic model per iteration: CSR matrix and the loop's vectors
    bytes += (f32 ? 8 * hs->nnz + 4 * (hs->n + 1) + (jac ? 52 : 44) * hs->n
                  : 12 * hs->nnz + 4 * (hs->n + 1) + (jac ? 104 : 88) * hs->n) * (int64_t)k;
  }
  cg_solve_info& I = h->last;
  I.status = worst_err ? (cg_status)worst_err : (nconv ? CG_NOT_CONVERGED : CG_OK);
  I.iters = maxk;
  I.restarts = rmax;
  I.grid_ctas = G;
  I.relres_true = relmax;
  I.relres_rec = relmax;
  I.kernel_ms = ms;
  I.bytes_moved = bytes;
  I.kernel_bytes_per_iter = 0;
  I.loop_form = B->ran_graph ? 2 : 1;
  I.kernel_launches = 4;  // gather, init, the persistent kernel, scatter
  if (worst_err)
    return bfail(h, (cg_status)I.status, std::string("cg_solve_batch: at least one system ended with ") +
                                             cg_status_string(worst_err));
  return (cg_status)I.status;
}

cg_status cg_batch_get_system(const cg_handle* h, int32_t s, int32_t* status, int32_t* iters, int32_t* restarts,
                              double* relres) {
  if (!h || !h->batch || s < 0 || s >= h->batch->nsys) return CG_ERR_INVALID;
  const BatchData* B = h->batch;
  if (status) *status = B->host_status[(size_t)s];
  if (iters) *iters = B->host_iters[(size_t)s];
  if (restarts) *restarts = B->host_restarts[(size_t)s];
  if (relres) *relres = B->host_relres[(size_t)s];
  return CG_OK;
}

cg_status cg_batch_get_tuning(const cg_handle* h, int32_t precond, int32_t precision, int32_t* count,
                              int32_t* grids, int32_t* ctas_per_sm, float* ms, int32_t* chosen) {
  if (!h || !h->batch || (precond != CG_PRECOND_NONE && precond != CG_PRECOND_JACOBI)) return CG_ERR_INVALID;
  if (precision != CG_PREC_FP64 && precision != CG_PREC_FP32_IR && precision != CG_PREC_FP32_RU)
    return CG_ERR_INVALID;
  const BatchData* B = h->batch;
  const int j = tune_slot(precond == CG_PRECOND_JACOBI, precision != CG_PREC_FP64);
  if (count) *count = B->tune_count[j];
  for (int c = 0; c < B->tune_count[j]; ++c) {
    if (grids) grids[c] = B->tune_grid[j][c];
    if (ctas_per_sm) ctas_per_sm[c] = B->tune_minb[j][c];
    if (ms) ms[c] = B->tune_ms[j][c];
  }
  if (chosen) *chosen = B->tune_chosen[j];
  return CG_OK;
}

}  // extern "C"
