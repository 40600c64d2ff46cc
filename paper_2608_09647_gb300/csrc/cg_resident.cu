// The fp64 CG loop of a stencil system (sliced-diagonal loop matrix) too large for one
// thread-block cluster and small enough for the SMs together: one CTA per SM keeps
// its rows of x^, r^, q and p, and where they fit its rows of the loop matrix, in
// shared memory for the whole solve (CG_OPT_LOOP_MODE 1; cg_solve's readings R1-R5,
// scaling and stopping test as in cg_kernels.cuh).
//
// What bounds an iteration at these sizes is latency: three grid-wide exchanges, the
// fp64 scalars between them, and the loads of each phase.  Here the r update and the
// x / p update touch no global memory, the SpMV reads only the p of other CTAs' rows
// (L2; its own from shared memory), and a thread meets the same rows in every phase.
// p is also written to global memory, for the other CTAs; the exchange after that is
// the only one that orders global writes, so the other two need no fence.  The form
// with all vectors in global memory, ~2 rows a thread over 304 CTAs, spent 12 of its
// 17 us an iteration on exchanges and most of the rest on L2 round trips: 17.3 us an
// iteration at 301^2 rows, 9 points, now 11.3 (8 of them the exchanges); 43 us at 97^3
// rows, 7 points, now 25.6 (10.6 the SpMV, at the fp64 unit's rate).
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "cg_handle.cuh"

using namespace cg;

namespace {

constexpr int kThreads = 512;  // one CTA per SM, four warps per sub-partition for the fp64 unit
constexpr int kRWarps = kThreads / 32;
constexpr int kVecs = 4;       // x^, r^, q, p of a CTA's rows
constexpr int kGroup = 4;      // rows of a thread together in the vector phases: a store to shared memory
                               // holds back the next row's loads (13.7 K clocks for 12 rows a thread)

struct ResidentParams {
  SolveParams P;
  int spc;  // 32-row slices per CTA
};

// A row's gathered entries: this CTA's rows from shared memory, the others from L2
// (never from L1: other CTAs write them every iteration).
struct Gather {
  unsigned own;  // shared-memory address of the CTA's first row
  const double* all;
  int r0, nr, nm1;
  __device__ __forceinline__ double operator()(int c) const {
    c = min(max(c, 0), nm1);
    const unsigned l = (unsigned)(c - r0);
    return ld_own_or_l2(own + 8u * l, all + c, l < (unsigned)nr);
  }
};

// acc + the off-diagonal part of the row with slots vp[0], vp[32], ... (W slots at
// compile time, all loads before the first product; W = 0: w of them, eight at a time).
template <int W>
__device__ __forceinline__ double row_sum(const Sell<double>& S, const double* vp, const Gather& p, int i, double acc) {
  constexpr int CH = W > 0 ? W : 8;
  const int w = W > 0 ? W : S.uw;
  for (int m0 = 0; m0 < w; m0 += CH) {
    double v[CH], x[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      if (W > 0 || m0 + u < w) {
        v[u] = vp[(m0 + u) * 32];
        x[u] = p(i + S.delta[m0 + u]);
      }
    }
#pragma unroll
    for (int u = 0; u < CH; ++u)
      if (W > 0 || m0 + u < w) acc = fma(v[u], x[u], acc);
  }
  return acc;
}

// MS: the loop matrix's rows are in shared memory too (else streamed from L2).
template <bool JAC, int W, bool MS>
__global__ void __launch_bounds__(kThreads, 1) pcg64_resident_kernel(ResidentParams RP) {
  const SolveParams& P = RP.P;
  const Sell<double>& S = P.S64;
  extern __shared__ __align__(16) double sm[];
  __shared__ XState s_x;
  __shared__ double s_alpha, s_beta, s_rho, s_rr, s_inv_rho, s_sum[3];
  __shared__ int s_st, s_want, s_exact, s_conv;
  const int t = threadIdx.x, n = (int)S.n;
  const int r0 = (int)blockIdx.x * RP.spc * 32;
  const int nr = min(n - r0, RP.spc * 32), cap = RP.spc * 32;
  double* xs = sm;
  double* rs = xs + cap;
  double* qs = rs + cap;
  double* ps = qs + cap;
  double* pg = P.V64.p;
  const int w = W > 0 ? W : S.uw;
  const double* vals = S.val + (int64_t)blockIdx.x * RP.spc * w * 32;
  if (MS) {  // this CTA's slices, as they are
    double* ms = ps + cap;
    const int ne = (nr + 31) / 32 * w * 32;
    for (int k = t; k < ne; k += kThreads) ms[k] = __ldcs(vals + k);
    vals = ms;
  }
  // (fault injection: CTA 0 does not add to exchange number skip_seq)
  x_init(&s_x, P.st, P.xs, gridDim.x, blockIdx.x, blockIdx.x == 0 ? P.skip_seq : 0u, P.timeout_ns);
  const Gather gp{(unsigned)__cvta_generic_to_shared(ps), pg, r0, nr, n - 1};
  // an exchange of sums whose CTAs hand over no global writes, and one that orders them
  auto sum1 = [&](double a, int kind) { return grid_exchange<1, kRWarps, false>(&s_x, kind, a, 0.0); };
  auto sum2 = [&](double a, double b, int kind) { return grid_exchange<2, kRWarps, false>(&s_x, kind, a, b); };
  auto sync = [&]() { return __syncthreads_and(grid_exchange<0, kRWarps, true>(&s_x, 0, 0.0, 0.0).ok) != 0; };

  int status = kNotConverged, k = 0, restarts = 0;
  double relres_true = 0.0, rr = 0.0, bb = 0.0;
  bool first = true, report = false;
  for (;;) {
    // a5 / (re)start: r = b - A x; r^ = D^-1/2 r; x^ = D^1/2 x
    double v[3] = {0.0, 0.0, 0.0};
    for (int li = t; li < nr; li += kThreads) {
      const int i = r0 + li;
      double s = 0.0;
      const int e = __ldg(P.A.rowptr + i + 1);
#pragma unroll 4
      for (int kk = __ldg(P.A.rowptr + i); kk < e; ++kk)
        s = fma(__ldg(P.A.vals + kk), __ldcg(P.x + __ldg(P.A.colind + kk)), s);
      const double bi = P.b[i], ri = bi - s;
      v[1] = fma(ri, ri, v[1]);
      if (report) continue;
      const double rh = JAC ? ri * __ldg(P.disq + i) : ri;
      const double xi = __ldcg(P.x + i);
      rs[li] = rh;
      ps[li] = rh;
      pg[i] = rh;
      xs[li] = JAC ? xi * __ldg(P.dsq + i) : xi;
      v[0] = fma(rh, rh, v[0]);
      v[2] = fma(bi, bi, v[2]);
    }
    const XSums a = sum2(v[0], v[1], kKindRes);
    if (t == 0) {
      s_sum[0] = a.v0;
      s_sum[1] = a.v1;
    }
    if (!__syncthreads_and(a.ok)) { status = kTimeout; break; }
    const XSums c = grid_exchange<1, kRWarps, true>(&s_x, kKindRes + 2, v[2], 0.0);
    if (t == 0) s_sum[2] = c.v0;
    if (!__syncthreads_and(c.ok)) { status = kTimeout; break; }
    const double rho0 = s_sum[0], rr0 = s_sum[1];
    if (report) {
      relres_true = sqrt(rr0) / sqrt(bb);
      break;
    }
    if (first) {
      bb = s_sum[2];
      if (bb == 0.0) {  // b = 0: x = 0 solves it
        for (int li = t; li < nr; li += kThreads) P.x[r0 + li] = 0.0;
        status = kOk;
        break;
      }
    } else {
      relres_true = sqrt(rr0) / sqrt(bb);
      if (!isfinite(relres_true)) { status = kNumeric; break; }
      if (relres_true <= P.tol) { status = kOk; break; }
      if (k >= P.maxit || restarts >= P.max_restarts) { status = kNotConverged; break; }
      ++restarts;
    }
    const bool was_first = first;
    first = false;
    rr = rr0;
    const int k_before = k;
    const double stop = P.tol * sqrt(bb), stop2_hi = stop2_high(stop);
    double rho = rho0;
    int st = kNotConverged;
    bool done = sqrt(rr) <= stop || k >= P.maxit;  // a4: tested before every SpMV
    if (sqrt(rr) <= stop) st = kOk;
    while (!done) {
      // a1: q = A^ p; p.q
      double pq = 0.0;
      for (int li = t; li < nr; li += kThreads) {
        const double pi = ps[li];
        const double* vp = vals + (li >> 5) * (w * 32) + (li & 31);
        const double qi = row_sum<W>(S, vp, gp, r0 + li, JAC ? pi : __ldg(S.dg + r0 + li) * pi);
        qs[li] = qi;
        pq = fma(pi, qi, pq);
      }
      const XSums x1 = sum1(pq, kKindPQ);
      if (t == 0) {
        s_st = !x1.ok ? kTimeout : ((!isfinite(x1.v0) || !isfinite(rho)) ? kNumeric : (x1.v0 <= 0.0 ? kBreakdown : 0));
        s_alpha = rho / x1.v0;
        s_want = JAC && rr_wanted(S, rho, stop * stop);
      }
      __syncthreads();
      if (s_st) { st = s_st; break; }
      // a2: r^ -= alpha q; r.z, r.r (r.r only when the test needs it); 1 / rho for
      // this iteration's beta (beta_of) in warp 1 meanwhile
      const double alpha = s_alpha;
      const bool want_rr = s_want != 0;
      if (t == 32) s_inv_rho = 1.0 / rho;
      double a_rho = 0.0, a_rr = 0.0;
      for (int l0 = t; l0 < nr; l0 += kGroup * kThreads) {
        double q[kGroup], r[kGroup];
#pragma unroll
        for (int u = 0; u < kGroup; ++u) {
          const int li = l0 + u * kThreads;
          q[u] = li < nr ? qs[li] : 0.0;
          r[u] = li < nr ? rs[li] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kGroup; ++u) r[u] = fma(-alpha, q[u], r[u]);
#pragma unroll
        for (int u = 0; u < kGroup; ++u) {
          const int li = l0 + u * kThreads;
          if (li < nr) {
            rs[li] = r[u];
            a_rho = fma(r[u], r[u], a_rho);
            if (JAC && want_rr) a_rr = fma(__ldg(S.dn + r0 + li) * r[u], r[u], a_rr);
          }
        }
      }
      XSums x2 = JAC && want_rr ? sum2(a_rho, a_rr, kKindUpd) : sum1(a_rho, kKindUpd);
      if (!(JAC && want_rr)) x2.v1 = x2.v0;  // plain CG: r.z is r.r
      if (t == 0) {
        double rr_ = x2.v1;
        if (!x2.ok) s_st = kTimeout;
        s_exact = JAC && !want_rr && rr_bound_test(S, x2.v0, stop * stop, &rr_) < 0;
        s_beta = beta_of(x2.v0, rho, s_inv_rho);
        s_rho = x2.v0;
        s_rr = rr_;
        s_conv = below_stop(rr_, stop, stop2_hi);
      }
      __syncthreads();
      if (s_st) { st = s_st; break; }
      const double beta = s_beta;
      rho = s_rho;
      if (s_exact) {  // rho fell into the band early: exact r.r
        double e = 0.0;
        for (int li = t; li < nr; li += kThreads) e = fma(__ldg(S.dn + r0 + li) * rs[li], rs[li], e);
        const XSums x3 = sum1(e, kKindRr);
        if (t == 0) {
          if (!x3.ok) s_st = kTimeout;
          s_rr = x3.v0;
          s_conv = below_stop(x3.v0, stop, stop2_hi);
        }
        __syncthreads();
        if (s_st) { st = s_st; break; }
      }
      rr = s_rr;
      ++k;
      const bool conv = s_conv != 0;
      done = conv || k >= P.maxit;
      if (conv) st = kOk;
      // a3: x^ += alpha p; p = r^ + beta p (last iteration: the caller's x)
      for (int l0 = t; l0 < nr; l0 += kGroup * kThreads) {
        double p[kGroup], x[kGroup], r[kGroup];
#pragma unroll
        for (int u = 0; u < kGroup; ++u) {
          const int li = l0 + u * kThreads;
          p[u] = li < nr ? ps[li] : 0.0;
          x[u] = li < nr ? xs[li] : 0.0;
          r[u] = li < nr ? rs[li] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kGroup; ++u) {
          x[u] = fma(alpha, p[u], x[u]);
          if (!done) p[u] = fma(beta, p[u], r[u]);
        }
#pragma unroll
        for (int u = 0; u < kGroup; ++u) {
          const int li = l0 + u * kThreads;
          if (li < nr) {
            xs[li] = x[u];
            if (done) {
              P.x[r0 + li] = JAC ? x[u] * __ldg(S.disq + r0 + li) : x[u];
            } else {
              ps[li] = p[u];
              pg[r0 + li] = p[u];
            }
          }
        }
      }
      if (!sync()) { st = kTimeout; break; }
    }
    if (st == kTimeout) { status = kTimeout; break; }
    if (st == kNumeric || st == kBreakdown) {  // x gets the last iterate; its true residual is reported
      status = st;
      if (k > k_before)
        for (int li = t; li < nr; li += kThreads) P.x[r0 + li] = JAC ? xs[li] * __ldg(S.disq + r0 + li) : xs[li];
      if (!sync()) { status = kTimeout; break; }
      report = true;
      continue;
    }
    if (was_first && k == k_before && st == kOk) {  // x0 met tol: its true residual is known
      relres_true = sqrt(rr0) / sqrt(bb);
      status = kOk;
      break;
    }
    // kOk or kNotConverged: the true residual next
  }
  if (blockIdx.x == 0 && t == 0) {
    P.st->status = status;
    P.st->iters = k;
    P.st->restarts = restarts;
    P.st->relres_true = relres_true;
    P.st->relres_rec = bb > 0.0 ? sqrt(rr) / sqrt(bb) : 0.0;
  }
}

template <bool MS>
const void* kernel_for(int uw, bool jac) {
  switch (uw) {
    case 4: return jac ? (const void*)pcg64_resident_kernel<true, 4, MS> : (const void*)pcg64_resident_kernel<false, 4, MS>;
    case 6: return jac ? (const void*)pcg64_resident_kernel<true, 6, MS> : (const void*)pcg64_resident_kernel<false, 6, MS>;
    case 8: return jac ? (const void*)pcg64_resident_kernel<true, 8, MS> : (const void*)pcg64_resident_kernel<false, 8, MS>;
    default: return jac ? (const void*)pcg64_resident_kernel<true, 0, MS> : (const void*)pcg64_resident_kernel<false, 0, MS>;
  }
}

}  // namespace

// The most bytes of a loop matrix streamed by this form.  Past them the matrix no longer
// stays in the 126 MB L2 beside the vectors, and the 16 warps an SM that stream it are too
// few.  Only matrices of more than 8 diagonals get there before their vectors outgrow shared
// memory.  The line lies where the graph form overtakes, sooner for 27 points, whose 26
// slots have a product of their own there.  fp64 Jacobi to 1e-12, ms, graph form and this:
// 27 points 72^3 rows (78 MB) 5.74 and 5.56, 74^3 (84 MB) 6.06 and 6.32, 90^3 (152 MB) 9.41
// and 10.9; 19 points 70^3 (49 MB) 6.44 and 4.78, 90^3 (105 MB) 10.2 and 9.48, 100^3
// (144 MB) 12.3 and 12.2; 13 points 100^3 (96 MB) 10.4 and 9.42.
int64_t streamed_max_bytes(int diagonals) { return diagonals == 26 ? 80000000 : 144000000; }

cudaError_t cgi::resident_launch(const cg_handle* h, const SolveParams& P, bool jac, int* grid, bool* launched) {
  *launched = false;
  if (!h->dia || h->n < 1) return cudaSuccess;
  cudaError_t e;
  const int ctas = std::min(h->sm_count, kXCtas<kRWarps>);
  const int spc = (int)((h->nslices + ctas - 1) / ctas);
  for (int ms = 1; ms >= 0; --ms) {
    if (!ms && (int64_t)sizeof(double) * h->sell_entries > streamed_max_bytes(h->uniform_w)) continue;
    const void* fn = ms ? kernel_for<true>(h->uniform_w, jac) : kernel_for<false>(h->uniform_w, jac);
    size_t limit = 0;
    if ((e = allow_dynamic_smem(fn, &limit)) != cudaSuccess) return e;
    const size_t smem = sizeof(double) * 32 * (size_t)spc * (size_t)(kVecs + (ms ? h->uniform_w : 0));
    if (smem > limit) continue;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, smem)) != cudaSuccess) return e;
    const int G = (int)((h->nslices + spc - 1) / spc);
    if (per_sm < 1 || G > per_sm * h->sm_count) continue;
    *grid = G;
    if ((e = cudaMemsetAsync(h->st, 0, kStBytes, h->stream)) != cudaSuccess) return e;
    if ((e = cudaEventRecord(h->ev0, h->stream)) != cudaSuccess) return e;
    ResidentParams RP{P, spc};
    void* args[] = {&RP};
    *launched = true;
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)G), dim3(kThreads), args, smem, h->stream);
  }
  return cudaSuccess;
}
