// SpMV on the caller's CSR matrix (Sec. 3.1: y_i = sum_k vals[k] x[colind[k]]
// over row i's stored entries): cg_spmv, the residuals b - A x of the graph
// form, and the true residuals and refinement residuals of the persistent
// kernels.
//
// The rows are cut (on the device, at creation) into row blocks of at most kCapV nonzeros and
// kBlock rows; a row with more than kCapV nonzeros is a block of its own (a
// "long" block, which the CTA strides over and reduces).  spmv_rowblock_fma:
// the block's column indices and values are copied to shared memory with
// 16-byte loads (four indices, two pairs of values) starting at the 16-byte
// boundary at or below the block's first nonzero.  A block of even rows has them
// summed by one thread each (storage order, fused multiply-adds: one fp64 FMA per
// nonzero), or by two where it holds few long ones (27-point stencils); a block of
// uneven rows has them sorted by length first, its rows of more than kThreadRow
// entries summed by eight lanes each (long_row_sum); a row beyond the block cap is
// summed by the whole CTA.  GB300's fp64 pipe issues 2 FMAs per clock per SM, so a
// separate multiply and add per nonzero (two fp64 instructions) makes a
// 7-point SpMV pipe-bound; with one FMA the kernel is HBM-bound.
#pragma once

#include "cg_device.cuh"

namespace cg {

constexpr int kCap = 2048;                 // shared staging of one row block
constexpr int kCapV = kCap - 4;            // nonzeros of a row block: its 16-byte window fits kCap

// CSR matrix view plus its row-block schedule.  Row block b covers rows
// [rb[b], rb[b+1]).  vec != 0: colind and vals start on 16-byte boundaries, so
// the 16-byte loads of spmv_rowblock_fma are allowed.
template <typename T>
struct Csr {
  int64_t n;
  const int32_t* __restrict__ rowptr;
  const int32_t* __restrict__ colind;
  const T* __restrict__ vals;
  const int32_t* __restrict__ rb;
  int32_t nrb;
  int32_t vec;
};

constexpr int kQuadPasses = 2;
static_assert((kCapV + 3 + 3) / 4 <= kQuadPasses * kBlock, "a row block's window exceeds two quads per thread");
constexpr int kRowUnroll = 4;  // a row's nonzeros whose gathers are in flight together
// Rows with more nonzeros than a thread takes are summed by eight lanes each.  A
// thread takes a row of up to kThreadRow entries; in the caller's CSR, when
// more than kWideRows of a warp's 32 rows have kThreadRow + 1 .. kThreadRowWide
// entries (a 27-point stencil) it takes those too: one thread a row costs the warp
// one FMA step per entry, and no tree of fp64 additions per row; a few such rows
// among short ones go to eight lanes, so they do not hold a warp of short rows.
constexpr int kThreadRow = 16;
constexpr int kThreadRowWide = 32;
constexpr int kWideRows = 4;

// The longest row a thread of this warp keeps (all 32 lanes call it).
__device__ __forceinline__ int thread_row_limit(int len) {
  const unsigned wide = __ballot_sync(0xffffffffu, len > kThreadRow && len <= kThreadRowWide);
  return __popc(wide) > kWideRows ? kThreadRowWide : kThreadRow;
}

// The bounds of a row block: its positions [r0, r1) and entries [k0, k1).
struct BlockSpan {
  int r0, r1, k0, k1;
};
__device__ __forceinline__ BlockSpan block_span(const int32_t* __restrict__ rb, const int32_t* __restrict__ rptr, int b) {
  BlockSpan s;
  s.r0 = __ldg(rb + b);
  s.r1 = __ldg(rb + b + 1);
  s.k0 = __ldg(rptr + s.r0);
  s.k1 = __ldg(rptr + s.r1);
  return s;
}

// The sum of a row's len staged entries from a, in storage order, by one thread; every
// lane of the warp takes wlen steps, keeping its sum past its own row's end.
__device__ __forceinline__ double row_chain(const double* __restrict__ x, const int* s_col, const double* s_val, int a,
                                            int len, int wlen) {
  double s = 0.0;
  int k = 0;
  for (; k + kRowUnroll <= wlen; k += kRowUnroll) {  // kRowUnroll gathers in flight together
    double xv[kRowUnroll], vv[kRowUnroll];
#pragma unroll
    for (int u = 0; u < kRowUnroll; ++u) {
      const bool in = k + u < len;
      vv[u] = in ? s_val[a + k + u] : 0.0;
      xv[u] = in ? __ldg(x + s_col[a + k + u]) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kRowUnroll; ++u) {
      const double nx = fma(vv[u], xv[u], s);
      s = k + u < len ? nx : s;
    }
  }
  for (; k < wlen; ++k) {
    const bool in = k < len;
    const double nx = fma(in ? s_val[a + k] : 0.0, in ? __ldg(x + s_col[a + k]) : 0.0, s);
    s = in ? nx : s;
  }
  return s;
}

// The sum of a long row of len entries by eight lanes (t & 7), in each of them: CHAINS = 4
// chains a lane of every 32nd entry and a fixed tree, as a warp would sum it.  One chain a
// lane of every 8th entry is four times as long, and so are its rounding errors, which fp32
// refinement pays for in iterations (power-law graph of 60,000 rows: 94 against 88), and
// has one gather in flight.
template <int CHAINS, typename T, class Step>
__device__ __forceinline__ T long_row_sum(int len, Step step) {
  T s[CHAINS];
#pragma unroll
  for (int u = 0; u < CHAINS; ++u) s[u] = T(0);
  for (int k = threadIdx.x & 7; k < len; k += 8 * CHAINS) {
#pragma unroll
    for (int u = 0; u < CHAINS; ++u)
      if (k + 8 * u < len) s[u] = step(k + 8 * u, s[u]);
  }
  T acc = CHAINS == 4 ? (s[0] + s[2 % CHAINS]) + (s[1 % CHAINS] + s[3 % CHAINS]) : s[0];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

// One row block of y = A x with one fused multiply-add per nonzero (header
// comment).  The block's column indices and values are copied with 16-byte
// loads into s_col / s_val at their offset from the window start a0.  In a block
// of even rows thread t then sums row r0 + t, in storage order, gathering x itself
// (a warp's gathers for one term cover 32 consecutive rows' neighbours), or two
// threads a row sum its halves; in one of uneven rows s_med lists the rows by
// descending length, the long ones first, which eight lanes each sum, the others
// a thread each.
template <class Next>
__device__ __forceinline__ void spmv_rowblock_fma(const Csr<double>& A, const double* __restrict__ x,
                                                  double* __restrict__ y, const BlockSpan& B, int* s_col,
                                                  double* s_val, int* s_med, int* s_sort, Next next) {
  const int r0 = B.r0, r1 = B.r1, k0 = B.k0, k1 = B.k1;
  const int t = threadIdx.x;
  if (k1 - k0 > kCapV) {  // long row (r1 == r0 + 1 by construction): strided FMA, fixed tree
    double acc = 0.0;
    for (int k = k0 + t; k < k1; k += kBlock) acc = fma(__ldg(A.vals + k), __ldg(x + __ldg(A.colind + k)), acc);
    double v[1] = {acc};
    block_sum<1>(v);
    if (t == 0) y[r0] = v[0];
    next();
    return;
  }
  const int a0 = A.vec ? (k0 & ~3) : k0;
  const int nq = (k1 - a0 + 3) >> 2;
  int4 c4[kQuadPasses];
  double2 va[kQuadPasses], vb[kQuadPasses];
#pragma unroll
  for (int j = 0; j < kQuadPasses; ++j) {  // every load issued before the first store
    const int qd = t + j * kBlock;
    const int k = a0 + 4 * qd;
    c4[j] = make_int4(0, 0, 0, 0);
    va[j] = vb[j] = make_double2(0.0, 0.0);
    if (qd >= nq) continue;
    if (A.vec && k + 4 <= k1) {
      c4[j] = __ldg(reinterpret_cast<const int4*>(A.colind + k));
      va[j] = __ldg(reinterpret_cast<const double2*>(A.vals + k));
      vb[j] = __ldg(reinterpret_cast<const double2*>(A.vals + k + 2));
    } else {  // the ragged end of the block (or unaligned arrays): entries below k1 only
      int c[4] = {0, 0, 0, 0};
      double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u < k1) {
          c[u] = __ldg(A.colind + k + u);
          v[u] = __ldg(A.vals + k + u);
        }
      c4[j] = make_int4(c[0], c[1], c[2], c[3]);
      va[j] = make_double2(v[0], v[1]);
      vb[j] = make_double2(v[2], v[3]);
    }
  }
#pragma unroll
  for (int j = 0; j < kQuadPasses; ++j) {
    const int qd = t + j * kBlock;
    if (qd < nq) {
      *reinterpret_cast<int4*>(s_col + 4 * qd) = c4[j];
      *reinterpret_cast<double2*>(s_val + 4 * qd) = va[j];
      *reinterpret_cast<double2*>(s_val + 4 * qd + 2) = vb[j];
    }
  }
  const int i = r0 + t, nrows = r1 - r0;
  int a = 0, len = 0;
  if (i < r1) {
    a = __ldg(A.rowptr + i) - a0;
    len = __ldg(A.rowptr + i + 1) - a0 - a;
  }
  const bool med = len > thread_row_limit(len);
  // few rows of many entries (27-point stencils: 75 a block): two threads a row below
  const bool halves = 2 * nrows <= kBlock && k1 - k0 > kThreadRow * nrows;
  if (halves && i < r1) s_med[t] = (a << 12) | len;
  // the steps this warp's FMA chain would take beyond what its rows hold
  const int mine = med ? 0 : len;
  const int steps = __reduce_max_sync(0xffffffffu, mine), held = __reduce_add_sync(0xffffffffu, mine);
  const int live = __popc(__ballot_sync(0xffffffffu, i < r1 && !med));
  const bool uneven = __syncthreads_or(med || 4 * held < 3 * live * steps) != 0;
  next();
  if (uneven) {
    // Rows of mixed lengths: a warp of 32 consecutive ones runs to its longest (GB300
    // issues an fp64 warp instruction in full whatever its active lanes: ~14 steps a
    // warp where the rows of a power-law graph average 6, two thirds of the kernel's
    // time on the fp64 pipe), so the block's rows are sorted by length first (counting
    // sort, 32 keys).  Which thread sums a row does not change its sum.
    const int lane = t & 31;
    const int key = i < r1 ? (med ? 0 : 31 - min(len, 30)) : 31;
    const unsigned same = __match_any_sync(0xffffffffu, i < r1 ? key : 32);  // one atomic a key and warp
    const int lead = __ffs(same) - 1;
    int rank = 0;
    if (lane == lead && i < r1) rank = atomicAdd(s_sort + key, __popc(same));
    rank = __shfl_sync(0xffffffffu, rank, lead) + __popc(same & ((1u << lane) - 1u));
    __syncthreads();  // the counts, and the staged entries
    const int cnt = s_sort[lane];
    int before = cnt;  // rows of smaller keys
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += v;
    }
    before -= cnt;
    const int nmed = __shfl_sync(0xffffffffu, cnt, 0);
    const int pos = __shfl_sync(0xffffffffu, before, key) + rank;
    if (i < r1) s_med[pos] = (a << 20) | (len << 8) | t;  // a < 2^12, len < 2^12, t < 2^8
    __syncthreads();
    if (t < 32) s_sort[t] = 0;  // for the next block
    // the long rows by eight lanes each, 32 at a time
    for (int m = t >> 3; m < (nmed + 3) / 4 * 4; m += kBlock / 8) {
      const int e = m < nmed ? s_med[m] : 0;
      const int am = (unsigned)e >> 20, lm = (e >> 8) & 0xFFF;
      const double acc = long_row_sum<4, double>(
          lm, [&](int k, double s) { return fma(s_val[am + k], __ldg(x + s_col[am + k]), s); });
      if ((t & 7) == 0 && m < nmed) y[r0 + (e & 0xFF)] = acc;
    }
    const int at = nmed + t;
    const int e = at < nrows ? s_med[at] : 0;
    a = (unsigned)e >> 20;
    len = (e >> 8) & 0xFFF;
    const int wlen = __reduce_max_sync(0xffffffffu, len);
    const double s = row_chain(x, s_col, s_val, a, len, wlen);
    if (at < nrows) y[r0 + (e & 0xFF)] = s;
    __syncthreads();  // s_col / s_val / s_med are reused by the next row block
    return;
  }
  if (halves) {
    // two threads a row, each the chain of half its entries: with one, 75 of 256 threads
    // worked, each through 27 dependent steps
    const int r = t >> 1;
    const int e = r < nrows ? s_med[r] : 0;
    const int el = e & 0xFFF, h = (el + 1) >> 1;
    const int ea = ((unsigned)e >> 12) + ((t & 1) ? h : 0), en = (t & 1) ? el - h : h;
    double s = row_chain(x, s_col, s_val, ea, en, __reduce_max_sync(0xffffffffu, en));
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (!(t & 1) && r < nrows) y[r0 + r] = s;
    __syncthreads();  // s_col / s_val / s_med are reused by the next row block
    return;
  }
  // one row a thread; the warp's FMA chain runs to its longest row, each lane keeping
  // its sum past its own row's end
  const double s = row_chain(x, s_col, s_val, a, len, steps);
  if (i < r1) y[i] = s;
  __syncthreads();  // s_col / s_val are reused by the next row block
}

// Row blocks cta, cta + stride, ... of y = A x by one CTA (static shared memory of the caller).
// AHEAD: the next block's bounds are read while this one is summed, which two CTAs per SM
// need (FSAI refinement, 1000^2 rows: 4.74 ms without, 4.55 with) and six have no registers
// for (spmv_kernel spilled: 7 points, 150^3 rows, 82.6 us a product against 76.7).
template <bool AHEAD>
__device__ __forceinline__ void spmv_rowblocks(const Csr<double>& A, const double* x, double* y, int cta, int stride,
                                               int* s_col, double* s_val, int* s_med, int* s_sort) {
  if (threadIdx.x < 32) s_sort[threadIdx.x] = 0;
  __syncthreads();
  if constexpr (AHEAD) {
    BlockSpan B{0, 0, 0, 0}, ahead{0, 0, 0, 0};
    if (cta < A.nrb) B = block_span(A.rb, A.rowptr, cta);
    for (int b = cta; b < A.nrb; b += stride) {
      spmv_rowblock_fma(A, x, y, B, s_col, s_val, s_med, s_sort, [&] {
        if (b + stride < A.nrb) ahead = block_span(A.rb, A.rowptr, b + stride);
      });
      B = ahead;
    }
  } else {
    for (int b = cta; b < A.nrb; b += stride)
      spmv_rowblock_fma(A, x, y, block_span(A.rb, A.rowptr, b), s_col, s_val, s_med, s_sort, [] {});
  }
}

// Stand-alone y = A x over all row blocks (cg_spmv, the graph form's residuals);
// CTAs take blocks round-robin, so the grid works on one band of rows at a time
// and the gathers of neighbouring rows meet in L2.  fp64 only.
template <typename T>
__global__ void __launch_bounds__(kBlock, 6) spmv_kernel(Csr<T> A, const T* x, T* y) {
  static_assert(sizeof(T) == sizeof(double), "the stand-alone caller-CSR SpMV is fp64");
  __shared__ __align__(16) int s_col[kCap];
  __shared__ __align__(16) double s_val[kCap];
  __shared__ int s_med[kBlock];
  __shared__ int s_sort[32];
  spmv_rowblocks<false>(A, x, y, (int)blockIdx.x, (int)gridDim.x, s_col, s_val, s_med, s_sort);
}

}  // namespace cg
