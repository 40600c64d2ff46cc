// Device-side building blocks shared by the libcg kernels: exact sums, block and
// grid reductions, the grid exchange (a bounded barrier that carries sums).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "cg_exact.cuh"

namespace cg {

constexpr int kBlock = 256;          // threads per CTA of every libcg kernel
constexpr int kWarps = kBlock / 32;

// Device status words of one persistent launch (zeroed before each launch).
struct DevState {
  unsigned long long bar_arrivals;  // grid-barrier arrivals of this launch (only grows)
  int abort;             // set by any CTA that gave up; every CTA then leaves
  int status;            // cg_status of the solve
  int iters;
  int restarts;
  int err_cta;           // CTA that first timed out (-1 none)
  int err_barrier;       // barrier sequence number where it happened
  double relres_true;
  double relres_rec;
  unsigned long long tphase[6];  // CTA 0 time (ns): SpMV, wait, r update, wait, x/p update, wait
};

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Add without a returned value, ordered after this thread's earlier writes.
__device__ __forceinline__ void red_release_add_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ int ld_relaxed_s32(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid-wide barrier for a co-resident (cooperatively launched) grid.  Every
// wait is bounded: a CTA that waits longer than timeout_ns, or sees another
// CTA's abort flag, records CG_ERR_TIMEOUT (-4) and returns false; the caller
// must then leave the kernel.  `seq` numbers the barriers of the launch
// (1-based) for the fault-injection hook: when skip_seq == seq, CTA 0 does not
// arrive, so the barrier can never complete and every CTA's wait runs out.
// With a single CTA this is a plain __syncthreads().  Thread 32 runs `meanwhile` while
// thread 0 waits; what it writes to shared memory is visible to every thread afterwards.
struct Nothing {
  __device__ __forceinline__ void operator()() const {}
};
template <class F = Nothing>
__device__ __forceinline__ bool grid_barrier(DevState* st, unsigned nblocks, uint64_t timeout_ns,
                                             unsigned seq, unsigned skip_seq, F meanwhile = F()) {
  __shared__ int s_ok;
  if (nblocks == 1) {
    if (threadIdx.x == 32) meanwhile();
    __syncthreads();
    return true;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // barrier seq of this launch is complete when the arrivals reach
    // seq * nblocks: each CTA adds 1 with release order (its partials are
    // visible first) and waits for the total with acquire loads; there is no
    // last arriver to wait for and no reset
    int ok = 1;
    const unsigned long long target = (unsigned long long)seq * nblocks;
    const bool skip = (skip_seq != 0u && seq == skip_seq && blockIdx.x == 0);
    if (!skip) red_release_add_u64(&st->bar_arrivals, 1ull);
    const uint64_t t0 = global_timer_ns();
    unsigned spins = 0;
    while (ld_acquire_u64(&st->bar_arrivals) < target) {
      if (ld_relaxed_s32(&st->abort) != 0) { ok = 0; break; }
      if (((++spins) & 15u) == 0u && global_timer_ns() - t0 > timeout_ns) {
        if (atomicCAS(&st->abort, 0, 1) == 0) {
          st->err_cta = (int)blockIdx.x;
          st->err_barrier = (int)seq;
        }
        ok = 0;
        break;
      }
      __nanosleep(32);
    }
    s_ok = ok;
  }
  if (threadIdx.x == 32) meanwhile();
  __syncthreads();
  return s_ok != 0;
}

// One entry from shared memory (`own`) or from global memory through L2, by predicated
// loads: as a branch per gather the loads of a row waited for one another.  The
// address that is not taken is not touched.
__device__ __forceinline__ double ld_own_or_l2(unsigned smem, const double* global, bool own) {
  double v;
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n @p ld.shared.f64 %0, [%1];\n @!p ld.global.cg.f64 %0, [%2];\n}"
      : "=d"(v)
      : "r"(smem), "l"(global), "r"((unsigned)own)
      : "memory");
  return v;
}
__device__ __forceinline__ float ld_own_or_l2(unsigned smem, const float* global, bool own) {
  float v;
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n @p ld.shared.f32 %0, [%1];\n @!p ld.global.cg.f32 %0, [%2];\n}"
      : "=f"(v)
      : "r"(smem), "l"(global), "r"((unsigned)own)
      : "memory");
  return v;
}

// ---- exact sums on the integer pipes (cg_exact.cuh).  GB300's fp64 unit issues
// one warp instruction per ~64 clocks per SM sub-partition, so a tree of fp64
// adds in one warp (5 levels for a warp, 8 for a CTA) sits on every reduction's
// critical path; these sums use integer instructions and redux.sync, and give
// the exact sum rounded once, whatever the order of the terms.

// Sum over the warp of an integer with |S| < 2^72: four limbs (three unsigned
// 22-bit ones and the signed rest), each summed by one redux.sync, recombined exactly.
__device__ __forceinline__ cg_exact::i128 warp_sum_i128(cg_exact::i128 S) {
  using cg_exact::i128;
  const unsigned l0 = (unsigned)((unsigned long long)S & 0x3FFFFFull);
  const unsigned l1 = (unsigned)((unsigned long long)(S >> 22) & 0x3FFFFFull);
  const unsigned l2 = (unsigned)((unsigned long long)(S >> 44) & 0x3FFFFFull);
  const int l3 = (int)(S >> 66);
  const unsigned s0 = __reduce_add_sync(0xffffffffu, l0);
  const unsigned s1 = __reduce_add_sync(0xffffffffu, l1);
  const unsigned s2 = __reduce_add_sync(0xffffffffu, l2);
  const int s3 = __reduce_add_sync(0xffffffffu, l3);
  return (i128)s0 + (i128)s1 * ((i128)1 << 22) + (i128)s2 * ((i128)1 << 44) + (i128)s3 * ((i128)1 << 66);
}

// warp_sum_i128 for 64-bit terms: three limbs (two unsigned 22-bit ones and the signed rest).
__device__ __forceinline__ cg_exact::i128 warp_sum64(long long X) {
  using cg_exact::i128;
  const unsigned l0 = (unsigned)((unsigned long long)X & 0x3FFFFFull);
  const unsigned l1 = (unsigned)(((unsigned long long)X >> 22) & 0x3FFFFFull);
  const int l2 = (int)(X >> 44);
  const unsigned s0 = __reduce_add_sync(0xffffffffu, l0);
  const unsigned s1 = __reduce_add_sync(0xffffffffu, l1);
  const int s2 = __reduce_add_sync(0xffffffffu, l2);
  return (i128)s0 + (i128)s1 * ((i128)1 << 22) + (i128)s2 * ((i128)1 << 44);
}

// In every lane: the exact sum of the lanes' fp64 values at the warp's scale *E
// (the largest exponent field among them).
__device__ __forceinline__ cg_exact::i128 warp_exact_sum(double v, int* E, bool* bad) {
  const cg_exact::Parts p = cg_exact::parts(v);
  // one redux for the scale and the NaN flag (a bad sum is NaN; any scale >= every e will do)
  const unsigned eb = __reduce_max_sync(0xffffffffu, (unsigned)p.e | (p.bad ? 0x10000u : 0u));
  *bad = eb > 0xFFFFu;
  *E = *bad ? 2046 : (int)(eb & 0xFFFFu);
  return warp_sum64(cg_exact::to_fixed(p, *E));
}

// The same, packed with that scale.
__device__ __forceinline__ ulonglong2 warp_exact(double v) {
  int E;
  bool bad;
  const cg_exact::i128 S = warp_exact_sum(v, &E, &bad);
  unsigned long long lo, hi;
  cg_exact::pack(S, E, bad, &lo, &hi);
  return make_ulonglong2(lo, hi);
}

// In every lane: the exact sum of the lanes' fp64 values rounded once, with no
// fp64 instruction (for loops bound by GB300's fp64 pipe, where a 5-level fp64
// xor tree would take 5 of its warp instructions).
__device__ __forceinline__ double warp_sum_exact(double v) {
  const ulonglong2 w = warp_exact(v);
  int E;
  bool bad;
  const cg_exact::i128 S = cg_exact::unpack(w.x, w.y, &E, &bad);
  return cg_exact::to_fp64_int(S, E, bad);
}

// In every lane of a warp: the packed entries held by its lanes (lanes without
// one hold zero at scale 1) moved to their largest scale and added exactly.
__device__ __forceinline__ cg_exact::i128 sum_entries(const ulonglong2& w, bool has, int* Em, bool* bad) {
  int E = 1;
  bool b = false;
  const cg_exact::i128 S = has ? cg_exact::unpack(w.x, w.y, &E, &b) : (cg_exact::i128)0;
  *Em = (int)__reduce_max_sync(0xffffffffu, (unsigned)E);
  *bad = __reduce_or_sync(0xffffffffu, b ? 1u : 0u) != 0u;
  return warp_sum_i128(cg_exact::shift_down(S, *Em - E));
}

// Sum of v over the CTA, valid in warp 0: each warp's exact sum (warp_exact),
// then warp 0 adds the 8 warp sums exactly and rounds once to fp64.  The result
// does not depend on which thread held which value.
template <int NV>
__device__ __forceinline__ void cta_sum0(double (&v)[NV]) {
  __shared__ ulonglong2 s_w[NV][kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ulonglong2 w[NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) w[j] = warp_exact(v[j]);
  __syncthreads();  // s_w may still be read by warp 0 of a previous call
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) s_w[j][warp] = w[j];
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      int E;
      bool bad;
      const cg_exact::i128 T = sum_entries(s_w[j][lane < kWarps ? lane : 0], lane < kWarps, &E, &bad);
      v[j] = cg_exact::to_fp64(T, E, bad);
    }
  }
}

// beta = rho' / rho as rho' (1 / rho), a multiply on the critical path where a division
// would be (within 1.5 ulp of it); the division itself where 1 / rho is not a normal
// number (rho below about 2^-1024 would make it infinite, above 2^1022 lose bits).
__device__ __forceinline__ double beta_of(double rho1, double rho, double inv_rho) {
  const unsigned e = ((unsigned)__double2hiint(inv_rho) >> 20) & 0x7FFu;
  return e - 1u < 0x7FEu ? rho1 * inv_rho : rho1 / rho;
}

// Sum of v over the CTA in a fixed order (warp xor-tree, then warp 0 over the
// per-warp sums); the result is returned to every thread.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV]) {
  __shared__ double s_red[NV][kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
  }
  __syncthreads();  // s_red may still be read from a previous call
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) s_red[j][warp] = v[j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += s_red[j][w];
    v[j] = t;
  }
}

// The stopping test sqrt(rr) <= stop with the square root (a ~700-clock chain
// on GB300's fp64 pipe) taken only near the band.  stop2_hi = stop^2 (1 + 1e-12)
// rounded exceeds stop^2, and rr above it has sqrt(rr) above stop by ~5e-13
// relative (thousands of ulps), so the test is false without the root and the
// decision is the one sqrt(rr) <= stop gives.  A stop whose square under- or
// overflows (or NaN) gets stop2_hi = inf: always the exact test.
__device__ __forceinline__ double stop2_high(double stop) {
  const double s = stop * stop * (1.0 + 1e-12);
  return s >= 1e-300 ? s : INFINITY;
}
// The root stays inside its branch through a register dependence on an empty
// asm: the compiler had been computing it on every call.
__device__ __forceinline__ bool below_stop(double rr, double stop, double stop2_hi) {
  if (!(rr <= stop2_hi)) return false;
  double r = rr;
  asm volatile("" : "+d"(r));
  return sqrt(r) <= stop;
}

// Sum of the G per-CTA partials part[j*G + c], exact and rounded once, given to
// every thread.  Lane l of warp 0 takes partials l, l + 32, ..., kGridBatch loads
// in flight at a time, and adds them exactly at a running scale (the largest
// exponent seen: a larger one shifts the lane's sum down first); the 32 lane sums
// meet at the largest scale (sum_entries' alignment, one redux.sync a limb).
// Every CTA computes the identical value (same loads, same order), so decisions
// made from it agree across the grid without another barrier.
template <int NV>
__device__ __forceinline__ void grid_sum_lanes(const double* part, unsigned G, double (&out)[NV]) {
  constexpr int kGridBatch = NV <= 2 ? 8 : 1;  // NV > 2: the once-per-solve residual sums
  __shared__ double s_out[NV];
  if (threadIdx.x < 32) {
    const unsigned lane = threadIdx.x;
    cg_exact::i128 acc[NV];
    int Ea[NV];
    bool bad[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      acc[j] = 0;
      Ea[j] = 1;
      bad[j] = false;
    }
    for (unsigned c0 = lane; c0 < G; c0 += 32u * kGridBatch) {
      double v[kGridBatch][NV];
#pragma unroll
      for (int u = 0; u < kGridBatch; ++u) {
        const unsigned c = c0 + 32u * u;
#pragma unroll
        for (int j = 0; j < NV; ++j) v[u][j] = c < G ? __ldcg(part + (size_t)j * G + c) : 0.0;
      }
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        // the batch's largest exponent field from the bits, then one value at a
        // time (few registers live: the persistent kernels are register-budgeted)
        int Eb = Ea[j];
#pragma unroll
        for (int u = 0; u < kGridBatch; ++u) {
          const int f = (int)((cg_exact::bits_of(v[u][j]) >> 52) & 0x7FF);
          bad[j] = bad[j] || f == 0x7FF;
          Eb = max(Eb, f == 0x7FF ? 1 : max(f, 1));
        }
        if (Eb > Ea[j]) {
          acc[j] = cg_exact::shift_down(acc[j], Eb - Ea[j]);
          Ea[j] = Eb;
        }
#pragma unroll
        for (int u = 0; u < kGridBatch; ++u) acc[j] += (cg_exact::i128)cg_exact::to_fixed(cg_exact::parts(v[u][j]), Eb);
      }
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      unsigned long long lo, hi;
      cg_exact::pack(acc[j], Ea[j], bad[j], &lo, &hi);
      int E;
      bool bd;
      const cg_exact::i128 T = sum_entries(make_ulonglong2(lo, hi), true, &E, &bd);
      const double r = cg_exact::to_fp64(T, E, bd);
      if (lane == 0) s_out[j] = r;
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < NV; ++j) out[j] = s_out[j];
  __syncthreads();
}

// The same sum with every thread loading: thread t takes partials t, t + 256, ...
// (at most kPer = 4 of them, all loads in flight: one L2 round trip), each warp
// sums each of its kPer loads exactly (warp_exact), and warp 0 adds the warps'
// entries, one a lane, exactly and rounds once.  For G > 1024, or in the
// one-warp scalar kernels of the graph forms, the lane form.
template <int NV>
__device__ __forceinline__ void grid_sum(const double* part, unsigned G, double (&out)[NV]) {
  constexpr int kPer = 4;
  if (G > (unsigned)(kPer * kBlock) || blockDim.x != (unsigned)kBlock) {
    grid_sum_lanes<NV>(part, G, out);
    return;
  }
  __shared__ ulonglong2 s_w[NV][kPer * kWarps];
  __shared__ double s_out[NV];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (int)((G + kBlock - 1) / kBlock);  // loads a thread makes (uniform)
  double v[kPer][NV];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const unsigned c = threadIdx.x + (unsigned)(k * kBlock);
#pragma unroll
    for (int j = 0; j < NV; ++j) v[k][j] = (k < per && c < G) ? __ldcg(part + (size_t)j * G + c) : 0.0;
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (k < per) {
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        const ulonglong2 w = warp_exact(v[k][j]);
        if (lane == 0) s_w[j][k * kWarps + warp] = w;
      }
    }
  }
  __syncthreads();
  if (warp == 0) {
    const int ne = per * kWarps;  // <= 32 entries: one a lane
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      int E;
      bool bad;
      const cg_exact::i128 T = sum_entries(s_w[j][lane < ne ? lane : 0], lane < ne, &E, &bad);
      const double r = cg_exact::to_fp64(T, E, bad);
      if (lane == 0) s_out[j] = r;
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < NV; ++j) out[j] = s_out[j];
  __syncthreads();
}

// ---- exchanges of a co-resident (cooperatively launched) grid
//
// One exchange is a grid barrier that carries NV sums at no further cost: a CTA adds
// its exact sum, as an integer at a scale every CTA knows, to accumulators in L2,
// three words on lines of their own, and each word's top 9 bits count the CTAs that
// have added.  A CTA has the grid's sum when every count
// is complete: one reduction without a returned value and one poll, the round trip a
// plain arrival counter takes.  (Partials read back after a counter's wait cost a
// second round trip and a tree, ~4 us a sum of 304 CTAs; all CTAs polling all CTAs'
// slots 6-9 us, and in two levels of ~18 slots 4 us, most of it fences.)
//
// The accumulators only grow: a CTA subtracts the words it read when their last use
// was complete.  Exchanges alternate between two sets of words: nobody adds to a set
// again before every CTA has arrived at the exchange in between, so has read it.
//
// The scale is that of the last sum of the same kind, with room both ways.  A CTA
// whose sum does not fit (or is not finite) says so in the third word, and a total
// far below the last one would lack bits: then, the same in every CTA, the largest
// exponent is exchanged first and the sum is formed again at that scale.
template <int WARPS>                           // most CTAs, of WARPS warps, that exchange sums
constexpr int kXCtas = cg_exact::kMaxSums / WARPS < cg_exact::kMaxAddends ? cg_exact::kMaxSums / WARPS
                                                                          : cg_exact::kMaxAddends;
constexpr int kXVals = 2;                      // most sums per exchange
constexpr int kXKinds = 7;                     // kinds of sums whose scales are kept

// One word a 128-byte line: per set a plain counter (barriers without a sum) and
// three limbs a value, each in kXSplit words that every kXSplit-th CTA adds to and that
// a poll reads together (atomics on one address go one after the other: 152 of them
// took about as long as the round trip); then the largest-exponent word.
struct XWord {
  unsigned long long w;
  unsigned long long pad[15];
};
constexpr int kXSplit = 4;
constexpr int kXWords = kXSplit * (1 + 3 * kXVals);
constexpr int kXAll = 2 * kXWords + 1;
constexpr size_t kXBytes = sizeof(XWord) * kXAll;
static_assert(kXSplit * 3 * kXVals <= 32, "a lane a word");

// A CTA's exchanges, in shared memory: its grid (or group of a grid), the words at
// their last use and the scales of the last sums.
struct XState {
  DevState* st;
  XWord* words;
  uint64_t timeout_ns;
  unsigned G, rank;   // CTAs that exchange; this one's number among them
  unsigned seq;       // exchanges so far
  unsigned skip_seq;  // fault injection: do not add at this exchange (1-based; 0: never)
  int scale[kXKinds];  // exponent field of the last sum; 0: none yet
  unsigned long long prev[2][kXWords];
};

__device__ __forceinline__ void x_init(XState* x, DevState* st, XWord* words, unsigned G, unsigned rank,
                                       unsigned skip_seq, uint64_t timeout_ns) {
  for (int k = threadIdx.x; k < 2 * kXWords; k += blockDim.x) x->prev[k / kXWords][k % kXWords] = 0ull;
  for (int k = threadIdx.x; k < kXKinds; k += blockDim.x) x->scale[k] = 0;
  if (threadIdx.x == 0) {
    x->st = st;
    x->words = words;
    x->timeout_ns = timeout_ns;
    x->G = G;
    x->rank = rank;
    x->seq = 0;
    x->skip_seq = skip_seq;
  }
  __syncthreads();
}

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void red_add(XWord* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(&p->w), "l"(v) : "memory");
}
__device__ __forceinline__ void red_max(XWord* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.max.u64 [%0], %1;" ::"l"(&p->w), "l"(v) : "memory");
}
template <bool ORDER>
__device__ __forceinline__ unsigned long long ld_word(const XWord* p) {
  unsigned long long v;
  if (ORDER) asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(&p->w) : "memory");
  else asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(&p->w) : "memory");
  return v;
}

// Warp 0 adds add[w] to the n words w0 + w of the exchange's set (lane kXSplit w + k
// holds add[w] and word k of its split) and waits (bounded) until their counts, at bit
// `at`, say that all G CTAs have; *diff: what the CTAs added to the lane's word.
// False: a wait gave up.  ORDER: this CTA's global writes
// (before the caller's last __syncthreads) come before its words, and the other CTAs'
// writes before theirs are visible after the wait (acquiring polls: relaxed ones and a
// fence after the wait took ~0.3 us more).
template <bool ORDER>
__device__ __forceinline__ bool x_round(XState* c, unsigned seq, int w0, int n, int at, unsigned long long add,
                                        unsigned long long* diff) {
  const int lane = threadIdx.x & 31;
  bool ok = true;
  unsigned long long d = 0;
  if (ORDER) fence_gpu();
  if (lane < kXSplit * n) {
    const unsigned sub = (unsigned)lane % kXSplit;
    const unsigned G = (c->G + kXSplit - 1 - sub) / kXSplit;  // CTAs that add to this word
    XWord* w = c->words + (seq & 1u) * kXWords + kXSplit * w0 + lane;
    unsigned long long* prev = &c->prev[seq & 1u][kXSplit * w0 + lane];
    const unsigned long long was = *prev;
    if (c->rank % kXSplit == sub && c->skip_seq != seq) red_add(w, add);
    uint64_t t0 = 0;
    for (unsigned spins = 0;; ++spins) {
      const unsigned long long now = ld_word<ORDER>(w);
      d = now - was;
      if ((d >> at) == G) {
        *prev = now;
        break;
      }
      if (spins == 0) t0 = global_timer_ns();
      if ((spins & 15u) == 15u) {
        if (ld_relaxed_s32(&c->st->abort) != 0) { ok = false; break; }
        if (global_timer_ns() - t0 > c->timeout_ns) {
          if (atomicCAS(&c->st->abort, 0, 1) == 0) {
            c->st->err_cta = (int)blockIdx.x;
            c->st->err_barrier = (int)seq;
          }
          ok = false;
          break;
        }
      }
    }
  }
  *diff = d;
  return __all_sync(0xffffffffu, ok);
}

// The sum of value j from the lanes that hold its words.
__device__ __forceinline__ cg_exact::i128 x_join(unsigned long long d, int j, int* exceptions) {
#pragma unroll
  for (int o = 1; o < kXSplit; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  return cg_exact::join_limbs(__shfl_sync(0xffffffffu, d, kXSplit * 3 * j), __shfl_sync(0xffffffffu, d, kXSplit * (3 * j + 1)),
                              __shfl_sync(0xffffffffu, d, kXSplit * (3 * j + 2)), exceptions);
}

struct XSums {
  double v0, v1;
  bool ok;
};

// The next exchange of c, called by every thread.  Warp 0
// gets the sums over the grid of the threads' v0 and v1 (NV of them, of kinds `kind`,
// `kind` + 1; NV = 0 is a plain barrier, of any G), exact and rounded once, the same
// bits in every CTA, and whether it succeeded; the other warps return at once and meet
// warp 0 at the caller's next __syncthreads().  Global writes made by any CTA before
// the exchange are visible to every CTA after that.  Every wait is bounded: a CTA that
// waits longer than timeout_ns, or sees another's abort flag, records CG_ERR_TIMEOUT
// and gets ok = false; the caller must then leave the kernel.
// Not inlined: the 128-bit steps would cost the persistent kernels' loops registers.
template <int NV, int WARPS = kWarps, bool ORDER = true>
__device__ __noinline__ XSums grid_exchange(XState* c, int kind, double v0, double v1) {
  constexpr int kN = NV > 0 ? NV : 1;
  // the warps' sums at their own scales, and as limbs at the exchange's scale (all ones
  // in the third limb: it does not fit there)
  __shared__ ulonglong2 s_w[kN][WARPS];
  __shared__ unsigned long long s_l[3 * kN][WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double v[2] = {v0, v1};
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    int E;
    bool bad;
    cg_exact::i128 S = warp_exact_sum(v[j], &E, &bad);
    if (lane == 3) {
      unsigned long long lo, hi;
      cg_exact::pack(S, E, bad, &lo, &hi);
      s_w[j][warp] = make_ulonglong2(lo, hi);
    }
    const int e = c->scale[kind + j];
    const bool fits = e != 0 && cg_exact::to_scale(&S, E, bad, max(1, e - cg_exact::kRoom));
    if (lane < 3) s_l[3 * j + lane][warp] = fits ? cg_exact::limb(S, lane) : (lane == 2 ? ~0ull : 0ull);
  }
  __syncthreads();  // the warps' sums, and every global write of this CTA, before the words
  XSums r{0.0, 0.0, true};
  if (warp != 0) return r;
  unsigned s = c->seq + 1;
  __syncwarp();
  unsigned long long d;
  if (NV == 0) {
    if (c->G > 1) {
      r.ok = x_round<ORDER>(c, s, 0, 1, 0, 1ull, &d);
      if (lane == 0) c->seq = s;
    }
    return r;
  }
  double out[kN];
  if (c->G == 1) {
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      int E;
      bool bad;
      const cg_exact::i128 S = sum_entries(s_w[j][lane < WARPS ? lane : 0], lane < WARPS, &E, &bad);
      out[j] = cg_exact::to_fp64(S, E, bad);
    }
  } else {
    unsigned long long add = 0;
    if (lane < kXSplit * 3 * kN) {
      const int l = lane / kXSplit;
      bool out = false;
#pragma unroll
      for (int w = 0; w < WARPS; ++w) {
        const unsigned long long x = s_l[l][w];
        out = out || x == ~0ull;
        add += x == ~0ull ? 0ull : x;
      }
      add += (1ull << cg_exact::kCountAt) + (out ? 1ull << cg_exact::kExcAt : 0ull);
    }
    r.ok = x_round<ORDER>(c, s, 1, 3 * kN, cg_exact::kCountAt, add, &d);
    bool again = false;
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      const int B = max(1, c->scale[kind + j] - cg_exact::kRoom);
      int exc;
      out[j] = cg_exact::to_fp64(x_join(d, j, &exc), B, false);
      again = again || exc != 0 || !cg_exact::enough_bits(out[j], B);
    }
    if (again && r.ok) {  // the same decision in every CTA: the largest exponent first, then the sums
      XWord* mx = c->words + 2 * kXWords;
#pragma unroll 1
      for (int j = 0; j < kN; ++j) {
        int E;
        bool bad;
        cg_exact::i128 S = sum_entries(s_w[j][lane < WARPS ? lane : 0], lane < WARPS, &E, &bad);
        ++s;
        if (lane == 0) red_max(mx, ((unsigned long long)s << 32) | (unsigned)(bad ? 2047 : E));
        __syncwarp();
        r.ok = x_round<true>(c, s, 0, 1, 0, 1ull, &d) && r.ok;
        __syncwarp();
        const int Em = (int)(ld_word<true>(mx) & 0xFFFFull), B = max(1, Em - cg_exact::kRoom);
        ++s;
        const bool fits = cg_exact::to_scale(&S, E, bad, B);
        add = (1ull << cg_exact::kCountAt) + (fits ? cg_exact::limb(S, lane / kXSplit) : 0ull);
        r.ok = x_round<ORDER>(c, s, 1, 3, cg_exact::kCountAt, add, &d) && r.ok;
        int exc;
        const double o = cg_exact::to_fp64(x_join(d, 0, &exc), B, Em >= 2047);
        if (j == 0) out[0] = o;
        else out[kN - 1] = o;
      }
    }
    if (lane == 0) {
      c->seq = s;
#pragma unroll
      for (int j = 0; j < kN; ++j) {
        const int e = (int)((cg_exact::bits_of(out[j]) >> 52) & 0x7FF);
        c->scale[kind + j] = e == 0x7FF ? 0 : e;
      }
    }
  }
  r.v0 = out[0];
  r.v1 = out[kN - 1];
  return r;
}

}  // namespace cg
