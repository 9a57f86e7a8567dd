// CUDA kernels of one Parallel CFR iteration (sm_103a).
//
// The paper's seven stages (Section 4.1, Table 1) are regrouped by what couples them:
//   * every pass along the tree -- regret matching (Eq. rm), forward reach (Stage 1),
//     backward values (Stage 6, Eq. backward), the regret / average update (Stage 7) and
//     the best-response backward pass -- is independent per private hand.  k_hand gives
//     each CUDA block a chunk of hands and walks all tree levels for them, with only
//     __syncthreads() between levels; the chunk's per-node state sits in shared memory
//     when it fits, else in the global arrays (L2);
//   * terminal values need the opponent's whole reach vector: k_terminal gives each block
//     one fold or showdown node and evaluates it in O(hands) (Stages 2-4): card-blocker
//     inclusion-exclusion at folds, rank-sorted prefix sums with per-card corrections at
//     showdowns.
// One player's update is therefore two launches (terminal, then hand), recorded once in
// a CUDA graph.  Inside k_hand the FP64 regret / average update is one fully parallel pass
// over (row, hand) items after the backward levels, so GB300's long FP64 latency is paid
// once per launch rather than once per tree level.
//
// Precision: cumulative regrets R and average sums S are FP64 (GB300 runs FP64 at about
// 1/64 of the FP32 rate, so FP64 is kept to those updates).  Reach, strategies and values
// are either double-float pairs on the FP32 pipe (Pairs, the default: ~44-bit
// significands, so regrets that are small differences of large values keep their digits)
// or plain FP32 (Single).
#include <cuda_runtime.h>

#include <cstdio>
#include <type_traits>

#include "pcfr_internal.h"

namespace pcfr {

constexpr int kHandThreads = 256;
constexpr int kTermThreads = 512;


// ------------------------------------------------------------------ double-float arithmetic
//
// A value is hi + lo with |lo| <= ulp(hi) / 2.  Sums use Knuth's TwoSum (TAOCP vol. 2,
// section 4.2.2) on both halves followed by renormalisation (Dekker 1971; the "accurate"
// addition of Hida, Li and Bailey's double-double library); products use the FMA form of
// Dekker's exact product.  The _rn intrinsics stop the compiler from contracting or
// reassociating the error terms.

using ff = PairF;  // (hi, lo)

__device__ __forceinline__ ff ff_of(float x) { return {x, 0.f}; }
__device__ __forceinline__ ff ff_neg(ff a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {  // |a| >= |b|
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  float s1, s2, t1, t2;
  two_sum(a.hi, b.hi, s1, s2);
  two_sum(a.lo, b.lo, t1, t2);
  s2 = __fadd_rn(s2, t1);
  fast_two_sum(s1, s2, s1, s2);
  s2 = __fadd_rn(s2, t2);
  fast_two_sum(s1, s2, s1, s2);
  return {s1, s2};
}
__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }
// Sum of two double-floats of the same sign (no cancellation possible): TwoSum of the high
// parts, low parts added in FP32, one renormalisation -- about half the operations of ff_add.
__device__ __forceinline__ ff ff_add_pos(ff a, ff b) {
  float s, e, hi, lo;
  two_sum(a.hi, b.hi, s, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  fast_two_sum(s, e, hi, lo);
  return {hi, lo};
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  float hi, lo;
  fast_two_sum(p, e, hi, lo);
  return {hi, lo};
}
// Compensated accumulation (Ogita, Rump and Oishi 2005, "Accurate sum and dot product",
// Sum2 / Dot2): a running FP32 sum s, with every rounding error -- found exactly by TwoSum
// and by the FMA form of TwoProduct -- added into a separate FP32 error sum e.  The
// critical path is one FP32 addition per term, and s + e, kept as a pair, carries about
// twice the working precision.
struct acc2 {
  float s, e;
};
__device__ __forceinline__ acc2 acc_zero() { return {0.f, 0.f}; }
__device__ __forceinline__ void acc_add(acc2& a, ff x) {
  float t, err;
  two_sum(a.s, x.hi, t, err);
  a.s = t;
  a.e = __fadd_rn(a.e, __fadd_rn(err, x.lo));
}
__device__ __forceinline__ void acc_fma(acc2& a, ff x, ff y) {  // a += x * y
  const float p = __fmul_rn(x.hi, y.hi);
  const float pe = __fmaf_rn(x.hi, y.hi, -p);
  const float cross = __fmaf_rn(x.hi, y.lo, __fmul_rn(x.lo, y.hi));
  float t, err;
  two_sum(a.s, p, t, err);
  a.s = t;
  a.e = __fadd_rn(a.e, __fadd_rn(err, __fadd_rn(pe, cross)));
}
__device__ __forceinline__ void acc_merge(acc2& a, acc2 b) {
  float t, err;
  two_sum(a.s, b.s, t, err);
  a.s = t;
  a.e = __fadd_rn(a.e, __fadd_rn(err, b.e));
}
__device__ __forceinline__ ff acc_value(acc2 a) {
  float hi, lo;
  two_sum(a.s, a.e, hi, lo);
  return {hi, lo};
}

// 1 / b: the FP32 reciprocal refined by one Newton step in double-float.
__device__ __forceinline__ ff ff_recip(ff b) {
  const ff r = ff_of(__frcp_rn(b.hi));
  return ff_add(r, ff_mul(r, ff_sub(ff_of(1.f), ff_mul(b, r))));
}
__device__ __forceinline__ bool ff_gt(ff a, ff b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }

// Exact float -> double by exponent rebias on the integer pipe (IEEE 754 binary32 ->
// binary64; subnormal floats, below 1.2e-38, become zero).
__device__ __forceinline__ double f2d(float f) {
  const uint32_t u = __float_as_uint(f), a = u & 0x7fffffffu;
  uint32_t hi = (a >> 3) + 0x38000000u, lo = u << 29;  // exponent + 896, mantissa up by 29 bits
  if (a >= 0x7f800000u) hi += 0x38000000u;             // infinity and NaN: exponent 0x7ff
  if (a < 0x00800000u) hi = lo = 0u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)lo);
}
// double -> float, round to nearest even, on the integer pipe where the result is a normal float (or
// overflows by rounding): 29 mantissa bits off with the carry, exponent - 896.  A conversion holds the
// FP64 pipe as long as an addition; without it a row of the hand tiles' updates needs that pipe three
// times, not four: Leduc 5.44 -> 5.25 ms, resident river 4.12 -> 4.08, 256 rivers 69.4 -> 69.0.  The
// wide update, which waits on memory, keeps the conversion (without it the exact turn is 0.3 % slower).
__device__ __forceinline__ float d2f(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x), a = hi & 0x7fffffffu;
  if (a - 0x38100000u < 0x0fe00000u) {  // 2^-126 <= |x| < 2^128
    const uint64_t r = ((uint64_t)(a - 0x38000000u) << 32 | lo) + 0x0fffffffu + ((lo >> 29) & 1u);
    return __uint_as_float((uint32_t)(r >> 29) | (hi & 0x80000000u));
  }
  return __double2float_rn(x);  // zeros, results below the normal floats, infinities and NaN
}
__device__ __forceinline__ ff d2ff(double x) {
  const float hi = __double2float_rn(x);
  return {hi, __double2float_rn(x - f2d(hi))};
}
__device__ __forceinline__ double ff2d(ff a) { return f2d(a.hi) + f2d(a.lo); }

// ------------------------------------------------------------------ precision policies

struct Pairs {  // double-float values
  using V = ff;
  static __device__ __forceinline__ V zero() { return ff_of(0.f); }
  static __device__ __forceinline__ V add(V a, V b) { return ff_add(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return ff_sub(a, b); }
  static __device__ __forceinline__ V mul(V a, V b) { return ff_mul(a, b); }
  static __device__ __forceinline__ V vmax(V a, V b) { return ff_gt(b, a) ? b : a; }
  static __device__ __forceinline__ bool positive(V a) { return a.hi > 0.f; }
  static __device__ __forceinline__ V recip(V a) { return ff_recip(a); }
  static __device__ __forceinline__ V one() { return ff_of(1.f); }
  static __device__ __forceinline__ V uniform(int A) { return ff_recip(ff_of((float)A)); }  // 1 / A
  static __device__ __forceinline__ V of_double(double x) { return d2ff(x); }
  static __device__ __forceinline__ V of_double_int(double x) {  // the same value
    const float hi = d2f(x);
    return {hi, d2f(x - f2d(hi))};
  }
  static __device__ __forceinline__ double to_double(V a) { return ff2d(a); }
  static __device__ __forceinline__ V scale(ff u) { return u; }  // a payoff scale as a value
  using Acc = acc2;
  static __device__ __forceinline__ Acc acc0() { return acc_zero(); }
  static __device__ __forceinline__ void acc(Acc& a, V x) { acc_add(a, x); }
  static __device__ __forceinline__ void acc_mul(Acc& a, V x, V y) { acc_fma(a, x, y); }
  static __device__ __forceinline__ V value(Acc a) { return acc_value(a); }
};

struct Single {  // plain FP32 values
  using V = float;
  static __device__ __forceinline__ V zero() { return 0.f; }
  static __device__ __forceinline__ V add(V a, V b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ V mul(V a, V b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ V vmax(V a, V b) { return fmaxf(a, b); }
  static __device__ __forceinline__ bool positive(V a) { return a > 0.f; }
  // correctly rounded reciprocal: the same bits as 1 / a in IEEE division
  static __device__ __forceinline__ V recip(V a) { return __frcp_rn(a); }
  static __device__ __forceinline__ V one() { return 1.f; }
  static __device__ __forceinline__ V uniform(int A) { return __frcp_rn((float)A); }
  static __device__ __forceinline__ V of_double(double x) { return __double2float_rn(x); }
  static __device__ __forceinline__ V of_double_int(double x) { return d2f(x); }  // the same value
  static __device__ __forceinline__ double to_double(V a) { return f2d(a); }
  static __device__ __forceinline__ V scale(ff u) { return u.hi; }
  using Acc = float;
  static __device__ __forceinline__ Acc acc0() { return 0.f; }
  static __device__ __forceinline__ void acc(Acc& a, V x) { a = __fadd_rn(a, x); }
  static __device__ __forceinline__ void acc_mul(Acc& a, V x, V y) { a = fmaf(x, y, a); }
  static __device__ __forceinline__ V value(Acc a) { return a; }
};

// ------------------------------------------------------------------ block primitives (double-float)

__device__ __forceinline__ acc2 acc_shfl_up(acc2 a, int o) {
  return {__shfl_up_sync(0xffffffffu, a.s, o), __shfl_up_sync(0xffffffffu, a.e, o)};
}

// ------------------------------------------------------------------ bulk copies (TMA) into shared memory

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// Make the barrier's initialisation visible to the asynchronous (TMA) proxy.
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// One-dimensional bulk copy global -> shared; both addresses and the size are multiples of 16.
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Asynchronous element copies global -> shared (cp.async): every copy of a block is in
// flight at once instead of one load-then-store round trip per loop iteration.
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  static_assert(BYTES == 4 || BYTES == 8 || BYTES == 16, "cp.async copies 4, 8 or 16 bytes");
  if (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Programmatic dependent launch.  Every kernel first stages what launches two or more steps
// back produced, then waits for its immediate predecessor (griddepcontrol.wait returns once
// that grid has completed and its writes are visible), and only then lets its own dependent
// start.  So whenever a kernel is running, everything but its immediate predecessor has
// completed, which is what makes the early staging safe.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Bounded wait for phase `parity` of the barrier: false if it did not complete within
// `limit` polls.
constexpr long kWaitLimit = 1l << 20;
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity, long limit = kWaitLimit) {
  for (long k = 0; k < limit; ++k)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// Polls the terminal kernel's first bulk-copy wait of each block makes before it gives up:
// kWaitLimit, unless a test lowers it to exercise the timeout path (with 0 the block gives
// up before its copies can land, drains them with the full limit, sets the error flag and
// returns).  Every other wait keeps kWaitLimit.
__device__ long g_first_wait_polls = kWaitLimit;

// ------------------------------------------------------------------ terminal values (Stages 2-4)

// Whether hand h (its cards from the staged table: c1 | c2 << 8) holds a card of `board`.
__device__ __forceinline__ bool holds_board_card(const uint16_t* cards, int h, int k, uint64_t board) {
  const unsigned cw = cards[h];
  return (((board >> (cw & 0xffu)) | (k == 2 ? board >> (cw >> 8) : 0ull)) & 1ull) != 0;
}

// Values of player i at fold and showdown nodes (Stages 2-4) from the opponent's reach q there.
// kappa = 1/Z, and a node's payoff already carries the probability of the public cards dealt on its
// path, so every value is a counterfactual value in the sense of Eq. (cfv).
//   fold (Stage 3):   v_i(h) = u_i kappa (T - C[c1] - C[c2] + q[h]),  T = sum_o q[o],
//                     C[c] = sum_{o holds c} q[o]  (inclusion-exclusion over the two cards)
//   showdown (Stage 4): v_i(h) = c kappa (W(h) - L(h)), W / L the opponent reach of weaker /
//                     stronger hands that share no card with h, from exclusive prefix sums
//                     over the rank-sorted order minus per-card prefix sums; the tie group
//                     of h is excluded from both (a split pot pays 0).
// Sums and differences are double-float with FP32-pair values (whose folds take T and C[c] from
// the same prefix sums, in hand order), plain FP32 with FP32 values.

// Entries of a thread's run at most: kMaxHands over 160 threads (8) and twice as many over 352 (7) with
// FP32 values, over 256 (10) with pairs.
template <typename P>
struct ScanPer {
  static constexpr int n = std::is_same<P, Single>::value ? 8 : 10;
};

template <typename P, int NV>
struct alignas(NV * sizeof(typename P::V)) Vec {
  typename P::V v[NV];
};
template <typename P, int NV>
struct alignas(16) VecAcc {  // running sums: FP32, or compensated pairs
  typename P::Acc v[NV];
};
__device__ __forceinline__ float acc_up(float a, int o) { return __shfl_up_sync(0xffffffffu, a, o); }
__device__ __forceinline__ acc2 acc_up(acc2 a, int o) { return acc_shfl_up(a, o); }
__device__ __forceinline__ float acc_from(float a, int l) { return __shfl_sync(0xffffffffu, a, l); }
__device__ __forceinline__ acc2 acc_from(acc2 a, int l) {
  return {__shfl_sync(0xffffffffu, a.s, l), __shfl_sync(0xffffffffu, a.e, l)};
}
__device__ __forceinline__ void acc_join(float& a, float b) { a = __fadd_rn(a, b); }
__device__ __forceinline__ void acc_join(acc2& a, acc2 b) { acc_merge(a, b); }

// Exclusive prefix sums of NV arrays of n values by GT consecutive threads, in two halves with a block
// barrier between.  Each thread owns a run of ceil(n / GT) entries, entry e at at(e) -- in registers
// (REGS: ScanPer of them at most), or in the output array itself: first x receives the inclusive sum
// of its warp's runs up to its own, and the warp's total goes to red[warp].  Sums are plain FP32 with
// FP32 values, compensated with pairs.
template <typename P, int NV, bool REGS, typename F>
__device__ __forceinline__ void scan_runs(F at, int cnt, VecAcc<P, NV>* red, int gtid, VecAcc<P, NV>& x) {
  const int lane = gtid & 31;
#pragma unroll
  for (int v = 0; v < NV; ++v) x.v[v] = P::acc0();
  auto add = [&](int e) {
    const Vec<P, NV> y = at(e);
#pragma unroll
    for (int v = 0; v < NV; ++v) P::acc(x.v[v], y.v[v]);
  };
  if constexpr (REGS) {
#pragma unroll
    for (int e = 0; e < ScanPer<P>::n; ++e)
      if (e < cnt) add(e);
  } else {
    for (int e = 0; e < cnt; ++e) add(e);
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const typename P::Acc y = acc_up(x.v[v], o);
      if (lane >= o) acc_join(x.v[v], y);
    }
  if (lane == 31) red[gtid >> 5] = x;
}

// After the barrier: the exclusive prefix sums of the thread's run into out (out[place(n)] = totals).
// Every warp scans the GT / 32 warp totals itself.
template <typename P, int NV, int GT, bool REGS, typename F, typename M>
__device__ __forceinline__ void scan_write(F at, int begin, int cnt, int n, const VecAcc<P, NV>* red, int gtid,
                                           const VecAcc<P, NV>& x, Vec<P, NV>* out, M place) {
  const int lane = gtid & 31, warp = gtid >> 5;
  VecAcc<P, NV> run;
  Vec<P, NV> total;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    typename P::Acc w = lane < GT / 32 ? red[lane].v[v] : P::acc0();
#pragma unroll
    for (int o = 1; o < GT / 32; o <<= 1) {
      const typename P::Acc y = acc_up(w, o);
      if (lane >= o) acc_join(w, y);
    }
    run.v[v] = acc_up(x.v[v], 1);
    if (lane == 0) run.v[v] = P::acc0();
    const typename P::Acc before = acc_from(w, max(warp - 1, 0));
    if (warp > 0) acc_join(run.v[v], before);
    total.v[v] = P::value(acc_from(w, GT / 32 - 1));
  }
  auto put = [&](int e) {
    const Vec<P, NV> y = at(e);
    Vec<P, NV> o;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      o.v[v] = P::value(run.v[v]);
      P::acc(run.v[v], y.v[v]);
    }
    out[place(begin + e)] = o;
  };
  if constexpr (REGS) {
#pragma unroll
    for (int e = 0; e < ScanPer<P>::n; ++e)
      if (e < cnt) put(e);
  } else {
    for (int e = 0; e < cnt; ++e) put(e);
  }
  if (gtid == 0) out[place(n)] = total;
}

// ---- one node, all of a block of kTermThreads threads: the latency form

constexpr int kTermHands = 3;  // hands per thread
static_assert(kTermHands * kTermThreads >= kMaxHands, "every hand has a thread");

// The threads on the rank order (the others take the card lists), and a thread's run of them.
template <typename P>
struct TermRun {
  static constexpr int gp = std::is_same<P, Single>::value ? 5 * 32 : kTermThreads / 2;
  static_assert(ScanPer<P>::n * gp >= kMaxHands && ScanPer<P>::n * (kTermThreads - gp) >= 2 * kMaxHands,
                "a thread's run holds its share of the hands and of the card lists");
  int begin, cnt;
  __device__ __forceinline__ TermRun() : begin(0), cnt(0) {}
  __device__ __forceinline__ TermRun(int H, int k) {
    const int tid = threadIdx.x, n = tid < gp ? H : k * H, gn = tid < gp ? gp : kTermThreads - gp,
              per = (n + gn - 1) / gn;
    begin = min((tid < gp ? tid : tid - gp) * per, n);
    cnt = min(begin + per, n) - begin;
  }
};

// What a thread reads of a board table for the nodes of one kind: the hands of its run (in rank
// order, or along the card lists; pairs' folds: in hand order), two in a word, and its hands' records.
// It stays in registers while the block's nodes share the table and kind (resident schedule).
template <typename P>
struct TermLane {
  TermRun<P> run;
  uint32_t at[ScanPer<P>::n / 2];
  uint4 rec[kTermHands];
  __device__ __forceinline__ int hand(int e) const { return at[e / 2] >> (e & 1 ? 16 : 0) & 0xffffu; }
  __device__ __forceinline__ uint4 record(int s, int) const { return rec[s]; }
};

// The same read from the staged table when it is used (one-node launch: each block has one node).
template <typename P>
struct TermStaged {
  TermRun<P> run;
  const uint16_t *list, *perm, *cards, *gs, *ge, *lo, *hi;  // list: the thread's run, or null (hand order)
  __device__ __forceinline__ int hand(int e) const {
    return e >= run.cnt ? 0 : list ? list[run.begin + e] : run.begin + e;
  }
  __device__ __forceinline__ void set(const TermTab& tt, const uint16_t* tab, int H, int k, bool show) {
    run = TermRun<P>(H, k);
    perm = tab + tt.perm;
    list = (int)threadIdx.x >= run.gp ? tab + tt.clh : show ? perm : nullptr;
    cards = tab + tt.cards, gs = tab + tt.gs, ge = tab + tt.ge, lo = tab + tt.lo, hi = tab + tt.hi;
  }
  __device__ __forceinline__ uint4 record(int, int h) const {
    return make_uint4(cards[h] | (uint32_t)gs[h] << 16, ge[h] | (uint32_t)lo[2 * h] << 16,
                      hi[2 * h] | (uint32_t)lo[2 * h + 1] << 16, hi[2 * h + 1]);
  }
};

template <typename P>
__device__ __forceinline__ void term_lane_load(TermLane<P>& L, const GameDev& G, int table, bool show) {
  const int H = G.n_hands, k = G.hand_size, tid = threadIdx.x;
  if (!show && std::is_same<P, Single>::value) return;
  const TermTab tt(H, k, G.deck);
  const uint16_t* gt = G.term_tab + (size_t)table * tt.len;
  L.run = TermRun<P>(H, k);
#pragma unroll
  for (int e = 0; e < ScanPer<P>::n; ++e) {
    const int j = L.run.begin + e;
    const uint32_t h = e >= L.run.cnt ? 0 : tid >= L.run.gp ? __ldg(gt + tt.clh + j) : show ? __ldg(gt + tt.perm + j) : j;
    L.at[e / 2] = e & 1 ? L.at[e / 2] | h << 16 : h;
  }
#pragma unroll
  for (int s = 0; s < kTermHands; ++s)
    if (tid + s * kTermThreads < H) L.rec[s] = __ldg(G.term_rec + (size_t)table * H + tid + s * kTermThreads);
}

// Values at one node: q its reach row, ft the fold part of its board table (card lists, cards, list
// offsets) and CP [k H + 1], Ps [H + 1] in shared memory; put(h, value) takes the results.
template <typename P, bool REGS = true, bool SWAP = false, typename LT, typename F>
__device__ __forceinline__ void terminal_node(const LT& L, int H, int k, int deck, bool show, uint64_t board, ff u,
                                              const typename P::V* q, const uint16_t* ft, typename P::V* CP,
                                              typename P::V* Ps, F put) {
  using V = typename P::V;
  using V1 = Vec<P, 1>;
  constexpr bool single = std::is_same<P, Single>::value;
  constexpr int gp = TermRun<P>::gp;
  __shared__ VecAcc<P, 1> red[2][kTermThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31;
  const uint16_t* clh = ft;
  const uint16_t* cards = ft + k * H;
  const uint16_t* cloff = cards + H;
  if constexpr (single) {
    if (!show) {
      // T: warp 0 keeps 32 lane-strided partial sums of q and combines them by a fixed xor tree; C[c]:
      // one thread per card sums card c's list in list order
      __shared__ float Cs[kMaxDeck], Ts;
      if (tid < 32) {
        float t = 0.f;
#pragma unroll 8
        for (int h = lane; h < H; h += 32) t = __fadd_rn(t, q[h]);
        for (int o = 16; o > 0; o >>= 1) t = __fadd_rn(t, __shfl_xor_sync(0xffffffffu, t, o));
        if (lane == 0) Ts = t;
      } else if (tid - 32 < deck) {
        const int c = tid - 32, end = cloff[c + 1];
        float s = 0.f;
#pragma unroll 8
        for (int j = cloff[c]; j < end; ++j) s = __fadd_rn(s, q[clh[j]]);
        Cs[c] = s;
      }
      __syncthreads();
#pragma unroll
      for (int s = 0; s < kTermHands; ++s) {
        const int h = tid + s * kTermThreads;
        if (h < H) {
          const unsigned cw = cards[h], c1 = cw & 0xffu, c2 = cw >> 8;
          float m = __fsub_rn(Ts, Cs[c1]);
          bool blocked = (board >> c1) & 1ull;
          if (k == 2) {
            m = __fadd_rn(__fsub_rn(m, Cs[c2]), q[h]);
            blocked = blocked || ((board >> c2) & 1ull);
          }
          put(h, blocked ? 0.f : __fmul_rn(u.hi, m));
        }
      }
      return;
    }
  }
  // In place, threads walk the arrays a run apart: runs of a multiple of eight entries would meet in a few
  // banks, so with SWAP the entries of such an array swap places within each eight of them (by the number
  // of the eight; see scans_in_eights).
  constexpr int gc = kTermThreads - gp;
  const int pmask = SWAP && (H + gp - 1) / gp % 8 == 0 ? 7 : 0, cmask = SWAP && (k * H + gc - 1) / gc % 8 == 0 ? 7 : 0;
  auto pat = [&](int j) { return !SWAP ? j : j ^ (j >> 3 & pmask); };
  auto cat = [&](int j) { return !SWAP ? j : j ^ (j >> 3 & cmask); };
  {
    V1 a[REGS ? ScanPer<P>::n : 1];
    VecAcc<P, 1> x;
    V1* ps = reinterpret_cast<V1*>(Ps);
    V1* cp = reinterpret_cast<V1*>(CP);
    const int gtid = tid < gp ? tid : tid - gp;
    if constexpr (REGS) {
#pragma unroll
      for (int e = 0; e < ScanPer<P>::n; ++e) a[e].v[0] = q[L.hand(e)];
    } else {  // gathered into the arrays that the scan turns into prefix sums in place
      for (int j = tid; j < H; j += kTermThreads) ps[pat(j)].v[0] = q[show ? L.perm[j] : j];
      for (int j = tid; j < k * H; j += kTermThreads) cp[cat(j)].v[0] = q[clh[j]];
      __syncthreads();
    }
    V1* mine = tid < gp ? ps : cp;
    const int mask = tid < gp ? pmask : cmask, begin = L.run.begin;
    auto at = [&](int e) { return REGS ? a[REGS ? e : 0] : mine[!SWAP ? begin + e : (begin + e) ^ ((begin + e) >> 3 & mask)]; };
    scan_runs<P, 1, REGS>(at, L.run.cnt, red[tid >= gp], gtid, x);
    __syncthreads();
    if (tid < gp)
      scan_write<P, 1, gp, REGS>(at, L.run.begin, L.run.cnt, H, red[0], gtid, x, ps, pat);
    else
      scan_write<P, 1, gc, REGS>(at, L.run.begin, L.run.cnt, k * H, red[1], gtid, x, cp, cat);
  }
  __syncthreads();
  const V T = Ps[pat(H)], us = P::scale(u);
#pragma unroll
  for (int s = 0; s < kTermHands; ++s) {
    const int h = tid + s * kTermThreads;
    if (h < H) {
      const uint4 r = L.record(s, h);
      const unsigned c1 = r.x & 0xffu, c2 = (r.x >> 8) & 0xffu;
      bool blocked = (board >> c1) & 1ull;
      const V a0 = CP[cat(cloff[c1])], z0 = CP[cat(cloff[c1 + 1])];
      V d;
      if (show) {
        V Wn = Ps[pat(r.x >> 16)], Ln = P::sub(T, Ps[pat(r.y & 0xffffu)]);
        Wn = P::sub(Wn, P::sub(CP[cat(r.y >> 16)], a0));
        Ln = P::sub(Ln, P::sub(z0, CP[cat(r.z & 0xffffu)]));
        if (k == 2) {
          blocked = blocked || ((board >> c2) & 1ull);
          Wn = P::sub(Wn, P::sub(CP[cat(r.z >> 16)], CP[cat(cloff[c2])]));
          Ln = P::sub(Ln, P::sub(CP[cat(cloff[c2 + 1])], CP[cat(r.w & 0xffffu)]));
        }
        d = P::sub(Wn, Ln);
      } else {
        d = P::sub(T, P::sub(z0, a0));
        if (k == 2) {
          blocked = blocked || ((board >> c2) & 1ull);
          d = P::add(P::sub(d, P::sub(CP[cat(cloff[c2 + 1])], CP[cat(cloff[c2])])), q[h]);
        }
      }
      put(h, blocked ? P::zero() : P::mul(us, d));
    }
  }
}

// The player of a block of the terminal launch and its item of n (grid: (player, item)).
__device__ __forceinline__ int terminal_item(int n, int player_mask, int& i) {
  if (player_mask != 3) {
    i = player_mask == 1 ? 0 : 1;
    return blockIdx.x;
  }
  i = (int)blockIdx.x >= n;
  return blockIdx.x - i * n;
}

// Payoff for player i per unit of (opponent reach) x kappa at node n: the FP64 product as a pair
// of FP32 rounded once on the host (FP32 values use its high part): no FP64 work per thread.
__device__ __forceinline__ ff terminal_payoff(const GameDev& G, const NodeDev& nd, int n, int i) {
  const bool neg = nd.type == kFold && nd.player == i;
  return {neg ? -G.payoff_ff[2 * n] : G.payoff_ff[2 * n], neg ? -G.payoff_ff[2 * n + 1] : G.payoff_ff[2 * n + 1]};
}

// Terminal values (Stages 2-4), the one-node form for handles with few terminals.  One block per
// (player, node): its board table comes in by a bulk (TMA) copy that starts before the launch waits
// for its predecessor, the opponent's reach row by another after it.  A showdown below an all-in
// run-out reads the run-out's reach row (src) and zeroes the hands holding a dealt card itself
// (nobody acts below the run-out, so that is its reach).  The wait is bounded: on a timeout the
// block sets *err, lets its copies drain and leaves.
template <typename P>
__global__ void __launch_bounds__(kTermThreads, 2) k_terminal(const GameDev* __restrict__ games,
                                                            const Work* __restrict__ work,
                                                            const TermSrc* __restrict__ src, int n_work,
                                                            int player_mask, int use_bar, int* err) {
  using V = typename P::V;
  int i;
  const int first = terminal_item(n_work, player_mask, i), tid = threadIdx.x;
  const GameDev& G = games[work[first].game];
  const int n = work[first].unit, from = src[first].row[1 - i];
  const NodeDev nd = G.nodes[n];
  const int H = G.n_hands, k = G.hand_size;
  const size_t stride = (size_t)G.hstride;
  const TermTab tt(H, k, G.deck);
  const bool show = nd.type == kShowdown;
  const unsigned tab_bytes = (unsigned)(show ? tt.len : tt.fold_len) * 2u, q_bytes = (unsigned)(stride * sizeof(V));
  const V* qsrc = static_cast<const V*>(use_bar ? G.reach_bar : G.reach) + (size_t)(1 - i) * G.n_nodes * stride;
  V* dst = static_cast<V*>(use_bar ? G.cfv_br : G.cfv) + ((size_t)i * G.n_nodes + n) * stride;

  extern __shared__ __align__(128) unsigned char smt[];
  __shared__ __align__(8) uint64_t bar;
  const uint16_t* tab = reinterpret_cast<const uint16_t*>(smt);  // [tt.len]
  V* q = reinterpret_cast<V*>(smt + (size_t)tt.len * 2);          // [hstride]
  V* CP = q + stride;                                            // [k H + 1]
  V* Ps = CP + (k * H + 1);                                      // [H + 1]
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_barrier_init();
  }
  __syncthreads();
  if (tid == 0) {
    mbar_arrive_expect_tx(&bar, tab_bytes + q_bytes);
    bulk_copy_g2s(smt, G.term_tab + (size_t)(show ? nd.row : 0) * tt.len, tab_bytes, &bar);
  }
  pdl_wait();  // the reach rows come from the launch just before this one
  pdl_trigger();
  if (tid == 0) bulk_copy_g2s(q, qsrc + (size_t)term_src_node(from) * stride, q_bytes, &bar);
  const ff u = terminal_payoff(G, nd, n, i);
  TermStaged<P> L;
  L.set(tt, tab, H, k, show);
  const bool ok = tid >= 32 || mbar_wait_bounded(&bar, 0, g_first_wait_polls);  // one warp polls
  if (__syncthreads_or(!ok)) {  // a copy did not land: report, let the copies drain, leave
    if (tid == 0) {
      atomicExch(err, 1);
      mbar_wait_bounded(&bar, 0);
    }
    __syncthreads();
    return;
  }
  if (from < 0) {  // below an all-in run-out: its reach, without the hands holding a card dealt since
    for (int h = tid; h < H; h += kTermThreads)
      if (holds_board_card(L.cards, h, k, nd.board)) q[h] = P::zero();
    __syncthreads();
  }
  terminal_node<P>(L, H, k, G.deck, show, nd.board, u, q, tab, CP, Ps, [&](int h, V v) { dst[h] = v; });
}

// ---- the run form, for handles whose terminals fill the GPU many times over
//
// A block takes up to eight nodes of one game, board table and kind one after the other: the table is
// staged once, and each node's reach row lands (two buffers) while the node before is computed.  A
// node is a chain of four block barriers with little between them, so what counts is how many chains
// an SM holds: four blocks (with pairs up to about 950 hands, three above, whose arrays fill its shared
// memory), which the scans' in-place form leaves room for (32 registers; 64 with the
// entries in registers hold two).  Pairs always run so (groups of two nodes a thread spilled, and
// took 419 us a player on 256 rivers of 1,081 hands where this form takes 309); FP32 values where a
// board table has few showdown nodes (see create_impl).  Measured, one player: 256 rivers, pairs, 309
// us (317 held to three blocks' registers, 342 with the entries in registers); exact turn, pairs, 214;
// the 31,124-node flop of 513 hands, FP32 values 158, pairs 275.
template <typename P, bool SWAP>
__global__ void __launch_bounds__(kTermThreads, 4) k_terminal_run(const GameDev* __restrict__ games,
                                                            const Work* __restrict__ work,
                                                            const TermSrc* __restrict__ src,
                                                            const Work* __restrict__ runs, int n_runs,
                                                            int player_mask, int use_bar, int* err) {
  using V = typename P::V;
  int i;
  const Work r = runs[terminal_item(n_runs, player_mask, i)];  // (first entry of work, count)
  const int first = r.game, count = r.unit, tid = threadIdx.x;
  const GameDev& G = games[work[first].game];
  const NodeDev nd0 = G.nodes[work[first].unit];
  const int H = G.n_hands, k = G.hand_size;
  const size_t stride = (size_t)G.hstride;
  const TermTab tt(H, k, G.deck);
  const bool show = nd0.type == kShowdown;
  const unsigned tab_bytes = (unsigned)(show ? tt.len : tt.fold_len) * 2u, q_bytes = (unsigned)(stride * sizeof(V));
  const V* qsrc = static_cast<const V*>(use_bar ? G.reach_bar : G.reach) + (size_t)(1 - i) * G.n_nodes * stride;
  V* dst = static_cast<V*>(use_bar ? G.cfv_br : G.cfv) + (size_t)i * G.n_nodes * stride;

  extern __shared__ __align__(128) unsigned char smt[];
  __shared__ __align__(8) uint64_t bar[2];
  const uint16_t* tab = reinterpret_cast<const uint16_t*>(smt);  // [tt.len]
  V* rows = reinterpret_cast<V*>(smt + (size_t)tt.len * 2);       // [2][hstride]
  V* CP = rows + 2 * stride;                                     // [k H + 1], with SWAP in eights
  V* Ps = CP + (SWAP ? TermTab::round8(k * H + 1) : k * H + 1);  // [H + 1]
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_barrier_init();
  }
  __syncthreads();
  auto copy_row = [&](int j) {
    bulk_copy_g2s(rows + (j & 1) * stride, qsrc + (size_t)term_src_node(src[first + j].row[1 - i]) * stride, q_bytes, &bar[j & 1]);
  };
  if (tid == 0) {
    mbar_arrive_expect_tx(&bar[0], tab_bytes + q_bytes);
    bulk_copy_g2s(smt, G.term_tab + (size_t)(show ? nd0.row : 0) * tt.len, tab_bytes, &bar[0]);
  }
  pdl_wait();  // the reach rows come from the launch just before this one
  pdl_trigger();
  if (tid == 0) copy_row(0);
  TermStaged<P> L;
  L.set(tt, tab, H, k, show);
  for (int j = 0; j < count; ++j) {
    const int n = work[first + j].unit, from = src[first + j].row[1 - i];
    const uint64_t board = G.nodes[n].board;
    const ff u = terminal_payoff(G, G.nodes[n], n, i);
    if (tid == 0 && j + 1 < count) {
      // the other buffer's last readers are behind the barrier that closed node j - 1; the block's own
      // writes there (zeroed hands) come before the copy
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive_expect_tx(&bar[(j + 1) & 1], q_bytes);
      copy_row(j + 1);
    }
    const bool ok = tid >= 32 || mbar_wait_bounded(&bar[j & 1], (j >> 1) & 1, j == 0 ? g_first_wait_polls : kWaitLimit);
    if (__syncthreads_or(!ok)) {  // a copy did not land: report, let the copies drain, leave
      if (tid == 0) {
        atomicExch(err, 1);
        mbar_wait_bounded(&bar[j & 1], (j >> 1) & 1);
        if (j + 1 < count) mbar_wait_bounded(&bar[(j + 1) & 1], ((j + 1) >> 1) & 1);
      }
      __syncthreads();
      return;
    }
    V* q = rows + (j & 1) * stride;
    if (from < 0) {  // below an all-in run-out: its reach, without the hands holding a card dealt since
      for (int h = tid; h < H; h += kTermThreads)
        if (holds_board_card(L.cards, h, k, board)) q[h] = P::zero();
      __syncthreads();
    }
    V* out = dst + (size_t)n * stride;
    terminal_node<P, false, SWAP>(L, H, k, G.deck, show, board, u, q, tab, CP, Ps, [&](int h, V v) { out[h] = v; });
    __syncthreads();  // the row and the scan arrays are free
  }
}

// ---- several nodes at once: the throughput form of FP32 values
//
// A group is up to NV nodes of one game, one kind (folds or showdowns) and one board table.  The
// scan arrays of terminal_node become arrays of NV values (16 bytes), so each table entry and
// each address is read and computed once for NV nodes and a gather is one 16-byte shared-memory
// access.  Component v runs exactly the one-node form's operations in its order (the same runs
// of entries per thread, the same combination of threads and warps), so the bits are the same.
//
// Blocks are persistent: two per SM, each walking its own contiguous stretch of the groups, so
// that the board table is reloaded only when it changes, descriptors are staged once, and the
// reach rows of the next group are in flight (bulk copies, two buffers) while the current one
// is computed.  A showdown group takes three block barriers: rows landed; each thread has
// gathered its run of entries into registers and summed it; the prefix sums are written.
// Bound by random shared-memory gathers (5060 wavefronts a group of four, 45 % of the pipe's rate).
// Measured against blocks that take their nodes one by one: exact turn 119 -> 88 us per player,
// 256 rivers 132 -> 129, with one block per group and its descriptors read node by node 147.

template <int NV>
__global__ void __launch_bounds__(kTermThreads, 2) k_terminal_vec(const GameDev* __restrict__ games,
                                                                const TermGroup* __restrict__ groups,
                                                                const Work* __restrict__ segments, int n_segments,
                                                                int player_mask, int use_bar, int* err) {
  using P = Single;
  using VV = Vec<P, NV>;
  constexpr int kScanPer = ScanPer<P>::n;
  constexpr int gp = TermRun<P>::gp;  // threads on the rank order; the rest on the card lists
  int i;
  const Work seg = segments[terminal_item(n_segments, player_mask, i)];  // (first group, count <= kTermSegment)
  const int tid = threadIdx.x, lane = tid & 31;

  extern __shared__ __align__(128) unsigned char smt[];
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ VecAcc<P, NV> red[2][kTermThreads / 32];
  __shared__ float Cs[NV][kMaxDeck], Ts[NV];  // fold groups
  TermGroup* desc = reinterpret_cast<TermGroup*>(smt);
  const uint4* gsrc = reinterpret_cast<const uint4*>(groups + seg.game);
  for (int k = tid; k < seg.unit * (int)(sizeof(TermGroup) / 16); k += kTermThreads)
    reinterpret_cast<uint4*>(desc)[k] = __ldg(gsrc + k);
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_barrier_init();
  }
  __syncthreads();

  // per (game, table, kind), reloaded when it changes; shared memory by offsets into smt: the table's
  // fold part (card lists, cards, list offsets) at kTab, then rows [2][NV][hstride], CP [k H + 1],
  // Ps [H + 1]
  constexpr int kTab = kTermSegment * (int)sizeof(TermGroup);
  int game = -1, table = -1, kind = -1, H = 0, k = 0, stride = 0, begin = 0, cnt = 0, rows = 0;
  float* dst = nullptr;
  const uint4* rec = nullptr;
  uint32_t at[kScanPer / 2];  // hands of the thread's run (rank order or card lists), two in a word

  auto copy_rows = [&](int g) {  // one thread: the reach rows of group g into buffer g & 1
    const TermGroup& d = desc[g];
    const GameDev& Gg = games[d.game];
    const size_t S = (size_t)Gg.hstride;
    const unsigned bytes = (unsigned)(S * sizeof(float));
    const TermTab tg(Gg.n_hands, Gg.hand_size, Gg.deck);
    unsigned char* buf = smt + kTab + tg.fold_len * 2 + (g & 1) * NV * bytes;
    const float* q = static_cast<const float*>(use_bar ? Gg.reach_bar : Gg.reach) + (size_t)(1 - i) * Gg.n_nodes * S;
    // the block's own writes there (zeroed hands, another game's arrays) come before the copies
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_expect_tx(&bar[g & 1], NV * bytes);  // a short group repeats its last node
    for (int v = 0; v < NV; ++v) bulk_copy_g2s(buf + v * bytes, q + (size_t)term_src_node(d.src[v].row[1 - i]) * S, bytes, &bar[g & 1]);
  };

  pdl_wait();  // the reach rows come from the launch just before this one
  pdl_trigger();
  for (int g = 0; g < seg.unit; ++g) {
    const TermGroup& d = desc[g];
    const bool show = d.kind == kShowdown, other = d.game != game;
    if (other) {
      // the rows of a game's first group start once the shared memory of the game before is free
      // (each game lays it out by its own hand count)
      if (g > 0) __syncthreads();
      if (tid == 0) copy_rows(g);
    }
    if (other || d.table != table || d.kind != kind) {
      const GameDev& G = games[d.game];
      H = G.n_hands, k = G.hand_size;
      const TermTab tt(H, k, G.deck);
      if (other) {
        stride = G.hstride;
        rows = kTab + tt.fold_len * 2;
        dst = static_cast<float*>(use_bar ? G.cfv_br : G.cfv) + (size_t)i * G.n_nodes * stride;
      }
      const uint16_t* gt = G.term_tab + (size_t)d.table * tt.len;
      if (other || d.table != table) {
        if (!other) __syncthreads();  // the last group's readers of the table are done
        table = d.table;
        for (int x = tid; x < tt.fold_len / 8; x += kTermThreads)
          reinterpret_cast<uint4*>(smt + kTab)[x] = __ldg(reinterpret_cast<const uint4*>(gt) + x);
        rec = G.term_rec + (size_t)table * H;
      }
      game = d.game;
      kind = d.kind;
      if (show) {
        const int n = tid < gp ? H : k * H, gt_n = tid < gp ? gp : kTermThreads - gp, gtid = tid < gp ? tid : tid - gp;
        const int per = (n + gt_n - 1) / gt_n;
        begin = min(gtid * per, n);
        cnt = min(begin + per, n) - begin;
#pragma unroll
        for (int e = 0; e < kScanPer; ++e) {
          const int j = begin + e;
          const uint32_t h = e >= cnt ? 0 : gt[(tid >= gp ? tt.clh : tt.perm) + j];
          at[e / 2] = e & 1 ? at[e / 2] | h << 16 : h;
        }
      }
    }
    const bool ok = tid >= 32 || mbar_wait_bounded(&bar[g & 1], (g >> 1) & 1, g == 0 ? g_first_wait_polls : kWaitLimit);
    if (__syncthreads_or(!ok)) {  // a copy did not land: report, let the copies drain, leave
      if (tid == 0) {
        atomicExch(err, 1);
        mbar_wait_bounded(&bar[g & 1], (g >> 1) & 1);
      }
      __syncthreads();
      return;
    }
    // the other buffer's last readers are behind the barrier above
    if (tid == 0 && g + 1 < seg.unit && desc[g + 1].game == game) copy_rows(g + 1);
    const uint16_t* clh = reinterpret_cast<const uint16_t*>(smt + kTab);
    const uint16_t* cards = clh + k * H;
    const uint16_t* cloff = cards + H;
    float* q = reinterpret_cast<float*>(smt + rows) + (g & 1) * NV * stride;  // node v's row at q + v * stride
    VV* CP = reinterpret_cast<VV*>(reinterpret_cast<float*>(smt + rows) + 2 * NV * stride);
    VV* Ps = CP + (k * H + 1);
    if (d.below >> (1 - i) & 1) {  // nodes below an all-in run-out: its reach, without the hands holding a card dealt since
      for (int v = 0; v < NV; ++v)
        if (d.src[v].row[1 - i] < 0)
          for (int h = tid; h < H; h += kTermThreads)
            if (holds_board_card(cards, h, k, d.board[v])) q[v * stride + h] = 0.f;
      __syncthreads();
    }

    if (!show) {  // terminal_node's fold sums: T of node v by warp v, C[c] of (v, c) by one thread
      const int deck = games[game].deck;
      if (tid < 32 * NV) {
        const float* qv = q + (tid >> 5) * stride;
        float t = 0.f;
#pragma unroll 8
        for (int h = lane; h < H; h += 32) t = __fadd_rn(t, qv[h]);
        for (int o = 16; o > 0; o >>= 1) t = __fadd_rn(t, __shfl_xor_sync(0xffffffffu, t, o));
        if (lane == 0) Ts[tid >> 5] = t;
      } else if (tid - 32 * NV < NV * deck) {
        const int x = tid - 32 * NV, v = x / deck, c = x - v * deck;
        const float* qv = q + v * stride;
        float s = 0.f;
#pragma unroll 8
        for (int j = cloff[c]; j < cloff[c + 1]; ++j) s = __fadd_rn(s, qv[clh[j]]);
        Cs[v][c] = s;
      }
      __syncthreads();
      for (int h = tid; h < H; h += kTermThreads) {
        const unsigned cw = cards[h];
        const unsigned c1 = cw & 0xffu, c2 = cw >> 8;
        const uint64_t own = (1ull << c1) | (k == 2 ? 1ull << c2 : 0ull);
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (v < d.count) {
            float m = __fsub_rn(Ts[v], Cs[v][c1]);
            if (k == 2) m = __fadd_rn(__fsub_rn(m, Cs[v][c2]), q[v * stride + h]);
            dst[(size_t)d.node[v] * stride + h] = (d.board[v] & own) ? 0.f : __fmul_rn(d.pay[i][v], m);
          }
      }
      continue;
    }
    {  // the reach in rank order and along the card lists
      VV a[kScanPer];
      VecAcc<P, NV> x;
#pragma unroll
      for (int e = 0; e < kScanPer; ++e)
        if (e < cnt) {
          const float* qe = q + (at[e / 2] >> (e & 1 ? 16 : 0) & 0xffffu);
#pragma unroll
          for (int v = 0; v < NV; ++v) a[e].v[v] = qe[v * stride];
        }
      const int gtid = tid < gp ? tid : tid - gp;
      auto entry = [&](int e) { return a[e]; };
      auto same = [](int j) { return j; };
      scan_runs<P, NV, true>(entry, cnt, red[tid >= gp], gtid, x);
      __syncthreads();
      if (tid < gp)
        scan_write<P, NV, gp, true>(entry, begin, cnt, H, red[0], gtid, x, Ps, same);
      else
        scan_write<P, NV, kTermThreads - gp, true>(entry, begin, cnt, k * H, red[1], gtid, x, CP, same);
    }
    __syncthreads();
    for (int h = tid; h < H; h += kTermThreads) {
      const uint4 hr = __ldg(rec + h);
      const unsigned c1 = hr.x & 0xffu, c2 = (hr.x >> 8) & 0xffu;
      uint64_t own = 1ull << c1;
      const VV T = Ps[H];
      VV Wn = Ps[hr.x >> 16], Ln = Ps[hr.y & 0xffffu];
#pragma unroll
      for (int v = 0; v < NV; ++v) Ln.v[v] = P::sub(T.v[v], Ln.v[v]);
      auto one = [&](unsigned c, unsigned lo, unsigned hi) {
        const VV a = CP[lo], a0 = CP[cloff[c]], z0 = CP[cloff[c + 1]], z = CP[hi];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          Wn.v[v] = P::sub(Wn.v[v], P::sub(a.v[v], a0.v[v]));
          Ln.v[v] = P::sub(Ln.v[v], P::sub(z0.v[v], z.v[v]));
        }
      };
      one(c1, hr.y >> 16, hr.z & 0xffffu);
      if (k == 2) {
        one(c2, hr.z >> 16, hr.w & 0xffffu);
        own |= 1ull << c2;
      }
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (v < d.count)
          dst[(size_t)d.node[v] * stride + h] = (d.board[v] & own) ? 0.f : P::mul(d.pay[i][v], P::sub(Wn.v[v], Ln.v[v]));
    }
  }
}

// ------------------------------------------------------------------ per-hand passes

// One column of a [rows][*] array: shared memory (row stride W, column w) or global
// memory (row stride hstride, column h).
template <typename T>
struct Col {
  T* base;
  size_t rs;
  __device__ __forceinline__ T& operator[](int row) const { return base[(size_t)row * rs]; }
};

__host__ __device__ inline size_t round16(size_t x) { return (x + 15) / 16 * 16; }

// Shared memory of the per-hand kernel for one game (must match the layout in k_hand):
// nodes, level offsets, row -> node map, decision-node list (fewer entries than rows), R and
// S rows, then values, reach and strategy.
__host__ __device__ inline size_t hand_smem_bytes(int n_nodes, int n_levels, int rows_max, int W, size_t es) {
  return round16((size_t)n_nodes * sizeof(NodeDev)) + round16((size_t)(n_levels + 1) * 4) +
         2 * round16((size_t)rows_max * 4) + 2 * round16((size_t)rows_max * W * 8) +
         (size_t)(2 * n_nodes + rows_max) * W * es;
}

// The per-hand passes of one chunk of W hands of player p, on whichever arrays hold the
// chunk's columns (shared memory, or the global arrays at column h).  Each node and each row
// is computed by one thread in a fixed order, so the result does not depend on how many
// threads share the work (slot / nslots): the level and resident schedules give the same bits.
template <typename P>
struct HandView {
  const NodeDev* nodes;
  const int* ls;      // level offsets [L + 1]
  const int* rown;    // node of each row of p
  const int* decs;    // decision nodes of p
  int L, ndec, nrows, rb, p;
  int slot, nslots;   // this thread's slot and the block's slot count
  bool valid;         // a real hand (h < n_hands)
  bool wr;            // this lane may write its column of the working arrays
  uint64_t hmask;     // cards of the hand
  Col<typename P::V> v, rch, sg;
  Col<double> Rc, Sc;
};

// Value of one inner node from its children's stored values (Stage 6, Eq. backward);
// MODE = kModeBR takes the max over p's actions (best response).
template <int MODE, typename P>
__device__ __forceinline__ typename P::V node_value(const HandView<P>& hv, const NodeDev& nd) {
  using V = typename P::V;
  const int A = nd.n_kids, k0 = nd.first_kid;
  if (MODE == kModeBR && nd.type == kDecision && nd.player == hv.p) {
    V val = hv.v[k0];
    for (int a = 1; a < A; ++a) val = P::vmax(val, hv.v[k0 + a]);
    return val;
  }
  typename P::Acc acc = P::acc0();
  if (nd.type == kChance) {
    // children values already carry the card probabilities; cards in the hand are out
    for (int a = 0; a < A; ++a)
      if (!((hv.hmask >> hv.nodes[k0 + a].deal) & 1ull)) P::acc(acc, hv.v[k0 + a]);
  } else if (nd.player != hv.p) {
#pragma unroll 4  // the children's loads go out together; the sum keeps its order
    for (int a = 0; a < A; ++a) P::acc(acc, hv.v[k0 + a]);
  } else {
    const int r0 = nd.row - hv.rb;
#pragma unroll 4
    for (int a = 0; a < A; ++a) P::acc_mul(acc, hv.sg[r0 + a], hv.v[k0 + a]);
  }
  return P::value(acc);
}

// Backward values (Stage 6, Eq. backward), level by level from the leaves.
template <int MODE, typename P>
__device__ __forceinline__ void hand_backward(const HandView<P>& hv) {
  for (int l = hv.L - 1; l >= 0; --l) {
    const int a0 = hv.ls[l], cnt = hv.ls[l + 1] - a0;
    for (int idx = hv.slot; idx < cnt; idx += hv.nslots) {
      const int n = a0 + idx;
      const NodeDev nd = hv.nodes[n];
      if (is_end(nd.type)) continue;
      const typename P::V val = node_value<MODE, P>(hv, nd);
      if (hv.wr) hv.v[n] = val;
    }
    __syncthreads();
  }
}

// Positive parts of the strategy source into sg, one (row, hand) item per thread:
//   update: the Stage 7 update of R and S (new rows to Rout / Sout where out_ok, the
//           prediction to M where the hand is real), then the positive part of the new R;
//   init: the positive part of R (+ M);  average: S.
// (sign tests of FP64 values read the sign bit on the integer pipe: x > 0 exactly when the
// bits, as a signed integer, are positive)
template <int MODE, typename P>
__device__ __forceinline__ void hand_rows(const HandView<P>& hv, const Discount& d, int variant, Col<double> Rout,
                                          Col<double> Sout, bool out_ok, Col<double> M) {
  using V = typename P::V;
  for (int r = hv.slot; r < hv.nrows; r += hv.nslots) {
    double x;
    if (MODE == kModeUpdate) {
      const int n = hv.rown[r];
      const NodeDev nd = hv.nodes[n];
      const V rr = P::sub(hv.v[nd.first_kid + (hv.rb + r - nd.row)], hv.v[n]);  // instantaneous regret
      const double contrib = P::to_double(P::mul(hv.rch[n], hv.sg[r]));      // pi_i(I) sigma(I, a)
      const double rd = P::to_double(rr);
      x = hv.Rc[r] + rd;
      if (variant == 2) x *= __double_as_longlong(x) > 0 ? d.dpos : d.dneg;
      if ((variant == 1 || variant == 3) && __double_as_longlong(x) < 0) x = 0.0;  // CFR+, Predictive CFR+
      const double sn = fma(hv.Sc[r], d.dS, (variant == 1 || variant == 3) ? d.wS * contrib : contrib);
      if (out_ok) {
        Rout[r] = x;
        Sout[r] = sn;
      }
      if (variant == 3 && hv.valid) M[r] = rd;  // the prediction of the next regret
      if (variant == 3) x += rd;                // Predictive CFR+ matches R + M
    } else {
      x = MODE == kModeInit ? hv.Rc[r] : hv.Sc[r];
      if (MODE == kModeInit && M.base) x += hv.valid ? M[r] : 0.0;
    }
    if (hv.wr) hv.sg[r] = __double_as_longlong(x) > 0 ? P::of_double(x) : P::zero();
  }
  __syncthreads();
}

// Regret matching (Eq. rm) / normalisation of the average, per decision node of p.
template <typename P>
__device__ __forceinline__ void hand_rm(const HandView<P>& hv) {
  using V = typename P::V;
  for (int k = hv.slot; k < hv.ndec; k += hv.nslots) {
    const NodeDev nd = hv.nodes[hv.decs[k]];
    const int A = nd.n_kids, r0 = nd.row - hv.rb;
    V tot = P::zero();
    int npos = 0, last = 0;
    for (int a = 0; a < A; ++a) {
      const V x = hv.sg[r0 + a];
      if (P::positive(x)) ++npos, last = a;
      tot = P::add(tot, x);
    }
    if (!hv.wr) continue;
    if (npos == 1) {  // x / x = 1 exactly, as the definition gives
      for (int a = 0; a < A; ++a) hv.sg[r0 + a] = a == last ? P::one() : P::zero();
    } else if (npos > 1) {
      const V inv = P::recip(tot);
      for (int a = 0; a < A; ++a) hv.sg[r0 + a] = P::mul(hv.sg[r0 + a], inv);
    } else {
      const V uni = P::uniform(A);
      for (int a = 0; a < A; ++a) hv.sg[r0 + a] = uni;
    }
  }
  __syncthreads();
}

// Forward reach of player p (Stages 1-2) under the strategy in sg, from the root reach `root`.
template <typename P>
__device__ __forceinline__ void hand_forward(const HandView<P>& hv, typename P::V root) {
  using V = typename P::V;
  if (hv.slot == 0 && hv.wr) hv.rch[0] = root;
  __syncthreads();
  for (int l = 1; l < hv.L; ++l) {
    const int a0 = hv.ls[l], cnt = hv.ls[l + 1] - a0;
    for (int idx = hv.slot; idx < cnt; idx += hv.nslots) {
      const int n = a0 + idx;
      const NodeDev nd = hv.nodes[n];
      V x = hv.wr ? hv.rch[nd.parent] : P::zero();
      if (nd.aplayer == hv.p) x = P::mul(x, hv.sg[nd.arow - hv.rb]);
      if (nd.deal != kNoCard && ((hv.hmask >> nd.deal) & 1ull)) x = P::zero();
      if (hv.wr) hv.rch[n] = x;
    }
    __syncthreads();
  }
}

// Per-hand tree passes for one chunk of W hands of player p (grid: (player, chunk)).
//   kModeInit:   sigma_p = RM(R_p) (Eq. rm), forward reach of p (Stage 1).
//   kModeUpdate: backward values of p (Stage 6, Eq. backward) from the terminal values,
//                regret and average update (Stage 7), new sigma_p, forward reach of p.
//   kModeAvg:    average strategy S / sum S of p, forward reach of p under it.
//   kModeBR:     best-response backward pass of p (max over p's actions) and the FP64
//                root sum r_p(h) v*_p(root, h), reduced by the last block of each game.
// With G.smem set the block stages the tree and its hands' state in shared memory;
// otherwise it works on the global arrays directly (trees too large to stage).
template <int MODE, typename P, bool SM>
__global__ void __launch_bounds__(kHandThreads, 1) k_hand(const GameDev* __restrict__ games,
                                                       const Work* __restrict__ work, int n_work, int player_mask,
                                                       int advance, int* iter, unsigned* done,
                                                       const Discount* __restrict__ disc_tab, int variant) {
  using V = typename P::V;
  int item = blockIdx.x;
  int p;
  if (player_mask == 3) {
    p = item >= n_work;
    item -= p * n_work;
  } else {
    p = player_mask == 1 ? 0 : 1;
  }
  const Work wk = work[item];
  const GameDev& G = games[wk.game];
  const int W = G.chunk;
  const int tid = threadIdx.x;
  const int w = tid % W;
  const int slot = tid / W;
  const int nslots = kHandThreads / W;
  const int h = wk.unit * W + w;  // < hstride: hstride is a multiple of 32 and W divides 32
  const bool valid = h < G.n_hands;
  const int N = G.n_nodes, L = G.n_levels;
  const size_t stride = (size_t)G.hstride;
  const int rb = G.row_begin[p], re = G.row_begin[p + 1];
  const int nrows = re - rb;
  const int rows_max = max(G.row_begin[1] - G.row_begin[0], G.row_begin[2] - G.row_begin[1]);
  const uint64_t hmask = valid ? G.hand_mask[h] : 0ull;
  constexpr bool sm = SM;       // the launch stages every game in shared memory
  const bool wr = sm || valid;  // this lane may write its column of the working arrays

  // global arrays of this player, at column h
  V* gv = static_cast<V*>(MODE == kModeBR ? G.cfv_br : G.cfv) + (size_t)p * N * stride + h;
  V* grch = static_cast<V*>(MODE == kModeAvg ? G.reach_bar : G.reach) + (size_t)p * N * stride + h;
  V* gsg = static_cast<V*>(MODE == kModeAvg ? G.sigbar : G.sigma) + (size_t)rb * stride + h;
  double* gR = G.R + (size_t)rb * stride + h;
  double* gS = G.S + (size_t)rb * stride + h;

  // shared layout (see hand_smem_bytes)
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* cur = smraw;
  NodeDev* snodes = reinterpret_cast<NodeDev*>(cur);
  cur += round16((size_t)N * sizeof(NodeDev));
  int* sls = reinterpret_cast<int*>(cur);
  cur += round16((size_t)(L + 1) * 4);
  int* srow = reinterpret_cast<int*>(cur);
  cur += round16((size_t)rows_max * 4);
  int* sdec = reinterpret_cast<int*>(cur);
  cur += round16((size_t)rows_max * 4);
  double* sR = reinterpret_cast<double*>(cur);
  cur += round16((size_t)rows_max * W * 8);
  double* sS = reinterpret_cast<double*>(cur);
  cur += round16((size_t)rows_max * W * 8);
  V* sv = reinterpret_cast<V*>(cur);
  V* srch = sv + (size_t)N * W;
  V* ssg = srch + (size_t)N * W;

  const NodeDev* nodes = sm ? snodes : G.nodes;
  const int* ls = sm ? sls : G.level_start;
  const int* rown = sm ? srow : G.row_node + rb;
  const int db = G.dec_begin[p], ndec = G.dec_begin[p + 1] - db;
  const int* decs = sm ? sdec : G.dec_nodes + db;
  const Col<V> v = sm ? Col<V>{sv + w, (size_t)W} : Col<V>{gv, stride};
  const Col<V> rch = sm ? Col<V>{srch + w, (size_t)W} : Col<V>{grch, stride};
  const Col<V> sg = sm ? Col<V>{ssg + w, (size_t)W} : Col<V>{gsg, stride};
  const Col<double> Rc = sm ? Col<double>{sR + w, (size_t)W} : Col<double>{gR, stride};
  const Col<double> Sc = sm ? Col<double>{sS + w, (size_t)W} : Col<double>{gS, stride};
  __shared__ Discount disc;
  __shared__ int s_last;
  __shared__ double red64[kHandThreads];

  // ---- stage: every load is independent of the others, so they are all in flight at once
  if (MODE == kModeUpdate && tid == 0) disc = disc_tab[*iter];
  if constexpr (SM) {
    constexpr int VB = (int)sizeof(V);
    const int4* gn = reinterpret_cast<const int4*>(G.nodes);
    int4* sn = reinterpret_cast<int4*>(snodes);
    for (int k = tid; k < 2 * N; k += kHandThreads) cp_async<16>(sn + k, gn + k);
    for (int k = tid; k <= L; k += kHandThreads) cp_async<4>(sls + k, G.level_start + k);
    for (int k = tid; k < nrows; k += kHandThreads) cp_async<4>(srow + k, G.row_node + rb + k);
    for (int k = tid; k < ndec; k += kHandThreads) cp_async<4>(sdec + k, G.dec_nodes + db + k);
    if (MODE == kModeUpdate) {
      for (int n = slot; n < N; n += nslots) cp_async<VB>(&rch[n], grch + (size_t)n * stride);
      for (int r = slot; r < nrows; r += nslots) {
        cp_async<VB>(&sg[r], gsg + (size_t)r * stride);
        cp_async<8>(&Rc[r], gR + (size_t)r * stride);
        cp_async<8>(&Sc[r], gS + (size_t)r * stride);
      }
    }
    if (MODE == kModeInit)
      for (int r = slot; r < nrows; r += nslots) cp_async<8>(&Rc[r], gR + (size_t)r * stride);
    if (MODE == kModeAvg)
      for (int r = slot; r < nrows; r += nslots) cp_async<8>(&Sc[r], gS + (size_t)r * stride);
  }
  pdl_wait();  // terminal values come from the launch just before this one
  pdl_trigger();
  if constexpr (SM) {
    constexpr int VB = (int)sizeof(V);
    if (MODE == kModeUpdate || MODE == kModeBR)
      for (int n = slot; n < N; n += nslots) cp_async<VB>(&v[n], gv + (size_t)n * stride);
    cp_async_wait_all();
  }
  __syncthreads();

  const HandView<P> hv{nodes, ls, rown, decs, L, ndec, nrows, rb, p, slot, nslots, valid, wr, hmask, v, rch, sg, Rc, Sc};

  // ---- backward pass (Stage 6), level by level from the leaves
  if (MODE == kModeUpdate || MODE == kModeBR) {
    hand_backward<MODE, P>(hv);
    if (sm && valid)
      for (int n = slot; n < N; n += nslots) gv[(size_t)n * stride] = v[n];
  }

  // ---- best response: FP64 root sum of this chunk, then the last block of the game
  //      reduces all chunks of both players in a fixed order
  if (MODE == kModeBR) {
    if (tid < W) {  // slot 0: one lane per hand of the chunk, all in warp 0
      double x = valid ? G.range64[(size_t)p * stride + h] * P::to_double(v[0]) : 0.0;
      const unsigned mask = W == 32 ? 0xffffffffu : (1u << W) - 1u;
      for (int o = W / 2; o > 0; o >>= 1) x += __shfl_down_sync(mask, x, o, W);
      if (tid == 0) G.br_partial[(size_t)p * G.n_chunks + wk.unit] = x;
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      s_last = atomicAdd(G.br_done, 1u) == (unsigned)(2 * G.n_chunks - 1);
    }
    __syncthreads();
    if (s_last) {
      __threadfence();
      for (int q = 0; q < 2; ++q) {
        double x = 0.0;
        for (int c = tid; c < G.n_chunks; c += kHandThreads) x += G.br_partial[(size_t)q * G.n_chunks + c];
        red64[tid] = x;
        __syncthreads();
        for (int o = kHandThreads / 2; o > 0; o >>= 1) {
          if (tid < o) red64[tid] += red64[tid + o];
          __syncthreads();
        }
        if (tid == 0) G.br_out[q] = red64[0];
        __syncthreads();
      }
      if (tid == 0) *G.br_done = 0u;
    }
    return;
  }

  // ---- positive parts of the strategy source (the update writes R and S to the global rows)
  hand_rows<MODE, P>(hv, disc, variant, Col<double>{gR, stride}, Col<double>{gS, stride}, valid,
                     Col<double>{G.M ? G.M + (size_t)rb * stride + h : nullptr, stride});
  // ---- regret matching (Eq. rm) / normalisation of the average, per decision node of p
  hand_rm<P>(hv);
  // ---- forward reach of player p (Stages 1-2) under the strategy in sg
  hand_forward<P>(hv, valid ? static_cast<const V*>(G.range_v)[(size_t)p * stride + h] : P::zero());
  if (sm && valid) {
    for (int n = slot; n < N; n += nslots) grch[(size_t)n * stride] = rch[n];
    for (int r = slot; r < nrows; r += nslots) gsg[(size_t)r * stride] = sg[r];
  }

  if (MODE == kModeUpdate && advance) {
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      const unsigned prev = atomicAdd(done, 1u);
      if (prev == gridDim.x - 1) {  // last block of the launch: every block has read *iter
        *done = 0u;
        *iter += 1;
        __threadfence();
      }
    }
  }
}


// ------------------------------------------------------------------ hand tiles
//
// The throughput form of the per-hand passes for handles of many subgames whose trees fit a
// block's shared memory a few times per SM (batches of rivers).  One block owns W hands (32, 16
// or 8: the most that fit) of one subgame and one player:
//   A  the values of the tree's end nodes and the stored strategy come in by cp.async; the inner
//      nodes' values (Stage 6) are computed level by level in shared memory;
//   B  the regret and average update (Stage 7) of every row of the player: a flat loop over (row,
//      hand) items with no order between them, four in flight a thread, so that the FP64 pipe
//      (64 cycles a warp instruction and scheduler) and the R and S streams stay busy; the
//      positive parts of the new regrets replace the strategy in shared memory;
//   C  level by level from the root: regret matching of the player's nodes (Eq. rm) and the
//      reach of their children (Stage 1), in the array of A.
// R and S are read and written once, straight from registers; L2 is asked for their lines at the
// start, before the launch waits for its predecessor.  The arithmetic is k_hand's, in its order.
// Bound: the FP64 pipe (three operations a row and hand: 66 us on the batch below) and issue slots.
// Measured, one player's update: 256 rivers, FP32 values 267 -> 180 us against the one-warp walk;
// 64 rivers, pairs, Predictive CFR+ 321 -> 110 us.  Average pass 780 -> 167, best response 943 ->
// 150 us (256 rivers, both players; k_hand before).

constexpr int kTileThreads = 256;  // at most; 128 where the tiles are small (see create_impl)

__host__ __device__ inline size_t tile_smem_bytes(int tab16, int n_nodes, int rows_max, int W, size_t es) {
  return (size_t)tab16 * 16 + (size_t)(n_nodes + rows_max) * W * es;
}

// Copies rows of W values (count of them, row k of the source at row_at(k)) into the tile.
template <typename V, typename F, typename T>
__device__ __forceinline__ void tile_copy(V* tile, const V* __restrict__ src, size_t stride, int wlog, int count, F row_at,
                                          T tile_at) {
  const int pl = wlog + (sizeof(V) == 8 ? 3 : 2) - 4;  // log2 of a row's 16-byte pieces
  for (int k = threadIdx.x; k < count << pl; k += blockDim.x) {
    const int r = k >> pl, part = k & ((1 << pl) - 1);
    cp_async<16>(reinterpret_cast<unsigned char*>(tile + (tile_at(r) << wlog)) + part * 16,
                 reinterpret_cast<const unsigned char*>(src + (size_t)row_at(r) * stride) + part * 16);
  }
}

// One lane's place in a tile: its column of the tile's arrays (node n or row r at [n << wlog]) and
// the threads that walk the levels.
struct TileLane {
  const TileHead* head;
  const uint16_t* tab;      // the table the head opens
  int p, wlog, slot, h, stride;
  int group;                // threads taking part in the level walks: fewer wait less at their barriers
  bool valid;               // a real hand
  uint64_t hmask;           // its cards
};

// Value of a chance node for one lane: the sum over its A children c[a * W] but those whose card is in
// the hand (children values carry the card probabilities).  One thread adds up to 49 children, so the
// cards are in the tile's table and several children are loaded ahead of the sum: with the cards in
// global memory an update of a 537-node turn with FP32 values took 27.1 us, now 18.5.  FP32 values take
// eight a step.  Pairs take four, added to a copy of the sum that the card's test then keeps or drops
// (turn to a leaf network, 997 hands: 24.0 us an update with eight and a branch at each, 19.1 so), and
// so does FP32 in the resident kernel, where the longer code costs rivers that have no such node
// (187 hands: 13.7 and 13.5 us an iteration).
template <typename P, bool LEAN>
__device__ __forceinline__ typename P::V tile_chance(const TileLane& T, const TileNode& nd, const typename P::V* c, int W) {
  const uint8_t* deal = reinterpret_cast<const uint8_t*>(T.tab + T.head->deal) + nd.first_kid;
  const int A = nd.kids & 63;
  typename P::Acc acc = P::acc0();
  if constexpr (LEAN || std::is_same<P, Pairs>::value) {
    constexpr int kAhead = 4;
    for (int a0 = 0; a0 < A; a0 += kAhead) {
      typename P::V y[kAhead];
      int card[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int a = min(a0 + u, A - 1);
        y[u] = c[a * W], card[u] = deal[a];
      }
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        typename P::Acc with = acc;
        P::acc(with, y[u]);
        if (a0 + u < A && !((T.hmask >> card[u]) & 1ull)) acc = with;
      }
    }
  } else {
#pragma unroll 8
    for (int a = 0; a < A; ++a)
      if (!((T.hmask >> deal[a]) & 1ull)) P::acc(acc, c[a * W]);
  }
  return P::value(acc);
}

// Barrier of the first `group` threads of the block.
__device__ __forceinline__ void group_barrier(int group) {
  if (group == (int)blockDim.x)
    __syncthreads();
  else
    asm volatile("barrier.sync 1, %0;" ::"r"(group) : "memory");
}

// Phase A: the inner nodes' values from the deepest level up (Stage 6, Eq. backward; kModeBR: the
// best response's), by the first `group` threads.  gv: the player's value rows; the values are
// stored there when `store` is set, the root's always.
template <int MODE, typename P, bool LEAN = false>
__device__ __forceinline__ void tile_values(const TileLane& T, typename P::V* val, const typename P::V* sg,
                                            typename P::V* gv, bool store) {
  using V = typename P::V;
  const TileNode* inner = reinterpret_cast<const TileNode*>(T.tab + T.head->inner);
  const uint16_t* level = T.tab + T.head->level;  // inner nodes of level l: [level[l], level[l + 1])
  const int wlog = T.wlog, nslots = T.group >> wlog;
  for (int l = T.head->levels - 1; l >= 0; --l) {
    const int last = level[l + 1];
    for (int k = level[l] + T.slot; k < last; k += nslots) {
      const TileNode nd = inner[k];
      const int A = nd.kids & 63, kind = nd.kids >> 6;
      const V* c = val + (nd.first_kid << wlog);
      V x;
      if (kind == 2) {
        x = tile_chance<P, LEAN>(T, nd, c, 1 << wlog);
      } else if (MODE == kModeBR && kind == T.p) {
        x = c[0];
        for (int a = 1; a < A; ++a) x = P::vmax(x, c[a << wlog]);
      } else {
        typename P::Acc acc = P::acc0();
        if (kind != T.p) {
#pragma unroll 4
          for (int a = 0; a < A; ++a) P::acc(acc, c[a << wlog]);
        } else {
          const V* s = sg + (nd.row << wlog);
#pragma unroll 4
          for (int a = 0; a < A; ++a) P::acc_mul(acc, s[a << wlog], c[a << wlog]);
        }
        x = P::value(acc);
      }
      val[nd.id << wlog] = x;
      if (T.valid && (store || l == 0)) gv[(size_t)nd.id * T.stride + T.h] = x;
    }
    group_barrier(T.group);
  }
}

// tile_values for tiles of 8 hands in the latency forms, where a level is a few nodes and every
// instruction of its chain counts: fixed offsets, the first four children loaded together (past a
// node's last child they are not used; the tile ends with slack for them), and the next level's
// node read before the barrier.  With tile_reach8, iterations against the forms for any width: resident
// river of 1,081 hands and 75 nodes 16.6 -> 16.2 us, with pairs 31.7 -> 27.1, of 27 nodes 14.0 -> 13.0;
// 165-node river of 300 hands with pairs, level schedule, 32.8 -> 30.7.
constexpr int kTileSlack = 4;  // rows of slack behind a tile's strategy
template <int MODE, typename P, bool LEAN = false>
__device__ __forceinline__ void tile_values8(const TileLane& T, typename P::V* val, const typename P::V* sg,
                                             typename P::V* gv, bool store) {
  using V = typename P::V;
  const TileNode* inner = reinterpret_cast<const TileNode*>(T.tab + T.head->inner);
  const uint16_t* level = T.tab + T.head->level;
  const int nslots = T.group >> 3;
  int l = T.head->levels - 1, first = level[l], last = level[l + 1];
  TileNode nd = inner[min(first + T.slot, last - 1)];
  for (;; --l) {
    for (int k = first + T.slot; k < last;) {
      const int A = nd.kids & 63, kind = nd.kids >> 6;
      const V* c = val + nd.first_kid * 8;
      V x;
      if (kind == 2) {
        x = tile_chance<P, LEAN>(T, nd, c, 8);
      } else {
        V cc[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) cc[e] = c[e * 8];
        typename P::Acc acc = P::acc0();
        if (kind != T.p) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (e < A) P::acc(acc, cc[e]);
          for (int a = 4; a < A; ++a) P::acc(acc, c[a * 8]);
          x = P::value(acc);
        } else if (MODE == kModeBR) {
          x = cc[0];
#pragma unroll
          for (int e = 1; e < 4; ++e)
            if (e < A) x = P::vmax(x, cc[e]);
          for (int a = 4; a < A; ++a) x = P::vmax(x, c[a * 8]);
        } else {
          const V* s = sg + nd.row * 8;
          V ss[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) ss[e] = s[e * 8];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (e < A) P::acc_mul(acc, ss[e], cc[e]);
          for (int a = 4; a < A; ++a) P::acc_mul(acc, s[a * 8], c[a * 8]);
          x = P::value(acc);
        }
      }
      val[nd.id * 8] = x;
      if (T.valid && (store || l == 0)) gv[(size_t)nd.id * T.stride + T.h] = x;
      k += nslots;
      if (k < last) nd = inner[k];
    }
    if (l == 0) break;
    last = first;
    first = level[l - 1];
    nd = inner[min(first + T.slot, last - 1)];
    group_barrier(T.group);
  }
  group_barrier(T.group);
}

// Stage 7 of one row and hand (sign tests of FP64 values read the sign bit on the integer pipe): the
// new R and S in place, rd the instantaneous regret (the next prediction of Predictive CFR+);
// returns what regret matching takes.  rr: child value less node value; contrib: pi sigma(a).
template <typename P, bool DCFR>
__device__ __forceinline__ double tile_row(double& R, double& S, typename P::V rr, typename P::V contrib, const Discount& d,
                                           int variant, double& rd) {
  rd = P::to_double(rr);
  const double c = P::to_double(contrib);
  R += rd;
  if constexpr (DCFR) {
    R *= __double_as_longlong(R) > 0 ? d.dpos : d.dneg;
    S = fma(S, d.dS, c);
  } else {
    if (variant == 2) R *= __double_as_longlong(R) > 0 ? d.dpos : d.dneg;
    const bool plus = variant == 1 || variant == 3;  // CFR+, Predictive CFR+
    if (plus && __double_as_longlong(R) < 0) R = 0.0;
    S = fma(S, d.dS, plus ? d.wS * c : c);
  }
  return !DCFR && variant == 3 ? R + rd : R;  // Predictive CFR+ matches R + M
}

// Regret matching (Eq. rm) at a decision node of the player with NA actions from the positive parts
// s, and the reach of its children c from the node's reach x (regret_match_n's operations).
// put_sigma(row, value) and put_reach(node, value) take the results.
template <typename P, int NA, typename FS, typename FR>
__device__ __forceinline__ void tile_match(const TileNode& nd, const typename P::V* s, typename P::V* c, int wlog,
                                           typename P::V x, FS put_sigma, FR put_reach) {
  using V = typename P::V;
  V y[NA], tot = P::zero();
  int npos = 0;
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    y[a] = s[a << wlog];
    npos += P::positive(y[a]);
    tot = P::add(tot, y[a]);
  }
  const V inv = P::recip(tot);  // unused (and possibly not finite) unless npos > 1
  const V uni = P::uniform(NA);
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    const V many = P::mul(y[a], inv);
    y[a] = npos > 1 ? many : npos == 1 ? (P::positive(y[a]) ? P::one() : P::zero()) : uni;
    put_sigma(nd.row + a, y[a]);
    const V r = P::mul(x, y[a]);
    c[a << wlog] = r;
    put_reach(nd.first_kid + a, r);
  }
}

// Phase C: regret matching and reach from the root down (rch[0] set) by the first `group` threads, over
// the nodes that make new reach rows: the children of the player's decisions and of chance nodes
// (every other node shares a row above it).
template <typename P, typename FS, typename FR>
__device__ __forceinline__ void tile_reach(const TileLane& T, typename P::V* rch, const typename P::V* sg, FS put_sigma,
                                           FR put_reach) {
  using V = typename P::V;
  const TileNode* fwd = reinterpret_cast<const TileNode*>(T.tab + T.head->fwd[T.p]);
  const uint16_t* flevel = T.tab + T.head->flevel[T.p];
  const uint8_t* deal = reinterpret_cast<const uint8_t*>(T.tab + T.head->deal);
  const int wlog = T.wlog, nslots = T.group >> wlog, levels = T.head->flevels[T.p];
  for (int l = 0; l < levels; ++l) {
    const int last = flevel[l + 1];
    for (int k = flevel[l] + T.slot; k < last; k += nslots) {
      const TileNode nd = fwd[k];
      const int A = nd.kids & 63;
      const V x = rch[nd.id << wlog];
      V* c = rch + (nd.first_kid << wlog);
      const V* s = sg + (nd.row << wlog);
      if (nd.kids >> 6 == 2) {
        for (int a = 0; a < A; ++a) {
          const V y = ((T.hmask >> deal[nd.first_kid + a]) & 1ull) ? P::zero() : x;
          c[a << wlog] = y;
          put_reach(nd.first_kid + a, y);
        }
        continue;
      }
      switch (A) {
        case 1: tile_match<P, 1>(nd, s, c, wlog, x, put_sigma, put_reach); break;
        case 2: tile_match<P, 2>(nd, s, c, wlog, x, put_sigma, put_reach); break;
        case 3: tile_match<P, 3>(nd, s, c, wlog, x, put_sigma, put_reach); break;
        case 4: tile_match<P, 4>(nd, s, c, wlog, x, put_sigma, put_reach); break;
        case 5: tile_match<P, 5>(nd, s, c, wlog, x, put_sigma, put_reach); break;
        case 6: tile_match<P, 6>(nd, s, c, wlog, x, put_sigma, put_reach); break;
        case 7: tile_match<P, 7>(nd, s, c, wlog, x, put_sigma, put_reach); break;
        case 8: tile_match<P, 8>(nd, s, c, wlog, x, put_sigma, put_reach); break;
        default: {  // up to kMaxActions
          V tot = P::zero();
          int npos = 0;
          for (int a = 0; a < A; ++a) {
            const V y = s[a << wlog];
            npos += P::positive(y);
            tot = P::add(tot, y);
          }
          const V inv = P::recip(tot), uni = P::uniform(A);
          for (int a = 0; a < A; ++a) {
            V y = s[a << wlog];
            y = npos > 1 ? P::mul(y, inv) : npos == 1 ? (P::positive(y) ? P::one() : P::zero()) : uni;
            put_sigma(nd.row + a, y);
            const V r = P::mul(x, y);
            c[a << wlog] = r;
            put_reach(nd.first_kid + a, r);
          }
        }
      }
    }
    group_barrier(T.group);
  }
}

// Whether the walk's regret matching runs ahead of it: with pairs, but not on trees of one or two such
// levels, where the barrier costs as much as it saves (river of 275 hands with pairs, resident, 18.8 us an
// iteration inside the walk, 20.6 ahead).
template <typename P>
__device__ __forceinline__ bool match_ahead(const TileLane& T) {
  return std::is_same<P, Pairs>::value && T.head->flevels[T.p] > 2;
}

// Regret matching of all the player's nodes ahead of the walk, by nslots slots of W lanes (slot, from
// them, this lane's): the strategy replaces the positive parts in sg.  The latency forms take it with
// pairs: a node's reciprocal and products are a long chain in double-float arithmetic, paid once here
// instead of once a level (the walk then only multiplies).  FP32 values match inside the walk, which
// saves the barrier.  Iterations with pairs: 165-node river of 300 hands 30.8 -> 28.7 us, Leduc 46.4 ->
// 45.1 (matching inside the walk before).
template <typename P, typename FS>
__device__ __forceinline__ void tile_match_all(const TileLane& T, typename P::V* sg, int slot, int nslots, FS put_sigma) {
  using V = typename P::V;
  const TileNode* fwd = reinterpret_cast<const TileNode*>(T.tab + T.head->fwd[T.p]);
  const uint16_t* flevel = T.tab + T.head->flevel[T.p];
  const int wlog = T.wlog, last = flevel[T.head->flevels[T.p]];
  for (int k = slot; k < last; k += nslots) {
    const TileNode nd = fwd[k];
    const int A = nd.kids & 63;
    if (nd.kids >> 6 == 2) continue;
    V* s = sg + (nd.row << wlog);
    V tot = P::zero();
    int npos = 0;
#pragma unroll 4
    for (int a = 0; a < A; ++a) {
      const V y = s[a << wlog];
      npos += P::positive(y);
      tot = P::add(tot, y);
    }
    const V inv = P::recip(tot), uni = P::uniform(A);  // inv is unused (and may not be finite) unless npos > 1
#pragma unroll 4
    for (int a = 0; a < A; ++a) {
      V y = s[a << wlog];
      const V many = P::mul(y, inv);
      y = npos > 1 ? many : npos == 1 ? (P::positive(y) ? P::one() : P::zero()) : uni;
      s[a << wlog] = y;
      put_sigma(nd.row + a, y);
    }
  }
}

// The walk after tile_match_all: the reach of each child is the node's times the action's probability.
template <typename P, typename FR>
__device__ __forceinline__ void tile_reach_matched(const TileLane& T, typename P::V* rch, const typename P::V* sg,
                                                   FR put_reach) {
  using V = typename P::V;
  const TileNode* fwd = reinterpret_cast<const TileNode*>(T.tab + T.head->fwd[T.p]);
  const uint16_t* flevel = T.tab + T.head->flevel[T.p];
  const uint8_t* deal = reinterpret_cast<const uint8_t*>(T.tab + T.head->deal);
  const int wlog = T.wlog, nslots = T.group >> wlog, levels = T.head->flevels[T.p];
  for (int l = 0; l < levels; ++l) {
    const int last = flevel[l + 1];
    for (int k = flevel[l] + T.slot; k < last; k += nslots) {
      const TileNode nd = fwd[k];
      const int A = nd.kids & 63;
      const bool chance = nd.kids >> 6 == 2;
      const V x = rch[nd.id << wlog];
      V* c = rch + (nd.first_kid << wlog);
      const V* s = sg + (nd.row << wlog);
#pragma unroll 4
      for (int a = 0; a < A; ++a) {
        const V y = chance ? ((T.hmask >> deal[nd.first_kid + a]) & 1ull ? P::zero() : x) : P::mul(x, s[a << wlog]);
        c[a << wlog] = y;
        put_reach(nd.first_kid + a, y);
      }
    }
    group_barrier(T.group);
  }
}

// tile_reach for tiles of 8 hands in the latency forms, as tile_values8.
template <typename P, typename FS, typename FR>
__device__ __forceinline__ void tile_reach8(const TileLane& T, typename P::V* rch, const typename P::V* sg, FS put_sigma,
                                            FR put_reach) {
  using V = typename P::V;
  const TileNode* fwd = reinterpret_cast<const TileNode*>(T.tab + T.head->fwd[T.p]);
  const uint16_t* flevel = T.tab + T.head->flevel[T.p];
  const uint8_t* deal = reinterpret_cast<const uint8_t*>(T.tab + T.head->deal);
  const int nslots = T.group >> 3, levels = T.head->flevels[T.p];
  if (levels == 0) return;
  int first = 0, last = flevel[1];
  TileNode nd = fwd[min(T.slot, last - 1)];
  for (int l = 0;;) {
    for (int k = first + T.slot; k < last;) {
      const int A = nd.kids & 63;
      const V x = rch[nd.id * 8];
      V* c = rch + nd.first_kid * 8;
      if (nd.kids >> 6 == 2) {
        for (int a = 0; a < A; ++a) {
          const V y = ((T.hmask >> deal[nd.first_kid + a]) & 1ull) ? P::zero() : x;
          c[a * 8] = y;
          put_reach(nd.first_kid + a, y);
        }
      } else {
        const V* s = sg + nd.row * 8;
        V y[4], tot = P::zero();
        int npos = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) y[e] = s[e * 8];
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e < A) npos += P::positive(y[e]), tot = P::add(tot, y[e]);
        for (int a = 4; a < A; ++a) {
          const V z = s[a * 8];
          npos += P::positive(z), tot = P::add(tot, z);
        }
        const V inv = P::recip(tot), uni = P::uniform(A);  // inv is unused (and may not be finite) unless npos > 1
        auto one = [&](int a, V z) {
          const V many = P::mul(z, inv);
          z = npos > 1 ? many : npos == 1 ? (P::positive(z) ? P::one() : P::zero()) : uni;
          put_sigma(nd.row + a, z);
          const V r = P::mul(x, z);
          c[a * 8] = r;
          put_reach(nd.first_kid + a, r);
        };
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e < A) one(e, y[e]);
        for (int a = 4; a < A; ++a) one(a, s[a * 8]);
      }
      k += nslots;
      if (k < last) nd = fwd[k];
    }
    if (++l == levels) break;
    first = last;
    last = flevel[l + 1];
    nd = fwd[min(first + T.slot, last - 1)];
    group_barrier(T.group);
  }
  group_barrier(T.group);
}

// LAT: the latency form, for handles of few blocks (one subgame): R and S are staged in shared
// memory with the strategy, before the launch waits for its predecessor, and every inner node's
// value is stored (the level and wide schedules keep them readable).  Bound by the instruction latency
// of a few warps per phase.  Measured, whole solves: Leduc (100 iterations, a launch per tree level
// before) 14.0 -> 5.4 ms; 8 rivers of 403 hands 1.81 -> 1.50 ms (50 iterations).
template <int MODE, typename P, bool DCFR, bool LAT>
__global__ void __launch_bounds__(LAT ? 2 * kTileThreads : kTileThreads, LAT ? 2 : 4) k_tile(const GameDev* __restrict__ games,
                                                       const Work* __restrict__ work, int n_work, int player_mask,
                                                       int advance, int* iter, unsigned* done,
                                                       const Discount* __restrict__ disc_tab, int variant) {
  using V = typename P::V;
  constexpr int kTileRows = LAT ? 1 : 4;  // (row, hand) items of phase B in flight per thread
  extern __shared__ __align__(16) unsigned char smx[];
  __shared__ Discount disc;
  int p;
  const Work wk = work[terminal_item(n_work, player_mask, p)];
  const GameDev& G = games[wk.game];
  const int wlog = G.tile_wlog, W = 1 << wlog, tid = threadIdx.x, w = tid & (W - 1), slot = tid >> wlog,
            nslots = blockDim.x >> wlog;
  const int h0 = wk.unit << wlog, h = h0 + w;  // < hstride: hstride is a multiple of 32 and W divides 32
  const bool valid = h < G.n_hands;
  const int N = G.n_nodes, stride = G.hstride, rb = G.row_begin[p], nrows = G.row_begin[p + 1] - rb;
  const int tab16 = G.tile_tab16;
  const TileHead* head = reinterpret_cast<const TileHead*>(smx);
  const uint16_t* tab = reinterpret_cast<const uint16_t*>(smx);
  const TileLane T{head, tab, p, wlog, slot, h, stride, LAT ? G.tile_group : (int)blockDim.x, valid,
                   valid ? G.hand_mask[h] : 0ull};

  // shared: the tile table, values / reach [N][W], strategy [rows][W], LAT: R and S [rows][W]
  V* tval = reinterpret_cast<V*>(smx + (size_t)tab16 * 16);
  V* tsg = tval + ((size_t)N << wlog);
  double* tR = reinterpret_cast<double*>(tsg + ((size_t)nrows << wlog));
  double* tS = tR + ((size_t)nrows << wlog);
  V* val = tval + w;  // this lane's column: node n at val[n << wlog]
  V* sg = tsg + w;    // row r at sg[r << wlog]
  const size_t plane = (size_t)p * N * stride;
  V* gv = static_cast<V*>(MODE == kModeBR ? G.cfv_br : G.cfv) + plane;
  V* grch = static_cast<V*>(MODE == kModeAvg ? G.reach_bar : G.reach) + plane;
  V* gsg = static_cast<V*>(MODE == kModeAvg ? G.sigbar : G.sigma) + (size_t)rb * stride;
  double* gR = G.R + (size_t)rb * stride;
  double* gS = G.S + (size_t)rb * stride;

  // ---- what older launches wrote: the table, the strategy, and R and S (or their L2 lines)
  for (int k = tid; k < tab16; k += blockDim.x)
    reinterpret_cast<uint4*>(smx)[k] = __ldg(reinterpret_cast<const uint4*>(G.tile_tab) + k);
  auto same = [](int r) { return r; };
  if (MODE == kModeUpdate) {
    if (tid == 0) disc = disc_tab[*iter];
    tile_copy(tsg, static_cast<const V*>(gsg) + h0, (size_t)stride, wlog, nrows, same, same);
  }
  if (LAT) {
    if (MODE == kModeUpdate || MODE == kModeInit) tile_copy(tR, static_cast<const double*>(gR) + h0, (size_t)stride, wlog, nrows, same, same);
    if (MODE == kModeUpdate || MODE == kModeAvg) tile_copy(tS, static_cast<const double*>(gS) + h0, (size_t)stride, wlog, nrows, same, same);
  } else if (MODE != kModeBR) {
    const int ll = wlog == 5;  // lines of 16 doubles per row: 2, or 1
    for (int k = tid; k < nrows << ll; k += blockDim.x) {
      const size_t at = (size_t)(k >> ll) * stride + h0 + (k & ll) * 16;
      if (MODE != kModeAvg) asm volatile("prefetch.global.L2 [%0];" ::"l"(gR + at));
      if (MODE != kModeInit) asm volatile("prefetch.global.L2 [%0];" ::"l"(gS + at));
    }
  }
  pdl_wait();  // terminal values come from the launch just before this one
  pdl_trigger();
  __syncthreads();

  if (MODE == kModeUpdate || MODE == kModeBR) {
    // ---- A: end values in, then inner values
    const uint16_t* ends = tab + head->ends;
    auto end = [&](int e) { return (int)ends[e]; };
    tile_copy(tval, static_cast<const V*>(gv) + h0, (size_t)stride, wlog, head->n_ends, end, end);
    cp_async_wait_all();
    __syncthreads();
    if (!LAT) {
      tile_values<MODE, P>(T, val, sg, gv, MODE == kModeBR);
    } else {
      if (tid < T.group) {
        if (wlog == 3) tile_values8<MODE, P>(T, val, sg, gv, true);
        else tile_values<MODE, P>(T, val, sg, gv, true);
      }
      __syncthreads();
    }
  } else if (LAT) {
    cp_async_wait_all();
    __syncthreads();
  }
  if constexpr (MODE == kModeBR) {
    // FP64 root sums of the tile's chunks, reduced by the game's last block as in k_hand
    __shared__ int s_last;
    __shared__ double red64[kHandThreads];
    const int C = G.chunk;  // <= W
    if (tid < W) {
      double x = valid ? G.range64[(size_t)p * stride + h] * P::to_double(val[0]) : 0.0;
      const unsigned mask = W == 32 ? 0xffffffffu : (1u << W) - 1u;
      for (int o = C / 2; o > 0; o >>= 1) x += __shfl_down_sync(mask, x, o, C);
      if (w % C == 0 && valid) G.br_partial[(size_t)p * G.n_chunks + h / C] = x;
      __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
      const unsigned chunks = (unsigned)((min(h0 + W, G.n_hands) - h0 + C - 1) / C);
      s_last = atomicAdd(G.br_done, chunks) + chunks == (unsigned)(2 * G.n_chunks);
    }
    __syncthreads();
    if (s_last) {  // the sums of kHandThreads threads, as k_hand's last block forms them
      __threadfence();
      for (int q = 0; q < 2; ++q) {
        for (int t = tid; t < kHandThreads; t += blockDim.x) {
          double x = 0.0;
          for (int c = t; c < G.n_chunks; c += kHandThreads) x += __ldcg(&G.br_partial[(size_t)q * G.n_chunks + c]);
          red64[t] = x;
        }
        __syncthreads();
        for (int o = kHandThreads / 2; o > 0; o >>= 1) {
          for (int t = tid; t < o; t += blockDim.x) red64[t] += red64[t + o];
          __syncthreads();
        }
        if (tid == 0) G.br_out[q] = red64[0];
        __syncthreads();
      }
      if (tid == 0) *G.br_done = 0u;
    }
    return;
  }

  // ---- B: every row of the player
  {
    const TileRow* rowmap = reinterpret_cast<const TileRow*>(tab + head->rows[p]);
    double* gM = G.M ? G.M + (size_t)rb * stride + h : nullptr;
    const double* src = LAT ? (MODE == kModeAvg ? tS : tR) + w : (MODE == kModeAvg ? gS : gR) + h;
    const double* srcS = LAT ? tS + w : gS + h;
    const size_t rs = LAT ? (size_t)W : (size_t)stride;
    for (int r0 = slot; r0 < nrows; r0 += kTileRows * nslots) {
      double R[kTileRows], S[kTileRows];
      V pi[kTileRows];
      TileRow m[kTileRows];
#pragma unroll
      for (int e = 0; e < kTileRows; ++e) {
        const int r = r0 + e * nslots;
        if (r < nrows) {
          R[e] = src[r * rs];
          if (MODE == kModeUpdate) {
            m[e] = rowmap[r];
            S[e] = srcS[r * rs];
            pi[e] = grch[(size_t)m[e].src * stride + h];
          }
        }
      }
#pragma unroll
      for (int e = 0; e < kTileRows; ++e) {
        const int r = r0 + e * nslots;
        if (r < nrows) {
          double x = R[e];
          if (MODE == kModeUpdate) {
            double rd;
            x = tile_row<P, DCFR>(R[e], S[e], P::sub(val[m[e].kid << wlog], val[m[e].node << wlog]),
                                  P::mul(pi[e], sg[r << wlog]), disc, variant, rd);
            if (valid) {
              gR[(size_t)r * stride + h] = R[e];
              gS[(size_t)r * stride + h] = S[e];
              if (!DCFR && variant == 3) gM[(size_t)r * stride] = rd;
            }
          } else if (MODE == kModeInit && gM) {
            x += gM[(size_t)r * stride];
          }
          sg[r << wlog] = __double_as_longlong(x) > 0 ? P::of_double_int(x) : P::zero();
        }
      }
    }
  }
  __syncthreads();  // the positive parts are there, and the values have been read: their array takes the reach

  // ---- C.  An update stores the reach rows it makes; the other passes every node's
  if (tid < W) val[0] = valid ? static_cast<const V*>(G.range_v)[(size_t)p * stride + h] : P::zero();
  __syncthreads();
  auto put_sigma = [&](int r, V y) {
    if (valid) gsg[(size_t)r * stride + h] = y;
  };
  auto put_reach = [&](int n, V y) {
    if (MODE == kModeUpdate && valid) grch[(size_t)n * stride + h] = y;
  };
  if (LAT && match_ahead<P>(T)) {
    tile_match_all<P>(T, sg, slot, nslots, put_sigma);
    __syncthreads();
    if (tid < T.group) tile_reach_matched<P>(T, val, sg, put_reach);
  } else if (!LAT) {
    tile_reach<P>(T, val, sg, put_sigma, put_reach);
  } else if (tid < T.group) {
    if (wlog == 3) tile_reach8<P>(T, val, sg, put_sigma, put_reach);
    else tile_reach<P>(T, val, sg, put_sigma, put_reach);
  }
  if (MODE != kModeUpdate) {
    if (LAT) __syncthreads();
    const uint16_t* all = tab + head->all[p];
    for (int n = slot; valid && n < N; n += nslots) grch[(size_t)n * stride + h] = val[all[n] << wlog];
  }

  if (MODE == kModeUpdate && advance) {
    if (LAT) __syncthreads();
    if (tid == 0) {
      __threadfence();
      const unsigned prev = atomicAdd(done, 1u);
      if (prev == gridDim.x - 1) {  // last block of the launch: every block has read *iter
        *done = 0u;
        *iter += 1;
        __threadfence();
      }
    }
  }
}

// ------------------------------------------------------------------ resident schedule
//
// The latency form of whole iterations, for handles whose hand chunks all fit the GPU at
// once (a single subgame): one cooperative launch runs n iterations.  Block b owns hand chunk
// b of both players and keeps its R, S, strategy and reach rows in shared memory for the whole
// launch, beside what it needs of the board table of the terminal nodes it evaluates.  An
// iteration's phases -- the terminal values of player i (Stages 2-4), then i's update (Stages 6, 7
// and 1, as hand tiles) -- each read what the whole grid wrote in the phase before: values carrying
// their iteration's stamp when updates alternate (below), the global rows with a grid barrier
// between phases when both players update at once.  The arithmetic is that of k_terminal and
// k_tile, and the global state left at the end is theirs: the level and resident schedules give
// the same bits.  Bound by the latency of the chain of phases.  Measured on the 1081-hand river, FP32
// values: 21.9 us an iteration with grid barriers and the per-hand kernel's passes, 16.4 now.

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int ld_relaxed_s32(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
template <typename V>
__device__ __forceinline__ V ld_cg(const V* p);
template <>
__device__ __forceinline__ float ld_cg<float>(const float* p) { return __ldcg(p); }
template <>
__device__ __forceinline__ ff ld_cg<ff>(const ff* p) {
  const float2 x = __ldcg(reinterpret_cast<const float2*>(p));
  return {x.x, x.y};
}

// Bounded grid barrier: after a block barrier, one thread counts the block's arrival with a
// release reduction (the block's writes of the phase, ordered before it by the block barrier,
// are visible to whoever acquires the count) and polls with acquire loads until `target`
// arrivals (a multiple of the grid size) have been counted; the block barrier after it orders
// the other threads' reads after that acquire.  Those reads of other blocks' data go past L1
// (ld.global.cg), so no stale line is read.  False when the wait gave up, after `limit` polls
// or because another block gave up: the error flag is then set and the caller leaves.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned target, int* err, long limit) {
  __shared__ int s_ok;
  __syncthreads();  // the block's writes of this phase are done
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    int ok = 1;
    for (long k = 0; ld_acquire_u32(count) < target; ++k)
      if (k >= limit || ld_relaxed_s32(err) != 0) {
        ok = 0;
        break;
      }
    if (!ok) atomicExch(err, 1);
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

__host__ __device__ inline size_t resident_term_bytes(int H, int k, int deck, int hstride, size_t es) {
  return (size_t)TermTab(H, k, deck).fold_len * 2 + ((size_t)hstride + (size_t)(k * H + 1 + H + 1)) * es;
}

// Shared memory of the resident kernel's hand region for one game (must match k_resident): the tile
// table, per player R and S, the values (one player at a time), and per player reach and strategy.
__host__ __device__ inline size_t resident_hand_bytes(int tab16, int n_nodes, int rows_max, int W, size_t es) {
  return (size_t)tab16 * 16 + 4 * round16((size_t)rows_max * W * 8) + 3 * round16((size_t)n_nodes * W * es) +
         2 * round16((size_t)rows_max * W * es) + (size_t)4 * W * es;  // slack for tile_values8's loads
}

// What crosses blocks inside a launch of alternating updates goes as stamped words: a value and the
// iteration's stamp in one 64-bit store (two for a pair), which a reader polls until the stamp is
// there.  A value is then one store-to-load trip (770 cycles) away from its reader, where a grid
// barrier takes about 2,900 (its release, 152 arrivals at one counter, the poll) and a load after it
// another 400.  No word is overwritten before its readers are done: a terminal's values of player
// i are rewritten once its block has read a whole reach row of the next update of the opponent, to
// which every chunk contributes after having read those values; a reach row is rewritten once the
// chunk has read the next values of every terminal of its subgame, whose blocks evaluate their
// items in order, the opponent's of the iteration before among them.
__device__ __forceinline__ void stamp_put(uint64_t* w, float v, uint32_t stamp) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"((uint64_t)stamp << 32 | __float_as_uint(v)) : "memory");
}
__device__ __forceinline__ void stamp_put(uint64_t* w, ff v, uint32_t stamp) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(w), "l"((uint64_t)stamp << 32 | __float_as_uint(v.hi)),
               "l"((uint64_t)stamp << 32 | __float_as_uint(v.lo))
               : "memory");
}
__device__ __forceinline__ bool stamp_get(const uint64_t* w, uint32_t stamp, float& v) {
  uint64_t x;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(w) : "memory");
  v = __uint_as_float((uint32_t)x);
  return (uint32_t)(x >> 32) == stamp;
}
__device__ __forceinline__ bool stamp_get(const uint64_t* w, uint32_t stamp, ff& v) {
  uint64_t x, y;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(w) : "memory");
  v = {__uint_as_float((uint32_t)x), __uint_as_float((uint32_t)y)};
  return (uint32_t)(x >> 32) == stamp && (uint32_t)(y >> 32) == stamp;
}
// Bounded poll: false (and the error flag set) after `limit` polls, or once another block gave up.
template <typename V>
__device__ __forceinline__ bool stamp_wait(const uint64_t* w, uint32_t stamp, V& v, long limit, int* err) {
  for (long k = 0; k < limit; ++k) {
    if (stamp_get(w, stamp, v)) return true;
    if ((k & 63) == 63 && ld_relaxed_s32(err) != 0) return false;
  }
  atomicExch(err, 1);
  return false;
}

// A terminal node in the resident kernel: what does not change from iteration to iteration, kept
// while the block's next item is the same node.
template <typename P>
struct ResidentTerm {
  int item;  // its term_work entry, or -1
  const GameDev* G;
  int H, k, deck, N, stride, node, table;
  bool show;
  uint64_t board;
  TermSrc src;
  ff u[2];
  int tab_game, tab_table, tab_show;  // what ft and lane hold
  TermLane<P> lane;
};

// Values of player i at terminal item e (Stages 2-4).  The opponent's reach row comes from the global
// rows (written by an earlier launch, or before a grid barrier) or, when `get` is set, with the stamp
// `from_stamp` from xreach; the values go to the global rows when `plain` is set, and with the stamp
// `stamp` to xval when `put` is.  False when a wait gave up.  Ends with a block barrier.
template <typename P>
__device__ __forceinline__ bool resident_terminal(const GameDev* __restrict__ games, const Work* __restrict__ term_work,
                                                  const TermSrc* __restrict__ term_src, int e, int i, unsigned char* smr,
                                                  ResidentTerm<P>& R, bool get, uint32_t from_stamp, bool put,
                                                  uint32_t stamp, bool plain, long limit, int* err) {
  using V = typename P::V;
  constexpr int words = (int)sizeof(V) / 4;  // stamped words per value
  const int tid = threadIdx.x;
  uint16_t* ft = reinterpret_cast<uint16_t*>(smr);
  if (R.item != e) {
    R.item = e;
    const Work wk = term_work[e];
    R.G = games + wk.game;
    const NodeDev nd = R.G->nodes[wk.unit];
    R.H = R.G->n_hands, R.k = R.G->hand_size, R.deck = R.G->deck, R.N = R.G->n_nodes, R.stride = R.G->hstride;
    R.node = wk.unit;
    R.src = term_src[e];
    R.show = nd.type == kShowdown;
    // a fold reads table 0, as in k_terminal (each table orders its per-card hand lists by its
    // own board's ranks, so another table's lists would sum the same reach in another order)
    R.table = R.show ? nd.row : 0;
    R.board = nd.board;
    for (int p = 0; p < 2; ++p) R.u[p] = terminal_payoff(*R.G, nd, wk.unit, p);
    if (R.tab_game != wk.game || R.tab_table != R.table || R.tab_show != R.show) {
      const TermTab tt(R.H, R.k, R.deck);
      const uint4* gt = reinterpret_cast<const uint4*>(R.G->term_tab + (size_t)R.table * tt.len);
      for (int x = tid; x < tt.fold_len / 8; x += kTermThreads) reinterpret_cast<uint4*>(ft)[x] = __ldg(gt + x);
      term_lane_load(R.lane, *R.G, R.table, R.show);
      R.tab_game = wk.game, R.tab_table = R.table, R.tab_show = R.show;
    }
  }
  const int H = R.H, k = R.k, stride = R.stride, from = R.src.row[1 - i];
  const TermTab tt(H, k, R.deck);
  V* q = reinterpret_cast<V*>(smr + (size_t)tt.fold_len * 2);
  V* CP = q + stride;
  V* Ps = CP + (k * H + 1);
  const size_t row = ((size_t)(1 - i) * R.N + term_src_node(from)) * stride;
  bool ok = true;
  if (!get) {
    const V* src = static_cast<const V*>(R.G->reach) + row;
    for (int h = tid; h < H; h += kTermThreads) q[h] = ld_cg(src + h);
  } else {
    const uint64_t* src = R.G->xreach + row * words;
    V v[kTermHands];
    bool got[kTermHands];
#pragma unroll
    for (int s = 0; s < kTermHands; ++s) {  // the first polls go out together
      const int h = tid + s * kTermThreads;
      got[s] = h >= H || (limit > 0 && stamp_get(src + (size_t)h * words, from_stamp, v[s]));
    }
#pragma unroll
    for (int s = 0; s < kTermHands; ++s) {
      const int h = tid + s * kTermThreads;
      if (!got[s]) ok = stamp_wait(src + (size_t)h * words, from_stamp, v[s], limit, err) && ok;
      if (h < H) q[h] = v[s];
    }
  }
  if (!__syncthreads_and(ok)) return false;
  if (from < 0) {  // below an all-in run-out: zero the hands holding a card dealt on the way
    for (int h = tid; h < H; h += kTermThreads)
      if (holds_board_card(ft + tt.cards, h, k, R.board)) q[h] = P::zero();
    __syncthreads();
  }
  const size_t out = ((size_t)i * R.N + R.node) * stride;
  V* dst = static_cast<V*>(R.G->cfv) + out;
  uint64_t* xdst = R.G->xval + out * words;
  terminal_node<P>(R.lane, H, k, R.deck, R.show, R.board, R.u[i], q, ft, CP, Ps, [&](int h, V v) {
    if (put) stamp_put(xdst + (size_t)h * words, v, stamp);
    if (plain) dst[h] = v;
  });
  __syncthreads();  // the row buffer and the scan arrays are free again
  return true;
}

// n_iters iterations (alternating: terminal and update of player 0, then of player 1;
// otherwise both players' terminals, then both updates).  Launched cooperatively, every block
// resident: grid >= n_chunk_work.  Alternating updates pass values and reach as stamped words (the
// stamp of iteration it of this launch is sync[2] + it + 1); simultaneous ones through the global
// rows, a grid barrier between phases.  sync[0] counts barrier arrivals, sync[1] blocks that have
// finished; the last block to finish resets both and advances *iter and sync[2] by n_iters.  The
// stamps are counted on the device, over the handle's life, so that a launch replayed from a
// captured graph takes new ones too; every word is rewritten every iteration, so they may wrap.
// AHEAD: some tree of the handle has its regrets matched ahead of the walk (match_ahead).  Handles without
// such trees are faster without that code (river of 789 hands and two levels with pairs 23.7 -> 22.1 us an
// iteration).
template <typename P, bool AHEAD>
__global__ void __launch_bounds__(kTermThreads, 1) k_resident(
    const GameDev* __restrict__ games, const Work* __restrict__ chunk_work, int n_chunk_work,
    const Work* __restrict__ term_work, const TermSrc* __restrict__ term_src, int n_term_work, int alternating,
    int n_iters, int* iter, const Discount* __restrict__ disc_tab, int variant, unsigned* sync, int* err,
    unsigned term_bytes) {
  using V = typename P::V;
  constexpr size_t es = sizeof(V);
  constexpr int words = (int)sizeof(V) / 4;
  extern __shared__ __align__(16) unsigned char smr[];
  const int tid = threadIdx.x;
  const bool owner = (int)blockIdx.x < n_chunk_work;
  const Work wk = owner ? chunk_work[blockIdx.x] : Work{0, 0};
  const GameDev& G = games[wk.game];
  const int wlog = G.tile_wlog, W = 1 << wlog, w = tid & (W - 1), slot = tid >> wlog, nslots = kTermThreads >> wlog;
  const int h = wk.unit * W + w;  // < hstride
  const bool valid = owner && h < G.n_hands;
  const int N = G.n_nodes, stride = G.hstride, tab16 = G.tile_tab16;
  const int rows_max = max(G.row_begin[1] - G.row_begin[0], G.row_begin[2] - G.row_begin[1]);

  // hand region (see resident_hand_bytes), after the terminal region; columns of this lane
  unsigned char* cur = smr + term_bytes;
  unsigned char* stab = cur;
  cur += (size_t)tab16 * 16;
  const size_t rd8 = round16((size_t)rows_max * W * 8);
  double* sR[2] = {reinterpret_cast<double*>(cur) + w, reinterpret_cast<double*>(cur + rd8) + w};
  cur += 2 * rd8;
  double* sS[2] = {reinterpret_cast<double*>(cur) + w, reinterpret_cast<double*>(cur + rd8) + w};
  cur += 2 * rd8;
  const size_t nv = round16((size_t)N * W * es), rv = round16((size_t)rows_max * W * es);
  V* val = reinterpret_cast<V*>(cur) + w;
  cur += nv;
  V* srch[2] = {reinterpret_cast<V*>(cur) + w, reinterpret_cast<V*>(cur + nv) + w};
  cur += 2 * nv;
  V* ssg[2] = {reinterpret_cast<V*>(cur) + w, reinterpret_cast<V*>(cur + rv) + w};
  const TileHead* head = reinterpret_cast<const TileHead*>(stab);
  const uint16_t* tab = reinterpret_cast<const uint16_t*>(stab);

  // ---- stage the tree and the chunk's state of both players (written by earlier launches)
  if (owner) {
    for (int k = tid; k < tab16; k += kTermThreads)
      reinterpret_cast<uint4*>(stab)[k] = __ldg(reinterpret_cast<const uint4*>(G.tile_tab) + k);
    for (int p = 0; p < 2; ++p) {
      const int rb = G.row_begin[p], nrows = G.row_begin[p + 1] - rb;
      for (int r = slot; r < nrows; r += nslots) {
        const size_t g = (size_t)(rb + r) * stride + h;
        sR[p][r << wlog] = G.R[g];
        sS[p][r << wlog] = G.S[g];
        ssg[p][r << wlog] = static_cast<const V*>(G.sigma)[g];
      }
      const V* grch = static_cast<const V*>(G.reach) + (size_t)p * N * stride + h;
      for (int n = slot; n < N; n += nslots) srch[p][n << wlog] = grch[(size_t)n * stride];
    }
  }
  __syncthreads();

  const int it0 = *iter;             // written only by the last block to finish
  const uint32_t stamp0 = sync[2];  // too
  const int steps = alternating ? 2 : 1;
  // A step's terminal items, of the one or both players.  Each block takes neighbours of the list, which
  // is sorted by board table and kind, so that what it keeps of the table stays (taking every
  // gridDim.x-th, Leduc's blocks met a fold and a showdown in turn: 38.4 against 34.6 us an iteration,
  // with pairs 56.0 against 50.2).
  const int items = (alternating ? 1 : 2) * n_term_work, share = items / (int)gridDim.x, over = items % (int)gridDim.x;
  const int item0 = (int)blockIdx.x * share + min((int)blockIdx.x, over),
            item1 = item0 + share + ((int)blockIdx.x < over);
  unsigned nbar = 0;
  bool ok = true;
  ResidentTerm<P> term;
  term.item = term.tab_game = term.tab_table = term.tab_show = -1;
  for (int it = 0; it < n_iters && ok; ++it) {
    const Discount d = disc_tab[it0 + it];
    const bool last = it == n_iters - 1;
    const uint32_t stamp = stamp0 + (uint32_t)it + 1u;
    for (int step = 0; step < steps && ok; ++step) {
      const int pm = alternating ? 1 << step : 3;
      const int p0 = pm == 2 ? 1 : 0, np = pm == 3 ? 2 : 1;
      const long limit = it == 0 ? g_first_wait_polls : kWaitLimit;
      // ---- terminal values of the player(s) of this step (Stages 2-4)
      for (int item = item0; item < item1 && ok; ++item) {
        const int e = item < n_term_work ? item : item - n_term_work, i = p0 + (item >= n_term_work);
        // player 0's first terminals read what the launch before left
        ok = resident_terminal<P>(games, term_work, term_src, e, i, smr, term, alternating && (it > 0 || step > 0),
                                  step == 0 ? stamp - 1u : stamp, alternating != 0, stamp, !alternating || last, limit, err);
      }
      if (!ok) break;
      if (!alternating) {
        ++nbar;
        ok = grid_barrier(&sync[0], nbar * gridDim.x, err, nbar == 1 ? g_first_wait_polls : kWaitLimit);
        if (!ok) break;
      }
      // ---- the update of the chunk's hands (Stages 6, 7, then 1 with the new strategy)
      if (owner) {
        for (int p = p0; p < p0 + np && ok; ++p) {
          const int rb = G.row_begin[p], nrows = G.row_begin[p + 1] - rb;
          const TileLane T{head, tab, p, wlog, slot, h, stride, G.tile_group, valid,
                           valid ? G.hand_mask[h] : 0ull};
          const size_t plane = (size_t)p * N * stride;
          V* gv = static_cast<V*>(G.cfv) + plane;
          V* grch = static_cast<V*>(G.reach) + plane;
          const uint64_t* xv = G.xval + plane * words;
          uint64_t* xr = G.xreach + plane * words;
          const uint16_t* ends = tab + head->ends;
          bool got = true;
          const int n_ends = head->n_ends;
          if (!alternating || n_ends <= nslots) {
            for (int e = slot; e < n_ends; e += nslots) {
              const int n = ends[e];
              const size_t at = (size_t)n * stride + h;
              V x = P::zero();
              if (!alternating) x = ld_cg(gv + at);
              else if (valid) got = stamp_wait(xv + at * words, stamp, x, limit, err) && got;
              val[n << wlog] = x;
            }
          } else {  // several values a thread: their first polls go out together (165-node river 20.4 -> 20.0 us)
            constexpr int kPolls = 4;
            for (int e0 = slot; e0 < n_ends; e0 += kPolls * nslots) {
              V x[kPolls];
              bool have[kPolls];
#pragma unroll
              for (int u = 0; u < kPolls; ++u) {
                const int e = e0 + u * nslots;
                x[u] = P::zero();
                have[u] = !valid || e >= n_ends ||
                          (limit > 0 && stamp_get(xv + ((size_t)ends[e] * stride + h) * words, stamp, x[u]));
              }
#pragma unroll
              for (int u = 0; u < kPolls; ++u) {
                const int e = e0 + u * nslots;
                if (!have[u]) got = stamp_wait(xv + ((size_t)ends[e] * stride + h) * words, stamp, x[u], limit, err) && got;
                if (e < n_ends) val[ends[e] << wlog] = x[u];
              }
            }
          }
          ok = __syncthreads_and(got);
          if (!ok) break;
          // A: later iterations of the launch overwrite the inner values, so only the last stores them
          if (tid < T.group) {
            if (wlog == 3) tile_values8<kModeUpdate, P, true>(T, val, ssg[p], gv, last);
            else tile_values<kModeUpdate, P, true>(T, val, ssg[p], gv, last);
          }
          __syncthreads();
          // B
          const TileRow* rowmap = reinterpret_cast<const TileRow*>(tab + head->rows[p]);
          for (int r = slot; r < nrows; r += nslots) {
            const TileRow m = rowmap[r];
            double rd, R = sR[p][r << wlog], S = sS[p][r << wlog];
            const double x = tile_row<P, false>(R, S, P::sub(val[m.kid << wlog], val[m.node << wlog]),
                                                P::mul(srch[p][m.src << wlog], ssg[p][r << wlog]), d, variant, rd);
            sR[p][r << wlog] = R;
            sS[p][r << wlog] = S;
            if (variant == 3 && valid) G.M[(size_t)(rb + r) * stride + h] = rd;
            ssg[p][r << wlog] = __double_as_longlong(x) > 0 ? P::of_double_int(x) : P::zero();
          }
          __syncthreads();
          // C: the opponent's terminal values read the new reach rows (the root's never changes, but its
          // stamp tells that this update is done)
          auto put_reach = [&](int n, V y) {
            if (!valid) return;
            const size_t at = (size_t)n * stride + h;
            if (alternating) stamp_put(xr + at * words, y, stamp);
            if (!alternating || last) grch[at] = y;
          };
          if (tid < W) put_reach(0, srch[p][0]);
          auto put_sigma = [&](int r, V y) { ssg[p][r << wlog] = y; };
          if (AHEAD && match_ahead<P>(T)) {
            tile_match_all<P>(T, ssg[p], slot, nslots, [](int, V) {});
            __syncthreads();
            if (tid < T.group) tile_reach_matched<P>(T, srch[p], ssg[p], put_reach);
          } else if (tid < T.group) {
            if (wlog == 3) tile_reach8<P>(T, srch[p], ssg[p], put_sigma, put_reach);
            else tile_reach<P>(T, srch[p], ssg[p], put_sigma, put_reach);
          }
          if (np == 2) __syncthreads();  // the values are free for the other player
        }
      }
      if (!alternating) {
        ++nbar;
        ok = ok && grid_barrier(&sync[0], nbar * gridDim.x, err, kWaitLimit);
      } else {
        __syncthreads();  // the strategy and reach rows of this update are in place
      }
    }
  }

  // ---- the chunk's R, S and strategy rows back to global memory
  if (ok && valid) {
    for (int p = 0; p < 2; ++p) {
      const int rb = G.row_begin[p], nrows = G.row_begin[p + 1] - rb;
      for (int r = slot; r < nrows; r += nslots) {
        const size_t g = (size_t)(rb + r) * stride + h;
        G.R[g] = sR[p][r << wlog];
        G.S[g] = sS[p][r << wlog];
        static_cast<V*>(G.sigma)[g] = ssg[p][r << wlog];
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(&sync[1], 1u) == gridDim.x - 1) {  // every other block has left its waits
      sync[0] = 0u;
      sync[1] = 0u;
      sync[2] = stamp0 + (uint32_t)n_iters;
      *iter += n_iters;
      __threadfence();
    }
  }
}

// ------------------------------------------------------------------ stream schedule
//
// The throughput form of the update launch (Stages 6, 7 and then 1 of one player), for
// handles whose hands fill the GPU many times over (batches of subgames).  One warp owns 32
// consecutive hands of one subgame and walks the subgame's depth-first program alone: no
// block barriers, every access to an R, S, reach or value row is one coalesced 32-lane
// segment, and the only per-node state kept is a stack per lane in shared memory.
//   1. bottom-up over the program in reverse: values of Eq. (backward) from the terminal
//      values, and at each of the player's decision nodes the regrets and the Stage 7
//      update of R and S with sigma = RM(R) (Eq. rm) and the player's reach there (stored
//      by the previous update of this player, or by the initial pass);
//   2. top-down over the program with the new strategy RM(R'): the player's reach at its
//      decision nodes (for its next update) and at the terminals (for the opponent's next
//      terminal launch).
// Strategies and the values of inner nodes never go to DRAM.  Every address a pass reads
// is fixed by the program, so each pass is cut into chunks (stream_tables) that are loaded
// into a per-lane ring in shared memory with cp.async one chunk ahead of the computation.
// The arithmetic (regret matching, child order of every sum, the update) is that of k_hand,
// so both schedules give the same bits.


// Regret matching of one node's A rows (Eq. rm), as k_hand computes it: positive parts in
// the value type, their sum in action order, exactly 1 for a lone positive action.
template <typename P>
__device__ __forceinline__ void regret_match(const double (&Rv)[kStreamMaxActions], int A,
                                             typename P::V (&sg)[kStreamMaxActions]) {
  using V = typename P::V;
  V tot = P::zero();
  int npos = 0, last = 0;
#pragma unroll
  for (int a = 0; a < kStreamMaxActions; ++a) {
    if (a < A) {
      const V x = __double_as_longlong(Rv[a]) > 0 ? P::of_double(Rv[a]) : P::zero();
      sg[a] = x;
      if (P::positive(x)) ++npos, last = a;
      tot = P::add(tot, x);
    }
  }
  if (npos == 1) {
#pragma unroll
    for (int a = 0; a < kStreamMaxActions; ++a) sg[a] = a == last ? P::one() : P::zero();
  } else if (npos > 1) {
    const V inv = P::recip(tot);
#pragma unroll
    for (int a = 0; a < kStreamMaxActions; ++a)
      if (a < A) sg[a] = P::mul(sg[a], inv);
  } else {
    const V uni = P::uniform(A);
#pragma unroll
    for (int a = 0; a < kStreamMaxActions; ++a) sg[a] = uni;
  }
}

// regret_match with a compile-time action count (same arithmetic, no per-action guards), with
// the three cases selected per lane instead of branched on: the hands of a warp often fall
// in different cases, and a branch would run all three paths for them.
template <typename P, int NA>
__device__ __forceinline__ void regret_match_n(const double (&Rv)[NA], typename P::V (&sg)[NA]) {
  using V = typename P::V;
  V tot = P::zero();
  int npos = 0, last = 0;
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    const V x = __double_as_longlong(Rv[a]) > 0 ? P::of_double(Rv[a]) : P::zero();
    sg[a] = x;
    if (P::positive(x)) ++npos, last = a;
    tot = P::add(tot, x);
  }
  const V inv = P::recip(tot);  // unused (and possibly not finite) unless npos > 1
  const V uni = P::uniform(NA);
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    const V many = P::mul(sg[a], inv);
    sg[a] = npos > 1 ? many : npos == 1 ? (a == last ? P::one() : P::zero()) : uni;
  }
}

__device__ __forceinline__ void load_rows(const double* __restrict__ base, size_t stride, int A,
                                          double (&out)[kStreamMaxActions]) {
#pragma unroll
  for (int a = 0; a < kStreamMaxActions; ++a) out[a] = a < A ? base[(size_t)a * stride] : 0.0;
}

// A program node, decoded.
struct Op {
  int node_off, row_off, type, player, A, deal, tmask, first_kid;
};
__device__ __forceinline__ Op decode(const ProgOp& o) {
  return {o.node_off,
          o.row_off,
          (int)(o.code & 3u),
          (int)((o.code >> 2) & 1u),
          (int)((o.code >> 3) & 63u),
          (int)((o.code >> 9) & 0xffu),
          (int)((o.code >> 17) & 0xffu),
          o.first_kid};
}

// One lane's view of its subgame for the stream passes.  A warp owns 32 * HP consecutive
// hands; lane l holds hands l, l + 32, ..., l + 32 (HP - 1) of them (HP = 1 or 2), so the
// walk's control work (program decode, branches, stack and ring bookkeeping, load issue)
// is shared by HP hands per lane and each lane has HP independent arithmetic chains.
template <typename P, int HP>
struct StreamLane {
  using V = typename P::V;
  const GameDev& G;
  const ProgOp* prog;     // the program (shared memory when staged)
  const uint32_t* units;  // this player's loads, bottom-up pass then top-down pass
  int p;
  bool valid[HP];         // hand l + 32 k exists
  uint64_t hmask[HP];
  size_t stride;
  double* R;        // column of the lane's first hand of R (hand k: + 32 k)
  double* S;
  double* M;        // the same of the Predictive CFR+ prediction (null otherwise)
  V* reach;         // column of the lane's first hand in player p's reach plane
  V* cfv;           // the same in player p's value plane
  uint64_t* ring;   // this lane's entry of the prefetch ring: unit u of half k at
                    // ring[(k * half + u) * 32 * HP], its hand k at + 32 k
  int half;         // units in each half of the ring
  V* st;            // this lane's stack: slot s, hand k at st[(s * HP + k) * 32]
};

// Issue loads [u0, u1) of a pass into ring half `half` (one commit group).  A unit is the
// warp's segment of 32 * HP consecutive elements of one row (256 * HP bytes of FP64 or pair
// values, 128 * HP of FP32 ones), landing at slot u - u0 of the ring half.  The warp's lanes
// split the units into 16-byte pieces (16 * HP per FP64 unit), so that one copy instruction
// moves pieces of several units.
template <typename P, int HP>
__device__ __forceinline__ void stream_issue(const StreamLane<P, HP>& L, const uint32_t* units, int u0, int u1,
                                             int half) {
  using V = typename P::V;
  constexpr int kPieces = 16 * HP;  // 16-byte pieces of one unit
  const int lane = threadIdx.x & 31;
  unsigned char* ring = reinterpret_cast<unsigned char*>(L.ring - lane + (size_t)half * L.half * 32 * HP);
  const int pieces = (u1 - u0) * kPieces;
  for (int k = lane; k < pieces; k += 32) {
    const int u = u0 + k / kPieces, part = k % kPieces;
    const uint32_t d = units[u];
    const uint32_t arr = d >> kArrShift, off = d & kArrOffMask;
    // the row's segment starts at the warp's first hand: the lane's column pointer minus its lane
    const void* src;
    if (arr == kArrR)
      src = L.R - lane + off + 2 * part;
    else if (arr == kArrS)
      src = L.S - lane + off + 2 * part;
    else if (arr == kArrM)
      src = L.M - lane + off + 2 * part;
    else if (part * 16 >= 32 * HP * (int)sizeof(V))  // FP32 rows fill half a slot
      continue;
    else
      src = reinterpret_cast<const unsigned char*>((arr == kArrReach ? L.reach : L.cfv) - lane + off) + part * 16;
    cp_async<16>(ring + (size_t)(u - u0) * 256 * HP + (size_t)part * 16, src);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// This lane's value of its hand k in a ring unit (slot: the lane's entry of the unit):
// 8-byte values sit at entry lane + 32 k, FP32 values packed at float lane + 32 k.
template <typename P, int HP>
__device__ __forceinline__ typename P::V ring_value(const uint64_t* slot, int k) {
  using V = typename P::V;
  if constexpr (sizeof(V) == 4) {
    const int lane = threadIdx.x & 31;
    return reinterpret_cast<const V*>(slot - lane)[lane + 32 * k];
  } else {
    return *reinterpret_cast<const V*>(slot + 32 * k);
  }
}

// Bottom-up work at one of the player's decision nodes with NA actions (Stages 6-7), for
// each of the lane's HP hands: the children's values (ring or stack), regret matching of R
// (R + M for Predictive CFR+), the node value, and the new R, S (and M) rows.  NA is a
// compile-time constant so that the actions' FP64 update chains are straight-line code the
// compiler can interleave.
template <typename P, int NA, int HP>
__device__ __forceinline__ void decision_back(const StreamLane<P, HP>& L, const Op& nd, const uint64_t* ring, int& u,
                                              int& sp, const Discount& d, int variant, typename P::V (&val)[HP]) {
  using V = typename P::V;
  constexpr int U = 32 * HP;  // ring entries per unit
  V* st = L.st;
  V c[NA][HP];
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    if ((nd.tmask >> a) & 1) {
#pragma unroll
      for (int k = 0; k < HP; ++k) c[a][k] = ring_value<P, HP>(ring + (size_t)u * U, k);
      ++u;
    } else {
      --sp;
#pragma unroll
      for (int k = 0; k < HP; ++k) c[a][k] = st[(sp * HP + k) * 32];
    }
  }
  const bool pred = L.M != nullptr;  // Predictive CFR+: R, M, S, reach
  const double* Rr = reinterpret_cast<const double*>(ring + (size_t)u * U);
  const double* Mr = reinterpret_cast<const double*>(ring + (size_t)(u + NA) * U);
  const double* Sr = reinterpret_cast<const double*>(ring + (size_t)(u + (pred ? 2 : 1) * NA) * U);
  const uint64_t* pislot = ring + (size_t)(u + (pred ? 3 : 2) * NA) * U;
  u += (pred ? 3 : 2) * NA + 1;
#pragma unroll
  for (int k = 0; k < HP; ++k) {
    const V pi = ring_value<P, HP>(pislot, k);
    double Rv[NA];
    V sg[NA];
    {
      double Rm[NA];
#pragma unroll
      for (int a = 0; a < NA; ++a) Rv[a] = Rm[a] = Rr[(size_t)a * U + 32 * k];
      if (pred) {  // Predictive CFR+ matches R + M (no FP64 add for the other variants)
#pragma unroll
        for (int a = 0; a < NA; ++a) Rm[a] = Rv[a] + Mr[(size_t)a * U + 32 * k];
      }
      regret_match_n<P, NA>(Rm, sg);
    }
    typename P::Acc acc = P::acc0();
#pragma unroll
    for (int a = 0; a < NA; ++a) P::acc_mul(acc, sg[a], c[a][k]);
    val[k] = P::value(acc);
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      const V rr = P::sub(c[a][k], val[k]);                    // instantaneous regret
      const double contrib = P::to_double(P::mul(pi, sg[a]));  // pi_i(I) sigma(I, a)
      const double rd = P::to_double(rr);
      double x = Rv[a] + rd;
      if (variant == 2) x *= __double_as_longlong(x) > 0 ? d.dpos : d.dneg;
      if ((variant == 1 || variant == 3) && __double_as_longlong(x) < 0) x = 0.0;
      const double sn =
          fma(Sr[(size_t)a * U + 32 * k], d.dS, (variant == 1 || variant == 3) ? d.wS * contrib : contrib);
      if (L.valid[k]) {
        const size_t at = (size_t)nd.row_off + (size_t)a * L.stride + 32 * k;
        L.R[at] = x;
        L.S[at] = sn;
        if (pred) L.M[at] = rd;
      }
    }
  }
}

// Top-down work at one of the player's decision nodes with NA actions: the reach x there is
// recorded, sigma = RM(R) (of R + M for Predictive CFR+) is formed from the ring, and each
// child's reach x sigma(a) goes to the terminal's row or onto the stack (child 0 on top).  NA
// is a compile-time constant, as in decision_back.
template <typename P, int NA, int HP>
__device__ __forceinline__ void decision_fwd(const StreamLane<P, HP>& L, const Op& nd, const uint64_t* ring, int& u,
                                             int& sp, const typename P::V (&x)[HP]) {
  using V = typename P::V;
  constexpr int U = 32 * HP;
  V* st = L.st;
  const bool pred = L.M != nullptr;  // Predictive CFR+: R then M
  const double* Rr = reinterpret_cast<const double*>(ring + (size_t)u * U);
  const double* Mr = reinterpret_cast<const double*>(ring + (size_t)(u + NA) * U);
  u += (pred ? 2 : 1) * NA;
  V sg[NA][HP];
#pragma unroll
  for (int k = 0; k < HP; ++k) {
    if (L.valid[k]) L.reach[(size_t)nd.node_off + 32 * k] = x[k];
    double Rv[NA];
    V s1[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) Rv[a] = Rr[(size_t)a * U + 32 * k];
    if (pred) {  // Predictive CFR+ matches R + M
#pragma unroll
      for (int a = 0; a < NA; ++a) Rv[a] += Mr[(size_t)a * U + 32 * k];
    }
    regret_match_n<P, NA>(Rv, s1);
#pragma unroll
    for (int a = 0; a < NA; ++a) sg[a][k] = s1[a];
  }
#pragma unroll
  for (int a = NA - 1; a >= 0; --a) {
    if ((nd.tmask >> a) & 1) {
#pragma unroll
      for (int k = 0; k < HP; ++k)
        if (L.valid[k]) L.reach[(size_t)(nd.first_kid + a) * L.stride + 32 * k] = P::mul(x[k], sg[a][k]);
    } else {
#pragma unroll
      for (int k = 0; k < HP; ++k) st[(sp * HP + k) * 32] = P::mul(x[k], sg[a][k]);
      ++sp;
    }
  }
}

// Bottom-up pass over chunk [k0, k1) (program positions counted from its end).  A node's
// children values come from the ring (terminal children, in child order) or from the stack
// (inner children, child 0 on top).
template <typename P, int HP>
__device__ __forceinline__ void stream_backward_chunk(const StreamLane<P, HP>& L, int k0, int k1, int half, int& sp,
                                                      const Discount& d, int variant) {
  using V = typename P::V;
  constexpr int U = 32 * HP;
  const int N = L.G.prog_len;
  const uint64_t* ring = L.ring + (size_t)half * L.half * U;
  V* st = L.st;
  int u = 0;
  for (int k = k0; k < k1; ++k) {
    const Op nd = decode(L.prog[N - 1 - k]);
    const int A = nd.A;
    V val[HP];
    if (nd.type == kChance || nd.player != L.p) {
      // chance: children values carry the card probabilities (a hand holding the card gets
      // nothing from that child); opponent: the plain sum
      const bool chance = nd.type == kChance;
      const bool term_all = nd.tmask & 1;  // chance: all children terminal (after an all-in) or all inner
      typename P::Acc acc[HP];
#pragma unroll
      for (int j = 0; j < HP; ++j) acc[j] = P::acc0();
      for (int a = 0; a < A; ++a) {
        const bool term = chance ? term_all : ((nd.tmask >> a) & 1);
        const int deal = chance ? L.G.nodes[nd.first_kid + a].deal : 0;
        if (!term) --sp;
#pragma unroll
        for (int j = 0; j < HP; ++j) {
          const V x = term ? ring_value<P, HP>(ring + (size_t)u * U, j) : st[(sp * HP + j) * 32];
          if (!chance || !((L.hmask[j] >> deal) & 1ull)) P::acc(acc[j], x);
        }
        if (term) ++u;
      }
#pragma unroll
      for (int j = 0; j < HP; ++j) val[j] = P::value(acc[j]);
    } else {  // the player's decision node: its action count as a compile-time constant
      switch (A) {
        case 1: decision_back<P, 1, HP>(L, nd, ring, u, sp, d, variant, val); break;
        case 2: decision_back<P, 2, HP>(L, nd, ring, u, sp, d, variant, val); break;
        case 3: decision_back<P, 3, HP>(L, nd, ring, u, sp, d, variant, val); break;
        case 4: decision_back<P, 4, HP>(L, nd, ring, u, sp, d, variant, val); break;
        case 5: decision_back<P, 5, HP>(L, nd, ring, u, sp, d, variant, val); break;
        case 6: decision_back<P, 6, HP>(L, nd, ring, u, sp, d, variant, val); break;
        case 7: decision_back<P, 7, HP>(L, nd, ring, u, sp, d, variant, val); break;
        default: decision_back<P, kStreamMaxActions, HP>(L, nd, ring, u, sp, d, variant, val); break;
      }
    }
#pragma unroll
    for (int j = 0; j < HP; ++j) st[(sp * HP + j) * 32] = val[j];
    ++sp;
  }
}

// Top-down pass over chunk [k0, k1) with sigma = RM(R): records the reach at the player's
// decision nodes, at chance nodes and, for the terminal children, at the terminals; pushes
// the reach of the inner children (child 0 on top).
template <typename P, int HP>
__device__ __forceinline__ void stream_forward_chunk(const StreamLane<P, HP>& L, int k0, int k1, int half, int& sp) {
  using V = typename P::V;
  constexpr int U = 32 * HP;
  const uint64_t* ring = L.ring + (size_t)half * L.half * U;
  V* st = L.st;
  int u = 0;
  for (int k = k0; k < k1; ++k) {
    const Op nd = decode(L.prog[k]);
    --sp;
    V x[HP];
#pragma unroll
    for (int j = 0; j < HP; ++j) {
      x[j] = st[(sp * HP + j) * 32];
      if (nd.deal != kNoCard && ((L.hmask[j] >> nd.deal) & 1ull)) x[j] = P::zero();
    }
    const int A = nd.A;
    if (nd.type == kDecision && nd.player == L.p) {  // its action count as a compile-time constant
      switch (A) {
        case 1: decision_fwd<P, 1, HP>(L, nd, ring, u, sp, x); break;
        case 2: decision_fwd<P, 2, HP>(L, nd, ring, u, sp, x); break;
        case 3: decision_fwd<P, 3, HP>(L, nd, ring, u, sp, x); break;
        case 4: decision_fwd<P, 4, HP>(L, nd, ring, u, sp, x); break;
        case 5: decision_fwd<P, 5, HP>(L, nd, ring, u, sp, x); break;
        case 6: decision_fwd<P, 6, HP>(L, nd, ring, u, sp, x); break;
        case 7: decision_fwd<P, 7, HP>(L, nd, ring, u, sp, x); break;
        default: decision_fwd<P, kStreamMaxActions, HP>(L, nd, ring, u, sp, x); break;
      }
    } else if (nd.type == kChance) {  // the player's reach passes through to each card
#pragma unroll
      for (int j = 0; j < HP; ++j)
        if (L.valid[j]) L.reach[(size_t)nd.node_off + 32 * j] = x[j];  // read by an all-in run-out's showdowns
      if (nd.tmask & 1) {  // terminal children: their reach, zero where the hand holds the card
        for (int a = 0; a < A; ++a) {
          const int deal = L.G.nodes[nd.first_kid + a].deal;
#pragma unroll
          for (int j = 0; j < HP; ++j)
            if (L.valid[j])
              L.reach[(size_t)(nd.first_kid + a) * L.stride + 32 * j] = ((L.hmask[j] >> deal) & 1ull) ? P::zero() : x[j];
        }
      } else {  // inner children apply their own card when they pop it
        for (int a = 0; a < A; ++a) {
#pragma unroll
          for (int j = 0; j < HP; ++j) st[(sp * HP + j) * 32] = x[j];
          ++sp;
        }
      }
    } else {  // opponent decision: the player's reach passes through
      for (int a = A - 1; a >= 0; --a) {
        if ((nd.tmask >> a) & 1) {
#pragma unroll
          for (int j = 0; j < HP; ++j)
            if (L.valid[j]) L.reach[(size_t)(nd.first_kid + a) * L.stride + 32 * j] = x[j];
        } else {
#pragma unroll
          for (int j = 0; j < HP; ++j) st[(sp * HP + j) * 32] = x[j];
          ++sp;
        }
      }
    }
  }
}

// One pass (list q of the load tables): chunk c + 1 loads while chunk c computes.
template <typename P, int HP, typename F>
__device__ __forceinline__ void stream_pass(const StreamLane<P, HP>& L, int q, const uint32_t* units, F compute) {
  const int32_t* ch = L.G.chunks + 2 * (size_t)L.G.chunk_off[q];  // (node, unit) pairs
  const int nch = L.G.chunk_count[q];
  stream_issue<P, HP>(L, units, ch[1], ch[3], 0);
  for (int c = 0; c < nch; ++c) {
    if (c + 1 < nch)
      stream_issue<P, HP>(L, units, ch[2 * c + 3], ch[2 * c + 5], (c + 1) & 1);
    else
      asm volatile("cp.async.commit_group;" ::: "memory");
    cp_async_wait_group<1>();  // chunk c has landed: this lane's pieces
    __syncwarp();              // and the other lanes' (each lane reads its own column of every piece)
    compute(ch[2 * c], ch[2 * c + 2], c & 1);
  }
  cp_async_wait_group<0>();
}

// Grid: one block per (player, work item); a work item is a game and the first of the
// kStreamWarps consecutive groups of 32 * HP hands its warps own.
template <typename P, int HP>
__global__ void __launch_bounds__(kStreamWarps * 32) k_stream_update(
    const GameDev* __restrict__ games, const Work* __restrict__ work, int n_work, int player_mask, int advance,
    int* iter, unsigned* done, const Discount* __restrict__ disc_tab, int variant, int depth, int prog_nodes,
    int prog_units, int half_units) {
  using V = typename P::V;
  extern __shared__ __align__(16) unsigned char sms[];
  __shared__ Discount disc;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int item = blockIdx.x;
  int p = player_mask == 2 ? 1 : 0;
  if (player_mask == 3 && item >= n_work) p = 1, item -= n_work;
  const Work wk = work[item];
  const GameDev& G = games[wk.game];
  const int unit = wk.unit + warp;
  const bool active = unit * 32 * HP < G.n_hands;
  if (threadIdx.x == 0) disc = disc_tab[*iter];
  // shared memory: the program, then per warp a prefetch ring (2 halves of half_units
  // units of 32 * HP 8-byte entries) and a stack (depth slots of HP values per lane)
  const size_t tables = (size_t)prog_nodes * sizeof(ProgOp) + (size_t)prog_units * 4;  // multiple of 16
  ProgOp* sprog = reinterpret_cast<ProgOp*>(sms);
  uint32_t* sunits = reinterpret_cast<uint32_t*>(sms + (size_t)prog_nodes * sizeof(ProgOp));
  uint64_t* ring = reinterpret_cast<uint64_t*>(sms + tables) + (size_t)warp * 2 * half_units * 32 * HP + lane;
  V* st = reinterpret_cast<V*>(sms + tables + (size_t)kStreamWarps * 2 * half_units * 32 * HP * 8) +
          (size_t)warp * depth * 32 * HP + lane;
  // this player's loads: the bottom-up pass's, then the top-down pass's
  const uint32_t* gunits_b = G.units + G.unit_off[p];
  const uint32_t* gunits_f = G.units + G.unit_off[2 + p];
  const int nb = G.unit_count[p], nf = G.unit_count[2 + p];
  if (prog_nodes > 0) {  // static: staged while the previous launch finishes
    const int4* src = reinterpret_cast<const int4*>(G.prog);
    int4* dst = reinterpret_cast<int4*>(sprog);
    for (int k = threadIdx.x; k < G.prog_len; k += blockDim.x) dst[k] = __ldg(src + k);
    for (int k = threadIdx.x; k < nb; k += blockDim.x) sunits[k] = __ldg(gunits_b + k);
    for (int k = threadIdx.x; k < nf; k += blockDim.x) sunits[nb + k] = __ldg(gunits_f + k);
  }
  pdl_wait();  // the terminal values come from the launch just before this one
  pdl_trigger();
  __syncthreads();  // disc, program
  if (active) {
    const int h = unit * 32 * HP + lane;  // hand k is h + 32 k < hstride (a multiple of 32 * HP)
    const size_t stride = (size_t)G.hstride;
    const size_t plane = (size_t)p * G.n_nodes * stride + h;
    const bool staged = prog_nodes > 0;
    StreamLane<P, HP> L{G, staged ? sprog : G.prog, staged ? sunits : gunits_b, p, {}, {}, stride,
                        G.R + h, G.S + h, G.M ? G.M + h : nullptr, static_cast<V*>(G.reach) + plane,
                        static_cast<V*>(G.cfv) + plane, ring, half_units, st};
#pragma unroll
    for (int k = 0; k < HP; ++k) {
      L.valid[k] = h + 32 * k < G.n_hands;
      L.hmask[k] = L.valid[k] ? G.hand_mask[h + 32 * k] : 0ull;
    }
    const Discount d = disc;
    int sp = 0;
    stream_pass<P, HP>(L, p, L.units, [&](int k0, int k1, int half) {
      stream_backward_chunk<P, HP>(L, k0, k1, half, sp, d, variant);
    });
#pragma unroll
    for (int k = 0; k < HP; ++k)
      if (L.valid[k]) L.cfv[32 * k] = st[k * 32];  // root value (read-back)
    __threadfence_block();  // the new R rows are read back by the warp's copies below
    __syncwarp();
#pragma unroll
    for (int k = 0; k < HP; ++k)
      st[k * 32] = L.valid[k] ? static_cast<const V*>(G.range_v)[(size_t)p * stride + h + 32 * k] : P::zero();
    sp = 1;
    stream_pass<P, HP>(L, 2 + p, staged ? sunits + nb : gunits_f,
                       [&](int k0, int k1, int half) { stream_forward_chunk<P, HP>(L, k0, k1, half, sp); });
  }

  if (advance) {
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      const unsigned prev = atomicAdd(done, 1u);
      if (prev == gridDim.x - 1) {  // last block of the launch: every block has read *iter
        *done = 0u;
        *iter += 1;
        __threadfence();
      }
    }
  }
}

// sigma = RM(R) at every decision node of every game (current strategy, for read-back when
// the update launches do not store it).
template <typename P>
__global__ void k_current_rows(const GameDev* __restrict__ games, int n_games) {
  using V = typename P::V;
  for (int g = 0; g < n_games; ++g) {
    const GameDev& G = games[g];
    const size_t stride = (size_t)G.hstride;
    const int total = G.n_nodes * G.n_hands;
    V* out = static_cast<V*>(G.sigma);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
      const int n = e / G.n_hands, h = e - n * G.n_hands;
      const NodeDev nd = G.nodes[n];
      if (nd.type != kDecision || nd.n_kids > kStreamMaxActions) continue;
      double Rv[kStreamMaxActions];
      V sg[kStreamMaxActions];
      load_rows(G.R + (size_t)nd.row * stride + h, stride, nd.n_kids, Rv);
      if (G.M) {  // Predictive CFR+: regret matching of R + M
        double Mv[kStreamMaxActions];
        load_rows(G.M + (size_t)nd.row * stride + h, stride, nd.n_kids, Mv);
#pragma unroll
        for (int a = 0; a < kStreamMaxActions; ++a) Rv[a] += Mv[a];
      }
      regret_match<P>(Rv, nd.n_kids, sg);
#pragma unroll
      for (int a = 0; a < kStreamMaxActions; ++a)
        if (a < nd.n_kids) out[(size_t)(nd.row + a) * stride + h] = sg[a];
    }
  }
}

// Average strategy S / sum S of every decision node of every game (for read-back).
template <typename P>
__global__ void k_average_rows(const GameDev* __restrict__ games, int n_games) {
  using V = typename P::V;
  for (int g = 0; g < n_games; ++g) {
    const GameDev& G = games[g];
    const size_t stride = (size_t)G.hstride;
    const int total = G.n_nodes * G.n_hands;
    V* out = static_cast<V*>(G.sigbar);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
      const int n = e / G.n_hands, h = e - n * G.n_hands;
      const NodeDev nd = G.nodes[n];
      if (nd.type != kDecision) continue;
      double tot = 0.0;
      for (int a = 0; a < nd.n_kids; ++a) tot += G.S[(size_t)(nd.row + a) * stride + h];
      for (int a = 0; a < nd.n_kids; ++a)
        out[(size_t)(nd.row + a) * stride + h] =
            P::of_double(tot > 0.0 ? G.S[(size_t)(nd.row + a) * stride + h] / tot : 1.0 / nd.n_kids);
    }
  }
}

// ------------------------------------------------------------------ wide schedule
//
// For one tree too large to stage in shared memory, each pass of the per-hand kernel becomes one
// launch per level over all of that level's (node, hand) pairs.  In the bottom-up step a block takes
// one node (or, when its hands are more than 512, an even share of them), two consecutive hands a
// thread: the node's description is one 16-byte load, branches are the block's, and rows are read and
// written 16 bytes a thread (FP64) or 8 (FP32 values); the row passes lay the nodes' hands end to end
// (wide_at).  The arithmetic per (node, hand) -- the order of every sum over children, regret matching,
// the Stage 7 update -- is the per-hand kernel's, so the schedules agree bit for bit.  Bound by DRAM
// where a level holds many nodes and by the launches' latency where it does not.  Measured, one
// player's update with FP32 values: exact turn 354 -> 211 us, learned flop 204 -> 135 us against one
// thread per (node, hand) that found its node by division and stored every node's reach; average pass
// of the turn (both players) 271 -> 142, best response 190 -> 98.  Three blocks of 80 registers per SM
// beat two without spills.

constexpr int kWideThreads = 256;  // at most (k_wide_back: LaunchCtx::wide_threads)
constexpr int kWideKids = 8;

template <typename P>
struct alignas(2 * sizeof(typename P::V)) V2 {  // two consecutive hands' values
  typename P::V v[2];
};

// The node of a list and the first of the two hands of this thread of the passes that only read and
// write rows: the nodes' `pairs` of hands laid end to end over the blocks.  (k_wide_back keeps a block
// to a node: its branches and action counts differ from node to node.)  Average pass of the 31,124-node
// flop of 12 hands 53 -> 20 us, of a 43,509-node turn of 200 hands 123 -> 92, against a block a node.
struct WideAt {
  int node, h;
};
__device__ __forceinline__ WideAt wide_at(int pairs) {
  // (below 2^32: a node and pair of hands takes more than 64 bytes of device memory)
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x, node = e / (unsigned)pairs;
  return {(int)node, 2 * (int)(e - node * (unsigned)pairs)};
}

// Two hands of a row; `both`: the second exists (it is not stored otherwise).
template <typename T2, typename T>
__device__ __forceinline__ T2 load2(const T* p) { return *reinterpret_cast<const T2*>(p); }
template <typename P>
__device__ __forceinline__ void store2(typename P::V* p, const V2<P>& x, bool both) {
  if (both) *reinterpret_cast<V2<P>*>(p) = x;
  else p[0] = x.v[0];
}
__device__ __forceinline__ void store2(double* p, double2 x, bool both) {
  if (both) *reinterpret_cast<double2*>(p) = x;
  else p[0] = x.x;
}

// The update at one of the player's decision nodes with NA actions, for two hands: the value under
// the current strategy, then Stage 7 and the new strategy RM(R') (Eq. rm).
template <typename P, int NA>
__device__ __forceinline__ V2<P> wide_decision(const typename P::V* __restrict__ c, typename P::V* __restrict__ sgp,
                                               const typename P::V* __restrict__ pip, double* __restrict__ Rp,
                                               double* __restrict__ Sp, double* __restrict__ Mp, size_t S,
                                               const Discount& d, int variant, bool both) {
  using V = typename P::V;
  if constexpr (NA > 3) {
    // more actions: their rows would not fit the registers, so each is read when its turn comes (the
    // children's values and the strategy twice, the second time from L1).  Update of a 1,581-node river
    // of 1,081 hands and up to 7 actions, FP32 values 69 -> 50 us, pairs 101 -> 80; exact turn 238 ->
    // 226 (every row loaded first, spilling, before)
    const bool plus = variant == 1 || variant == 3;
    typename P::Acc a0 = P::acc0(), a1 = P::acc0();
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      const V2<P> s = load2<V2<P>>(sgp + (size_t)a * S), x = load2<V2<P>>(c + (size_t)a * S);
      P::acc_mul(a0, s.v[0], x.v[0]);
      P::acc_mul(a1, s.v[1], x.v[1]);
    }
    V2<P> val;
    val.v[0] = P::value(a0), val.v[1] = P::value(a1);
    const V2<P> pi = load2<V2<P>>(pip);
    V2<P> y[NA];
    V tot[2] = {P::zero(), P::zero()};
    int npos[2] = {0, 0};
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      const V2<P> s = load2<V2<P>>(sgp + (size_t)a * S), x = load2<V2<P>>(c + (size_t)a * S);
      double2 R = load2<double2>(Rp + (size_t)a * S), Sv = load2<double2>(Sp + (size_t)a * S), rd;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const double r = P::to_double(P::sub(x.v[j], val.v[j]));
        const double contrib = P::to_double(P::mul(pi.v[j], s.v[j]));
        double z = (j ? R.y : R.x) + r;
        if (variant == 2) z *= __double_as_longlong(z) > 0 ? d.dpos : d.dneg;
        if (plus && __double_as_longlong(z) < 0) z = 0.0;
        (j ? Sv.y : Sv.x) = fma(j ? Sv.y : Sv.x, d.dS, plus ? d.wS * contrib : contrib);
        (j ? R.y : R.x) = z;
        (j ? rd.y : rd.x) = r;
        const double m = variant == 3 ? z + r : z;  // Predictive CFR+ matches R + M
        const V p = __double_as_longlong(m) > 0 ? P::of_double(m) : P::zero();
        y[a].v[j] = p;
        npos[j] += P::positive(p);
        tot[j] = P::add(tot[j], p);
      }
      store2(Rp + (size_t)a * S, R, both);
      store2(Sp + (size_t)a * S, Sv, both);
      if (variant == 3) store2(Mp + (size_t)a * S, rd, both);
    }
    const V inv[2] = {P::recip(tot[0]), P::recip(tot[1])}, uni = P::uniform(NA);
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      V2<P> o;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const V z = y[a].v[j], many = P::mul(z, inv[j]);
        o.v[j] = npos[j] > 1 ? many : npos[j] == 1 ? (P::positive(z) ? P::one() : P::zero()) : uni;
      }
      store2<P>(sgp + (size_t)a * S, o, both);
    }
    return val;
  }
  V2<P> cc[NA], sg[NA];
  double2 R[NA], Sv[NA];
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    cc[a] = load2<V2<P>>(c + (size_t)a * S);
    sg[a] = load2<V2<P>>(sgp + (size_t)a * S);
    R[a] = load2<double2>(Rp + (size_t)a * S);
    Sv[a] = load2<double2>(Sp + (size_t)a * S);
  }
  const V2<P> pi = load2<V2<P>>(pip);
  V2<P> val;
  const bool plus = variant == 1 || variant == 3;  // CFR+, Predictive CFR+
  double2 rd[NA];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    typename P::Acc acc = P::acc0();
#pragma unroll
    for (int a = 0; a < NA; ++a) P::acc_mul(acc, sg[a].v[j], cc[a].v[j]);
    val.v[j] = P::value(acc);
    double Rm[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      const double r = P::to_double(P::sub(cc[a].v[j], val.v[j]));                // instantaneous regret
      const double contrib = P::to_double(P::mul(pi.v[j], sg[a].v[j]));          // pi_i(I) sigma(I, a)
      double x = (j ? R[a].y : R[a].x) + r;
      if (variant == 2) x *= __double_as_longlong(x) > 0 ? d.dpos : d.dneg;
      if (plus && __double_as_longlong(x) < 0) x = 0.0;
      const double sn = fma(j ? Sv[a].y : Sv[a].x, d.dS, plus ? d.wS * contrib : contrib);
      (j ? R[a].y : R[a].x) = x;
      (j ? Sv[a].y : Sv[a].x) = sn;
      (j ? rd[a].y : rd[a].x) = r;
      Rm[a] = variant == 3 ? x + r : x;  // Predictive CFR+ matches R + M
    }
    V y[NA];
    regret_match_n<P, NA>(Rm, y);
#pragma unroll
    for (int a = 0; a < NA; ++a) sg[a].v[j] = y[a];
  }
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    store2(Rp + (size_t)a * S, R[a], both);
    store2(Sp + (size_t)a * S, Sv[a], both);
    if (variant == 3) store2(Mp + (size_t)a * S, rd[a], both);  // the prediction of the next regret
    store2<P>(sgp + (size_t)a * S, sg[a], both);
  }
  return val;
}

// Bottom-up step at the inner nodes of one level (Stage 6, Eq. backward) for player p =
// blockIdx.y when both players are in the launch.  kModeUpdate: at p's decision nodes also
// the regrets, the Stage 7 update of R and S and the new strategy RM(R') (Eq. rm);
// kModeBR: the best-response value max_a v(child a) at p's decision nodes.
template <int MODE, typename P>
__global__ void __launch_bounds__(kWideThreads, 3) k_wide_back(const GameDev* __restrict__ games,
                                                            const WideNode* __restrict__ inner, int segments,
                                                            int player_mask, const int* __restrict__ iter,
                                                            const Discount* __restrict__ disc_tab, int variant) {
  using V = typename P::V;
  const int p = player_mask == 3 ? (int)blockIdx.y : (player_mask == 1 ? 0 : 1);
  const WideNode w = inner[blockIdx.x / (unsigned)segments];
  const int h = 2 * ((int)(blockIdx.x % (unsigned)segments) * (int)blockDim.x + (int)threadIdx.x);
  pdl_wait();
  pdl_trigger();
  const GameDev& G = games[0];
  if (h >= G.n_hands) return;
  const bool both = h + 1 < G.n_hands;
  const size_t S = (size_t)G.hstride, N = (size_t)G.n_nodes;
  V* v = static_cast<V*>(MODE == kModeBR ? G.cfv_br : G.cfv) + (size_t)p * N * S + h;
  const int n = w.node(), A = w.kids(), kind = w.kind();
  const V* c = v + (size_t)w.first_kid * S;
  V2<P> val;
  if (kind == 2) {
    // children values already carry the card probabilities; cards in the hand are out
    const uint64_t m0 = G.hand_mask[h], m1 = both ? G.hand_mask[h + 1] : 0ull;
    typename P::Acc a0 = P::acc0(), a1 = P::acc0();
    // up to 49 children in one thread's sum: eight children's loads go out together (best response of the
    // 31,124-node flop of 33 hands with pairs 93 -> 67 us)
    for (int a = 0; a < A; a += kWideKids) {
      int deal[kWideKids];
      V2<P> x[kWideKids];
#pragma unroll
      for (int e = 0; e < kWideKids; ++e) {
        const int k = min(a + e, A - 1);
        deal[e] = G.nodes[w.first_kid + k].deal;
        x[e] = load2<V2<P>>(c + (size_t)k * S);
      }
#pragma unroll
      for (int e = 0; e < kWideKids; ++e) {
        if (a + e < A && !((m0 >> deal[e]) & 1ull)) P::acc(a0, x[e].v[0]);
        if (a + e < A && !((m1 >> deal[e]) & 1ull)) P::acc(a1, x[e].v[1]);
      }
    }
    val.v[0] = P::value(a0), val.v[1] = P::value(a1);
  } else if (kind != p) {
    typename P::Acc a0 = P::acc0(), a1 = P::acc0();
#pragma unroll 4
    for (int a = 0; a < A; ++a) {
      const V2<P> x = load2<V2<P>>(c + (size_t)a * S);
      P::acc(a0, x.v[0]);
      P::acc(a1, x.v[1]);
    }
    val.v[0] = P::value(a0), val.v[1] = P::value(a1);
  } else if (MODE == kModeBR) {
    val = load2<V2<P>>(c);
    for (int a = 1; a < A; ++a) {
      const V2<P> x = load2<V2<P>>(c + (size_t)a * S);
      val.v[0] = P::vmax(val.v[0], x.v[0]);
      val.v[1] = P::vmax(val.v[1], x.v[1]);
    }
  } else {
    const size_t at = (size_t)w.row * S + h;
    V* sg = static_cast<V*>(G.sigma) + at;
    const V* pi = static_cast<const V*>(G.reach) + ((size_t)p * N + w.src) * S + h;
    double* Mp = G.M ? G.M + at : nullptr;
    const Discount d = disc_tab[*iter];
    switch (A) {  // the block's, at most kStreamMaxActions
      case 1: val = wide_decision<P, 1>(c, sg, pi, G.R + at, G.S + at, Mp, S, d, variant, both); break;
      case 2: val = wide_decision<P, 2>(c, sg, pi, G.R + at, G.S + at, Mp, S, d, variant, both); break;
      case 3: val = wide_decision<P, 3>(c, sg, pi, G.R + at, G.S + at, Mp, S, d, variant, both); break;
      case 4: val = wide_decision<P, 4>(c, sg, pi, G.R + at, G.S + at, Mp, S, d, variant, both); break;
      case 5: val = wide_decision<P, 5>(c, sg, pi, G.R + at, G.S + at, Mp, S, d, variant, both); break;
      case 6: val = wide_decision<P, 6>(c, sg, pi, G.R + at, G.S + at, Mp, S, d, variant, both); break;
      case 7: val = wide_decision<P, 7>(c, sg, pi, G.R + at, G.S + at, Mp, S, d, variant, both); break;
      default: val = wide_decision<P, 8>(c, sg, pi, G.R + at, G.S + at, Mp, S, d, variant, both); break;
    }
  }
  store2<P>(v + (size_t)n * S, val, both);
}

// Strategy rows of player p = blockIdx.y: RM(R) (+ M for Predictive CFR+) into sigma (avg = 0), or the
// average S / sum S into sigbar (avg = 1), as the per-hand kernel computes them: positive parts in
// the value type, their sum in action order.
template <typename P>
__global__ void __launch_bounds__(kWideThreads) k_wide_rows(const GameDev* __restrict__ games, int pairs, int avg) {
  using V = typename P::V;
  pdl_wait();
  pdl_trigger();
  const GameDev& G = games[0];
  const WideAt at0 = wide_at(pairs);
  const int p = blockIdx.y, k = at0.node, h0 = at0.h;
  const int db = G.dec_begin[p], ndec = G.dec_begin[p + 1] - db;
  if (k >= ndec || h0 >= G.n_hands) return;
  const size_t S = (size_t)G.hstride;
  const NodeDev nd = G.nodes[G.dec_nodes[db + k]];
  for (int h = h0; h < min(h0 + 2, G.n_hands); ++h) {
    double x[kStreamMaxActions];
    load_rows((avg ? G.S : G.R) + (size_t)nd.row * S + h, S, nd.n_kids, x);
    if (!avg && G.M) {
      double m[kStreamMaxActions];
      load_rows(G.M + (size_t)nd.row * S + h, S, nd.n_kids, m);
#pragma unroll
      for (int a = 0; a < kStreamMaxActions; ++a) x[a] += m[a];
    }
    V sg[kStreamMaxActions];
    regret_match<P>(x, nd.n_kids, sg);
    V* out = static_cast<V*>(avg ? G.sigbar : G.sigma) + (size_t)nd.row * S + h;
#pragma unroll
    for (int a = 0; a < kStreamMaxActions; ++a)
      if (a < nd.n_kids) out[(size_t)a * S] = sg[a];
  }
}

// Top-down step (Stages 1-2) of player p = blockIdx.y (or the one of the launch) over the nodes that
// make new reach rows at one depth: its row is the one above it times p's probability of the
// action, or without the hands holding the dealt card.  The root takes p's range.
template <typename P>
__global__ void __launch_bounds__(kWideThreads) k_wide_fwd(const GameDev* __restrict__ games,
                                                           const WideReach* __restrict__ list0, int cnt0,
                                                           const WideReach* __restrict__ list1, int cnt1, int pairs,
                                                           int player_mask, int avg) {
  using V = typename P::V;
  const int p = player_mask == 3 ? (int)blockIdx.y : (player_mask == 1 ? 0 : 1);
  const WideAt at0 = wide_at(pairs);
  const int k = at0.node, h = at0.h;
  if (k >= (p ? cnt1 : cnt0)) return;  // (a launch's blocks may leave before its trigger)
  const WideReach w = (p ? list1 : list0)[k];
  pdl_wait();
  pdl_trigger();
  const GameDev& G = games[0];
  if (h >= G.n_hands) return;
  const bool both = h + 1 < G.n_hands;
  const size_t S = (size_t)G.hstride;
  V* rch = static_cast<V*>(avg ? G.reach_bar : G.reach) + (size_t)p * G.n_nodes * S + h;
  V2<P> x;
  if (w.src < 0) {
    x = load2<V2<P>>(static_cast<const V*>(G.range_v) + (size_t)p * S + h);
  } else {
    x = load2<V2<P>>(rch + (size_t)w.src * S);
    if (w.arow >= 0) {
      const V2<P> s = load2<V2<P>>(static_cast<const V*>(avg ? G.sigbar : G.sigma) + (size_t)w.arow * S + h);
      x.v[0] = P::mul(x.v[0], s.v[0]);
      x.v[1] = P::mul(x.v[1], s.v[1]);
    }
    if (w.deal >= 0) {
      if ((G.hand_mask[h] >> w.deal) & 1ull) x.v[0] = P::zero();
      if (both && ((G.hand_mask[h + 1] >> w.deal) & 1ull)) x.v[1] = P::zero();
    }
  }
  store2<P>(rch + (size_t)w.node * S, x, both);
}

// FP64 root sums of the best response, one block per player: sum_h r_p(h) v*_p(root, h),
// each thread over a fixed stride of hands, then a fixed-order tree in shared memory.
template <typename P>
__global__ void __launch_bounds__(kWideThreads) k_wide_root(const GameDev* __restrict__ games) {
  __shared__ double red[kWideThreads];
  pdl_wait();
  const GameDev& G = games[0];
  const int p = blockIdx.x;
  const size_t S = (size_t)G.hstride;
  using V = typename P::V;
  const V* v = static_cast<const V*>(G.cfv_br) + (size_t)p * G.n_nodes * S;
  double x = 0.0;
  for (int h = threadIdx.x; h < G.n_hands; h += kWideThreads) x += G.range64[(size_t)p * S + h] * P::to_double(v[h]);
  red[threadIdx.x] = x;
  __syncthreads();
  for (int o = kWideThreads / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) G.br_out[p] = red[0];
}

__global__ void k_wide_advance(int* iter) {
  pdl_wait();
  *iter += 1;
}

// ------------------------------------------------------------------ launchers

static int check_launch(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    fprintf(stderr, "pcfr: launch of %s failed: %s\n", what, cudaGetErrorString(e));
    return -1;
  }
  return 0;
}

int hand_kernel_smem_limit() { return 227 * 1024; }

size_t hand_smem_size(int n_nodes, int n_levels, int rows_max, int W, size_t es) {
  return hand_smem_bytes(n_nodes, n_levels, rows_max, W, es);
}

bool scans_in_eights(int n_hands, int hand_size, size_t es) {
  const int gp = es == 4 ? TermRun<Single>::gp : TermRun<Pairs>::gp, gc = kTermThreads - gp;
  return (n_hands + gp - 1) / gp % 8 == 0 || (hand_size * n_hands + gc - 1) / gc % 8 == 0;
}

size_t terminal_smem_size(int n_hands, int hand_size, int deck, int hstride, size_t es, int nv, bool runs) {
  const TermTab tt(n_hands, hand_size, deck);
  const size_t scan = (size_t)(hand_size * n_hands + 1 + n_hands + 1);
  if (runs)
    return (size_t)tt.len * 2 + 2 * (size_t)hstride * es +
           (size_t)(TermTab::round8(hand_size * n_hands + 1) + TermTab::round8(n_hands + 1)) * es;
  if (nv == 1) return (size_t)tt.len * 2 + (size_t)hstride * es + scan * es;
  return kTermSegment * sizeof(TermGroup) + (size_t)tt.fold_len * 2 + 2 * (size_t)nv * hstride * es + scan * nv * es;
}

size_t tile_smem_size(int tab16, int n_nodes, int rows_max, int W, size_t es, int staged) {
  const size_t slack = staged ? (size_t)kTileSlack * W * es : 0;
  return tile_smem_bytes(tab16, n_nodes, rows_max, W, es) + (staged ? (size_t)2 * rows_max * W * 8 : 0) + slack;
}

size_t resident_term_size(int n_hands, int hand_size, int deck, int hstride, size_t es) {
  return round16(resident_term_bytes(n_hands, hand_size, deck, hstride, es));
}
size_t resident_hand_size(int tab16, int n_nodes, int rows_max, int W, size_t es) {
  return resident_hand_bytes(tab16, n_nodes, rows_max, W, es);
}
int resident_blocks_per_sm(int precision, size_t smem) {
  int n = 0, m = 0;
  cudaError_t e;
  if (precision == kPrecisionSingle) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_resident<Single, false>, kTermThreads, smem);
  } else {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_resident<Pairs, false>, kTermThreads, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, k_resident<Pairs, true>, kTermThreads, smem);
    n = n < m ? n : m;
  }
  return e == cudaSuccess ? n : 0;
}

// Every kernel asks for the same shared-memory carveout (the maximum), so the SMs never
// have to be reconfigured between the terminal and per-hand launches of an iteration.
template <typename K>
static cudaError_t configure_one(K kernel, int smem) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  return e;
}

template <typename P, bool SM>
static cudaError_t configure_hand() {
  const int smem = hand_kernel_smem_limit() - 4096;
  cudaError_t e = configure_one(k_hand<kModeInit, P, SM>, smem);
  if (e == cudaSuccess) e = configure_one(k_hand<kModeUpdate, P, SM>, smem);
  if (e == cudaSuccess) e = configure_one(k_hand<kModeAvg, P, SM>, smem);
  if (e == cudaSuccess) e = configure_one(k_hand<kModeBR, P, SM>, smem);
  return e;
}

template <typename P>
static cudaError_t configure_precision() {
  cudaError_t e = configure_hand<P, true>();
  if (e == cudaSuccess) e = configure_hand<P, false>();
  if (e == cudaSuccess) e = configure_one(k_terminal<P>, 200 * 1024);
  if (e == cudaSuccess) e = configure_one(k_terminal_run<P, false>, 200 * 1024);
  if (e == cudaSuccess) e = configure_one(k_terminal_run<P, true>, 200 * 1024);
  if (e == cudaSuccess) e = configure_one(k_average_rows<P>, 0);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeInit, P, false, false>, kTileSmem);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeUpdate, P, false, false>, kTileSmem);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeUpdate, P, true, false>, kTileSmem);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeAvg, P, false, false>, kTileSmem);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeBR, P, false, false>, kTileSmem);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeInit, P, false, true>, kTileSmemStaged);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeUpdate, P, false, true>, kTileSmemStaged);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeAvg, P, false, true>, kTileSmemStaged);
  if (e == cudaSuccess) e = configure_one(k_tile<kModeBR, P, false, true>, kTileSmemStaged);
  if (e == cudaSuccess) e = configure_one(k_stream_update<P, 1>, 200 * 1024);
  if (e == cudaSuccess) e = configure_one(k_stream_update<P, 2>, 200 * 1024);
  if (e == cudaSuccess) e = configure_one(k_current_rows<P>, 0);
  if (e == cudaSuccess) e = configure_one(k_resident<P, false>, 200 * 1024);
  if (e == cudaSuccess && std::is_same<P, Pairs>::value) e = configure_one(k_resident<Pairs, true>, 200 * 1024);
  return e;
}

int set_first_wait_polls(long polls) {
  const long v = polls < 0 ? kWaitLimit : polls;
  return cudaMemcpyToSymbol(g_first_wait_polls, &v, sizeof(v)) == cudaSuccess ? 0 : -1;
}

int configure_kernels() {
  cudaError_t e = configure_precision<Pairs>();
  if (e == cudaSuccess) e = configure_precision<Single>();
  if (e == cudaSuccess) e = configure_one(k_terminal_vec<2>, 200 * 1024);
  if (e == cudaSuccess) e = configure_one(k_terminal_vec<4>, 200 * 1024);
  if (e != cudaSuccess) {
    fprintf(stderr, "pcfr: kernel attribute setup failed: %s\n", cudaGetErrorString(e));
    return -1;
  }
  return 0;
}

// Launch with programmatic stream serialisation (c.pdl) so the kernel may start while its
// predecessor finishes; kernels order their reads with pdl_wait().
template <typename... KArgs, typename... Args>
static cudaError_t launch_kernel(void (*kernel)(KArgs...), int grid, int block, size_t smem, void* stream, bool pdl,
                                 Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = pdl ? attr : nullptr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <int MODE, typename P>
static int launch_hand_p(const LaunchCtx& c, int player_mask, int advance, void* stream, bool pdl) {
  const int players = player_mask == 3 ? 2 : 1;
  const int grid = c.n_chunk_work * players;
  cudaError_t e;
  if (c.smem_hand > 0)
    e = launch_kernel(k_hand<MODE, P, true>, grid, kHandThreads, c.smem_hand, stream, pdl, c.games, c.chunk_work,
                      c.n_chunk_work, player_mask, advance, c.iter, c.done, c.disc, c.variant);
  else
    e = launch_kernel(k_hand<MODE, P, false>, grid, kHandThreads, 0, stream, pdl, c.games, c.chunk_work,
                      c.n_chunk_work, player_mask, advance, c.iter, c.done, c.disc, c.variant);
  if (e != cudaSuccess) {
    fprintf(stderr, "pcfr: launch of k_hand failed: %s\n", cudaGetErrorString(e));
    return -1;
  }
  return check_launch("k_hand");
}

template <int MODE>
static int launch_hand(const LaunchCtx& c, int player_mask, int advance, void* stream, bool pdl) {
  return c.precision == kPrecisionSingle ? launch_hand_p<MODE, Single>(c, player_mask, advance, stream, pdl)
                                         : launch_hand_p<MODE, Pairs>(c, player_mask, advance, stream, pdl);
}

// ---- wide schedule: a pass is a sequence of per-level launches (host loop over levels)

template <typename... KArgs, typename... Args>
static cudaError_t launch_wide(void (*kernel)(KArgs...), unsigned blocks, int players, int threads, void* stream, bool pdl,
                               Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks, (unsigned)players);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = pdl ? attr : nullptr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Blocks of the row passes over cnt nodes (wide_at).
static unsigned wide_blocks(const LaunchCtx& c, int cnt) {
  return (unsigned)(((size_t)cnt * c.wide_pairs + kWideThreads - 1) / kWideThreads);
}

template <int MODE, typename P>
static cudaError_t wide_backward(const LaunchCtx& c, int player_mask, void* stream) {
  const int players = player_mask == 3 ? 2 : 1;
  for (int l = c.wide_levels - 1; l >= 0; --l) {
    const int cnt = c.wide_inner_off[l + 1] - c.wide_inner_off[l];
    if (cnt == 0) continue;
    const cudaError_t e =
        launch_wide(k_wide_back<MODE, P>, (unsigned)cnt * c.wide_segments, players, c.wide_threads, stream, c.pdl != 0,
                    c.games, c.wide_inner + c.wide_inner_off[l], c.wide_segments, player_mask, c.iter, c.disc, c.variant);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The nodes of depth d of the players in the mask that make new reach rows.
static int wide_fwd_count(const LaunchCtx& c, int p, int d) {
  return d < c.wide_fwd_levels[p] ? c.wide_fwd_off[p][d + 1] - c.wide_fwd_off[p][d] : 0;
}

template <typename P>
static cudaError_t wide_forward(const LaunchCtx& c, int player_mask, int avg, int first_level, void* stream) {
  const int players = player_mask == 3 ? 2 : 1;
  for (int d = first_level; d < c.wide_fwd_levels[0] || d < c.wide_fwd_levels[1]; ++d) {
    const int c0 = player_mask & 1 ? wide_fwd_count(c, 0, d) : 0, c1 = player_mask & 2 ? wide_fwd_count(c, 1, d) : 0;
    const int cnt = c0 > c1 ? c0 : c1;
    if (cnt == 0) continue;
    const cudaError_t e = launch_wide(k_wide_fwd<P>, wide_blocks(c, cnt), players, kWideThreads, stream,
                                      c.pdl != 0, c.games, c.wide_fwd[0] + (c0 ? c.wide_fwd_off[0][d] : 0), c0,
                                      c.wide_fwd[1] + (c1 ? c.wide_fwd_off[1][d] : 0), c1, c.wide_pairs, player_mask, avg);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename P>
static cudaError_t wide_rows(const LaunchCtx& c, int avg, void* stream) {
  // rows of both players: the larger player's decision-node count sizes the grid
  return launch_wide(k_wide_rows<P>, wide_blocks(c, c.wide_max_dec), 2, kWideThreads, stream, c.pdl != 0, c.games,
                     c.wide_pairs, avg);
}

template <typename P>
static int wide_pass(const LaunchCtx& c, int which, int player_mask, int advance, void* stream) {
  cudaError_t e = cudaSuccess;
  if (which == kModeUpdate) {
    e = wide_backward<kModeUpdate, P>(c, player_mask, stream);
    if (e == cudaSuccess) e = wide_forward<P>(c, player_mask, 0, 1, stream);
    if (e == cudaSuccess && advance) e = launch_wide(k_wide_advance, 1, 1, 1, stream, c.pdl != 0, c.iter);
  } else if (which == kModeInit || which == kModeAvg) {
    const int avg = which == kModeAvg;
    e = wide_rows<P>(c, avg, stream);
    if (e == cudaSuccess) e = wide_forward<P>(c, 3, avg, 0, stream);
  } else {  // kModeBR
    e = wide_backward<kModeBR, P>(c, 3, stream);
    if (e == cudaSuccess) e = launch_wide(k_wide_root<P>, 2, 1, kWideThreads, stream, c.pdl != 0, c.games);
  }
  if (e != cudaSuccess) {
    fprintf(stderr, "pcfr: launch of a wide-schedule kernel failed: %s\n", cudaGetErrorString(e));
    return -1;
  }
  return check_launch("wide schedule");
}

static int launch_wide_pass(const LaunchCtx& c, int which, int player_mask, int advance, void* stream) {
  return c.precision == kPrecisionSingle ? wide_pass<Single>(c, which, player_mask, advance, stream)
                                         : wide_pass<Pairs>(c, which, player_mask, advance, stream);
}

int wide_launch_count(const LaunchCtx& c, int which, int player_mask, int advance) {
  int back = 0, fwd = 0;
  for (int l = 0; l < c.wide_levels; ++l) back += c.wide_inner_off[l + 1] > c.wide_inner_off[l];
  for (int d = which == kModeUpdate; d < c.wide_fwd_levels[0] || d < c.wide_fwd_levels[1]; ++d)
    fwd += (player_mask & 1 && wide_fwd_count(c, 0, d)) || (player_mask & 2 && wide_fwd_count(c, 1, d));
  if (which == kModeUpdate) return back + fwd + (advance ? 1 : 0);
  if (which == kModeInit || which == kModeAvg) return 1 + fwd;
  return back + 1;
}

template <int MODE, typename P>
static cudaError_t launch_tile_p(const LaunchCtx& c, int player_mask, int advance, void* stream, bool pdl) {
  auto go = [&](auto kernel) {
    return launch_kernel(kernel, c.n_tile_work * (player_mask == 3 ? 2 : 1), c.tile_threads, c.smem_tile, stream, pdl,
                         c.games, c.tile_work, c.n_tile_work, player_mask, advance, c.iter, c.done, c.disc, c.variant);
  };
  constexpr bool upd = MODE == kModeUpdate;  // the other passes do not depend on the variant
  if (c.tile_staged) return go(k_tile<MODE, P, false, true>);
  return upd && c.variant == 2 ? go(k_tile<MODE, P, upd, false>) : go(k_tile<MODE, P, false, false>);
}

template <int MODE>
static int launch_tile(const LaunchCtx& c, int player_mask, int advance, void* stream, bool pdl) {
  const cudaError_t e = c.precision == kPrecisionSingle ? launch_tile_p<MODE, Single>(c, player_mask, advance, stream, pdl)
                                                        : launch_tile_p<MODE, Pairs>(c, player_mask, advance, stream, pdl);
  if (e != cudaSuccess) {
    fprintf(stderr, "pcfr: launch of k_tile failed: %s\n", cudaGetErrorString(e));
    return -1;
  }
  return check_launch("k_tile");
}

int launch_init(const LaunchCtx& c, void* stream) {
  if (c.n_tile_work > 0) return launch_tile<kModeInit>(c, 3, 0, stream, false);
  if (c.schedule == kScheduleWide) return launch_wide_pass(c, kModeInit, 3, 0, stream);
  return launch_hand<kModeInit>(c, 3, 0, stream, false);
}
template <typename P, int HP>
static int launch_stream_p(const LaunchCtx& c, int player_mask, int advance, void* stream) {
  const int players = player_mask == 3 ? 2 : 1;
  const int grid = c.n_warp_work * players;
  const size_t smem =
      stream_smem_size(c.stream_prog, c.stream_units, c.stream_half, c.stream_depth, sizeof(typename P::V), HP);
  const cudaError_t e = launch_kernel(k_stream_update<P, HP>, grid, kStreamWarps * 32, smem, stream, c.pdl != 0,
                                      c.games, c.warp_work, c.n_warp_work, player_mask, advance, c.iter, c.done,
                                      c.disc, c.variant, c.stream_depth, c.stream_prog, c.stream_units,
                                      c.stream_half);
  if (e != cudaSuccess) {
    fprintf(stderr, "pcfr: launch of k_stream_update failed: %s\n", cudaGetErrorString(e));
    return -1;
  }
  return check_launch("k_stream_update");
}

int launch_update(const LaunchCtx& c, int player_mask, int advance, void* stream) {
  if (c.n_tile_work == 0 && c.schedule == kScheduleWide) return launch_wide_pass(c, kModeUpdate, player_mask, advance, stream);
  if (c.n_tile_work > 0) return launch_tile<kModeUpdate>(c, player_mask, advance, stream, c.pdl != 0);
  if (c.schedule == kScheduleStream)
    return c.precision == kPrecisionSingle
               ? (c.stream_hp == 2 ? launch_stream_p<Single, 2>(c, player_mask, advance, stream)
                                   : launch_stream_p<Single, 1>(c, player_mask, advance, stream))
               : (c.stream_hp == 2 ? launch_stream_p<Pairs, 2>(c, player_mask, advance, stream)
                                   : launch_stream_p<Pairs, 1>(c, player_mask, advance, stream));
  return launch_hand<kModeUpdate>(c, player_mask, advance, stream, c.pdl != 0);
}

int launch_current_rows(const LaunchCtx& c, void* stream) {
  if (c.precision == kPrecisionSingle)
    k_current_rows<Single><<<152, 256, 0, (cudaStream_t)stream>>>(c.games, c.n_games);
  else
    k_current_rows<Pairs><<<152, 256, 0, (cudaStream_t)stream>>>(c.games, c.n_games);
  return check_launch("k_current_rows");
}
int launch_avg_reach(const LaunchCtx& c, void* stream) {
  if (c.n_tile_work > 0) return launch_tile<kModeAvg>(c, 3, 0, stream, false);
  if (c.schedule == kScheduleWide) return launch_wide_pass(c, kModeAvg, 3, 0, stream);
  return launch_hand<kModeAvg>(c, 3, 0, stream, false);
}
int launch_br(const LaunchCtx& c, void* stream) {
  if (c.n_tile_work > 0) return launch_tile<kModeBR>(c, 3, 0, stream, c.pdl != 0);
  if (c.schedule == kScheduleWide) return launch_wide_pass(c, kModeBR, 3, 0, stream);
  return launch_hand<kModeBR>(c, 3, 0, stream, c.pdl != 0);
}

int launch_terminal(const LaunchCtx& c, int player_mask, int use_bar, void* stream) {
  if (c.n_term_work == 0) return 0;
  const int players = player_mask == 3 ? 2 : 1;
  const bool pdl = c.pdl != 0;
  auto one = [&](auto kernel) {
    return launch_kernel(kernel, c.n_term_work * players, kTermThreads, c.smem_term, stream, pdl, c.games, c.term_work,
                         c.term_src, c.n_term_work, player_mask, use_bar, c.err);
  };
  auto vec = [&](auto kernel) {
    return launch_kernel(kernel, c.n_term_segments * players, kTermThreads, c.smem_term, stream, pdl, c.games,
                         c.term_groups, c.term_segments, c.n_term_segments, player_mask, use_bar, c.err);
  };
  auto run = [&](auto kernel) {
    return launch_kernel(kernel, c.n_term_runs * players, kTermThreads, c.smem_term, stream, pdl, c.games, c.term_work,
                         c.term_src, c.term_runs, c.n_term_runs, player_mask, use_bar, c.err);
  };
  const bool single = c.precision == kPrecisionSingle;
  cudaError_t e;
  if (c.n_term_runs > 0)
    e = c.term_swap ? (single ? run(k_terminal_run<Single, true>) : run(k_terminal_run<Pairs, true>))
                    : (single ? run(k_terminal_run<Single, false>) : run(k_terminal_run<Pairs, false>));
  else if (c.term_nv > 1)
    e = c.term_nv == 4 ? vec(k_terminal_vec<4>) : vec(k_terminal_vec<2>);
  else
    e = single ? one(k_terminal<Single>) : one(k_terminal<Pairs>);
  if (e != cudaSuccess) {
    fprintf(stderr, "pcfr: launch of k_terminal failed: %s\n", cudaGetErrorString(e));
    return -1;
  }
  return check_launch("k_terminal");
}

// One cooperative launch: every block is resident at once, which the grid barriers need
// (the launch fails rather than run a grid that does not fit).
template <typename P, bool AHEAD>
static cudaError_t launch_resident_p(const LaunchCtx& c, int n_iters, void* stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c.resident_grid);
  cfg.blockDim = dim3(kTermThreads);
  cfg.dynamicSmemBytes = c.smem_resident;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_resident<P, AHEAD>, c.games, c.chunk_work, c.n_chunk_work, c.term_work,
                            c.term_src, c.n_term_work, c.alternating, n_iters, c.iter,
                            c.disc, c.variant, c.resident_sync, c.err, c.resident_term);
}

int launch_resident(const LaunchCtx& c, int n_iters, void* stream) {
  const cudaError_t e = c.precision == kPrecisionSingle ? launch_resident_p<Single, false>(c, n_iters, stream)
                        : c.resident_ahead              ? launch_resident_p<Pairs, true>(c, n_iters, stream)
                                                        : launch_resident_p<Pairs, false>(c, n_iters, stream);
  if (e != cudaSuccess) {
    fprintf(stderr, "pcfr: launch of k_resident failed: %s\n", cudaGetErrorString(e));
    return -1;
  }
  return check_launch("k_resident");
}

int launch_average_rows(const LaunchCtx& c, void* stream) {
  if (c.precision == kPrecisionSingle)
    k_average_rows<Single><<<152, 256, 0, (cudaStream_t)stream>>>(c.games, c.n_games);
  else
    k_average_rows<Pairs><<<152, 256, 0, (cudaStream_t)stream>>>(c.games, c.n_games);
  return check_launch("k_average_rows");
}

}  // namespace pcfr
