// k_tree.cu -- the priority sum-tree of prioritized replay (Schaul et al.,
// ICLR'16; the replay-state callback of Appendix C, Invariant 2):
// refresh of ancestor sums, stratified inverse-CDF sampling by descent, and
// the priority update with last-occurrence-wins duplicate handling.
//
// Layout: a 32-ary tree in fixed point.  Leaves are the uint32 priorities of
// the ring slots (physical order, zero-padded to 32^D); level d < D holds
// 32^d uint64 sums, node n of level d covering leaves [n*32^(D-d),
// (n+1)*32^(D-d)).  Integer sums make every result independent of the order
// in which threads add, so sums, targets and indices are bit-exact.
//
// A level is one load of a node's 32 children (whole cache lines: 256 bytes of
// sums, 128 of leaves), a shuffle prefix sum and a ballot -- D dependent loads
// per descent instead of the 5*D of a binary tree.  A refresh gives a node a
// warp; a descent gives it eight lanes, four children each.
#include "edp_internal.cuh"

namespace edp {
namespace {

// Internal levels are stored back to back from the root: level d starts at
// node (32^d - 1) / 31.
struct TreeView {
  uint64_t *nodes;
  uint32_t *leaves;
  uint32_t depth;
  __device__ __forceinline__ uint64_t *lvl(uint32_t d) const {
    return nodes + (((1ull << (5 * d)) - 1) / 31);
  }
};

TreeView view(edp_ctx *c) {
  TreeView t{};
  t.nodes = c->level[0];
  t.leaves = c->leaves;
  t.depth = c->depth;
  return t;
}

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Recompute nodes [a0, a0+n0) and [a1, a1+n1) of level d from level d+1.
__global__ void k_tree_level(uint64_t *out, const uint64_t *child64, const uint32_t *child32,
                             uint64_t a0, uint64_t n0, uint64_t a1, uint64_t n1) {
  pdl_wait();
  pdl_launch();
  const uint64_t w = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n0 + n1) return;
  const uint64_t node = w < n0 ? a0 + w : a1 + (w - n0);
  const uint64_t c = node * kFanout + lane;
  uint64_t v = child64 ? child64[c] : (uint64_t)child32[c];
  v = warp_sum_u64(v);
  if (lane == 0) out[node] = v;
}

// Stratified proportional sampling: eight lanes per stratum k, so a warp
// descends for four at a time.  The CTA first copies the top of the tree
// (levels 1 and 2: 32 + 1024 sums, 8.2 KiB) into shared memory, so a descent of
// a 1M-leaf tree makes two dependent global loads (level 3, then the leaf row)
// instead of four, and the sampled priority is the child that the last level
// loaded.  Bound by those round trips (small batches) or by issue (a stratum
// costs a quarter of what a warp of its own does).  Calls in a row, 1,000,000
// leaves, in us, and (before) with a warp per stratum: 512 strata 3.1 (3.3),
// 4,096 3.1 (5.5), 32,768 8.8 (25.4).  The delivery behind it, a grid of many
// waves, is released at once: a round of 512 stacks of 84x84 frames 31.4 us,
// 33.8 released at the end.
constexpr int kSmemLevels = 2;
constexpr int kSmemNodes = 32 + 1024;
constexpr int kGroup = 8;                  // lanes per descent
constexpr int kChildren = kFanout / kGroup;  // of a lane
constexpr int kSampleThreads = 256;
constexpr int kSamplePerCta = kSampleThreads / kGroup;

__device__ __forceinline__ ulonglong2 ld_keep2(const uint64_t *p, uint64_t pol) {
  ulonglong2 v;
  asm volatile("ld.global.L2::cache_hint.v2.u64 {%0, %1}, [%2], %3;"
               : "=l"(v.x), "=l"(v.y) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ uint4 ld_keep4(const uint32_t *p, uint64_t pol) {
  uint4 v;
  asm volatile("ld.global.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol));
  return v;
}

// Copies levels 1 .. cached of the tree into top (all loads issued before
// any use); returns the number of cached levels.
__device__ __forceinline__ uint32_t cache_top(const TreeView &t, uint64_t *top,
                                              uint64_t keep) {
  const uint32_t cached = t.depth - 1 < (uint32_t)kSmemLevels ? t.depth - 1 : kSmemLevels;
  const uint32_t pairs = (cached == 0 ? 0 : (cached == 1 ? 32 : 32 + 1024)) / 2;
  constexpr int kEach = (kSmemNodes / 2 + kSampleThreads - 1) / kSampleThreads;
  ulonglong2 v[kEach];
#pragma unroll
  for (int u = 0; u < kEach; ++u) {
    const uint32_t i = threadIdx.x + u * kSampleThreads;
    if (i < pairs) v[u] = ld_keep2(t.nodes + 1 + 2 * i, keep);
  }
#pragma unroll
  for (int u = 0; u < kEach; ++u) {
    const uint32_t i = threadIdx.x + u * kSampleThreads;
    if (i < pairs) reinterpret_cast<ulonglong2 *>(top)[i] = v[u];
  }
  return cached;
}

// Descent of one target by a group of kGroup lanes (all lanes of the warp call
// it, each group with its own target): the leaf whose prefix range
// [prefix(i), prefix(i) + q_i) holds `target`, for target < S, and its
// priority *q.  Per level each lane sums four of the 32 children, a prefix sum
// over the group places them, and a ballot names the lane that holds the
// target.  *ok is cleared if the sums disagree with the children (the leaf
// then stays in range).
__device__ __forceinline__ uint64_t descend(const TreeView &t, const uint64_t *top,
                                            uint32_t cached, uint64_t target, int lane,
                                            uint64_t keep, bool *ok, uint32_t *q) {
  const int sub = lane % kGroup, base = lane - sub;
  uint64_t node = 0;
  for (uint32_t d = 1; d <= t.depth; ++d) {
    const uint64_t c = node * kFanout + sub * kChildren;
    uint64_t v[kChildren];
    if (d <= cached) {
      const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(top + (d == 1 ? 0 : 32) + c);
      const ulonglong2 x = p[0], y = p[1];
      v[0] = x.x, v[1] = x.y, v[2] = y.x, v[3] = y.y;
    } else if (d < t.depth) {
      const ulonglong2 x = ld_keep2(t.lvl(d) + c, keep), y = ld_keep2(t.lvl(d) + c + 2, keep);
      v[0] = x.x, v[1] = x.y, v[2] = y.x, v[3] = y.y;
    } else {
      const uint4 x = ld_keep4(t.leaves + c, keep);
      v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
    }
    const uint64_t sum = v[0] + v[1] + v[2] + v[3];
    uint64_t incl = sum;
#pragma unroll
    for (int o = 1; o < kGroup; o <<= 1) {
      const uint64_t y = __shfl_up_sync(kFull, incl, o, kGroup);
      if (sub >= o) incl += y;
    }
    uint32_t m = (__ballot_sync(kFull, target < incl) >> base) & ((1u << kGroup) - 1);
    if (m == 0) {  // sums disagree with children: report, stay in range
      *ok = false;
      m = 1u << (kGroup - 1);
    }
    // in the lane that holds it: the last child that starts at or below the
    // target (the first one when none does)
    uint64_t excl = incl - sum, child = v[0];
    uint32_t f = 0;
#pragma unroll
    for (int j = 1; j < kChildren; ++j) {
      if (target >= excl + child) {
        excl += child;
        child = v[j];
        f = j;
      }
    }
    const int from = base + __ffs(m) - 1;
    excl = __shfl_sync(kFull, excl, from);
    f = __shfl_sync(kFull, f, from) + (from - base) * kChildren;
    if (d == t.depth) *q = (uint32_t)__shfl_sync(kFull, (uint32_t)child, from);
    target = target >= excl ? target - excl : 0;
    node = node * kFanout + f;
  }
  return node;
}

// floor(x / B) with inv = floor((2^64 - 1) / B): the high product is at most
// two below the quotient.
__device__ __forceinline__ uint64_t div_by(uint64_t x, uint32_t B, uint64_t inv) {
  uint64_t q = __umul64hi(x, inv);
  uint64_t r = x - q * B;
  if (r >= B) r -= B, ++q;
  if (r >= B) ++q;
  return q;
}

__global__ void __launch_bounds__(kSampleThreads)
k_sample_prio(TreeView t, uint32_t B, uint64_t inv_b, uint64_t seed, uint64_t round,
              int64_t *idx, uint32_t *qout, Ctrl *ctrl) {
  __shared__ __align__(16) uint64_t top[kSmemNodes];
  const int lane = threadIdx.x & 31;
  const uint64_t keep = policy_keep();
  // Philox and nothing else before the wait
  uint64_t k = (uint64_t)blockIdx.x * kSamplePerCta + threadIdx.x / kGroup;
  uint64_t u = philox_u64(seed, (uint32_t)k, round, 1);
  pdl_wait();
  pdl_launch();
  const uint64_t S = t.nodes[0];  // issued beside the loads of the top levels
  const uint32_t cached = cache_top(t, top, keep);
  __syncthreads();
  const uint64_t a = div_by(S, B, inv_b), b = S - a * B;
  // a warp's groups stay together: the loop ends for all of them at once
  for (uint64_t k0 = k - lane / kGroup; k0 < B; k0 += (uint64_t)gridDim.x * kSamplePerCta) {
    const bool mine = k < B;
    // stratum_target() with the divisions by B as products
    const uint64_t lo = a * k + div_by(b * k, B, inv_b);
    const uint64_t hi = a * (k + 1) + div_by(b * (k + 1), B, inv_b);
    const uint64_t target = lo + mulhi64(u, hi - lo);
    bool ok = true;
    uint32_t q = 0;
    const uint64_t node = descend(t, top, cached, target, lane, keep, &ok, &q);
    if (mine && lane % kGroup == 0) {
      if (S == 0) flag(ctrl, DEVERR_EMPTY, k);
      else if (!ok) flag(ctrl, DEVERR_TREE, k);
      idx[k] = S == 0 ? -1 : (int64_t)node;
      if (qout) qout[k] = S == 0 ? 0 : q;
    }
    k += (uint64_t)gridDim.x * kSamplePerCta;
    u = philox_u64(seed, (uint32_t)k, round, 1);
  }
}

// Descent of given targets (the shard side of a sharded buffer: targets
// routed here by edp_route_prioritized, each below this tree's total):
// eight lanes per target.  A target >= S is reported (DEVERR_INDEX) and
// gives idx -1, q 0.
__global__ void __launch_bounds__(kSampleThreads)
k_sample_targets(TreeView t, const uint64_t *targets, uint32_t n, int64_t *idx, uint32_t *qout,
                 Ctrl *ctrl) {
  __shared__ __align__(16) uint64_t top[kSmemNodes];
  const int lane = threadIdx.x & 31;
  const uint64_t keep = policy_keep();
  pdl_wait();
  pdl_launch();
  const uint64_t S = t.nodes[0];  // issued beside the loads of the top levels
  const uint64_t first =
      (uint64_t)blockIdx.x * kSamplePerCta + threadIdx.x / 32 * (32 / kGroup);
  uint64_t target = first + lane / kGroup < n ? targets[first + lane / kGroup] : 0;  // likewise
  const uint32_t cached = cache_top(t, top, keep);
  __syncthreads();
  for (uint64_t k0 = first; k0 < n; k0 += (uint64_t)gridDim.x * kSamplePerCta) {
    const uint64_t k = k0 + lane / kGroup;
    const bool mine = k < n;
    if (k0 != first) target = mine ? targets[k] : 0;
    const bool in = target < S;
    bool ok = true;
    uint32_t q = 0;
    const uint64_t node = descend(t, top, cached, in ? target : 0, lane, keep, &ok, &q);
    if (mine && lane % kGroup == 0) {
      if (!in) flag(ctrl, DEVERR_INDEX, target);
      else if (!ok) flag(ctrl, DEVERR_TREE, k);
      idx[k] = in ? (int64_t)node : -1;
      if (qout) qout[k] = in ? q : 0;
    }
  }
}

// PER priority from a TD error: clamp(rn((|td| + eps)^alpha * 2^20), 1,
// 2^32 - 1) (the rule is defined in fp64).  The exponent, eps and the
// constants of the fast path travel as double-float splits made on the host.
struct PrioRule {
  double alpha, eps;
  float a_hi, a_lo, e_hi, e_lo;
  int fast;  // alpha in (0, 1], eps in [0, 2^90]: the double-float path applies
};

PrioRule prio_rule(double alpha, double eps) {
  PrioRule r{};
  r.alpha = alpha;
  r.eps = eps;
  r.a_hi = (float)alpha;
  r.a_lo = (float)(alpha - (double)r.a_hi);
  r.e_hi = (float)eps;
  r.e_lo = (float)(eps - (double)r.e_hi);
  r.fast = alpha > 0.0 && alpha <= 1.0 && eps >= 0.0 && eps <= 0x1p90;
  return r;
}

// x^a * 2^20 for x in [2^-100, 2^100] and a in (0, 1], rounded to the nearest
// integer and clamped, in double-float arithmetic.  An fp64 instruction
// occupies this GPU's fp64 pipe for about 64 cycles whatever the number of
// active lanes, so the fp64 evaluation of the rule costs ~4,000 cycles per
// warp; this one issues fp32 and integer work only.
//   log: x = 2^e m with m in [sqrt(1/2), sqrt(2)); ln m = 2 atanh(s),
//   s = (m - 1)/(m + 1), |s| <= 0.1716, by its series through s^17 (the
//   terms beyond s^7 in fp32: they are below 2^-17 relative to the sum);
//   exp: Cody and Waite's reduction t = n ln 2 + r, |r| <= ln(2)/2, with
//   ln 2 split into three floats (the first with 15 significant bits, so
//   that n times it is exact), and Taylor's series of e^r through r^12
//   (terms from r^7 on in fp32).
// Relative error below 2^-40: against the fp64 rule evaluated with the C
// library's pow, the integer differs in about one case per million, by one.
constexpr double kLn2 = 0.69314718055994530942;
constexpr float kLn2A = 0.693145751953125f;  // 0x3f317200
constexpr float kLn2B = (float)(kLn2 - (double)kLn2A);
constexpr float kLn2C = (float)(kLn2 - (double)kLn2A - (double)kLn2B);
#define EDP_DF_CONST(v) df{(float)(v), (float)((v) - (double)(float)(v))}

__device__ __forceinline__ df df_div(df a, df b) {
  const float q1 = __fdiv_rn(a.hi, b.hi);
  df r = df_add(a, df_mul_f(b, -q1));
  const float q2 = __fdiv_rn(r.hi, b.hi);
  r = df_add(r, df_mul_f(b, -q2));
  const float q3 = __fdiv_rn(r.hi, b.hi);
  return df_add_f(quick_two_sum(q1, q2), q3);
}

__device__ __forceinline__ df df_two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ uint32_t prio_df(df x, df a) {
  const int bits = __float_as_int(x.hi);
  int e = ((bits >> 23) & 0xff) - 127;
  if ((bits & 0x7fffff) > 0x3504f3) e += 1;  // mantissa above sqrt(2)
  const float sc = __int_as_float((127 - e) << 23);
  const df m{__fmul_rn(x.hi, sc), __fmul_rn(x.lo, sc)};
  const df s = df_div(df_add_f(m, -1.0f), df_add_f(m, 1.0f));
  const df s2 = df_mul(s, s);
  float tail = 1.0f / 17;
  tail = __fmaf_rn(tail, s2.hi, 1.0f / 15);
  tail = __fmaf_rn(tail, s2.hi, 1.0f / 13);
  tail = __fmaf_rn(tail, s2.hi, 1.0f / 11);
  tail = __fmaf_rn(tail, s2.hi, 1.0f / 9);
  df p = df_add(EDP_DF_CONST(1.0 / 7), df_mul_f(s2, tail));
  p = df_add(EDP_DF_CONST(1.0 / 5), df_mul(s2, p));
  p = df_add(EDP_DF_CONST(1.0 / 3), df_mul(s2, p));
  p = df_add_f(df_mul(s2, p), 1.0f);
  df lnm = df_mul(s, p);
  lnm.hi = __fmul_rn(lnm.hi, 2.0f);
  lnm.lo = __fmul_rn(lnm.lo, 2.0f);
  const float ef = (float)e;
  df el{__fmul_rn(ef, kLn2A), 0.0f};
  el = df_add(el, df_two_prod(ef, kLn2B));
  el = df_add_f(el, __fmul_rn(ef, kLn2C));
  const df t = df_mul(a, df_add(el, lnm));
  const float nf = rintf(__fmul_rn(t.hi, 1.44269504f));
  df r = df_add_f(t, -__fmul_rn(nf, kLn2A));
  r = df_add(r, df_two_prod(-nf, kLn2B));
  r = df_add_f(r, -__fmul_rn(nf, kLn2C));
  float qt = 1.0f / 479001600;
  qt = __fmaf_rn(qt, r.hi, 1.0f / 39916800);
  qt = __fmaf_rn(qt, r.hi, 1.0f / 3628800);
  qt = __fmaf_rn(qt, r.hi, 1.0f / 362880);
  qt = __fmaf_rn(qt, r.hi, 1.0f / 40320);
  qt = __fmaf_rn(qt, r.hi, 1.0f / 5040);
  df q = df_add(EDP_DF_CONST(1.0 / 720), df_mul_f(r, qt));
  q = df_add(EDP_DF_CONST(1.0 / 120), df_mul(r, q));
  q = df_add(EDP_DF_CONST(1.0 / 24), df_mul(r, q));
  q = df_add(EDP_DF_CONST(1.0 / 6), df_mul(r, q));
  q = df_add_f(df_mul(r, q), 0.5f);
  q = df_add_f(df_mul(r, q), 1.0f);
  q = df_add_f(df_mul(r, q), 1.0f);
  const float sc2 = __int_as_float((127 + (int)nf + 20) << 23);  // 2^(n + 20)
  const float vh = __fmul_rn(q.hi, sc2), vl = __fmul_rn(q.lo, sc2);
  if (vh >= 4294967296.0f) return 0xffffffffu;
  const float rh = rintf(vh);
  const float d = __fadd_rn(__fsub_rn(vh, rh), vl);
  long long res = (long long)rh + (long long)rintf(d);
  if (res < 1) res = 1;
  if (res > 4294967295ll) res = 4294967295ll;
  return (uint32_t)res;
}
#undef EDP_DF_CONST

__device__ __forceinline__ uint32_t prio_td(float td, const PrioRule &rule) {
  if (rule.fast) {
    const df x = df_add_f(df{rule.e_hi, rule.e_lo}, fabsf(td));
    if (x.hi >= 0x1p-100f && x.hi <= 0x1p100f) return prio_df(x, df{rule.a_hi, rule.a_lo});
  }
  // the fp64 evaluation: exponents outside (0, 1], and arguments far from 1
  const double x = fabs((double)td) + rule.eps;
  double p = (x > 1e-300 && x < 1e300) ? pow_pos<true>(x, rule.alpha) * 1048576.0
                                       : pow(x, rule.alpha) * 1048576.0;
  double r = rint(p);
  if (!(r >= 1.0)) r = 1.0;
  if (r > 4294967295.0) r = 4294967295.0;
  return (uint32_t)r;
}

__global__ void k_prio_from_td(const float *__restrict__ td, uint32_t n, PrioRule rule,
                               uint32_t *__restrict__ q) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += gridDim.x * blockDim.x)
    q[i] = prio_td(td[i], rule);
}

constexpr uint32_t kEmpty = 0xffffffffu;

__device__ __forceinline__ uint32_t tab_hash(uint32_t x, uint32_t mask) {
  x ^= x >> 16;
  x *= 0x45d9f3bu;
  x ^= x >> 16;
  return x & mask;
}

// The pair's slot holds a transition; *k = its logical offset.
__device__ __forceinline__ bool slot_holds(int64_t sl, uint64_t cap, uint64_t oldest,
                                           uint64_t size, uint64_t *k) {
  if (sl < 0 || (uint64_t)sl >= cap) return false;
  *k = (uint64_t)sl >= oldest ? (uint64_t)sl - oldest : (uint64_t)sl + cap - oldest;
  return *k < size;
}

// Priority update of a large batch (more than kUpdSmallMax pairs; smaller
// ones take k_update_small below).  The slots are split over the CTAs by a
// hash, so a slot has one owner and repeats of it meet in one CTA: no
// scratch, no second phase, no CTA waits for another.  Every CTA reads the
// low words of the whole batch's slots (out of the L2), kUpdLow in flight per
// thread, and lists the positions of its own.  The owner test is a product on
// the low word, so that a foreign pair costs a few instructions; all else is
// done for the listed pairs, whose lanes are full.  They enter a shared-memory
// hash table that holds, per slot, the largest batch position (atomicMax): the
// last pair wins.  The CTA then evaluates the priority of each winner (a list
// of the occupied entries), writes its leaf and adds the exact signed delta to
// the ancestors (two's complement wrap makes negative deltas exact): deeper
// nodes rarely collide and take one 64-bit atomic per pair, level 1 (32 nodes)
// and the root are summed on chip first.  A batch of more pairs per CTA than
// half of the list, or with more pairs of one owner than the list holds, is
// entered in batch order, a part at a time where its pairs outgrow the table (a
// part's leaves are read again by the next).  The running maximum
// counts every pair, the overwritten ones too, so each warp evaluates a stripe
// of the batch for it.
//
// Bound by latency up to ~10,000 pairs, by the scan above.  Calls in a row from
// TD errors, 1,000,000 slots, and (one CTA that applied the batch 1,024 pairs at
// a time): 4,096 pairs 6.4 us (28.5), 32,768 pairs 9.0 (214.6), 131,072 pairs
// 19.5 (849.5).  With every pair tested in full and entered where it was found,
// at one pair in 32 lanes: 7.0, 13.6 and 40; halves of the scan by pairs of CTAs
// that enter each other's tables over the cluster: no gain over that.
constexpr int kUpdThreads = 1024;
constexpr int kUpdLoads = 8;                         // slots in flight per thread
constexpr int kUpdChunk = kUpdThreads * kUpdLoads;   // pairs scanned at a time
constexpr int kUpdGroup = 2;                         // loads applied at a time when a table fills
constexpr uint32_t kUpdTable = 4096;                 // open addressing, at most 3/4 full
constexpr uint32_t kUpdMost = kUpdTable / 4 * 3;
constexpr int kUpdLow = 8;                          // low words in flight per thread
constexpr uint32_t kUpdList = 2048;                  // pairs of an owner listed by the scan
static_assert(kUpdLoads % kUpdGroup == 0 && kUpdThreads * kUpdGroup <= kUpdMost,
              "a group of loads fits an empty table");
static_assert(kUpdList <= kUpdMost, "the listed pairs fit an empty table");

__device__ __noinline__ uint32_t prio_td_call(float td, const PrioRule &rule) {
  return prio_td(td, rule);
}

__global__ void __launch_bounds__(kUpdThreads, 1)
k_update(TreeView t, const int64_t *idx, const uint32_t *q, const float *td,
         const __grid_constant__ PrioRule rule, uint32_t n,
         uint64_t cap, uint64_t oldest, uint64_t size, int defer, Ctrl *ctrl) {
  __shared__ uint32_t hkey[kUpdTable];
  __shared__ uint32_t hpos[kUpdTable];
  __shared__ uint16_t used[kUpdMost];  // occupied entries, in any order
  __shared__ uint32_t list[kUpdList];   // batch positions
  __shared__ uint32_t s_used, s_listed;
  __shared__ uint32_t acc_lo[32], acc_hi[32];
  __shared__ unsigned long long warp_root[kUpdThreads / 32];
  __shared__ uint32_t s_sel, s_qmax;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t i = threadIdx.x; i < kUpdTable; i += kUpdThreads) {
    hkey[i] = kEmpty;
    hpos[i] = 0;
  }
  if (threadIdx.x < 32) {
    acc_lo[threadIdx.x] = 0;
    acc_hi[threadIdx.x] = 0;
  }
  if (threadIdx.x == 0) {
    s_sel = 0;
    s_used = 0;
    s_listed = 0;
    s_qmax = 0;
  }
  // Nothing in memory is read or written before the wait on the preceding
  // kernel: it may be the one that writes the TD errors.
  pdl_wait();
  pdl_launch();
  __syncthreads();
  // this warp's stripe of the batch: the running maximum, and bad slots
  uint32_t qmax = 0;
  for (uint64_t p = ((uint64_t)warp * gridDim.x + blockIdx.x) * 32 + lane; p < n;
       p += (uint64_t)gridDim.x * kUpdThreads) {
    const int64_t sl = idx[p];
    uint64_t k = 0;
    if (slot_holds(sl, cap, oldest, size, &k))
      qmax = max(qmax, td ? prio_td_call(td[p], rule) : q[p]);
    else if (sl < 0 || (uint64_t)sl >= cap)
      flag(ctrl, DEVERR_INDEX, (unsigned long long)sl);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) qmax = max(qmax, __shfl_xor_sync(kFull, qmax, o));
  if (lane == 0 && qmax) atomicMax(&s_qmax, qmax);

  unsigned long long root_sum = 0;
  auto insert = [&](uint32_t key, uint32_t pos) {
    uint32_t h = tab_hash(key, kUpdTable - 1);
    for (uint32_t probe = 0; probe < kUpdTable; ++probe) {
      const uint32_t prev = atomicCAS(&hkey[h], kEmpty, key);
      if (prev == kEmpty) used[atomicAdd(&s_used, 1u)] = (uint16_t)h;
      if (prev == kEmpty || prev == key) {
        atomicMax(&hpos[h], pos);
        break;
      }
      h = (h + 1) & (kUpdTable - 1);
    }
  };
  // applies the table's pairs and empties it
  auto apply = [&]() {
    __syncthreads();
    const uint32_t n_used = s_used;
    for (uint32_t i = threadIdx.x; i < n_used; i += kUpdThreads) {
      const uint32_t h = used[i];
      const uint32_t key = hkey[h];
      const uint32_t p = hpos[h];
      hkey[h] = kEmpty;
      hpos[h] = 0;
      const uint32_t old = __ldcg(t.leaves + key);
      const uint32_t qv = td ? prio_td_call(td[p], rule) : q[p];
      uint64_t k = 0;
      slot_holds((int64_t)key, cap, oldest, size, &k);
      if (defer && k == size - 1) {
        ctrl->pending_q = qv;
        continue;
      }
      const unsigned long long delta = (unsigned long long)((long long)qv - (long long)old);
      if (!delta) continue;
      t.leaves[key] = qv;
      root_sum += delta;
      if (t.depth >= 2) {
        // level 1 as two 32-bit halves with an explicit carry (exact mod 2^64)
        const uint32_t n1 = key >> (5 * (t.depth - 1));
        const uint32_t lo = (uint32_t)delta, hi = (uint32_t)(delta >> 32);
        const uint32_t was = atomicAdd(&acc_lo[n1], lo);
        atomicAdd(&acc_hi[n1], hi + (was + lo < was ? 1u : 0u));
      }
      for (uint32_t d = 2; d < t.depth; ++d)
        atomicAdd((unsigned long long *)&t.lvl(d)[key >> (5 * (t.depth - d))], delta);
    }
    __syncthreads();  // s_used and the list have been read
    if (threadIdx.x == 0) s_sel = s_used = 0;
    __syncthreads();
  };

  auto owned = [&](uint32_t low) {
    return __umulhi(low * 0x9E3779B1u, gridDim.x) == blockIdx.x;
  };
  // The scan lists the positions of the pairs owned here; no warp waits for
  // another until the batch has been read.
  const bool scan = n <= gridDim.x * (kUpdList / 2);
  if (scan) {
    const uint2 *slots = reinterpret_cast<const uint2 *>(idx);
    for (uint32_t base = 0; base < n; base += kUpdThreads * kUpdLow) {
      uint32_t low[kUpdLow], mine = 0;
      if (base + kUpdThreads * kUpdLow <= n) {
#pragma unroll
        for (int u = 0; u < kUpdLow; ++u)
          low[u] = __ldg(&slots[base + u * kUpdThreads + threadIdx.x].x);
#pragma unroll
        for (int u = 0; u < kUpdLow; ++u) mine |= owned(low[u]) ? 1u << u : 0u;
      } else {
#pragma unroll
        for (int u = 0; u < kUpdLow; ++u) {
          const uint32_t p = base + u * kUpdThreads + threadIdx.x;
          low[u] = p < n ? __ldg(&slots[p].x) : 0u;
        }
#pragma unroll
        for (int u = 0; u < kUpdLow; ++u)
          mine |= owned(low[u]) && base + u * kUpdThreads + threadIdx.x < n ? 1u << u : 0u;
      }
      if (!mine) continue;
      uint32_t at = atomicAdd(&s_listed, (uint32_t)__popc(mine));
      do {
        if (at < kUpdList) list[at] = base + (__ffs(mine) - 1) * kUpdThreads + threadIdx.x;
        ++at;
        mine &= mine - 1;
      } while (mine);
    }
    __syncthreads();
  }
  if (scan && s_listed <= kUpdList) {
    for (uint32_t i = threadIdx.x; i < s_listed; i += kUpdThreads) {
      const int64_t sl = idx[list[i]];
      uint64_t k = 0;
      if (slot_holds(sl, cap, oldest, size, &k)) insert((uint32_t)sl, list[i]);
    }
  } else {
    // A batch beyond the list, or most of it on few owners: in order, as many
    // pairs at a time as the table holds.
    for (uint64_t base = 0; base < n; base += kUpdChunk) {
      int64_t s[kUpdLoads];
#pragma unroll
      for (int u = 0; u < kUpdLoads; ++u) {
        const uint64_t p = base + u * kUpdThreads + threadIdx.x;
        s[u] = p < n ? idx[p] : -1;
      }
      uint32_t mine = 0;  // bit u: slot u is owned here
#pragma unroll
      for (int u = 0; u < kUpdLoads; ++u) {
        uint64_t k = 0;
        if (owned((uint32_t)s[u]) && slot_holds(s[u], cap, oldest, size, &k)) mine |= 1u << u;
      }
      if (mine) atomicAdd(&s_sel, (uint32_t)__popc(mine));
      __syncthreads();
      const bool fits = s_sel <= kUpdMost;
      __syncthreads();  // every thread has read s_sel
      if (fits) {
#pragma unroll
        for (int u = 0; u < kUpdLoads; ++u)
          if ((mine >> u) & 1u)
            insert((uint32_t)s[u], (uint32_t)base + u * kUpdThreads + threadIdx.x);
        continue;
      }
      apply();  // the earlier pairs, then this chunk's a group at a time
#pragma unroll
      for (int g = 0; g < kUpdLoads; g += kUpdGroup) {
#pragma unroll
        for (int u = g; u < g + kUpdGroup; ++u)
          if ((mine >> u) & 1u)
            insert((uint32_t)s[u], (uint32_t)base + u * kUpdThreads + threadIdx.x);
        apply();
      }
    }
  }
  apply();

#pragma unroll
  for (int o = 16; o; o >>= 1) root_sum += __shfl_xor_sync(kFull, root_sum, o);
  if (lane == 0) warp_root[warp] = root_sum;
  __syncthreads();
  if (warp == 0) {
    if (t.depth >= 2) {
      const unsigned long long v = ((unsigned long long)acc_hi[lane] << 32) | acc_lo[lane];
      if (v) atomicAdd((unsigned long long *)&t.lvl(1)[lane], v);
    }
    const unsigned long long root = warp_sum_u64(warp_root[lane]);
    if (lane == 0) {
      if (root) atomicAdd((unsigned long long *)&t.nodes[0], root);
      if (s_qmax) atomicMax(&ctrl->max_q, s_qmax);
    }
  }
}
static_assert(kUpdThreads / 32 == 32, "one warp sums the warps' root deltas");

// Priority update of a small batch (n <= kUpdSmallMax pairs): one CTA per 32
// pairs and a single pass, with no ticket and no second phase.  Each CTA
// stages the slots of the whole batch in shared memory and checks, for each
// of its own 32 pairs, whether a later pair of the batch sets the same slot
// (the table warps split the batch between them; every comparison reads one
// broadcast word).  The pairs that are the last occurrence of their slot
// write their leaves and add their exact deltas to the ancestors with
// atomics: each slot has exactly one writer in the batch, and integer sums
// do not depend on the order of the additions, so the tree equals the one
// the sequential application gives.  Warp 0 holds the CTA's pairs and
// evaluates their priorities meanwhile.
constexpr int kUpdSmallMax = 2048;
constexpr int kUpdSmallThreads = 256;
constexpr int kUpdScan = kUpdSmallThreads - 32;                        // scanning threads
constexpr int kUpdScanPer = (kUpdSmallMax + kUpdScan - 1) / kUpdScan;  // slots each loads

__global__ void __launch_bounds__(kUpdSmallThreads)
k_update_small(TreeView t, const int64_t *idx, const uint32_t *q, const float *td,
               PrioRule rule, uint32_t n, uint64_t cap, uint64_t oldest,
               uint64_t size, int defer, Ctrl *ctrl) {
  __shared__ uint32_t bkey[kUpdSmallMax];  // slot of each pair, kEmpty if it sets none
  __shared__ uint32_t later;               // bit l: a later pair sets pair l's slot
  __shared__ unsigned long long acc1[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t p0 = blockIdx.x * 32, p = p0 + lane;  // warp 0's pair
  pdl_wait();
  pdl_launch();
  int64_t sl = -1;
  uint64_t k = 0;
  bool holds = false;
  uint32_t qv = 0, old = 0;
  if (warp == 0) {
    float tdv = 0.f;
    if (p < n) {
      sl = idx[p];
      if (td) tdv = td[p];
      else qv = q[p];
      const bool valid = sl >= 0 && (uint64_t)sl < cap;
      if (!valid) flag(ctrl, DEVERR_INDEX, (unsigned long long)sl);
      k = !valid ? 0
          : (uint64_t)sl >= oldest ? (uint64_t)sl - oldest : (uint64_t)sl + cap - oldest;
      holds = valid && k < size;  // the slot holds a transition
      if (holds) old = t.leaves[sl];
    }
    if (holds && td) qv = prio_td(tdv, rule);
    if (!holds) qv = 0;
  } else {
    // the slots of the whole batch, every load in flight at once
    const uint32_t f = threadIdx.x - 32;
#pragma unroll
    for (int j = 0; j < kUpdScanPer; ++j) {
      const uint32_t i = f + j * kUpdScan;
      if (i < n) {
        const int64_t s2 = idx[i];
        uint32_t key = kEmpty;
        if (s2 >= 0 && (uint64_t)s2 < cap) {
          const uint64_t k2 = (uint64_t)s2 >= oldest ? (uint64_t)s2 - oldest
                                                     : (uint64_t)s2 + cap - oldest;
          if (k2 < size) key = (uint32_t)s2;
        }
        bkey[i] = key;
      }
    }
    if (f == 0) later = 0;
    asm volatile("bar.sync 1, %0;" :: "r"(kUpdScan) : "memory");
    // scanning warp w - 1 compares the CTA's pairs (one per lane) with the
    // later pairs among [j0, j1); every lane reads the same word (a
    // broadcast), and the loop is the same for all lanes
    const uint32_t mine = p < n ? bkey[p] : kEmpty;
    const uint32_t per = (n + (kUpdScan / 32) - 1) / (kUpdScan / 32);
    const uint32_t j0 = (warp - 1) * per;
    const uint32_t j1 = min(n, j0 + per);
    uint32_t j = max(j0, p0 + 1);
    bool dup = false;
    for (; j + 8 <= j1; j += 8) {
#pragma unroll
      for (int u = 0; u < 8; ++u) dup |= (bkey[j + u] == mine) & (j + u > p);
    }
    for (; j < j1; ++j) dup |= (bkey[j] == mine) & (j > p);
    const unsigned m = __ballot_sync(kFull, dup && mine != kEmpty);
    if (lane == 0 && m) atomicOr(&later, m);
  }
  __syncthreads();
  if (warp != 0) return;
  bool win = holds && !((later >> lane) & 1u);  // no later pair sets this slot
  if (win && defer && k == size - 1) {
    ctrl->pending_q = qv;
    win = false;
  }
  unsigned long long delta = 0;
  if (win) {
    t.leaves[sl] = qv;
    delta = (unsigned long long)((long long)qv - (long long)old);
  }
  if (delta) {
    uint64_t first = 33;  // level d starts at node (32^d - 1) / 31
    for (uint32_t d = 2; d < t.depth; ++d, first = first * 32 + 1)
      atomicAdd((unsigned long long *)&t.nodes[first + ((uint64_t)sl >> (5 * (t.depth - d)))],
                delta);
  }
  if (t.depth >= 2) {  // level 1 (32 nodes): the warp's deltas per node first
    acc1[lane] = 0;
    __syncwarp();
    if (delta) atomicAdd(&acc1[(uint64_t)sl >> (5 * (t.depth - 1))], delta);
    __syncwarp();
    if (acc1[lane]) atomicAdd((unsigned long long *)&t.nodes[1 + lane], acc1[lane]);
  }
  const unsigned long long root = warp_sum_u64(delta);
  uint32_t qmax = qv;  // 0 for a pair that sets no leaf
#pragma unroll
  for (int o = 16; o; o >>= 1) qmax = max(qmax, __shfl_xor_sync(kFull, qmax, o));
  if (lane == 0) {
    if (root) atomicAdd((unsigned long long *)&t.nodes[0], root);
    if (qmax) atomicMax(&ctrl->max_q, qmax);
  }
}

}  // namespace

void tree_ranges(const edp_ctx *c, uint64_t first, uint64_t count, TreeRanges *out) {
  // leaf ranges [a0, b0) and [a1, b1) (the second only on ring wrap)
  uint64_t a0 = first, b0 = first + count, a1 = 0, b1 = 0;
  if (b0 > c->cap) {
    b1 = b0 - c->cap;
    b0 = c->cap;
  }
  for (int d = (int)c->depth - 1; d >= 0; --d) {
    const unsigned shift = 5u * (c->depth - d);
    uint64_t x0 = a0 >> shift, y0 = ((b0 - 1) >> shift) + 1;
    uint64_t x1 = 0, y1 = 0;
    if (b1 > a1) {
      x1 = a1 >> shift;
      y1 = ((b1 - 1) >> shift) + 1;
      if (y1 >= x0) {  // ranges meet: one range covers both
        x0 = x1 < x0 ? x1 : x0;
        y0 = y1 > y0 ? y1 : y0;
        x1 = y1 = 0;
      }
    }
    out->a0[d] = x0;
    out->n0[d] = y0 - x0;
    out->a1[d] = x1;
    out->n1[d] = y1 - x1;
  }
}

cudaError_t launch_tree_refresh(edp_ctx *c, uint64_t first, uint64_t count,
                                cudaStream_t s) {
  if (!c->depth || !count) return cudaSuccess;
  TreeRanges r;
  tree_ranges(c, first, count, &r);
  for (int d = (int)c->depth - 1; d >= 0; --d) {
    const uint64_t nodes = r.n0[d] + r.n1[d];
    const uint64_t threads = nodes * 32;
    const unsigned blocks = (unsigned)((threads + 255) / 256);
    const bool leaves_below = (uint32_t)(d + 1) == c->depth;
    cudaError_t e = launch_pdl(k_tree_level, dim3(blocks), dim3(256), s, c->level[d],
                               leaves_below ? (const uint64_t *)nullptr
                                            : (const uint64_t *)c->level[d + 1],
                               leaves_below ? (const uint32_t *)c->leaves
                                            : (const uint32_t *)nullptr,
                               r.a0[d], r.n0[d], r.a1[d], r.n1[d]);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_tree_build_all(edp_ctx *c, cudaStream_t s) {
  return launch_tree_refresh(c, 0, c->cap, s);
}

namespace {
// A round of descents per CTA, at most eight CTAs per SM.
dim3 sample_grid(const edp_ctx *c, uint32_t n) {
  uint64_t blocks = ((uint64_t)n + kSamplePerCta - 1) / kSamplePerCta;
  if (blocks > 8u * (unsigned)c->coop_sms) blocks = 8u * (unsigned)c->coop_sms;
  return dim3((unsigned)blocks);
}
}  // namespace

cudaError_t launch_sample_targets(edp_ctx *c, const uint64_t *targets, uint32_t n,
                                  int64_t *idx, uint32_t *q, cudaStream_t s) {
  samples_on(c, s);
  return launch_pdl(k_sample_targets, sample_grid(c, n), dim3(kSampleThreads), s, view(c),
                    targets, n, idx, q, c->ctrl);
}

cudaError_t launch_sample_prioritized(edp_ctx *c, uint32_t B, uint64_t seed,
                                      uint64_t round, int64_t *idx, uint32_t *q,
                                      cudaStream_t s) {
  samples_on(c, s);
  return launch_pdl(k_sample_prio, sample_grid(c, B), dim3(kSampleThreads), s, view(c), B,
                    ~0ull / B, seed, round, idx, q, c->ctrl);
}

cudaError_t launch_update(edp_ctx *c, const int64_t *idx, const uint32_t *q,
                          const float *td, double alpha, double eps, uint32_t n,
                          cudaStream_t s) {
  samples_on(c, s);
  const uint64_t size = c->total < c->cap ? c->total : c->cap;
  const uint64_t oldest = (c->total - size) % c->cap;
  if (n <= (uint32_t)kUpdSmallMax)
    return launch_pdl(k_update_small, dim3((n + 31) / 32), dim3(kUpdSmallThreads), s,
                      view(c), idx, q, td, prio_rule(alpha, eps), n, c->cap, oldest,
                      size, c->defer, c->ctrl);
  // one CTA per SM, down to 64 pairs each: fewer CTAs read less but apply more
  // in turn (8,192 pairs at 64, 128, 256 each: 7.4, 7.8, 8.8 us)
  uint32_t grid = (n + 63) / 64;
  if (grid > (uint32_t)c->coop_sms) grid = (uint32_t)c->coop_sms;
  return launch_pdl(k_update, dim3(grid), dim3(kUpdThreads), s, view(c), idx, q, td,
                    prio_rule(alpha, eps), n, c->cap, oldest, size, c->defer, c->ctrl);
}

cudaError_t launch_prio_from_td(const float *td, uint32_t n, double alpha,
                                double eps, uint32_t *q, cudaStream_t s) {
  const unsigned blocks = (n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024;
  k_prio_from_td<<<blocks, 256, 0, s>>>(td, n, prio_rule(alpha, eps), q);
  return cudaGetLastError();
}

}  // namespace edp

// ---------------------------------------------------------------------------
// Allocation-free priority update: the kernels of edp_update_priorities_td,
// neither of which needs memory beyond its arguments, for at most
// kStaticMaxPairs pairs (the entry point's fixed limit).
// ---------------------------------------------------------------------------
extern "C" edp_status edp_update_priorities_td_static(
    edp_ctx *ctx, const int64_t *idx, const float *td, uint32_t n,
    double alpha, double eps, edp_stream stream) {
  using namespace edp;
  static const char who[] = "edp_update_priorities_td_static";
  constexpr uint32_t kStaticMaxPairs = 16384;
  if (ctx && n && !td) return fail(ctx, EDP_ERR_INVALID, "%s: td NULL", who);
  const edp_status st = update_args(ctx, who, idx, nullptr, td, n, alpha, eps);
  if (st != EDP_OK || n == 0) return st;
  if (n > kStaticMaxPairs)
    return fail(ctx, EDP_ERR_INVALID,
                "%s: n exceeds the fixed maximum of 16384 pairs (use "
                "edp_update_priorities_td)", who);
  DeviceGuard dg(ctx->cfg.device);
  EDP_TRACE(who);
  const cudaError_t e =
      launch_update(ctx, idx, nullptr, td, alpha, eps, n, (cudaStream_t)stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(ctx, EDP_ERR_CUDA, "%s: %s", who, cudaGetErrorString(e));
  }
  return EDP_OK;
}
