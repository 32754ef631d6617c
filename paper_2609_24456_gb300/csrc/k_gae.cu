// k_gae.cu -- generalized advantage estimation with global advantage
// normalisation (Schulman et al., ICLR'16; the return / advantage and
// normalisation steps of on-policy ingestion, Sec. 2.2).
//
//   delta_t = r_t + gamma V_{t+1} (1 - d_t) - V_t
//   A_t = delta_t + c_t A_{t+1},  c_t = gamma lambda (1 - d_t),  A_T = 0
//
// The recurrence is a composition of affine maps x -> b + a x, which is
// associative, so a CTA scans kE environments' steps in parallel: thread
// (s, e) composes the maps of kL consecutive steps of environment e (segment
// s), shuffles compose the segments of a warp, the warps' composites meet in
// shared memory, and each thread then replays its own steps from the value
// handed over by the later ones.  Chunks of as many steps as the CTA holds
// (2,048 / kE at most) are processed from the end of the rollout backwards,
// carrying A across; the next chunk's inputs are loaded beside a chunk's
// arithmetic.  With kE = 8 every access of a time-major row moves whole
// 32-byte sectors; rollouts of few environments use fewer per CTA, so that more
// SMs and longer chunks share the steps (gae_shape).
//
// Arithmetic: GB300's fp64 pipe is narrow (a dependent fp64 FMA costs ~64
// cycles, fp32 ~4), so the scan runs in double-float arithmetic -- a value
// is an unevaluated pair hi + lo of fp32 numbers, combined with the
// error-free transformations TwoSum (Knuth) and TwoProd via FMA (Dekker),
// as in the double-double arithmetic of Hida, Li and Bailey -- which keeps
// ~44 significant bits (relative error ~2^-44 per operation); gamma and
// gamma*lambda enter as pairs split from fp64.  The sums of A and A^2 carry three
// words and round once per CTA, to fp64 (in double-float the variance lost up to
// a digit against fp64: 24 rollouts of 2,048 steps, mean 1e5 deviations, 1.3e-5
// off, 7.8e-7 so).  The mean and the variance are formed in fp64 from the CTAs'
// sums; the normalisation of an element takes the mean in three fp32 words and
// the scale in two (norm_value), fp64 where a value is out of their range.
// Outputs are rounded to fp32.
//
// Bound by latency (a chunk's loads, then its dependent chain) up to ~10^6
// values, then by HBM.  Calls in a row with all three outputs, in us, and
// (before) with one warp per environment: 8 x 2,048 steps 10.3 (43.0), 4,096 x
// 64 11.9 (28.4), 1,024 x 1,024 24.6 (107), 64 x 8,192 36.9 (557), 8 x 128 6.8
// (9.2), 8 x 512 7.0 (16.0).
//
// Two kernels chained with programmatic dependent launch: the scan writes A,
// the returns and per-CTA sums of A and A^2; the normalisation kernel
// forms mean and the unbiased standard deviation (every CTA reduces the
// partials in the same fixed order, so all agree bit for bit) and writes
// the normalised values; a small rollout is scanned and normalised by one CTA,
// without a second kernel.  With the environments
// sharded over several ranks, the scan's sums are reduced to this rank's
// (n, sum A, sum A^2) instead (k_gae_stats), the caller sums those over the
// ranks, and the normalisation reads the totals.
#include <type_traits>

#include "edp_internal.cuh"

namespace edp {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kL = 4;               // steps per thread and chunk
constexpr int kGaeThreads = 512;    // at most per CTA
constexpr int kGaeWarps = kGaeThreads / 32;
static_assert(kGaeWarps <= 16, "half a warp adds the warps' sums");
constexpr int kNormThreads = 256;
constexpr int kNormLoads = 8;       // values in flight per thread of a single CTA

__device__ __forceinline__ df df_shfl_down(df a, int o) {
  return {__shfl_down_sync(kFull, a.hi, o), __shfl_down_sync(kFull, a.lo, o)};
}

// A sum of three fp32 numbers, for the sums over a CTA's values: each addition
// keeps about 70 significant bits (the errors of two_sum are carried in full, only
// the third words' sum rounds), so the total rounds once, to fp64.  fp64 itself
// would take 16 instructions a warp of the narrow pipe, about 64 cycles each.  In
// us, environments x steps, and with sums and trees in double-float: 262,144 x 1
// 60.4 (83.3: A and A^2 share a tree, half a warp each), 8 x 2,048 10.3 (10.7),
// 1,024 x 1,024 24.6 (24.3); long rollouts in many CTAs pay for the third word,
// most at 977 x 2,048 41.7 (40.9).
struct tf {
  float a, b, c;
};
__device__ __forceinline__ tf tf_norm(tf x) {
  const df p = two_sum(x.a, x.b);
  const df q = two_sum(p.lo, x.c);
  return {p.hi, q.hi, q.lo};
}
__device__ __forceinline__ tf tf_add(tf x, tf y) {
  const df s = two_sum(x.a, y.a), t = two_sum(x.b, y.b);
  const df m = two_sum(s.lo, t.hi);
  return tf_norm({s.hi, m.hi, __fadd_rn(__fadd_rn(x.c, y.c), __fadd_rn(t.lo, m.lo))});
}
// x + y for a running sum, in the operations of a double-float addition: the
// words overlap by the logarithm of the number of values, which tf_norm takes up
// before it counts.
__device__ __forceinline__ tf tf_acc(tf x, df y) {
  const df s = two_sum(x.a, y.hi), t = two_sum(x.b, y.lo);
  const df m = two_sum(s.lo, t.hi);
  return {s.hi, m.hi, __fadd_rn(x.c, __fadd_rn(t.lo, m.lo))};
}
__device__ __forceinline__ tf tf_shfl_down16(tf x, int o) {  // within half a warp
  return {__shfl_down_sync(kFull, x.a, o, 16), __shfl_down_sync(kFull, x.b, o, 16),
          __shfl_down_sync(kFull, x.c, o, 16)};
}
__device__ __forceinline__ tf tf_shfl_xor16(tf x) {
  return {__shfl_xor_sync(kFull, x.a, 16), __shfl_xor_sync(kFull, x.b, 16),
          __shfl_xor_sync(kFull, x.c, 16)};
}
__device__ __forceinline__ double tf_to_d(tf x) {
  return (double)x.a + ((double)x.b + (double)x.c);
}

// The value 2^e (|e| < 127).
__device__ __forceinline__ float exp2_int(int e) { return __int_as_float((127 + e) << 23); }

// What the normalisation needs of the whole rollout.
struct NormStat {
  double mean, inv;  // inv = 1 / (std + 1e-8); 0 for a single value
  // -mean in three fp32 words, exactly, and inv in two: with integers, which
  // run beside the fp64 chain
  float m[3];
  df inv_df;
  bool narrow;  // both within the words' range
};

// From n values with sums s1 (of A) and s2 (of A^2).
__device__ __forceinline__ NormStat norm_stat(double nn, double s1, double s2) {
  NormStat st;
  st.mean = s1 / nn;
  const uint64_t mb = (uint64_t)__double_as_longlong(st.mean);
  const int me = (int)((mb >> 52) & 0x7ff) - 1023;
  const uint64_t mm = (mb & 0x000fffffffffffffull) | (1ull << 52);
  const bool zero = (mb << 1) == 0;
  const bool m_in = zero || (me >= -70 && me < 60);
  const int e = zero || !m_in ? 0 : me;
  const float sg = zero ? 0.f : (mb >> 63) ? 1.f : -1.f;
  st.m[0] = sg * (float)(uint32_t)(mm >> 29) * exp2_int(e - 23);            // 24 bits
  st.m[1] = sg * (float)((uint32_t)(mm >> 5) & 0xffffffu) * exp2_int(e - 47);  // the next 24
  st.m[2] = sg * (float)((uint32_t)mm & 31u) * exp2_int(e - 52);            // and 5
  double var = nn > 1.0 ? (s2 - s1 * st.mean) / (nn - 1.0) : 0.0;
  if (var < 0.0) var = 0.0;
  // a single value equals its mean and normalises to exactly 0; the scale
  // is 0 so that the fp32 rounding of the stored A (A - mean ~ 2^-24 |A|
  // here) is not multiplied by 1 / 1e-8
  st.inv = nn > 1.0 ? 1.0 / (sqrt(var) + 1e-8) : 0.0;
  const uint64_t ib = (uint64_t)__double_as_longlong(st.inv);
  const int ie = (int)((ib >> 52) & 0x7ff) - 1023;
  const uint64_t im = (ib & 0x000fffffffffffffull) | (1ull << 52);
  const bool i_in = !(ib >> 63) && ie >= -60 && ie < 60;
  const int ix = i_in ? ie : 0;
  st.inv_df = {(float)(uint32_t)(im >> 29) * exp2_int(ix - 23),
               (float)((uint32_t)im & 0x1fffffffu) * exp2_int(ix - 52)};
  st.narrow = m_in && i_in;
  return st;
}

// (a - mean) inv, rounded once to fp32 but for 2^-45 of it: the difference is
// exact until its third word, however much of it cancels, so the result is at
// least as close as in fp64 (whose difference rounds at 2^-53 of the mean).  With
// the mean in two words split in fp64, values near it were off by 2^-48 of the
// mean, and the split took longer: gae_normalize of 4,096 values 2.9 us, now 2.7
// (2.7 with fp64 throughout, and 16.2 instead of 7.0 for 1,024 x 1,024).
__device__ __forceinline__ float norm_value(float a, const NormStat &st) {
  if (st.narrow && fabsf(a) < 1e18f) {
    const df s = two_sum(st.m[0], a), t = two_sum(s.hi, st.m[1]);
    const df x = two_sum(t.hi, __fadd_rn(__fadd_rn(s.lo, t.lo), st.m[2]));
    return df_mul(x, st.inv_df).hi;
  }
  return (float)(((double)a - st.mean) * st.inv);
}

// Inputs of one thread's kL steps and the value after each.
struct GaeIn {
  float r[kL], v[kL + 1];
  bool d[kL];
};
// Loads of a chunk [ts, te) by thread (seg, e) of `segs` segments.  With eight
// environments per CTA a warp's load of one step each touches four rows, whole
// sectors: the thread loads its own steps ts + seg kL ...  With fewer, adjacent
// threads load adjacent steps instead (x.r[i] is step ts + i segs + seg), since
// rows kL apart would take a cache line per lane, and the steps change hands
// through shared memory (gae_exchange).  A step at or past te reads a valid one
// instead, a value past te the one at te; x.v[kL] is the value after the
// thread's last step, or (staged) after the chunk.
template <bool STAGED>
__device__ __forceinline__ void gae_load(GaeIn &x, const float *r, const float *v,
                                         const uint8_t *d, uint32_t ts, uint32_t te,
                                         uint32_t seg, uint32_t segs, uint32_t E, uint32_t e) {
  // (T + 1) E < 2^32, and a step past te is less than a chunk past it.  The
  // eight-environment form keeps 64-bit indices: with fewer registers to hold,
  // ptxas takes it down to 64 with spills (1,024 x 1,024: 39 us, 29.5)
  using index = std::conditional_t<STAGED, uint32_t, uint64_t>;
#pragma unroll
  for (int i = 0; i < kL; ++i) {
    const index t = STAGED ? (index)ts + i * segs + seg : (index)ts + seg * kL + i;
    const index at = min(t, (index)(te - 1)) * E + e;
    x.r[i] = r[at];
    x.d[i] = d[at] != 0;
    x.v[i] = v[min(t, (index)te) * E + e];
  }
  x.v[kL] = v[(STAGED ? (index)te : min((index)ts + seg * kL + kL, (index)te)) * E + e];
}

// A chunk's inputs, [step * kE + e], the values one step more.
struct GaeStage {
  float r[kGaeThreads * kL];
  float v[kGaeThreads * kL + 8];
  bool d[kGaeThreads * kL];
};
template <int kE>
__device__ __forceinline__ void gae_exchange(GaeIn &x, GaeStage &s, uint32_t seg, uint32_t segs,
                                             uint32_t el) {
#pragma unroll
  for (int i = 0; i < kL; ++i) {
    const uint32_t at = (i * segs + seg) * kE + el;
    s.r[at] = x.r[i];
    s.v[at] = x.v[i];
    s.d[at] = x.d[i];
  }
  if (seg == 0) s.v[segs * kL * kE + el] = x.v[kL];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kL; ++i) {
    const uint32_t at = (seg * kL + i) * kE + el;
    x.r[i] = s.r[at];
    x.v[i] = s.v[at];
    x.d[i] = s.d[at];
  }
  x.v[kL] = s.v[(seg * kL + kL) * kE + el];
}

template <int kE>
__global__ void __launch_bounds__(kGaeThreads)
k_gae_scan(const float *r, const float *v, const uint8_t *d, uint32_t T, uint32_t E, float2 g2,
           float2 gl2, float *A_out, float *ret, double *partial, float *adv_norm) {
  __shared__ float4 agg[kGaeWarps][kE];  // a warp's composite: a.hi, a.lo, b.hi, b.lo
  __shared__ float2 s_carry[kE];         // A at the step after the chunk
  __shared__ tf s_sum[2][kGaeWarps];  // of A, of A^2
  __shared__ NormStat s_stat;
  constexpr bool kStaged = kE < 8;
  __shared__ std::conditional_t<kStaged, GaeStage, char> stage;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  const uint32_t el = threadIdx.x % kE, seg = threadIdx.x / kE;
  const uint32_t segs = blockDim.x / kE, chunk = segs * kL;
  const df one = {1.f, 0.f}, zero = {0.f, 0.f};
  const df g = {g2.x, g2.y}, gl = {gl2.x, gl2.y};  // gamma, gamma lambda
  pdl_wait();
  tf t1 = {0.f, 0.f, 0.f}, t2 = t1;  // this thread's sums of A and A^2
  for (uint32_t tile = blockIdx.x; (uint64_t)tile * kE < E; tile += gridDim.x) {
    const bool real = tile * kE + el < E;
    const uint32_t e = real ? tile * kE + el : E - 1;
    if (seg == 0) s_carry[el] = make_float2(0.f, 0.f);  // read after the barrier below
    GaeIn x;
    uint32_t te = T, ts = T > chunk ? T - chunk : 0;
    gae_load<kStaged>(x, r, v, d, ts, te, seg, segs, E, e);
    for (;;) {
      const uint64_t t0 = (uint64_t)ts + seg * kL;
      const uint32_t te2 = ts, ts2 = ts > chunk ? ts - chunk : 0;
      GaeIn next;
      if (te2) gae_load<kStaged>(next, r, v, d, ts2, te2, seg, segs, E, e);
      if constexpr (kStaged) gae_exchange<kE>(x, stage, seg, segs, el);
      df del[kL], cc[kL];
      df a = one, b = zero;  // this thread's steps composed: x -> b + a x
#pragma unroll
      for (int i = kL - 1; i >= 0; --i) {
        if (t0 + i < te) {
          // delta = r + gamma V' (1 - d) - V
          const df y = x.d[i] ? df{x.r[i], 0.f} : df_add_f(df_mul_f(g, x.v[i + 1]), x.r[i]);
          del[i] = df_add_f(y, -x.v[i]);
          cc[i] = x.d[i] ? zero : gl;
          b = df_add(del[i], df_mul(cc[i], b));
          a = df_mul(cc[i], a);
        } else {
          del[i] = zero;
          cc[i] = one;
        }
      }
      // inclusive suffix scan over the warp's segments of each environment
#pragma unroll
      for (int o = kE; o < 32; o <<= 1) {
        const df a2s = df_shfl_down(a, o);
        const df b2s = df_shfl_down(b, o);
        if (lane + o < 32) {
          b = df_add(b, df_mul(a, b2s));
          a = df_mul(a, a2s);
        }
      }
      if (lane < kE) agg[warp][el] = make_float4(a.hi, a.lo, b.hi, b.lo);
      __syncthreads();
      // A at the step after this warp's last one
      df A = {s_carry[el].x, s_carry[el].y};
      for (int w = nwarps - 1; w > warp; --w) {
        const float4 m = agg[w][el];
        A = df_add(df{m.z, m.w}, df_mul(df{m.x, m.y}, A));
      }
      // ... and after this thread's
      const df an = df_shfl_down(a, kE % 32), bn = df_shfl_down(b, kE % 32);
      if (lane < 32 - kE) A = df_add(bn, df_mul(an, A));
#pragma unroll
      for (int i = kL - 1; i >= 0; --i) {
        if (t0 + i < te) {
          A = df_add(del[i], df_mul(cc[i], A));
          if (real) {
            const uint64_t at = (t0 + i) * E + e;
            if (A_out) A_out[at] = A.hi;
            if (ret) ret[at] = df_add_f(A, x.v[i]).hi;
            t1 = tf_acc(t1, A);
            const float sq = __fmul_rn(A.hi, A.hi);
            t2 = tf_acc(t2, df{sq, __fmaf_rn(2.f * A.hi, A.lo, __fmaf_rn(A.hi, A.hi, -sq))});
          }
        }
      }
      __syncthreads();  // agg and s_carry have been read
      if (seg == 0) s_carry[el] = make_float2(A.hi, A.lo);
      if (!te2) break;
      // kL values since the last; ahead of the exchange above instead, under the
      // loads, it delayed a rollout of one chunk: an iteration of 256 x 128 with its
      // delivery 190.4 us, 188.7 so
      t1 = tf_norm(t1);
      t2 = tf_norm(t2);
      x = next;
      te = te2;
      ts = ts2;
    }
  }
  pdl_launch();
  if (!partial && !adv_norm) return;  // no normalisation requested
  // this CTA's sums in a fixed order: a shuffle tree per warp, then over the
  // warps, the lower half of a warp for A and the upper for A^2
  const int half = lane >> 4, hl = lane & 15;
  tf t = tf_add(half ? t2 : t1, tf_shfl_xor16(half ? t1 : t2));
#pragma unroll
  for (int o = 8; o; o >>= 1) t = tf_add(t, tf_shfl_down16(t, o));
  if (nwarps > 1) {
    if (hl == 0) s_sum[half][warp] = t;
    __syncthreads();
  }
  if (warp == 0) {
    if (nwarps > 1) {
      t = hl < nwarps ? s_sum[half][hl] : tf{0.f, 0.f, 0.f};
#pragma unroll
      for (int o = kGaeWarps / 2; o; o >>= 1)
        if (o < nwarps) t = tf_add(t, tf_shfl_down16(t, o));
    }
    const double sum = tf_to_d(t), other = __shfl_xor_sync(kFull, sum, 16);
    if (partial) {
      if (hl == 0) partial[2 * blockIdx.x + half] = sum;
    } else if (lane == 0) {
      s_stat = norm_stat((double)((uint64_t)T * E), sum, other);
    }
  }
  if (partial) return;
  // one CTA scanned everything: it normalises what it wrote
  __syncthreads();
  const NormStat st = s_stat;
  const uint64_t n = (uint64_t)T * E;
  for (uint64_t i0 = threadIdx.x; i0 < n; i0 += kNormLoads * blockDim.x) {
    float y[kNormLoads];
#pragma unroll
    for (int u = 0; u < kNormLoads; ++u) {
      const uint64_t i = i0 + u * blockDim.x;
      y[u] = i < n ? __ldcg(A_out + i) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kNormLoads; ++u) {
      const uint64_t i = i0 + u * blockDim.x;
      if (i < n) adv_norm[i] = norm_value(y[u], st);
    }
  }
}

// Sum of the per-CTA partials (sum A, sum A^2) in a fixed order; the totals
// end in *s1, *s2 of thread 0.  Every CTA that calls it gets the same bits.  Up
// to kFewParts one warp adds and shuffles them, without a barrier (a call of 8 x
// 2,048 takes 1.0 us longer with the tree); more take strided per-thread sums and
// a shared-memory tree, whose levels use fewer and fewer warps of the fp64 pipe
// (4,096 x 32: 1.4 us longer with shuffles in every warp).
constexpr uint32_t kFewParts = 128;
__device__ __forceinline__ void reduce_partials(const double *partial, uint32_t nparts,
                                                double *s1, double *s2) {
  __shared__ double r1[kNormThreads], r2[kNormThreads];
  double t1 = 0.0, t2 = 0.0;
  if (nparts <= kFewParts) {
    if (threadIdx.x < 32) {
      double p1[kFewParts / 32], p2[kFewParts / 32];
#pragma unroll
      for (uint32_t u = 0; u < kFewParts / 32; ++u) {
        const uint32_t i = threadIdx.x + 32 * u;
        p1[u] = i < nparts ? __ldcg(&partial[2 * i]) : 0.0;
        p2[u] = i < nparts ? __ldcg(&partial[2 * i + 1]) : 0.0;
      }
#pragma unroll
      for (uint32_t u = 0; u < kFewParts / 32; ++u) {
        if (32 * u >= nparts) break;
        t1 += p1[u];
        t2 += p2[u];
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        t1 += __shfl_down_sync(kFull, t1, o);
        t2 += __shfl_down_sync(kFull, t2, o);
      }
    }
  } else {
    for (uint32_t i = threadIdx.x; i < nparts; i += kNormThreads) {
      t1 += __ldcg(&partial[2 * i]);
      t2 += __ldcg(&partial[2 * i + 1]);
    }
    r1[threadIdx.x] = t1;
    r2[threadIdx.x] = t2;
    __syncthreads();
    for (int w = kNormThreads / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) {
        r1[threadIdx.x] += r1[threadIdx.x + w];
        r2[threadIdx.x] += r2[threadIdx.x + w];
      }
      __syncthreads();
    }
    t1 = r1[0];
    t2 = r2[0];
  }
  *s1 = t1;
  *s2 = t2;
}

// This rank's statistics of A for a normalisation over several ranks:
// stats = (n, sum A, sum A^2), reduced from the scan's partials in the same
// order as k_gae_norm reduces them (one CTA).
__global__ void __launch_bounds__(kNormThreads)
k_gae_stats(const double *partial, uint32_t nparts, uint64_t n, double *stats) {
  pdl_wait();
  pdl_launch();
  double s1, s2;
  reduce_partials(partial, nparts, &s1, &s2);
  if (threadIdx.x == 0) {
    stats[0] = (double)n;
    stats[1] = s1;
    stats[2] = s2;
  }
}

// Normalisation: every CTA reduces the per-CTA partials of the scan in the
// same fixed order (or reads the statistics (n, sum A, sum A^2) of all ranks
// when `stats` is given), then writes (A - mean) * inv_std, four elements per
// thread and load where both arrays allow it.  A is read from A_src (the
// caller's adv, or adv_norm itself); n is the number of elements here.
__global__ void __launch_bounds__(kNormThreads)
k_gae_norm(const float *A_src, float *adv_norm, uint64_t n, const double *partial,
           uint32_t nparts, const double *stats) {
  __shared__ NormStat s_stat;
  pdl_wait();
  pdl_launch();
  // this thread's first elements, loaded beside the partial sums
  const bool vec = (((uintptr_t)A_src | (uintptr_t)adv_norm) & 15u) == 0;
  const uint64_t nv = vec ? n / 4 : 0;
  const uint64_t i0 = blockIdx.x * (uint64_t)kNormThreads + threadIdx.x;
  const uint64_t stride = (uint64_t)gridDim.x * kNormThreads;
  const float4 *src = reinterpret_cast<const float4 *>(A_src);
  float4 x = i0 < nv ? __ldcg(src + i0) : make_float4(0.f, 0.f, 0.f, 0.f);
  double nn = (double)n, s1, s2;
  if (stats) {
    nn = __ldcg(&stats[0]);
    s1 = __ldcg(&stats[1]);
    s2 = __ldcg(&stats[2]);
  } else {
    reduce_partials(partial, nparts, &s1, &s2);  // of thread 0
  }
  if (threadIdx.x == 0) s_stat = norm_stat(nn, s1, s2);
  __syncthreads();
  const NormStat st = s_stat;
  for (uint64_t i = i0; i < nv; i += stride) {
    if (i != i0) x = __ldcg(src + i);
    x = make_float4(norm_value(x.x, st), norm_value(x.y, st), norm_value(x.z, st),
                    norm_value(x.w, st));
    reinterpret_cast<float4 *>(adv_norm)[i] = x;
  }
  for (uint64_t i = 4 * nv + i0; i < n; i += stride)
    adv_norm[i] = norm_value(__ldcg(&A_src[i]), st);
}

}  // namespace

namespace {

// Two sums per CTA: a CTA takes eight environments, or fewer while it makes
// fewer CTAs than SMs, which the least scratch block (ctx_scratch) covers.
size_t gae_scratch_bytes(uint32_t E) { return ((size_t)E + 3) / 4 * 2 * sizeof(double); }

// Environments per CTA, threads per CTA and CTAs of a scan.  A CTA of
// 512 threads is bound by issue (about 4 us per chunk whatever its shape), so
// the environments per CTA are halved from 8 while half of the SMs would idle:
// 8 x 512 steps with 8, 4, 2, 1 environments per CTA 12.7, 9.4, 7.8, 7.2 us
// per call, 8 x 2,048 35.9, 21.5, 13.8, 10.3, 256 x 128 7.6, 7.4, 7.6, 9.1.
struct GaeShape {
  uint32_t envs, threads, grid;
};
GaeShape gae_shape(const edp_ctx *c, uint32_t T, uint32_t E, bool one_cta) {
  GaeShape g;
  g.envs = 8;
  while (!one_cta && g.envs > 1 &&
         2 * (((uint64_t)E + g.envs - 1) / g.envs) < (uint64_t)c->coop_sms)
    g.envs /= 2;
  const uint64_t want = ((uint64_t)T + kL - 1) / kL * g.envs;
  g.threads = want < kGaeThreads ? (uint32_t)((want + 31) & ~31ull) : (uint32_t)kGaeThreads;
  g.grid = (uint32_t)(((uint64_t)E + g.envs - 1) / g.envs);
  return g;
}

cudaError_t launch_scan(const GaeShape &g, const float *r, const float *v, const uint8_t *d,
                        uint32_t T, uint32_t E, double gamma, double lambda, float *A_out,
                        float *ret, double *partial, float *adv_norm, cudaStream_t s) {
  auto kern = g.envs == 8 ? k_gae_scan<8> : g.envs == 4 ? k_gae_scan<4>
            : g.envs == 2 ? k_gae_scan<2> : k_gae_scan<1>;
  auto split = [](double x) {
    const float hi = (float)x;
    return make_float2(hi, (float)(x - (double)hi));
  };
  return launch_pdl(kern, dim3(g.grid), dim3(g.threads), s, r, v, d, T, E, split(gamma),
                    split(gamma * lambda), A_out, ret, partial, adv_norm);
}

// One CTA per SM while that leaves a thread a few elements: each CTA adds the
// partial sums again and forms the statistics, and several on one SM queue on
// its fp64 pipe (4,096 x 64: 12.7 us per call, 13.2 with four per SM); four per
// SM for the loads of more (1,024 x 1,024: 25.3 us, 29.6 with one).
unsigned norm_grid(const edp_ctx *c, uint64_t n) {
  const uint64_t sms = (uint64_t)c->coop_sms;
  const uint64_t want = (n + 4 * kNormThreads - 1) / (4 * kNormThreads);
  const uint64_t most = want <= 4 * sms ? sms : 4 * sms;
  return (unsigned)(want < most ? want : most);
}

}  // namespace

cudaError_t launch_gae(edp_ctx *c, const float *r, const float *v,
                       const uint8_t *d, uint32_t T, uint32_t E, double gamma,
                       double lambda, float *adv, float *ret, float *adv_norm,
                       cudaStream_t s) {
  // a rollout of one chunk of eight environments: one CTA scans and normalises
  // it (8 x 128: 6.8 us; equal either way from a graph, one launch instead of two)
  const bool one_cta = adv_norm && E <= 8 && T <= 128;
  const GaeShape g = gae_shape(c, T, E, one_cta);
  double *partial = nullptr;
  if (adv_norm) {
    void *blk = nullptr;
    const cudaError_t e = ctx_scratch(c, gae_scratch_bytes(E), s, &blk);
    if (e != cudaSuccess) return e;
    partial = (double *)blk;
  }
  // A is kept for the normalisation in adv, or in adv_norm itself (fp32; the
  // normalisation error this adds is below 2^-24 |A| / std)
  float *A_out = adv ? adv : adv_norm;
  if (one_cta)
    return launch_scan(g, r, v, d, T, E, gamma, lambda, A_out, ret, nullptr, adv_norm, s);
  const cudaError_t e =
      launch_scan(g, r, v, d, T, E, gamma, lambda, A_out, ret, partial, nullptr, s);
  if (e != cudaSuccess || !adv_norm) return e;
  const uint64_t n = (uint64_t)T * E;
  return launch_pdl(k_gae_norm, dim3(norm_grid(c, n)), dim3(kNormThreads), s,
                    (const float *)A_out, adv_norm, n, (const double *)partial, g.grid,
                    (const double *)nullptr);
}

cudaError_t launch_gae_stats(edp_ctx *c, const float *r, const float *v,
                             const uint8_t *d, uint32_t T, uint32_t E, double gamma,
                             double lambda, float *adv, float *ret, double *stats,
                             cudaStream_t s) {
  const GaeShape g = gae_shape(c, T, E, false);
  void *blk = nullptr;
  cudaError_t e = ctx_scratch(c, gae_scratch_bytes(E), s, &blk);
  if (e != cudaSuccess) return e;
  double *partial = (double *)blk;
  e = launch_scan(g, r, v, d, T, E, gamma, lambda, adv, ret, partial, nullptr, s);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_gae_stats, dim3(1), dim3(kNormThreads), s, (const double *)partial,
                    g.grid, (uint64_t)T * E, stats);
}

cudaError_t launch_gae_normalize(edp_ctx *c, const float *adv, uint64_t n,
                                 const double *stats, float *adv_norm, cudaStream_t s) {
  return launch_pdl(k_gae_norm, dim3(norm_grid(c, n)), dim3(kNormThreads), s, adv, adv_norm, n,
                    (const double *)nullptr, 0u, stats);
}

}  // namespace edp
