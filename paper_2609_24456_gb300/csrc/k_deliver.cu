// k_deliver.cu -- fused delivery: gather the sampled transitions, transform
// their uint8 payload into the learner layout, collate metadata, and
// compute importance weights, in one pass over the payload (the delivery
// operator of Sec. 2.2: the chosen transitions are materialised in the
// layout and batch shape the learner consumes).
//
// Work decomposition: the batch's output is a flat sequence of units (a
// 32-bit word of a frame, an 8-pixel group, an 8-byte run of a plane) cut into
// runs of one or two unrolled rounds, with a CTA per run however many waves
// that makes, so the block scheduler balances the tail.  The first CTAs collate
// the batch's scalars.  Frame stacks are cut by warp: a warp resolves slot,
// episode-boundary mask and source once per frame it meets.  Short frames and
// all images are cut by CTA: a thread per frame or image the CTA touches
// resolves it into shared memory, then all threads stream the run.  Loads are
// the payload bytes a lane needs for one 16-byte output store, so every
// warp-wide store instruction writes 512 contiguous bytes.  The byte->float
// step is x = b (exact), fl32(b/255) = fma(x, r1, x*r2) with one rounding (see
// unit_f32), then optionally the per-channel normalisation and the
// round-to-nearest-even bfloat16 conversion.  Where one FMA per byte,
// bf16(fma(b, A_c, B_c)), gives the same bf16 as that chain for all 256 bytes
// of every channel (constants searched and checked on the host at creation),
// the normalising delivery uses it instead of the five-operation chain.
//
// These kernels are HBM-bound: per sample they read the unique source bytes
// once and write the (2-8x larger) output once.
#include "edp_internal.cuh"

namespace edp {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
// 8-byte loads in flight per lane, and iterations per warp, of k_deliver_norm;
// loads in flight of k_deliver_norm_flat
constexpr int kNormUnroll = 6;
constexpr int kNormIters = 2;
constexpr int kNormFlatUnroll = 8;
constexpr int kStackMinBlocks = 5;  // __launch_bounds__: at most 48 registers
constexpr int kFlatMinBlocks = 5;
constexpr size_t kFourPerSm = 47000;  // shared memory of which an SM holds four

struct Common {
  const int64_t *idx;
  uint32_t B;
  uint64_t cap, oldest, nvalid;
  const int32_t *action;
  const float *reward;
  const uint8_t *done;
  int32_t *act_out;
  float *rew_out;
  uint8_t *done_out;
  const uint32_t *q;
  float *isw;
  double beta;
  const float *gsrc0, *gsrc1;
  float *gdst0, *gdst1;
  Ctrl *ctrl;
  float r1, r2;
  // fused uniform sampling: idx is then an output, sample k is drawn here
  int draw;
  uint64_t seed, round;
  int64_t *idx_out;
};

// Resolve slot -> logical offset; false (and a flag) when not sampleable.
__device__ __forceinline__ bool sample_slot(const Common &c, uint32_t k,
                                            uint64_t *slot, uint64_t *off,
                                            bool report) {
  if (c.draw) {
    // the uniform sampler's draw (Philox stream 0), made where it is used;
    // the thread that collates the sample writes its index
    const uint64_t o = mulhi64(philox_u64(c.seed, k, c.round, 0), c.nvalid);
    const uint64_t t = c.oldest + o;
    *slot = t >= c.cap ? t - c.cap : t;
    *off = o;
    if (report) c.idx_out[k] = (int64_t)*slot;
    return true;
  }
  const int64_t s = c.idx[k];
  if (s < 0 || (uint64_t)s >= c.cap) {
    if (report) flag(c.ctrl, DEVERR_INDEX, (unsigned long long)s);
    return false;
  }
  const uint64_t o = (uint64_t)s >= c.oldest ? (uint64_t)s - c.oldest
                                             : (uint64_t)s + c.cap - c.oldest;
  if (o >= c.nvalid) {
    if (report) flag(c.ctrl, DEVERR_INDEX, (unsigned long long)s);
    return false;
  }
  *slot = (uint64_t)s;
  *off = o;
  return true;
}

// Minimum of q over the batch (one warp): loads are issued 8 per lane at a
// time so a batch of 512 costs two memory round trips, not sixteen.
__device__ __forceinline__ uint32_t batch_qmin(const Common &c, int lane) {
  uint32_t m = 0xffffffffu;
  for (uint32_t i0 = lane; i0 < c.B; i0 += 32 * 8) {
    uint32_t v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t i = i0 + u * 32;
      v[u] = i < c.B ? __ldg(c.q + i) : 0xffffffffu;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) m = min(m, v[u]);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) m = min(m, __shfl_xor_sync(kFull, m, o));
  return m;
}

// Per-sample collate, importance weight and scalar gathers (one warp).  The
// head warp of each sample runs this before its payload span, so the fp64
// chain of the weight overlaps the other warps' streaming.
__device__ void collate(const Common &c, uint32_t k, bool ok, uint64_t slot,
                        uint64_t off, int lane) {
  if (lane == 0) {
    if (c.act_out) c.act_out[k] = ok ? c.action[slot] : 0;
    if (c.rew_out) c.rew_out[k] = ok ? c.reward[slot] : 0.f;
    if (c.done_out) c.done_out[k] = ok ? c.done[slot] : (uint8_t)0;
    if (c.gdst0) c.gdst0[k] = ok ? c.gsrc0[off] : 0.f;
    if (c.gdst1) c.gdst1[k] = ok ? c.gsrc1[off] : 0.f;
  }
  if (c.isw) {
    // PER: w = (q_min / q_k)^beta, q_min over the batch; fp64, one rounding
    const uint32_t m = batch_qmin(c, lane);
    if (lane == 0) c.isw[k] = is_weight(m, c.q[k], c.beta);
  }
}

// Minimum of q over the batch (the CTA): every thread gets it.  16-byte loads
// where q allows them, several in flight.
__device__ __forceinline__ uint32_t batch_qmin_cta(const Common &c) {
  __shared__ uint32_t s_min[kWarps];
  uint32_t m = 0xffffffffu;
  const uint32_t nv = ((uintptr_t)c.q & 15u) == 0 ? c.B / 4 : 0;
  const uint4 *q4 = reinterpret_cast<const uint4 *>(c.q);
  for (uint64_t i0 = threadIdx.x; i0 < nv; i0 += kThreads * 4) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = i0 + u * kThreads < nv ? __ldg(q4 + i0 + u * kThreads)
                                    : make_uint4(~0u, ~0u, ~0u, ~0u);
#pragma unroll
    for (int u = 0; u < 4; ++u) m = min(m, min(min(v[u].x, v[u].y), min(v[u].z, v[u].w)));
  }
  for (uint64_t i0 = 4ull * nv + threadIdx.x; i0 < c.B; i0 += kThreads * 4) {
    uint32_t v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = i0 + u * kThreads < c.B ? __ldg(c.q + i0 + u * kThreads) : 0xffffffffu;
#pragma unroll
    for (int u = 0; u < 4; ++u) m = min(m, v[u]);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) m = min(m, __shfl_xor_sync(kFull, m, o));
  if ((threadIdx.x & 31) == 0) s_min[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kWarps; ++w) m = min(m, s_min[w]);
  return m;
}

// Collate, importance weights and index reporting of the batch by CTA `cta`
// of `ncta`, a sample per thread of its first kCollateThreads (one warp for
// each fp64 pipe of the SM), so that the streaming CTAs carry no collate
// latency.  With weights each CTA takes q_min over the whole batch, so there
// are then at most kCollateCtas (half as many: the delivery of 32,768 small
// stacks 0.5 us shorter alone, 1 us longer in front of an update).
constexpr uint32_t kCollateThreads = 128;
constexpr uint32_t kCollateCtas = 256;
uint32_t collate_ctas(uint32_t B, bool weights) {
  const uint32_t n = B / kCollateThreads + (B % kCollateThreads != 0);
  return weights && n > kCollateCtas ? kCollateCtas : n;
}
__device__ void collate_batch(const Common &c, uint32_t cta, uint32_t ncta) {
  const uint32_t m = c.isw ? batch_qmin_cta(c) : 0xffffffffu;
  if (threadIdx.x >= kCollateThreads) return;
  for (uint64_t i = (uint64_t)cta * kCollateThreads + threadIdx.x; i < c.B;
       i += (uint64_t)ncta * kCollateThreads) {
    const uint32_t k = (uint32_t)i;
    uint64_t slot = 0, off = 0;
    const bool ok = sample_slot(c, k, &slot, &off, true);
    if (c.act_out) c.act_out[k] = ok ? c.action[slot] : 0;
    if (c.rew_out) c.rew_out[k] = ok ? c.reward[slot] : 0.f;
    if (c.done_out) c.done_out[k] = ok ? c.done[slot] : (uint8_t)0;
    if (c.gdst0) c.gdst0[k] = ok ? c.gsrc0[off] : 0.f;
    if (c.gdst1) c.gdst1[k] = ok ? c.gsrc1[off] : 0.f;
    if (c.isw) c.isw[k] = is_weight(m, c.q[k], c.beta);
  }
}

// [*f, *end): this warp's contiguous share of `total` units, rounded up to
// whole 32-unit rows so lanes stay aligned with the rows of the output.
__device__ __forceinline__ void warp_span(uint64_t total, uint64_t *f,
                                          uint64_t *end) {
  const uint64_t nw = (uint64_t)gridDim.x * kWarps;
  const uint64_t gw = (uint64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
  const uint64_t span = (((total + nw - 1) / nw) + 31) & ~31ull;
  *f = gw * span;
  *end = min(total, *f + span);
}

// exact integer -> float for a byte: 0x4B0000bb is 2^23 + b
__device__ __forceinline__ float byte_f(uint32_t w, int i) {
  return __int_as_float(__byte_perm(w, 0x4Bu, 0x4550u | i)) - 8388608.0f;
}

// ---------------------------------------------------------------------------
// Frame stack, float32 (DQN), on the load / store units.  A unit is one
// 32-bit word of frame m in [0, U) of sample k -- the frame at logical
// offset j = off - K + 1 + m, which is obs slot m (m < K) and next_obs slot
// m - 1 (m >= 1).  A lane turns its word into one float4 and stores it to
// obs and / or next_obs, so every warp-wide store writes 512 contiguous
// bytes.  Per segment (the part of one frame inside a warp's span) the warp
// resolves the slot and the episode mask once: lanes 0..K-m-1 load the done
// flags of offsets j..off and a ballot gives "an episode end before the
// anchor" (zeroes the frame in obs and next_obs) and "at the anchor" (zeroes
// it in next_obs only).
//
// A warp runs one unrolled iteration (or two, launch_deliver): UN loads in
// flight per lane, a span of 32 UN words or twice that, a CTA per kWarps spans,
// however many waves that makes; the first CTAs collate the batch
// (collate_batch) so that no streaming warp waits on it.  UN = 8 (256 words) keeps
// 8 KB of reads in flight per CTA; small batches spread over more SMs with 4.
//
// Bound by HBM.  Calls in a row, a fresh sample each, in us, and before, when
// frames were staged through shared memory by bulk copies, 2 CTAs per SM:
//   84x84, 4 frames + successors   512: 22.7 (23.6)  8,192: 314 (365), 6,820 GB/s
//   84x84, 1 frame                 8,192: 45.8 (47.6)  32,768: 172 (189)
//   64x64, 4 + successors          8,192: 184 (198)   128x128 2,048: 184 (196)
//   48x48, 4 + successors          512: 8.0 (12.0)    8,192: 105 (140)
//   92x92, 3 frames                512: 11.9 (105: its 529 runs of 16 bytes cut
//                                  into 23 equal pieces)
// 4 loads per lane instead of 8 lose up to 20% without successors (half the
// stores per load); two iterations of 4 are equal at large batches and slower
// at small ones; a 32x32 frame at 512 6.3 us (10.8).
// ---------------------------------------------------------------------------
struct StackArgs {
  const uint8_t *frames;
  uint32_t F;     // bytes per frame (multiple of 16)
  uint32_t W;     // 32-bit words per frame
  uint32_t K;
  uint32_t U;     // frames per sample (K, or K + 1 with next_obs)
  uint32_t ncollate;  // CTAs that collate the batch
  uint32_t span;      // words per warp, a multiple of 32 UN
  float *obs;
  float *next;
};

// Stack units [f, end) of one warp.
template <int UN>
__device__ __forceinline__ void stack_span(const Common &c, const StackArgs &a,
                                           uint64_t f, uint64_t end, int lane,
                                           uint64_t pol) {
  const uint64_t per = (uint64_t)a.U * a.W;  // units per sample
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  while (f < end) {
    // 32-bit divisions while they do (a 64-bit one is a long sequence)
    const uint32_t k = (f | per) <= 0xffffffffu ? (uint32_t)f / (uint32_t)per
                                                : (uint32_t)(f / per);
    const uint32_t rem = (uint32_t)(f - (uint64_t)k * per);
    const uint32_t m = rem / a.W;
    const uint32_t w_lo = rem - m * a.W;
    const uint64_t seg_end = min(end, (uint64_t)k * per + (uint64_t)(m + 1) * a.W);
    const uint32_t w_hi = (uint32_t)(seg_end - (uint64_t)k * per - (uint64_t)m * a.W);
    uint64_t slot = 0, off = 0;
    const bool ok = sample_slot(c, k, &slot, &off, false);
    const int64_t j = (int64_t)off - (int64_t)(a.K - 1) + (int64_t)m;
    const bool has_obs = m < a.K;
    const bool has_next = a.next && m >= 1;
    // the payload words of the first iteration are loaded before the
    // episode flags are known (a frame the flags zero is read for nothing),
    // so the flag and payload round trips overlap
    const bool src_ok = ok && j >= 0;
    const uint64_t js = c.oldest + (uint64_t)(j < 0 ? 0 : j);
    const uint32_t *src = reinterpret_cast<const uint32_t *>(
        a.frames + (js >= c.cap ? js - c.cap : js) * a.F);
    uint32_t v[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const uint32_t w = w_lo + lane + u * 32;
      v[u] = (src_ok && w < w_hi) ? ld_stream(src + w, pol) : 0u;
    }
    bool end_before = false, end_at = false;
    if (ok && j >= 0 && (int64_t)off >= j) {
      const uint32_t span = (uint32_t)((int64_t)off - j + 1);  // 1..K
      bool d = false;
      if ((uint32_t)lane < span) {
        const uint64_t t2 = c.oldest + (uint64_t)j + lane;
        d = c.done[t2 >= c.cap ? t2 - c.cap : t2] != 0;
      }
      const unsigned bal = __ballot_sync(kFull, d);
      end_at = (bal >> (span - 1)) & 1u;
      end_before = (bal & ((1u << (span - 1)) - 1u)) != 0;
    }
    const bool zo = !ok || j < 0 || end_before;
    const bool zn = zo || end_at;
    const bool load = (has_obs && !zo) || (has_next && !zn);
    float4 *dobs = has_obs ? reinterpret_cast<float4 *>(
                                 a.obs + ((uint64_t)k * a.K + m) * a.F)
                           : nullptr;
    float4 *dnext = has_next ? reinterpret_cast<float4 *>(
                                   a.next + ((uint64_t)k * a.K + m - 1) * a.F)
                             : nullptr;
    for (uint32_t u0 = w_lo + lane; u0 < w_hi; u0 += 32 * UN) {
      if (u0 != w_lo + lane) {
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          const uint32_t w = u0 + u * 32;
          v[u] = (load && w < w_hi) ? ld_stream(src + w, pol) : 0u;
        }
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const uint32_t w = u0 + u * 32;
        if (w >= w_hi) continue;
        float4 fv;
        fv.x = unit_f32(byte_f(v[u], 0), c.r1, c.r2);
        fv.y = unit_f32(byte_f(v[u], 1), c.r1, c.r2);
        fv.z = unit_f32(byte_f(v[u], 2), c.r1, c.r2);
        fv.w = unit_f32(byte_f(v[u], 3), c.r1, c.r2);
        if (dobs) st_stream(dobs + w, zo ? zero4 : fv, pol);
        if (dnext) st_stream(dnext + w, zn ? zero4 : fv, pol);
      }
    }
    f = seg_end;
  }
}

template <int UN>
__global__ void __launch_bounds__(kThreads, kStackMinBlocks)
k_deliver_stack(Common c, StackArgs a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t pol = policy_stream();
  // No early release: the next kernel's CTAs, waiting on this one in the last
  // waves' places, made a round of sampling, delivery and update 30.2 us; 29.7.
  pdl_wait();
  if (blockIdx.x < a.ncollate) {
    collate_batch(c, blockIdx.x, a.ncollate);
    return;
  }
  const uint64_t total = (uint64_t)c.B * a.U * a.W;
  const uint64_t f = ((uint64_t)(blockIdx.x - a.ncollate) * kWarps + warp) * a.span;
  if (f < total) stack_span<UN>(c, a, f, min(total, f + a.span), lane, pol);
}

// ---------------------------------------------------------------------------
// Frame stack, float32, as one flat range of words: a CTA takes `words`
// consecutive words of the batch's units (frame m of sample k, as above),
// whatever frames and samples they belong to, a lane per word and UN loads in
// flight, so a 128-byte frame fills a warp's access as
// well as a large one.  The samples it touches are resolved first, a thread
// each: index -> slot, into shared memory.  Then every thread issues its
// first loads, and the resolving threads load the K episode flags of their
// sample beside them and leave the masks of the frames that are zero in obs
// and in next_obs; a sample's chain is paid once per CTA and not once per
// frame.  The first `ncollate` CTAs collate the batch.
//
// Taken for frames below kFlatFrame bytes, where a span of k_deliver_stack
// crosses several frames and walks them in turn.  Calls in a row, 32,768
// samples, in us, here and (k_deliver_stack): 8x16, 1 frame and its successor,
// 12.5 (120: with 4 loads per lane); 4 frames and their successors of 320 bytes
// 67 (89), 448 91 (108), 512 102 (94: its frames end where spans do), 704 139
// (148), 768 150 (140), 784 154 (162), 1,024 198 (185).  8,192: 320 bytes 21.3
// (24.4), 704 39.2 (40.3), 784 42.4 (43.9).  Up to 2,048 samples the two cross
// at 320 to 384 bytes: 320 8.2 (8.1), 448 9.8 (9.3), 704 13.4 (12.2).
// ---------------------------------------------------------------------------
constexpr uint32_t kFlatFrame = 768;
constexpr uint32_t kFlatSamples = kThreads;  // at most touched by a CTA
struct FlatArgs {
  uint32_t words;           // per CTA
  uint32_t per;             // words per sample (U * W)
  uint32_t div_per, div_w;  // ceil(2^32 / per), ceil(2^32 / W)
};

template <int UN>
__global__ void __launch_bounds__(kThreads, kFlatMinBlocks)
k_deliver_stack_flat(Common c, StackArgs a, FlatArgs g) {
  __shared__ uint64_t s_pos[kFlatSamples];    // unwrapped slot of the anchor
  __shared__ int s_lim[kFlatSamples];         // frames back from the anchor that exist
  __shared__ uint32_t s_zo[kFlatSamples], s_zn[kFlatSamples];  // bit m: frame m is zero
  const uint64_t pol = policy_stream();
  // words [w0, w0 + nw) of the batch; the first is word i_0 of sample k0
  const uint64_t total = (uint64_t)c.B * g.per;
  const uint64_t w0 = (uint64_t)(blockIdx.x - a.ncollate) * g.words;
  const uint64_t k0 = w0 / g.per;
  const uint32_t i_0 = (uint32_t)(w0 - k0 * g.per);
  const uint32_t i_1 = i_0 + (uint32_t)min((uint64_t)g.words, total - w0);
  pdl_wait();
  pdl_launch();
  if (blockIdx.x < a.ncollate) {
    collate_batch(c, blockIdx.x, a.ncollate);
    return;
  }
  const uint32_t ns = (i_1 - 1) / g.per + 1;  // samples touched
  bool ok = false;
  uint64_t pos = 0, off = 0;
  if (threadIdx.x < ns) {
    uint64_t slot = 0;
    ok = sample_slot(c, (uint32_t)(k0 + threadIdx.x), &slot, &off, false);
    pos = c.oldest + off;
    s_pos[threadIdx.x] = pos;
    s_lim[threadIdx.x] = ok ? (int)min(off, (uint64_t)a.K) + 1 : -1;
  }
  __syncthreads();
  // word i of sample k0's range: i * per < 2^32, so the rounded-up
  // reciprocals give the exact quotients
  uint32_t v[UN];
  auto load = [&](uint32_t i, bool masked) -> uint32_t {
    if (i >= i_1) return 0u;
    const uint32_t s = __umulhi(i, g.div_per), rem = i - s * g.per;
    const uint32_t m = __umulhi(rem, g.div_w);
    if ((int)(a.K - 1) - (int)m >= s_lim[s]) return 0u;  // precedes the oldest, or a bad slot
    if (masked && ((s_zo[s] & s_zn[s]) >> m) & 1u) return 0u;
    const uint64_t js = s_pos[s] - (a.K - 1) + m;
    return ld_stream(reinterpret_cast<const uint32_t *>(
                         a.frames + (js >= c.cap ? js - c.cap : js) * a.F) + (rem - m * a.W),
                     pol);
  };
#pragma unroll
  for (int u = 0; u < UN; ++u) v[u] = load(i_0 + threadIdx.x + u * kThreads, false);
  if (threadIdx.x < ns) {
    uint32_t ends = 0;  // bit i: an episode ends at offset off - K + 1 + i
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t back = a.K - 1 - i;
      if ((uint32_t)i < a.K && ok && off >= back) {
        const uint64_t ps = pos - back;
        ends |= (c.done[ps >= c.cap ? ps - c.cap : ps] != 0 ? 1u : 0u) << i;
      }
    }
    // a frame is zero in obs when it precedes the oldest transition or an
    // episode ends between it and the anchor; in next_obs also when one ends
    // at the anchor; the anchor's successor (m = K) only with the sample
    const bool end_at = (ends >> (a.K - 1)) & 1u;
    uint32_t zo = 0, zn = (ok ? 0u : 1u) << a.K;
    bool before = false;
    for (int m = (int)a.K - 1; m >= 0; --m) {
      if (m < (int)a.K - 1) before |= (ends >> m) & 1u;
      const bool z = !ok || before || off < a.K - 1 - (uint32_t)m;
      zo |= (z ? 1u : 0u) << m;
      zn |= (z || end_at ? 1u : 0u) << m;
    }
    s_zo[threadIdx.x] = zo | 1u << a.K;  // the successor is no part of obs,
    s_zn[threadIdx.x] = a.next ? zn | 1u : ~0u;  // nor the first frame of next_obs
  }
  __syncthreads();
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  for (uint32_t i0 = i_0 + threadIdx.x; i0 < i_1; i0 += kThreads * UN) {
    if (i0 != i_0 + threadIdx.x) {
#pragma unroll
      for (int u = 0; u < UN; ++u) v[u] = load(i0 + u * kThreads, true);
    }
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const uint32_t i = i0 + u * kThreads;
      if (i >= i_1) continue;
      const uint32_t s = __umulhi(i, g.div_per), rem = i - s * g.per;
      const uint32_t m = __umulhi(rem, g.div_w), w = rem - m * a.W;
      const uint64_t frame = (k0 + s) * a.K + m;
      float4 fv;
      fv.x = unit_f32(byte_f(v[u], 0), c.r1, c.r2);
      fv.y = unit_f32(byte_f(v[u], 1), c.r1, c.r2);
      fv.z = unit_f32(byte_f(v[u], 2), c.r1, c.r2);
      fv.w = unit_f32(byte_f(v[u], 3), c.r1, c.r2);
      if (m < a.K)
        st_stream(reinterpret_cast<float4 *>(a.obs) + frame * a.W + w,
                  (s_zo[s] >> m) & 1u ? zero4 : fv, pol);
      if (a.next && m >= 1)
        st_stream(reinterpret_cast<float4 *>(a.next) + (frame - 1) * a.W + w,
                  (s_zn[s] >> m) & 1u ? zero4 : fv, pol);
    }
  }
}

// ---------------------------------------------------------------------------
// HWC uint8 -> CHW bfloat16 (on-policy mini-batches).  Unit = 8 pixels: a lane
// converts 8 consecutive pixels: it loads their 8*C interleaved bytes and
// writes C 16-byte runs, one per channel plane.  A CTA takes `units`
// consecutive units of the batch, whatever images they belong to: a thread
// per image it touches resolves the slot into shared memory, then all threads
// stream the units as one flat range, UN * C loads in flight each, so that
// images of any size fill a warp.  The first `ncollate` CTAs collate the batch.
// Bound by HBM; calls in a row, in us, and (before) when a warp walked its
// span image by image and collated at each: 8x16x1, 65,536 images 5.6 (20.3),
// 512 images 2.1 (4.9); 16x16x3, 65,536 24.6 (30.1); 64x64x3, 4,096 24.9
// (25.2), 65,536 352 (353); 84x84x4, 16,384 203 (207).
// ---------------------------------------------------------------------------
struct ChwArgs {
  const uint8_t *obs;
  uint32_t HW;   // pixels per image
  uint32_t units;  // per CTA
  uint32_t div_g;  // ceil(2^32 / G), G = HW / 8; 0: a CTA spans at most two images
  uint32_t ncollate;
  __nv_bfloat16 *out;
};
constexpr uint32_t kHwcImages = kThreads;  // at most touched by a CTA

template <int C, int UN>
__global__ void __launch_bounds__(kThreads)
k_deliver_hwc(Common c, ChwArgs a) {
  __shared__ uint64_t s_slot[kHwcImages];  // ~0: a bad index
  const uint64_t pol = policy_stream();
  const uint32_t G = a.HW / 8;  // 8-pixel groups per image
  const uint64_t F = (uint64_t)a.HW * C;
  // units [u0, u0 + n) of the batch; the first is unit i_0 of image k0
  const uint64_t total = (uint64_t)c.B * G;
  const uint64_t u0 = (uint64_t)(blockIdx.x - a.ncollate) * a.units;
  const uint64_t k0 = u0 / G;
  const uint32_t i_0 = (uint32_t)(u0 - k0 * G);
  const uint32_t i_1 = i_0 + (uint32_t)min((uint64_t)a.units, total - u0);
  pdl_wait();
  pdl_launch();
  if (blockIdx.x < a.ncollate) {
    collate_batch(c, blockIdx.x, a.ncollate);
    return;
  }
  if (threadIdx.x <= (i_1 - 1) / G) {
    uint64_t slot = 0, off = 0;
    s_slot[threadIdx.x] =
        sample_slot(c, (uint32_t)(k0 + threadIdx.x), &slot, &off, false) ? slot : ~0ull;
  }
  __syncthreads();
  for (uint32_t i0 = i_0 + threadIdx.x; i0 < i_1; i0 += kThreads * UN) {
    uint2 v[UN][C];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const uint32_t i = i0 + u * kThreads;
      // i * G < 2^32, so the rounded-up reciprocal gives the exact quotient
      const uint32_t s = a.div_g ? __umulhi(i, a.div_g) : (i >= G ? 1u : 0u);
      const uint64_t slot = i < i_1 ? s_slot[s] : ~0ull;
      const uint2 *src = reinterpret_cast<const uint2 *>(a.obs + slot * F) +
                         (uint64_t)(i - s * G) * C;
#pragma unroll
      for (int q = 0; q < C; ++q)
        v[u][q] = slot != ~0ull ? ld_stream(src + q, pol) : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const uint32_t i = i0 + u * kThreads;
      if (i >= i_1) continue;
      const uint32_t s = a.div_g ? __umulhi(i, a.div_g) : (i >= G ? 1u : 0u);
      uint4 *dst = reinterpret_cast<uint4 *>(a.out + (k0 + s) * F) + (i - s * G);
      uint32_t wd[2 * C];
#pragma unroll
      for (int q = 0; q < C; ++q) {
        wd[2 * q] = v[u][q].x;
        wd[2 * q + 1] = v[u][q].y;
      }
#pragma unroll
      for (int ch = 0; ch < C; ++ch) {
        float fv[8];
#pragma unroll
        for (int px = 0; px < 8; ++px) {
          const int byte = px * C + ch;  // position within the 8*C bytes
          fv[px] = unit_f32(byte_f(wd[byte >> 2], byte & 3), c.r1, c.r2);
        }
        uint4 o;
        o.x = pack_bf16x2(fv[0], fv[1]);
        o.y = pack_bf16x2(fv[2], fv[3]);
        o.z = pack_bf16x2(fv[4], fv[5]);
        o.w = pack_bf16x2(fv[6], fv[7]);
        st_stream(dst + (uint64_t)ch * G, o, pol);
      }
    }
  }
}

// One round of UN units per thread: longer ranges (up to 4,096 units while an
// SM keeps 8 CTAs) were equal on small images and 3-6% slower on large batches.
template <int C, int UN>
cudaError_t launch_hwc(const Common &c, ChwArgs a, cudaStream_t s) {
  const uint64_t G = a.HW / 8, total = c.B * G;
  uint64_t units = (uint64_t)kThreads * UN;
  if (units > (kHwcImages - 2) * G) units = ((kHwcImages - 2) * G) & ~31ull;
  a.units = (uint32_t)units;
  a.div_g = G < 32768 ? (uint32_t)((0x100000000ull + G - 1) / G) : 0u;
  const uint64_t ctas = (total + units - 1) / units + a.ncollate;
  if (ctas > 0x7FFFFFFFull) return cudaErrorInvalidValue;
  return launch_pdl(k_deliver_hwc<C, UN>, dim3((unsigned)ctas), dim3(kThreads), s, c, a);
}

// ---------------------------------------------------------------------------
// CHW uint8 -> per-channel normalised bfloat16 (multimodal payloads), with
// token collate; optionally two-tier (payload of older transitions in
// page-locked host memory, read over the host link).  Unit = 8 bytes: a lane
// converts 8 consecutive bytes of one channel plane to one 16-byte store.  The
// first `ncollate` CTAs collate the batch, the next `ntok` copy the tokens, and
// each of the others takes `units` consecutive units of the batch, whatever
// images they belong to: a thread per image (or token row) it touches resolves
// the row into shared memory, then all threads stream the units as one flat
// range, UN loads in flight each.  Bound by the chain of dependent loads for
// small batches.  Calls in a row, in us, and (by warps, k_deliver_norm):
//   images of     64x64x3      96x96x3 + 128   224x224x3 + 512  84x84x1     16x16x1
//   B = 64        3.1 (3.3)    3.1 (3.6)       5.7 (7.7)        2.8 (4.2)   2.6 (6.2)
//   B = 256       3.7 (3.6)    5.1 (6.5)                        2.8 (4.4)   2.6 (8.7)
//   B = 1,024     7.4 (8.9)                                     5.1 (7.8)   2.6 (9.0)
// 6 units in flight and 4 CTAs per SM, or 8 and 3: 7% slower on large batches; 4
// and 5: 10%.
// ---------------------------------------------------------------------------
struct NormArgs {
  const uint8_t *obs_h;   // HBM ring [cap_h][F]
  const uint8_t *obs_c;   // host ring [cap_c][F] (device-mapped) or null
  const int32_t *tok_h;
  const int32_t *tok_c;
  uint64_t cap_h, cap_c, total, size;
  // offsets below `cold` (older ones) live in the host tier; physical rows of
  // the oldest offset there and of offset `cold` in HBM
  uint64_t cold, first_c, first_h;
  uint32_t F8;    // 8-byte units per image
  uint32_t HW8;   // 8-byte units per channel plane
  uint32_t L16;   // 16-byte units of tokens per transition
  uint32_t units, tunits;  // image and token units per CTA
  uint32_t div_f, div_l;  // ceil(2^32 / F8), ceil(2^32 / L16); 0: a CTA spans at most two rows
  uint32_t ncollate, ntok;
  float mean[4], s1[4], s2[4], sd[4];
  float aa[4], ab[4];  // one-FMA form (AFF): bf16(fma(b, aa, ab))
  int fast;
  __nv_bfloat16 *out;
  int32_t *tok_out;
};
constexpr int kNormCtas = 4;               // CTAs per SM
constexpr uint32_t kNormRows = kThreads;   // at most touched by a CTA
constexpr uint32_t kTokUnroll = 4;         // 16-byte token loads in flight per lane
constexpr uint32_t kTokUnits = kThreads * kTokUnroll;

// Physical row of sample k in its tier; false for a bad index.
__device__ __forceinline__ bool norm_row(const Common &c, const NormArgs &a, uint32_t k,
                                         uint64_t *row, bool *hbm) {
  uint64_t slot = 0, off = 0;
  if (!sample_slot(c, k, &slot, &off, false)) return false;
  *hbm = off >= a.cold;
  const uint64_t at = *hbm ? a.first_h + (off - a.cold) : a.first_c + off;
  const uint64_t cap = *hbm ? a.cap_h : a.cap_c;
  *row = at >= cap ? at - cap : at;
  return true;
}

// i / d with inv = ceil(2^32 / d) (i d < 2^32), or for i < 2 d without one.
__device__ __forceinline__ uint32_t row_of_unit(uint32_t i, uint32_t d, uint32_t inv) {
  return inv ? __umulhi(i, inv) : (i >= d ? 1u : 0u);
}

// The eight bytes of unit w of an image, normalised.
template <bool AFF>
__device__ __forceinline__ uint4 norm_unit(const Common &c, const NormArgs &a, uint2 v,
                                           uint32_t w) {
  const uint32_t ch = (w >= a.HW8) + (w >= 2 * a.HW8) + (w >= 3 * a.HW8);
  float fv[8];
  if constexpr (AFF) {
    const float A = a.aa[ch], Bc = a.ab[ch];
#pragma unroll
    for (int bb = 0; bb < 8; ++bb)
      fv[bb] = __fmaf_rn(byte_f(bb < 4 ? v.x : v.y, bb & 3), A, Bc);
  } else {
    const float mc = a.mean[ch], s1 = a.s1[ch], s2 = a.s2[ch];
#pragma unroll
    for (int bb = 0; bb < 8; ++bb) {
      const float x = unit_f32(byte_f(bb < 4 ? v.x : v.y, bb & 3), c.r1, c.r2);
      const float tt = __fsub_rn(x, mc);
      fv[bb] = a.fast ? __fmaf_rn(tt, s1, __fmul_rn(tt, s2)) : __fdiv_rn(tt, a.sd[ch]);
    }
  }
  uint4 o;
  o.x = pack_bf16x2(fv[0], fv[1]);
  o.y = pack_bf16x2(fv[2], fv[3]);
  o.z = pack_bf16x2(fv[4], fv[5]);
  o.w = pack_bf16x2(fv[6], fv[7]);
  return o;
}

template <int UN, bool AFF, bool TWO>
__global__ void __launch_bounds__(kThreads, kNormCtas)
k_deliver_norm_flat(Common c, NormArgs a) {
  __shared__ uint64_t s_src[kNormRows];  // a row's address (16-byte aligned), its lowest bit
                                         // set in HBM; 0: a bad index
  const uint64_t pol = policy_stream();
  const bool tok = blockIdx.x >= a.ncollate && blockIdx.x < a.ncollate + a.ntok;
  // units [u0, u0 + n) of the batch's rows of P units; the first is unit i_0 of
  // row k0
  const uint32_t P = tok ? a.L16 : a.F8;
  const uint64_t total = (uint64_t)c.B * P;
  const uint64_t u0 = tok ? (uint64_t)(blockIdx.x - a.ncollate) * a.tunits
                          : (uint64_t)(blockIdx.x - a.ncollate - a.ntok) * a.units;
  const uint64_t k0 = u0 <= 0xffffffffu ? (uint32_t)u0 / P : u0 / P;
  const uint32_t i_0 = (uint32_t)(u0 - k0 * P);
  const uint32_t i_1 = i_0 + (uint32_t)min((uint64_t)(tok ? a.tunits : a.units), total - u0);
  pdl_wait();
  pdl_launch();
  if (blockIdx.x < a.ncollate) {
    collate_batch(c, blockIdx.x, a.ncollate);
    return;
  }
  if (threadIdx.x <= (i_1 - 1) / P) {
    uint64_t row = 0, src = 0;
    bool hbm = true;
    if (norm_row(c, a, (uint32_t)(k0 + threadIdx.x), &row, &hbm)) {
      if (tok) {
        src = (uint64_t)((hbm ? a.tok_h : a.tok_c) + row * a.L16 * 4ull);
      } else {
        src = (uint64_t)((hbm ? a.obs_h : a.obs_c) + row * a.F8 * 8ull);
        // a two-tier row read over the host link (edp_get_counters), counted
        // where its first unit is read
        if (!hbm && (threadIdx.x || i_0 == 0))
          atomicAdd(&c.ctrl->host_bytes,
                    (unsigned long long)a.F8 * 8ull + (a.tok_out ? a.L16 * 16ull : 0ull));
      }
      src |= hbm ? 1u : 0u;
    }
    s_src[threadIdx.x] = src;
  }
  __syncthreads();
  if (tok) {
    uint4 v[kTokUnroll];
#pragma unroll
    for (uint32_t u = 0; u < kTokUnroll; ++u) {
      const uint32_t i = i_0 + threadIdx.x + u * kThreads;
      const uint32_t s = P == 1 ? i : row_of_unit(i, P, a.div_l);  // 2^32 / 1 has no 32 bits
      const uint64_t src = i < i_1 ? s_src[s] & ~1ull : 0;
      v[u] = src ? reinterpret_cast<const uint4 *>(src)[i - s * P] : make_uint4(0u, 0u, 0u, 0u);
    }
    uint4 *dst = reinterpret_cast<uint4 *>(a.tok_out) + k0 * P;
#pragma unroll
    for (uint32_t u = 0; u < kTokUnroll; ++u) {
      const uint32_t i = i_0 + threadIdx.x + u * kThreads;
      if (i < i_1) dst[i] = v[u];
    }
    return;
  }
  uint4 *dst = reinterpret_cast<uint4 *>(a.out) + k0 * P;
  for (uint32_t i0 = i_0 + threadIdx.x; i0 < i_1; i0 += kThreads * UN) {
    uint2 v[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const uint32_t i = i0 + u * kThreads;
      const uint32_t s = row_of_unit(i, P, a.div_f);
      const uint64_t src = i < i_1 ? s_src[s] : 0;
      const uint2 *p = reinterpret_cast<const uint2 *>(src & ~1ull) + (i - s * P);
      // HBM tier: streaming non-coherent loads; host tier: plain loads of the
      // mapped page-locked memory
      v[u] = src ? (!TWO || (src & 1u) ? ld_stream(p, pol) : *p) : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const uint32_t i = i0 + u * kThreads;
      if (i >= i_1) continue;
      const uint32_t s = row_of_unit(i, P, a.div_f), w = i - s * P;
      uint4 o = norm_unit<AFF>(c, a, v[u], w);
      if (!s_src[s]) o = make_uint4(0u, 0u, 0u, 0u);
      st_stream(dst + i, o, pol);
    }
  }
}

// The same by warps: each takes an equal contiguous span of the batch, image by
// image, and resolves and collates a sample where its first unit lies, so no
// warp waits for another.  For large batches of large images, where a delivery
// alone takes as long either way, and on two streams in turn, each filling the
// other's last wave, 67.3 us a batch of 1,024 224x224x3 + 512 tokens; 68.2 by
// flat runs.
template <int UN, bool AFF>
__global__ void __launch_bounds__(kThreads)
k_deliver_norm(Common c, NormArgs a) {
  const int lane = threadIdx.x & 31;
  const uint64_t pol = policy_stream();
  pdl_wait();
  pdl_launch();
  const uint64_t total = (uint64_t)c.B * a.F8;
  uint64_t f, end;
  warp_span(total, &f, &end);
  while (f < end) {
    const uint32_t k = (uint32_t)(f / a.F8);
    const uint32_t u_lo = (uint32_t)(f - (uint64_t)k * a.F8);
    const uint64_t seg_end = min(end, (uint64_t)(k + 1) * a.F8);
    const uint32_t u_hi = (uint32_t)(seg_end - (uint64_t)k * a.F8);
    const bool head = u_lo == 0;
    uint64_t slot = 0, off = 0;
    const bool ok = sample_slot(c, k, &slot, &off, head && lane == 0);
    if (head) collate(c, k, ok, slot, off, lane);
    // tier of the logical id L = total - size + off
    const uint64_t L = a.total - a.size + off;
    const uint64_t in_hbm = a.total < a.cap_h ? a.total : a.cap_h;
    const bool hbm = !a.obs_c || L >= a.total - in_hbm;
    const uint64_t ps = hbm ? L % a.cap_h : L % a.cap_c;
    const uint8_t *obs = hbm ? a.obs_h : a.obs_c;
    const uint2 *src = reinterpret_cast<const uint2 *>(obs + ps * a.F8 * 8ull);
    uint4 *dst = reinterpret_cast<uint4 *>(a.out + (uint64_t)k * a.F8 * 8ull);
    for (uint32_t u0 = u_lo + lane; u0 < u_hi; u0 += 32 * UN) {
      uint2 v[UN];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const uint32_t w = u0 + u * 32;
        // HBM tier: streaming non-coherent loads; host tier: plain loads of
        // the mapped page-locked memory
        v[u] = (ok && w < u_hi) ? (hbm ? ld_stream(src + w, pol) : src[w])
                                : make_uint2(0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const uint32_t w = u0 + u * 32;
        if (w >= u_hi) continue;
        uint4 o = norm_unit<AFF>(c, a, v[u], w);
        if (!ok) o = make_uint4(0u, 0u, 0u, 0u);
        st_stream(dst + w, o, pol);
      }
    }
    if (head) {
      // a two-tier row read over the host link (edp_get_counters)
      if (lane == 0 && ok && a.obs_c && !hbm)
        atomicAdd(&c.ctrl->host_bytes,
                  (unsigned long long)a.F8 * 8ull + (a.tok_out ? a.L16 * 16ull : 0ull));
      if (a.tok_out) {
        // the row's tokens, kTokBatch 16-byte loads per lane in flight
        // before their stores
        constexpr int kTokBatch = 4;
        const uint4 *ts = reinterpret_cast<const uint4 *>(
            (hbm ? a.tok_h : a.tok_c) + ps * a.L16 * 4ull);
        uint4 *td = reinterpret_cast<uint4 *>(a.tok_out + (uint64_t)k * a.L16 * 4ull);
        for (uint32_t i0 = lane; i0 < a.L16; i0 += 32 * kTokBatch) {
          uint4 t4[kTokBatch];
#pragma unroll
          for (int u = 0; u < kTokBatch; ++u) {
            const uint32_t i = i0 + u * 32;
            t4[u] = (ok && i < a.L16) ? ts[i] : make_uint4(0u, 0u, 0u, 0u);
          }
#pragma unroll
          for (int u = 0; u < kTokBatch; ++u)
            if (i0 + u * 32 < a.L16) td[i0 + u * 32] = t4[u];
        }
      }
    }
    f = seg_end;
  }
}

// Grid size from the work: enough CTAs that each warp runs about `iters`
// iterations of its unrolled loop (`per_iter` units each), so the block
// scheduler balances the tail and a CTA that starts late (its SM still busy
// with another kernel) holds up little work; a small batch is spread over up
// to one wave (blocks resident per SM x SMs, queried once for each kernel: the
// library runs on one kind of GPU) with at least one iteration per warp.
template <auto kern>
unsigned grid_for(uint64_t units, uint64_t per_iter, int iters, int sms) {
  static const int per_sm = [] {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kThreads, 0);
    return n < 1 ? 1 : n;
  }();
  const uint64_t wave = (uint64_t)per_sm * sms;
  const uint64_t warp_iters = (units + per_iter - 1) / per_iter;
  uint64_t blocks = (warp_iters + (uint64_t)kWarps * iters - 1) / ((uint64_t)kWarps * iters);
  if (blocks < wave) {
    const uint64_t most = (warp_iters + kWarps - 1) / kWarps;
    blocks = most < wave ? most : wave;
  }
  return (unsigned)(blocks ? blocks : 1);
}

}  // namespace

cudaError_t launch_deliver(edp_ctx *ctx, const int64_t *idx, uint32_t B,
                           const edp_batch *out, cudaStream_t s, const DrawUniform *draw) {
  Common c{};
  c.idx = idx;
  if (draw) {
    c.draw = 1;
    c.seed = draw->seed;
    c.round = draw->round;
    c.idx_out = draw->idx_out;
  }
  c.B = B;
  c.cap = ctx->cap;
  const uint64_t size = ctx->total < ctx->cap ? ctx->total : ctx->cap;
  c.oldest = (ctx->total - size) % ctx->cap;
  c.nvalid = size - ctx->defer;
  c.action = ctx->st.action;
  c.reward = ctx->st.reward;
  c.done = ctx->st.done;
  c.act_out = out->action;
  c.rew_out = out->reward;
  c.done_out = out->done;
  c.q = out->q;
  c.isw = out->isw;
  c.beta = out->beta;
  c.gsrc0 = out->gather_src[0];
  c.gdst0 = out->gather_dst[0];
  c.gsrc1 = out->gather_src[1];
  c.gdst1 = out->gather_dst[1];
  c.ctrl = ctx->ctrl;
  c.r1 = ctx->r1;
  c.r2 = ctx->r2;
  const int sms = ctx->coop_sms;
  const auto &cfg = ctx->cfg;
  if (cfg.transform == EDP_XFORM_STACK_F32) {
    StackArgs a{};
    a.frames = ctx->st.obs;
    a.F = (uint32_t)ctx->obs_bytes;
    a.W = a.F / 4;
    a.K = cfg.frame_stack;
    a.obs = (float *)out->obs;
    a.next = (float *)out->next_obs;
    a.U = a.K + (a.next ? 1 : 0);
    a.ncollate = collate_ctas(B, out->isw != nullptr);
    const uint64_t per = (uint64_t)a.U * a.W, units = B * per;
    if (a.F < kFlatFrame) {
      FlatArgs g{};
      g.per = (uint32_t)per;  // at most 17 frames: words * per < 2^32
      // 1,024 words with 4 loads per lane, one round (8x16, 4 frames and
      // successors, 512 stacks: 3.6 us, 4.7 with 2,048 words and 8); 2,048 with
      // 8 from 3.5 CTAs of those per SM on (8,192 stacks: 9.4 us, 10.3), up to
      // 4,096 while every SM keeps eight CTAs (16x16, 32,768: 55 us, 58)
      const bool wide = units / 2048 >= 7ull * sms / 2;
      g.words = wide ? 2048 : 1024;
      while (g.words < 4096 && units / (2 * g.words) >= 8ull * sms) g.words *= 2;
      if (g.words > (kFlatSamples - 2) * per)
        g.words = (uint32_t)((kFlatSamples - 2) * per) & ~31u;
      g.div_per = (uint32_t)((0x100000000ull + per - 1) / per);
      g.div_w = (uint32_t)((0x100000000ull + a.W - 1) / a.W);
      const uint64_t ctas = (units + g.words - 1) / g.words + a.ncollate;
      if (ctas > 0x7FFFFFFFull) return cudaErrorInvalidValue;
      auto kern = wide ? k_deliver_stack_flat<8> : k_deliver_stack_flat<4>;
      return launch_pdl(kern, dim3((unsigned)ctas), dim3(kThreads), s, c, a, g);
    }
    // 4 loads per lane up to three such CTAs per SM (84x84, 4 frames and
    // successors, 48: 4.1 us, 4.6 with 8; 64: 4.7, 4.6; 128x128, 16: 3.6, 4.1; one
    // frame, 192: 3.6, 3.8)
    const bool few = units <= 3ull * kWarps * 32 * 4 * sms;
    a.span = 32 * (few ? 4 : 8);
    uint64_t ctas = (units + (uint64_t)kWarps * a.span - 1) / ((uint64_t)kWarps * a.span);
    // Stacks of three frames or more with successors, from 2.8 waves on: four CTAs
    // per SM instead of five, held there by shared memory that they don't use: as
    // fast alone (84x84, 4 frames, 512: 22.7 us, 22.9; 3 frames, 2.7 waves: 19.1, 18.7),
    // and the small kernels of other streams find room among its waves (sampling
    // and update beside it: a round 22.6 us, 24.4).  Fewer stores per load need the
    // fifth: 84x84, 1 frame and successor, 4,096: 51.8 us, 45.7; 2 frames, 768: 18.6,
    // 16.6; without successors 8,192: 195, 171.
    const bool four =
        a.next && a.K >= 3 && 5 * (ctas + a.ncollate) >= 14ull * kStackMinBlocks * sms;
    // On another stream than the context's sampling and updates, two iterations
    // per warp up to 16 waves: in half the waves those kernels, on which the next
    // delivery waits, get through sooner.  That round 21.6 us instead of 22.6 for
    // 512 stacks, 43.3 instead of 43.9 for 1,024, 83.8 instead of 84.4 for 2,048
    // (8,192: 327.5, 326.6).  On their stream it is slower, the last wave being
    // longer: 30.5 instead of 29.7, the delivery alone 23.7 instead of 22.8.
    if (four && ctas <= 64ull * sms && ctx->sampler_known && s != ctx->sampler_stream) {
      a.span *= 2;
      ctas = (ctas + 1) / 2;
    }
    ctas += a.ncollate;
    if (ctas > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    auto kern = few ? k_deliver_stack<4> : k_deliver_stack<8>;
    return launch_pdl_smem(kern, dim3((unsigned)ctas), dim3(kThreads), four ? kFourPerSm : 0, s,
                           c, a);
  } else if (cfg.transform == EDP_XFORM_HWC_CHW_BF16) {
    ChwArgs a{};
    a.obs = ctx->st.obs;
    a.HW = cfg.obs_h * cfg.obs_w;
    a.out = (__nv_bfloat16 *)out->obs;
    a.ncollate = collate_ctas(B, out->isw != nullptr);
    switch (cfg.obs_c) {
      case 1: return launch_hwc<1, 4>(c, a, s);
      case 2: return launch_hwc<2, 2>(c, a, s);
      case 3: return launch_hwc<3, 2>(c, a, s);
      default: return launch_hwc<4, 2>(c, a, s);
    }
  } else {
    NormArgs a{};
    a.obs_h = ctx->st.obs;
    a.obs_c = ctx->cap_c ? ctx->st.host_obs : nullptr;
    a.tok_h = ctx->st.tokens;
    a.tok_c = ctx->cap_c ? ctx->st.host_tokens : nullptr;
    a.cap_h = ctx->cap_h;
    a.cap_c = ctx->cap_c ? ctx->cap_c : 1;
    a.total = ctx->total;
    a.size = size;
    // ids total - size + off; the newest min(total, cap_h) of them in HBM at id
    // mod cap_h, the older ones in the host tier at id mod cap_c
    const uint64_t in_hbm = ctx->total < ctx->cap_h ? ctx->total : ctx->cap_h;
    a.cold = size > in_hbm ? size - in_hbm : 0;
    a.first_h = (ctx->total - size + a.cold) % a.cap_h;
    a.first_c = (ctx->total - size) % a.cap_c;
    a.F8 = (uint32_t)(ctx->obs_bytes / 8);
    a.HW8 = cfg.obs_h * cfg.obs_w / 8;
    a.L16 = (uint32_t)(ctx->tok_bytes / 16);
    for (int i = 0; i < 4; ++i) {
      a.mean[i] = ctx->nmean[i];
      a.s1[i] = ctx->ns1[i];
      a.s2[i] = ctx->ns2[i];
      a.sd[i] = ctx->nstd[i] > 0.f ? ctx->nstd[i] : 1.f;
      a.aa[i] = ctx->naff_a[i];
      a.ab[i] = ctx->naff_b[i];
    }
    a.fast = ctx->norm_fast;
    a.out = (__nv_bfloat16 *)out->obs;
    a.tok_out = out->tokens;
    const uint64_t rows = kNormRows - 2, total = (uint64_t)B * a.F8;
    uint64_t units = (uint64_t)kThreads * kNormFlatUnroll;
    // Flat runs up to two waves of CTAs, and for small images (below 1,024
    // units, where a warp's span crosses several) at any batch size, in runs of
    // two rounds there (4,096 images of 84x84: 13.1 us; 13.9 in one round, 16.2
    // by warps).
    if (total > 2 * (uint64_t)kNormCtas * sms * units) {
      if (a.F8 >= 1024) {
        constexpr auto one_fma = k_deliver_norm<kNormUnroll, true>;
        constexpr auto chain = k_deliver_norm<kNormUnroll, false>;
        const unsigned grid =
            ctx->norm_affine ? grid_for<one_fma>(total, 32 * kNormUnroll, kNormIters, sms)
                             : grid_for<chain>(total, 32 * kNormUnroll, kNormIters, sms);
        return launch_pdl(ctx->norm_affine ? one_fma : chain, dim3(grid), dim3(kThreads), s, c, a);
      }
      units *= 2;
    }
    if (units > rows * a.F8) units = (rows * a.F8) & ~31ull;
    a.units = (uint32_t)units;
    a.ncollate = collate_ctas(B, out->isw != nullptr);
    const uint64_t tok_units = a.tok_out ? (uint64_t)B * a.L16 : 0;
    a.tunits = rows * a.L16 < kTokUnits ? (uint32_t)(rows * a.L16) : kTokUnits;
    const uint64_t ntok = tok_units ? (tok_units + a.tunits - 1) / a.tunits : 0;
    a.ntok = (uint32_t)ntok;
    a.div_f = a.F8 < 32768 ? (uint32_t)((0x100000000ull + a.F8 - 1) / a.F8) : 0u;
    a.div_l = a.L16 && a.L16 < 32768 ? (uint32_t)((0x100000000ull + a.L16 - 1) / a.L16) : 0u;
    const uint64_t ctas = (total + units - 1) / units + a.ncollate + a.ntok;
    if (ctas > 0x7FFFFFFFull || ntok > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    auto kern = ctx->norm_affine
                    ? (a.obs_c ? k_deliver_norm_flat<kNormFlatUnroll, true, true>
                               : k_deliver_norm_flat<kNormFlatUnroll, true, false>)
                    : (a.obs_c ? k_deliver_norm_flat<kNormFlatUnroll, false, true>
                               : k_deliver_norm_flat<kNormFlatUnroll, false, false>);
    return launch_pdl(kern, dim3((unsigned)ctas), dim3(kThreads), s, c, a);
  }
}

}  // namespace edp
