// k_llm.cu -- LLM post-training on the experience path (Appendix A): the
// group-relative advantages of GRPO (Shao et al. 2024), computed during
// ingestion, and the packed delivery of variable-length token sequences
// with a per-sequence value broadcast to their tokens.
//
// Advantages: one warp per group, two warps per CTA so the groups spread
// over every SM (the fp64 pipe is narrow; eight warps on one SM queue on
// it); fp64 sums of r and of (r - mean)^2 (two passes), one rounding to fp32
// per output.  Packing: each batch entry's source start, length and value
// (one thread each, into the context's scratch) with a length sum per
// 256-entry chunk; then the copy forms each sequence's output offset -- the
// chunk sums before its chunk plus the lengths before it in the chunk -- and
// moves its tokens (neither the source nor the destination offset is aligned
// to more than a token), writing the value beside each token: a CTA per
// sequence, several CTAs per long sequence, or a warp per short one, the long
// ones among them by CTAs from a list (launch_gather).  Up to kDirectChunks
// chunks the copying CTAs add the chunk sums themselves; beyond that the last
// lengths CTA turns them into prefixes once.  The copy is HBM-bound.
#include "edp_internal.cuh"

namespace edp {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kGrpoThreads = 64;
constexpr int kGrpoWarps = kGrpoThreads / 32;
constexpr int kPackThreads = 256;
constexpr uint64_t kPackWaitNs = 1000000000ull;  // bound of the gather's wait for its copy
constexpr uint32_t kDirectChunks = 256;  // chunk sums a gather CTA adds itself
static_assert(kDirectChunks <= kPackThreads, "a gather CTA adds one chunk sum per thread");

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Groups g = first, first + stride, ... of one warp.
__device__ __forceinline__ void grpo_groups(const float *r, const uint64_t *goff, uint32_t ng,
                                            float eps, float *adv, uint64_t first,
                                            uint64_t stride) {
  const int lane = threadIdx.x & 31;
  for (uint64_t g = first; g < ng; g += stride) {
    const uint64_t lo = goff[g], hi = goff[g + 1];
    if (hi <= lo) continue;
    const uint64_t n = hi - lo;
    double s1 = 0.0;
    for (uint64_t i = lo + lane; i < hi; i += 32) s1 += (double)r[i];
    const double mean = warp_sum(s1) / (double)n;
    double s2 = 0.0;
    for (uint64_t i = lo + lane; i < hi; i += 32) {
      const double d = (double)r[i] - mean;
      s2 = fma(d, d, s2);
    }
    s2 = warp_sum(s2);
    const double var = n > 1 ? s2 / (double)(n - 1) : 0.0;
    const double den = sqrt(var) + (double)eps;
    for (uint64_t i = lo + lane; i < hi; i += 32)
      adv[i] = den > 0.0 ? (float)(((double)r[i] - mean) / den) : 0.f;
  }
}

__global__ void __launch_bounds__(kGrpoThreads)
k_grpo(const float *r, const uint64_t *goff, uint32_t ng, float eps, float *adv) {
  pdl_wait();
  pdl_launch();
  grpo_groups(r, goff, ng, eps, adv, (uint64_t)blockIdx.x * kGrpoWarps + (threadIdx.x >> 5),
              (uint64_t)gridDim.x * kGrpoWarps);
}

// What the copy of batch entry k needs, resolved once: where its tokens
// start, how many there are, and the sequence (for its value; kNoSeq when
// the index is out of range).
struct PackEntry {
  uint64_t src;
  uint32_t seq;
  uint32_t len;
};
constexpr uint32_t kNoSeq = 0xffffffffu;

// What k_pack_gather_short does with the long entries (above kShortTokens) of a
// CTA's `each` neighbouring ones: the first of them, up to `keep` tokens together,
// the CTA copies itself, the others the lengths kernel lists (in any order) for
// whichever CTA takes them.  entry null: no list is wanted.
constexpr uint32_t kShortTokens = 1024;
struct LongList {
  uint32_t *entry;  // [B]
  uint32_t each;    // 8, 16 or 32: lanes of a warp, and divides the 256-entry chunk
  uint32_t keep;    // 0: CTAs apart from the others take the list
};
enum class Copy { kWarp, kCta, kList };
// Lane i of a group of `each` lanes: how its entry of `len` tokens is copied.
__device__ __forceinline__ Copy copy_of(uint32_t len, const LongList &l) {
  const bool is_long = len > kShortTokens;
  if (!__any_sync(kFull, is_long)) return Copy::kWarp;
  const uint32_t g = threadIdx.x & (l.each - 1);
  uint64_t sum = is_long ? len : 0u;
#pragma unroll
  for (uint32_t o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(kFull, sum, o);
    if (g >= o) sum += y;
  }
  return !is_long ? Copy::kWarp : sum <= l.keep ? Copy::kCta : Copy::kList;
}

__device__ __forceinline__ uint64_t block_sum(uint64_t v, uint64_t *red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  __syncthreads();  // red may still be read by a previous call
  if (lane == 0) red[wid] = v;
  __syncthreads();
  uint64_t t = 0;
#pragma unroll
  for (int w = 0; w < kPackThreads / 32; ++w) t += red[w];
  return t;
}

// One thread per batch entry: its entry (0 tokens and a flag for an index
// out of range); per CTA the sum of its 256 lengths.  With `pre` (more than
// kDirectChunks chunks) the last CTA to finish (a ticket that the context's
// ordered packed deliveries share) turns those sums into exclusive prefixes
// and resets the ticket.
// Chunk `cta` of `ncta` (the CTA's role; the fused GRPO kernel runs it
// beside the advantages).
__device__ __forceinline__ void pack_lengths_cta(const uint64_t *soff, uint64_t nseq,
                                                 const int64_t *idx, uint32_t B, PackEntry *ent,
                                                 uint64_t *part, uint64_t *pre, LongList longs,
                                                 Ctrl *ctrl, uint32_t cta, uint32_t ncta) {
  __shared__ uint64_t red[kPackThreads / 32];
  __shared__ uint32_t ticket;
  const uint64_t k = (uint64_t)cta * kPackThreads + threadIdx.x;
  uint64_t len = 0;
  if (k < B) {
    const int64_t s = idx[k];
    uint64_t a = 0;
    uint32_t seq = kNoSeq;
    if (s >= 0 && (uint64_t)s < nseq) {
      a = soff[s];
      const uint64_t b = soff[s + 1];
      len = b > a ? b - a : 0;
      seq = (uint32_t)s;
    } else {
      flag(ctrl, DEVERR_INDEX, (unsigned long long)s);
    }
    ent[k] = PackEntry{a, seq, (uint32_t)len};
  }
  if (longs.entry) {  // one atomic per warp that has any
    const int lane = threadIdx.x & 31;
    const bool listed = copy_of((uint32_t)len, longs) == Copy::kList;  // the length as stored
    const unsigned m = __ballot_sync(kFull, listed);
    if (m) {
      uint32_t at = lane == 0 ? atomicAdd(&ctrl->pack_long, (uint32_t)__popc(m)) : 0u;
      at = __shfl_sync(kFull, at, 0) + __popc(m & ((1u << lane) - 1u));
      if (listed && at < B) longs.entry[at] = (uint32_t)k;
    }
  }
  const uint64_t sum = block_sum(len, red);
  if (!pre) {
    if (threadIdx.x == 0) part[cta] = sum;
    return;
  }
  if (threadIdx.x == 0) {
    part[cta] = sum;
    __threadfence();
    ticket = atomicAdd(&ctrl->pack_ticket, 1u);
  }
  __syncthreads();
  if (ticket != ncta - 1) return;
  __threadfence();
  // the last CTA: exclusive prefix of the per-CTA sums, kPackThreads at a time
  uint64_t carry = 0;
  for (uint32_t base = 0; base < ncta; base += kPackThreads) {
    const uint32_t i = base + threadIdx.x;
    const uint64_t v = i < ncta ? __ldcg(&part[i]) : 0;
    uint64_t incl = v;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t t = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += t;
    }
    __syncthreads();
    if (lane == 31) red[wid] = incl;
    __syncthreads();
    uint64_t before = carry;
    for (int w = 0; w < wid; ++w) before += red[w];
    if (i < ncta) pre[i] = before + incl - v;
    uint64_t tile = 0;
#pragma unroll
    for (int w = 0; w < kPackThreads / 32; ++w) tile += red[w];
    carry += tile;
  }
  if (threadIdx.x == 0) ctrl->pack_ticket = 0u;  // every CTA has taken its ticket
}

__global__ void __launch_bounds__(kPackThreads)
k_pack_lengths(const uint64_t *soff, uint64_t nseq, const int64_t *idx, uint32_t B, PackEntry *ent,
               uint64_t *part, uint64_t *pre, LongList longs, Ctrl *ctrl) {
  pdl_wait();
  pdl_launch();
  pack_lengths_cta(soff, nseq, idx, B, ent, part, pre, longs, ctrl, blockIdx.x, gridDim.x);
}

// The GRPO step's first kernel: CTAs [0, ngc) compute the group advantages
// (two warps each, so the groups spread over the SMs), the others the
// batch's length pass, which needs no advantage (the gather reads them).
__global__ void __launch_bounds__(kPackThreads)
k_grpo_pack_lengths(const float *r, const uint64_t *goff, uint32_t ng, float eps, float *adv,
                    uint32_t ngc, const uint64_t *soff, uint64_t nseq, const int64_t *idx,
                    uint32_t B, PackEntry *ent, uint64_t *part, uint64_t *pre, LongList longs,
                    Ctrl *ctrl) {
  pdl_wait();
  pdl_launch();
  if (blockIdx.x < ngc) {
    const uint32_t w = threadIdx.x >> 5;
    if (w < kGrpoWarps)
      grpo_groups(r, goff, ng, eps, adv, (uint64_t)blockIdx.x * kGrpoWarps + w,
                  (uint64_t)ngc * kGrpoWarps);
    return;
  }
  pack_lengths_cta(soff, nseq, idx, B, ent, part, pre, longs, ctrl, blockIdx.x - ngc,
                   gridDim.x - ngc);
}

// 4-byte store with the streaming (evict-first) L2 policy: the packed batch
// is written once and read by the learner, not by this kernel.
__device__ __forceinline__ void st_stream32(void *p, uint32_t v, uint64_t pol) {
  asm volatile("st.global.L1::no_allocate.L2::cache_hint.b32 [%0], %1, %2;"
               :: "l"(p), "r"(v), "l"(pol) : "memory");
}

constexpr uint32_t kPackChunk = 4096;  // tokens per bulk copy at most (16 KB of shared memory)
struct PackBuf {
  alignas(16) uint32_t tok[kPackChunk + 8];
  unsigned long long bar;
};

// One CTA copies tokens [c0, c0 + m) of a sequence whose tokens start at src
// to out + c0 (and the value to vout + c0), m <= kPackChunk: the source's
// 16-byte-aligned interior by one bulk copy into shared memory (completion on
// an mbarrier, waited for with a bound), its up to three unaligned tokens at
// either end by plain loads; the destination's aligned interior by 16-byte
// stores read from shared memory at the offset between the two alignments,
// its ends by 4-byte stores.  The value is a fill with the same split, written
// while the copy is in flight.  `uses`: completed phases of the mbarrier.
__device__ __forceinline__ void pack_copy_cta(PackBuf &sm, uint32_t &uses, const int32_t *src,
                                              int32_t *out, float *vout, uint32_t vbits,
                                              uint64_t c0, uint32_t m, uint32_t k, uint64_t pol,
                                              Ctrl *ctrl) {
  const int32_t *sc = src + c0;
  // source: tokens [0, head) and [head + body, m) by plain loads, the
  // 16-byte-aligned [head, head + body) by one bulk copy; token t sits at
  // tok[t + shift], which puts token `head` on a 16-byte boundary
  const uint32_t hs = (uint32_t)(((16u - ((uint32_t)(uintptr_t)sc & 15u)) & 15u) >> 2);
  const uint32_t head = min(hs, m);
  const uint32_t body = (m - head) & ~3u;
  const uint32_t shift = (4u - head) & 3u;
  if (threadIdx.x == 0 && body) {
    // the previous chunk's reads of tok (generic proxy) come before this
    // copy's writes (async proxy)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_tx(&sm.bar, body * 4);
    bulk_load(&sm.tok[head + shift], sc + head, body * 4, &sm.bar, pol);
  }
  const uint32_t tail0 = head + body;
  if (threadIdx.x < head) sm.tok[threadIdx.x + shift] = (uint32_t)sc[threadIdx.x];
  if (threadIdx.x < m - tail0)
    sm.tok[tail0 + threadIdx.x + shift] = (uint32_t)sc[tail0 + threadIdx.x];
  // values: the same split on the destination
  if (vout) {
    float *vo = vout + c0;
    const uint32_t hv = min((uint32_t)(((16u - ((uint32_t)(uintptr_t)vo & 15u)) & 15u) >> 2), m);
    const uint32_t qv = (m - hv) >> 2;
    if (threadIdx.x < hv) st_stream32(vo + threadIdx.x, vbits, pol);
    const uint4 v4 = make_uint4(vbits, vbits, vbits, vbits);
    for (uint32_t i = threadIdx.x; i < qv; i += kPackThreads)
      st_stream(reinterpret_cast<uint4 *>(vo + hv) + i, v4, pol);
    const uint32_t tv = hv + 4 * qv;
    if (threadIdx.x < m - tv) st_stream32(vo + tv + threadIdx.x, vbits, pol);
  }
  if (body) {
    if (!mbar_wait(&sm.bar, uses & 1u, kPackWaitNs)) {
      if (threadIdx.x == 0) flag(ctrl, DEVERR_TIMEOUT, k);
      mbar_wait(&sm.bar, uses & 1u, kPackWaitNs);  // bounded: the copy lands first
    }
    ++uses;
  }
  __syncthreads();
  // destination: 16-byte stores of its aligned interior
  int32_t *oc = out + c0;
  const uint32_t ho = min((uint32_t)(((16u - ((uint32_t)(uintptr_t)oc & 15u)) & 15u) >> 2), m);
  const uint32_t q = (m - ho) >> 2;
  if (threadIdx.x < ho) st_stream32(oc + threadIdx.x, sm.tok[threadIdx.x + shift], pol);
  // the four tokens of a store straddle two 16-byte words of shared memory,
  // which are read whole (four 4-byte reads would conflict four ways each)
  const uint32_t off = (ho + shift) & 3u;
  const uint4 *words = reinterpret_cast<const uint4 *>(sm.tok) + (ho + shift) / 4;
  for (uint32_t i = threadIdx.x; i < q; i += kPackThreads) {
    uint4 x = words[i];
    if (off) {
      const uint4 y = words[i + 1];
      x = off == 1 ? make_uint4(x.y, x.z, x.w, y.x)
        : off == 2 ? make_uint4(x.z, x.w, y.x, y.y) : make_uint4(x.w, y.x, y.y, y.z);
    }
    st_stream(reinterpret_cast<uint4 *>(oc + ho) + i, x, pol);
  }
  const uint32_t to = ho + 4 * q;
  if (threadIdx.x < m - to)
    st_stream32(oc + to + threadIdx.x, sm.tok[to + threadIdx.x + shift], pol);
  __syncthreads();  // tok is refilled by the next chunk
}

__device__ __forceinline__ void pack_buf_init(PackBuf &sm) {
  if (threadIdx.x == 0) {
    mbar_init(&sm.bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
}

// Output offset of batch entry k (the CTA): the prefix of its 256-entry chunk
// (from `pre`, or the chunk sums before it) plus the lengths before it in the
// chunk, in one round trip and a block sum.
__device__ __forceinline__ uint64_t pack_offset_cta(const PackEntry *ent, const uint64_t *part,
                                                    const uint64_t *pre, uint32_t k,
                                                    uint64_t *red) {
  const uint32_t c = k / kPackThreads;
  const uint32_t j = c * kPackThreads + threadIdx.x;
  uint64_t v = j < k ? ent[j].len : 0;
  if (pre) {
    if (threadIdx.x == 0) v += pre[c];
  } else if (threadIdx.x < c) {
    v += part[threadIdx.x];  // c <= kDirectChunks = the block size
  }
  return block_sum(v, red);
}

// A CTA per sequence, in chunks of kPackChunk tokens, or (SPLIT) gridDim.y
// CTAs that take its chunks of `chunk` tokens in turn.  The first CTA of each
// entry writes its output offset, that of the last entry out_off[batch] = the
// total, and flags an overflow.
// 32 registers, 16.5 KB: 8 CTAs per SM keep more copies in flight than 6 at 38
// registers (8,192 sequences of 128 to 4,096 tokens 34.4 us, 37.3).  Neither
// this kernel nor k_pack_gather_short releases the next one early: its CTAs, which
// can only wait, took places from the last waves (that call 33.6 us, with its
// lengths and advantages 37.3, 39.3 before; 65,536 short sequences 28.0, 28.9).
template <bool SPLIT>
__global__ void __launch_bounds__(kPackThreads, 8)
k_pack_gather(const int32_t *tokens, const PackEntry *ent, const uint64_t *part,
              const uint64_t *pre, uint32_t B, const float *sv, int32_t *otok, uint64_t *ooff,
              float *osv, uint64_t cap, uint32_t chunk, Ctrl *ctrl) {
  __shared__ uint64_t red[kPackThreads / 32];
  __shared__ PackBuf sm;
  pack_buf_init(sm);
  uint32_t uses = 0;
  const uint64_t pol = policy_stream();
  pdl_wait();
  const uint32_t k = blockIdx.x;
  const uint64_t first = SPLIT ? (uint64_t)blockIdx.y * chunk : 0;
  if (SPLIT && blockIdx.y && ent[k].len <= first) return;  // no chunk is left
  const PackEntry e = ent[k];
  const uint64_t dst = pack_offset_cta(ent, part, pre, k, red);
  if (threadIdx.x == 0 && (!SPLIT || blockIdx.y == 0)) {
    ooff[k] = dst;
    if (k == B - 1) {
      ooff[B] = dst + e.len;
      if (dst + e.len > cap) flag(ctrl, DEVERR_OVERFLOW, (unsigned long long)(dst + e.len));
    }
  }
  if (e.len == 0 || dst >= cap) return;
  const float value = osv && e.seq != kNoSeq ? __ldcg(&sv[e.seq]) : 0.f;
  const uint64_t n = min((uint64_t)e.len, cap - dst);
  const uint32_t each = SPLIT ? chunk : kPackChunk;
  for (uint64_t c0 = first; c0 < n; c0 += (uint64_t)(SPLIT ? gridDim.y : 1) * each)
    pack_copy_cta(sm, uses, tokens + e.src, otok + dst, osv ? osv + dst : nullptr,
                  __float_as_uint(value), c0, (uint32_t)min((uint64_t)each, n - c0), k, pol,
                  ctrl);
}

// Short sequences, many of them: a CTA takes 8, 16 or 32 neighbouring entries,
// resolves the output offset of the first as above and those of the others from
// their lengths, and each warp copies its entries by 4-byte loads and stores,
// kShortUnroll in flight per lane.  A long entry (above kShortTokens) is copied by
// a whole CTA as in k_pack_gather: by its own one while that has little of such
// work (LongList::keep), else by the one that its place in the lengths kernel's
// list names, so that long sequences run side by side however they lie in the
// batch; batches of less than a wave of CTAs get kServersPerSm CTAs per SM for the
// list alone.  Bound by the chain of a CTA (entries, offset, tokens) that few
// waves hide.  Calls in a row, in us, here, (with the long ones left to the CTA of
// their neighbours) and [a CTA each, k_pack_gather]:
//   lengths U[8, 256]        65,536: 22.9 (22.5) [171]     4,096: 5.0 (4.8) [13.4]
//   U[64, 1,024]              8,192: 12.0 (11.7) [25.8]
//   2% of 16,000, first, 64   1,024: 7.2 (26.7) [7.2]     65,536: 50 (430) [192]
//   10% of 8,000 at random    1,024: 5.9 (10.0) [8.7]      8,192: 14.1 (19.2) [30.0]
//   50% of 1,500 at random    8,192: 16.7 (15.6) [25.7]   65,536: 133 (116) [191]
// kKeepTokens 12,288 or 4,096: 5% slower on one of the last three or another.
constexpr int kShortUnroll = 8;
constexpr uint32_t kPackWarps = kPackThreads / 32;
constexpr uint32_t kShortEntries = 32;  // per CTA at most: the lanes of a warp
constexpr uint32_t kServersPerSm = 4;
constexpr uint32_t kKeepTokens = 6144;

__global__ void __launch_bounds__(kPackThreads, 6)
k_pack_gather_short(const int32_t *tokens, const PackEntry *ent, const uint64_t *part,
                    const uint64_t *pre, uint32_t B, const float *sv, int32_t *otok,
                    uint64_t *ooff, float *osv, uint64_t cap, uint32_t server0,
                    LongList longs, Ctrl *ctrl) {
  __shared__ uint64_t red[kPackThreads / 32];
  __shared__ PackBuf sm;
  __shared__ uint32_t s_listed;
  pack_buf_init(sm);
  uint32_t uses = 0;
  const int lane = threadIdx.x & 31;
  const uint32_t warp = threadIdx.x >> 5;
  const uint64_t pol = policy_stream();
  pdl_wait();
  const uint32_t each = longs.each, per_warp = each / kPackWarps;
  const uint64_t first = (uint64_t)blockIdx.x * each;
  const uint32_t k0 = (uint32_t)min(first, (uint64_t)B);
  const uint32_t ne = min(each, B - k0);  // 0: a CTA for the list alone
  const uint32_t server = blockIdx.x - server0, nserver = gridDim.x - server0;
  const uint32_t next = !ne && server < B ? longs.entry[server] : 0u;  // beside the length
  if (threadIdx.x == 0) s_listed = min(__ldcg(&ctrl->pack_long), B);
  if (!ne) __syncthreads();  // else one follows
  // lane i of every warp: entry k0 + i, and its value
  PackEntry mine{0, kNoSeq, 0};
  if ((uint32_t)lane < ne) mine = ent[k0 + lane];
  float value = 0.f;
  if (osv && mine.seq != kNoSeq) value = __ldcg(&sv[mine.seq]);
  if (ne) {
    uint64_t dst = mine.len;  // inclusive, then exclusive prefix
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(kFull, dst, o);
      if (lane >= o) dst += y;
    }
    dst += pack_offset_cta(ent, part, pre, k0, red) - mine.len;
    if (warp == 0 && (uint32_t)lane < ne) {
      ooff[k0 + lane] = dst;
      if (k0 + lane == B - 1) {
        ooff[B] = dst + mine.len;
        if (dst + mine.len > cap)
          flag(ctrl, DEVERR_OVERFLOW, (unsigned long long)(dst + mine.len));
      }
    }
    for (uint32_t i = warp * per_warp; i < min(ne, (warp + 1) * per_warp); ++i) {
      const uint32_t len = __shfl_sync(kFull, mine.len, i);
      const uint64_t d = __shfl_sync(kFull, dst, i);
      const uint64_t src = __shfl_sync(kFull, mine.src, i);
      const uint32_t vbits = __float_as_uint(__shfl_sync(kFull, value, i));
      if (len > kShortTokens || d >= cap) continue;
      const uint32_t n = (uint32_t)min((uint64_t)len, cap - d);
      const int32_t *sc = tokens + src;
      for (uint32_t t0 = lane; t0 < n; t0 += 32 * kShortUnroll) {
        int32_t v[kShortUnroll];
#pragma unroll
        for (int u = 0; u < kShortUnroll; ++u)
          if (t0 + u * 32 < n) v[u] = __ldg(sc + t0 + u * 32);
#pragma unroll
        for (int u = 0; u < kShortUnroll; ++u)
          if (t0 + u * 32 < n) {
            st_stream32(otok + d + t0 + u * 32, (uint32_t)v[u], pol);
            if (osv) st_stream32(osv + d + t0 + u * 32, vbits, pol);
          }
      }
    }
    const Copy how = copy_of(mine.len, longs);
    for (uint32_t left = __ballot_sync(kFull, how == Copy::kCta); left; left &= left - 1) {
      const int i = __ffs(left) - 1;  // the same in every warp
      const uint32_t len = __shfl_sync(kFull, mine.len, i);
      const uint64_t d = __shfl_sync(kFull, dst, i);
      const uint64_t src = __shfl_sync(kFull, mine.src, i);
      const float val = __shfl_sync(kFull, value, i);
      if (d >= cap) continue;
      const uint64_t n = min((uint64_t)len, cap - d);
      for (uint64_t c0 = 0; c0 < n; c0 += kPackChunk)
        pack_copy_cta(sm, uses, tokens + src, otok + d, osv ? osv + d : nullptr,
                      __float_as_uint(val), c0, (uint32_t)min((uint64_t)kPackChunk, n - c0), k0 + i,
                      pol, ctrl);
    }
  }
  if (blockIdx.x >= server0) {
    const uint32_t listed = s_listed;  // thread 0's, so that all of the CTA go by one value
    for (uint32_t i = server; i < listed; i += nserver) {
      const uint32_t k = !ne && i == server ? next : longs.entry[i];
      const PackEntry e = ent[k];
      const uint64_t d = pack_offset_cta(ent, part, pre, k, red);
      if (d >= cap) continue;
      const float val = osv && e.seq != kNoSeq ? __ldcg(&sv[e.seq]) : 0.f;
      const uint64_t n = min((uint64_t)e.len, cap - d);
      for (uint64_t c0 = 0; c0 < n; c0 += kPackChunk)
        pack_copy_cta(sm, uses, tokens + e.src, otok + d, osv ? osv + d : nullptr,
                      __float_as_uint(val), c0, (uint32_t)min((uint64_t)kPackChunk, n - c0), k,
                      pol, ctrl);
    }
    // the last CTA that is done with the list clears it for the next call
    if (listed && threadIdx.x == 0 && atomicInc(&ctrl->pack_left, nserver - 1) == nserver - 1)
      ctrl->pack_long = 0;
  }
}

}  // namespace

cudaError_t launch_grpo(edp_ctx *c, const float *r, const uint64_t *goff, uint32_t ng,
                        float eps, float *adv, cudaStream_t s) {
  uint64_t blocks = (ng + kGrpoWarps - 1) / kGrpoWarps;
  if (blocks > 16ull * c->coop_sms) blocks = 16ull * c->coop_sms;
  // Launched plainly (its pdl_wait / pdl_launch are then no-ops): released early
  // behind a gather of thousands of CTAs, advantages then delivery take 48.1 us
  // for 512 x 16 responses instead of 38.0.
  k_grpo<<<dim3((unsigned)blocks), dim3(kGrpoThreads), 0, s>>>(r, goff, ng, eps, adv);
  return cudaGetLastError();
}

namespace {

// A wave of gather CTAs.
uint64_t pack_wave(const edp_ctx *c) { return 6ull * (uint64_t)c->coop_sms; }

struct PackPlan {
  PackEntry *ent;
  uint64_t *part, *pre;
  LongList longs;  // entry null: k_pack_gather
  uint32_t G;
};

cudaError_t pack_plan(edp_ctx *c, uint32_t B, uint64_t cap, bool host_out, cudaStream_t s,
                      PackPlan *p) {
  p->G = (B + kPackThreads - 1) / kPackThreads;
  const size_t ent_bytes = ((size_t)B * sizeof(PackEntry) + 255) & ~(size_t)255;
  void *blk = nullptr;
  const cudaError_t e = ctx_scratch(
      c, ent_bytes + 2 * (size_t)p->G * sizeof(uint64_t) + (size_t)B * sizeof(uint32_t), s, &blk);
  if (e != cudaSuccess) return e;
  uint8_t *scr = (uint8_t *)blk;
  p->ent = (PackEntry *)scr;
  p->part = (uint64_t *)(scr + ent_bytes);
  p->pre = p->G > kDirectChunks ? p->part + p->G : nullptr;
  p->longs = LongList{};
  const uint64_t wave = pack_wave(c);
  if (B > wave && cap / B <= kShortTokens && !host_out) {  // k_pack_gather_short (launch_gather)
    p->longs.entry = (uint32_t *)(p->part + 2 * (size_t)p->G);
    uint32_t &each = p->longs.each = kShortEntries;
    while (each > kPackWarps && B < 2 * wave * each) each /= 2;
    p->longs.keep = (B + each - 1) / each < wave ? 0 : kKeepTokens;
  }
  return cudaSuccess;
}

// How the batch is copied follows from its size and from the room the caller
// gave it, which bounds the mean length (the lengths are on the device):
//  - more sequences than about a wave of CTAs, at most kShortTokens of room
//    each on average: k_pack_gather_short (1,024 sequences U[1, 256] 3.9 us, 4.9
//    with a CTA each; exponential lengths of mean 512 5.7, 5.4).  Not into
//    page-locked host memory, where its 4-byte stores of any alignment make more
//    and smaller writes on the link: 4,096 sequences U[64, 1,024] 154 us, 111 with a
//    CTA each, 16,384 U[8, 256] 153, 126;
//  - otherwise a CTA per sequence, and where that leaves the chip idle and
//    the room allows long sequences, several CTAs per sequence on chunks of
//    1,024 tokens or more (64 sequences U[2,048, 32,768]: 5.9 us, 12.3 with
//    one CTA each; 8 of them 3.9, 11.4).
cudaError_t launch_gather(edp_ctx *c, const PackPlan &p, const int32_t *tokens, uint32_t B,
                          const float *sv, int32_t *otok, uint64_t *ooff, float *osv,
                          uint64_t cap, cudaStream_t s) {
  const uint64_t wave = pack_wave(c);
  const uint64_t room = cap / B;
  if (p.longs.entry) {
    const uint32_t ctas = (B + p.longs.each - 1) / p.longs.each;
    const bool apart = !p.longs.keep;
    return launch_pdl(k_pack_gather_short,
                      dim3(apart ? ctas + kServersPerSm * (unsigned)c->coop_sms : ctas),
                      dim3(kPackThreads), s, tokens, (const PackEntry *)p.ent,
                      (const uint64_t *)p.part, (const uint64_t *)p.pre, B, sv, otok, ooff, osv,
                      cap, apart ? ctas : 0u, p.longs, c->ctrl);
  }
  uint32_t chunk = kPackChunk;
  while (chunk > 1024 && (uint64_t)B * ((room + chunk - 1) / chunk) < wave) chunk /= 2;
  uint64_t split = (room + chunk - 1) / chunk;
  const uint64_t most = 4 * wave / B;  // CTAs without a chunk leave at once
  if (split > most) split = most;
  if (split > 1024) split = 1024;
  auto kern = split > 1 ? k_pack_gather<true> : k_pack_gather<false>;
  return launch_pdl(kern, dim3(B, split > 1 ? (unsigned)split : 1u), dim3(kPackThreads), s, tokens,
                    (const PackEntry *)p.ent, (const uint64_t *)p.part,
                    (const uint64_t *)p.pre, B, sv, otok, ooff, osv, cap, chunk, c->ctrl);
}

}  // namespace

cudaError_t launch_pack(edp_ctx *c, const int32_t *tokens, const uint64_t *soff,
                        uint64_t nseq, const int64_t *idx, uint32_t B, const float *sv,
                        int32_t *otok, uint64_t *ooff, float *osv, uint64_t cap, bool host_out,
                        cudaStream_t s) {
  PackPlan p;
  cudaError_t e = pack_plan(c, B, cap, host_out, s, &p);
  if (e != cudaSuccess) return e;
  e = launch_pdl(k_pack_lengths, dim3(p.G), dim3(kPackThreads), s, soff, nseq, idx, B,
                 p.ent, p.part, p.pre, p.longs, c->ctrl);
  if (e != cudaSuccess) return e;
  return launch_gather(c, p, tokens, B, sv, otok, ooff, osv, cap, s);
}

cudaError_t launch_grpo_pack(edp_ctx *c, const float *r, const uint64_t *goff, uint32_t ng,
                             float eps, float *adv, const int32_t *tokens,
                             const uint64_t *soff, uint64_t nseq, const int64_t *idx,
                             uint32_t B, int32_t *otok, uint64_t *ooff, float *osv,
                             uint64_t cap, bool host_out, cudaStream_t s) {
  PackPlan p;
  cudaError_t e = pack_plan(c, B, cap, host_out, s, &p);
  if (e != cudaSuccess) return e;
  uint64_t ngc = (ng + kGrpoWarps - 1) / kGrpoWarps;
  if (ngc > 16ull * c->coop_sms) ngc = 16ull * c->coop_sms;
  e = launch_pdl(k_grpo_pack_lengths, dim3((unsigned)(ngc + p.G)), dim3(kPackThreads), s, r,
                 goff, ng, eps, adv, (uint32_t)ngc, soff, nseq, idx, B, p.ent, p.part, p.pre,
                 p.longs, c->ctrl);
  if (e != cudaSuccess) return e;
  return launch_gather(c, p, tokens, B, adv, otok, ooff, osv, cap, s);
}

}  // namespace edp
