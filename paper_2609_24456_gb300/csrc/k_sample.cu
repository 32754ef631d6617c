// k_sample.cu -- the uniform replay sampler and the on-policy shuffle.
//
// Uniform: index_k = slot(mulhi64(Philox(k; seed, round, stream 0), n_valid)),
// one thread per index, no shared state.
//
// Shuffle (mini-batch partition with shuffling, Sec. 2.2 on-policy
// delivery): a random-key sort of the logical offsets j < n by
// (Philox(j; seed, round, stream 2), j), as three kernels chained with
// programmatic dependent launch (no grid-wide barrier):
//   keys     draw key_j, count it into bucket key_j >> (64 - log2 nb); the
//            count it found is its place in the bucket
//   scatter  every CTA scans the nb <= 8192 counts in shared memory (the
//            bucket starts), then puts its (key, j) pairs in their places
//   rank     a CTA takes whole buckets (a few hundred pairs), which lie
//            side by side, into shared memory: rank_j = bucket start +
//            #{members < (key_j, j)}; idx[rank_j] = slot of offset j;
//            re-zero the counters for the next call
// With nb ~ n/4 buckets (up to 32,768 elements) a bucket holds ~4 keys; above
// that it holds n / 8192.  The result does not depend on the order of the
// counting.  Bound by the latency of the three kernels' chains up to ~100,000
// elements, by the counting atomics and the 16-byte scattered writes above.
// Calls in a row: 32,768 elements 7.8 us, 262,144 20.1 us, 1,048,576 78.6 us;
// 13.3, 238.5 and 3,366 us when every element read its bucket from the L2 and
// the counts were scanned from 4-byte loads.
#include "edp_internal.cuh"

namespace edp {
namespace {

__global__ void k_sample_uniform(uint32_t B, uint64_t seed, uint64_t round, uint64_t n_valid,
                                 uint64_t oldest, uint64_t cap, int64_t *idx) {
  pdl_wait();
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < B;
       k += gridDim.x * blockDim.x) {
    const uint64_t off = mulhi64(philox_u64(seed, k, round, 0), n_valid);
    idx[k] = (int64_t)((oldest + off) % cap);
  }
  pdl_launch();
}

constexpr int kPermThreads = 256;
constexpr uint32_t kMaxBuckets = 8192;  // bucket starts scanned in shared memory

}  // namespace

size_t perm_scratch_bytes(uint32_t n) {
  return 3 * (kMaxBuckets + 64) * sizeof(uint32_t) + (size_t)n * (8 + 8 + 4 + 8) + 256;
}
size_t perm_zeroed_bytes() { return kMaxBuckets * sizeof(uint32_t); }

namespace {

struct PermScratch {
  uint32_t *count;   // [nb], zero between calls
  uint32_t *start;   // [nb + 1] bucket starts
  uint4 *pairs;      // [n] bucketed: key (two words), offset
  uint64_t *keys;    // [n]
  uint32_t *place;   // [n] place within the bucket
};

__device__ __forceinline__ uint32_t bucket_of(uint64_t key, int lg) {
  return lg ? (uint32_t)(key >> (64 - lg)) : 0u;
}

// Elements per thread whose loads (and counts) are in flight together.
constexpr int kPermBatch = 4;

__global__ void __launch_bounds__(kPermThreads)
k_perm_keys(uint32_t n, uint64_t seed, uint64_t round, int lg, PermScratch sc) {
  pdl_wait();
  pdl_launch();
  const uint64_t stride = (uint64_t)gridDim.x * kPermThreads;
  for (uint64_t j0 = blockIdx.x * kPermThreads + threadIdx.x; j0 < n;
       j0 += kPermBatch * stride) {
    uint32_t place[kPermBatch];
#pragma unroll
    for (int u = 0; u < kPermBatch; ++u) {
      const uint64_t j = j0 + u * stride;
      if (j < n) {
        const uint64_t key = philox_u64(seed, (uint32_t)j, round, 2);
        sc.keys[j] = key;
        place[u] = atomicAdd(&sc.count[bucket_of(key, lg)], 1u);
      }
    }
#pragma unroll
    for (int u = 0; u < kPermBatch; ++u) {
      const uint64_t j = j0 + u * stride;
      if (j < n) sc.place[j] = place[u];
    }
  }
}

__global__ void __launch_bounds__(kPermThreads)
k_perm_scatter(uint32_t n, int lg, PermScratch sc) {
  // Exclusive scan of the bucket counts: a warp takes 1,024 consecutive ones as
  // rows of 16-byte vectors, all in flight before the first is used, and scans
  // the vectors' sums by shuffles (48 a lane; 96 loads and stores of shared
  // memory when each thread scanned 32 counts there).
  __shared__ __align__(16) uint32_t start[kMaxBuckets];
  __shared__ uint32_t warp_tot[kPermThreads / 32];
  const uint32_t nb = 1u << lg;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int kVecs = kMaxBuckets / 4 / kPermThreads;
  const uint32_t v0 = wid * 32 * kVecs + lane;
  pdl_wait();
  pdl_launch();
  uint4 c4[kVecs];
#pragma unroll
  for (int u = 0; u < kVecs; ++u) {
    const uint32_t i = 4 * (v0 + u * 32);
    // counts past nb stay zero between calls: whole vectors may be read
    c4[u] = i < nb ? __ldcg(reinterpret_cast<const uint4 *>(sc.count + i))
                   : make_uint4(0u, 0u, 0u, 0u);
  }
  uint32_t before[kVecs], run = 0;
#pragma unroll
  for (int u = 0; u < kVecs; ++u) {
    const uint32_t sum = c4[u].x + c4[u].y + c4[u].z + c4[u].w;
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    before[u] = run + incl - sum;
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) warp_tot[wid] = run;
  __syncthreads();
  uint32_t acc = 0;
#pragma unroll
  for (int w = 0; w < kPermThreads / 32; ++w) acc += w < wid ? warp_tot[w] : 0u;
#pragma unroll
  for (int u = 0; u < kVecs; ++u) {
    uint4 at;
    at.x = acc + before[u];
    at.y = at.x + c4[u].x;
    at.z = at.y + c4[u].y;
    at.w = at.z + c4[u].z;
    reinterpret_cast<uint4 *>(start)[v0 + u * 32] = at;
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    for (uint32_t i = threadIdx.x; i < nb; i += kPermThreads) sc.start[i] = start[i];
    if (threadIdx.x == 0) sc.start[nb] = n;
  }
  const uint64_t stride = (uint64_t)gridDim.x * kPermThreads;
  for (uint64_t j0 = blockIdx.x * kPermThreads + threadIdx.x; j0 < n;
       j0 += kPermBatch * stride) {
    uint64_t key[kPermBatch];
    uint32_t place[kPermBatch];
#pragma unroll
    for (int u = 0; u < kPermBatch; ++u) {
      const uint64_t j = j0 + u * stride;
      key[u] = j < n ? __ldcg(&sc.keys[j]) : 0;
      place[u] = j < n ? __ldcg(&sc.place[j]) : 0;
    }
#pragma unroll
    for (int u = 0; u < kPermBatch; ++u) {
      const uint64_t j = j0 + u * stride;
      if (j < n)
        sc.pairs[start[bucket_of(key[u], lg)] + place[u]] =
            make_uint4((uint32_t)key[u], (uint32_t)(key[u] >> 32), (uint32_t)j, 0u);
    }
  }
}

// The pairs that a CTA ranks are whole buckets, taken through shared memory
// kRankTile at a time (one tile unless the buckets are large; 1,024: 262,144
// elements 21.1 us instead of 20.1, 1,048,576 82.4 instead of 78.6).
constexpr uint32_t kRankTile = 512;
constexpr uint32_t kRankBuckets = 128;  // at most per CTA: a bucket holds over 2 pairs on average
// Pairs a CTA is given on average: more, smaller CTAs while the buckets are
// small (32,768 pairs: 7.8 us per shuffle with 128, 8.9 with 256, 8.2 with
// 64), a thread each above that (262,144: 20.1 with 256, 21.4 with 128).
constexpr uint32_t kRankFew = 65536;
constexpr uint32_t rank_want(uint32_t n) { return n <= kRankFew ? 128 : kPermThreads; }

__global__ void __launch_bounds__(kPermThreads)
k_perm_rank(uint32_t n, int lg, uint32_t per_cta, PermScratch sc, uint64_t oldest, uint64_t cap,
            int64_t *idx) {
  __shared__ uint64_t tkey[kRankTile];
  __shared__ __align__(16) uint32_t ttop[kRankTile];  // high words; ~0 past the pairs
  __shared__ uint32_t tj[kRankTile];
  __shared__ uint32_t bstart[kRankBuckets + 1];
  const uint32_t nb = 1u << lg;
  const uint32_t b0 = blockIdx.x * per_cta, b1 = min(nb, b0 + per_cta);
  pdl_wait();
  pdl_launch();
  for (uint32_t i = threadIdx.x; i <= b1 - b0; i += kPermThreads)
    bstart[i] = __ldcg(&sc.start[b0 + i]);
  __syncthreads();
  const uint32_t lo = bstart[0], hi = bstart[b1 - b0];
  constexpr int kEach = kRankTile / kPermThreads;
  for (uint64_t e0 = lo; e0 < hi; e0 += kRankTile) {  // the pairs being ranked
    uint64_t key[kEach];
    uint32_t j[kEach], blo[kEach], bhi[kEach], r[kEach];
#pragma unroll
    for (int u = 0; u < kEach; ++u) {
      const uint64_t p = e0 + u * kPermThreads + threadIdx.x;
      r[u] = blo[u] = bhi[u] = j[u] = 0;
      key[u] = 0;
      if (p < hi) {
        const uint4 v = __ldcg(&sc.pairs[p]);
        key[u] = ((uint64_t)v.y << 32) | v.x;
        j[u] = v.z;
        const uint32_t b = bucket_of(key[u], lg) - b0;
        blo[u] = bstart[b];
        bhi[u] = bstart[b + 1];
      }
    }
    for (uint64_t t0 = lo; t0 < hi; t0 += kRankTile) {  // the pairs compared with
      const uint32_t tlo = (uint32_t)t0, thi = (uint32_t)min((uint64_t)hi, t0 + kRankTile);
      __syncthreads();  // the tile before is no longer read
      if (t0 == e0) {
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
          tkey[u * kPermThreads + threadIdx.x] = key[u];
          tj[u * kPermThreads + threadIdx.x] = j[u];
          ttop[u * kPermThreads + threadIdx.x] = bhi[u] > blo[u] ? (uint32_t)(key[u] >> 32) : ~0u;
        }
      } else {
        for (uint32_t i = threadIdx.x; i < kRankTile; i += kPermThreads) {
          ttop[i] = ~0u;
          if (i >= thi - tlo) continue;
          const uint4 v = __ldcg(&sc.pairs[tlo + i]);
          tkey[i] = ((uint64_t)v.y << 32) | v.x;
          tj[i] = v.z;
          ttop[i] = v.y;
        }
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kEach; ++u) {
        if (max(blo[u], tlo) >= min(bhi[u], thi)) continue;
        const uint32_t a = max(blo[u], tlo) - tlo, z = min(bhi[u], thi) - tlo;
        // By the high words, four at a time: those before `a` in the first
        // four are of lower buckets, hence less, those from `z` on never.
        const uint32_t top = (uint32_t)(key[u] >> 32);
        uint32_t less = 0, most = 0;
        for (uint32_t i = a & ~3u; i < z; i += 4) {
          const uint4 v = *reinterpret_cast<const uint4 *>(ttop + i);
          less += (v.x < top) + (v.y < top) + (v.z < top) + (v.w < top);
          most += (v.x <= top) + (v.y <= top) + (v.z <= top) + (v.w <= top);
        }
        if (most - less == (t0 == e0 ? 1u : 0u)) {
          r[u] += less - (a & 3u);
        } else {  // another key with this high word: in full, equal ones by offset
          for (uint32_t i = a; i < z; ++i)
            r[u] += tkey[i] < key[u] || (tkey[i] == key[u] && tj[i] < j[u]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kEach; ++u)
      if (bhi[u] > blo[u]) {
        const uint64_t s2 = oldest + j[u];  // < 2 cap
        idx[blo[u] + r[u]] = (int64_t)(s2 >= cap ? s2 - cap : s2);
      }
  }
  // this kernel reads only the bucket starts: the counters can be cleared
  // for the next call
  for (uint32_t b = b0 + threadIdx.x; b < b1; b += kPermThreads) sc.count[b] = 0;
}

}  // namespace

cudaError_t launch_sample_uniform(edp_ctx *c, uint32_t B, uint64_t seed,
                                  uint64_t round, int64_t *idx, cudaStream_t s) {
  samples_on(c, s);
  const uint64_t size = c->total < c->cap ? c->total : c->cap;
  const uint64_t oldest = (c->total - size) % c->cap;
  const uint64_t nv = size - c->defer;
  const unsigned threads = 128;
  unsigned blocks = (B + threads - 1) / threads;
  if (blocks > 4096) blocks = 4096;
  return launch_pdl(k_sample_uniform, dim3(blocks), dim3(threads), s, B, seed,
                    round, nv, oldest, c->cap, idx);
}

cudaError_t launch_permute(edp_ctx *c, uint32_t n, uint64_t seed,
                           uint64_t round, int64_t *idx, cudaStream_t s) {
  int lg = 0;
  while ((1ull << (lg + 2)) < n && (1u << lg) < kMaxBuckets) ++lg;  // nb ~ n/4
  const uint32_t nb = 1u << lg;
  void *block = nullptr;
  const cudaError_t ge = ctx_perm_scratch(c, perm_scratch_bytes(n), s, &block);
  if (ge != cudaSuccess) return ge;
  uint8_t *base = (uint8_t *)block;
  PermScratch sc;
  sc.count = (uint32_t *)base;  // the zeroed head of the block
  sc.start = sc.count + kMaxBuckets;
  sc.pairs = (uint4 *)(base + 3 * (kMaxBuckets + 64) * sizeof(uint32_t));
  sc.keys = (uint64_t *)(sc.pairs + n);
  sc.place = (uint32_t *)(sc.keys + n);
  const uint64_t size = c->total < c->cap ? c->total : c->cap;
  const uint64_t oldest = (c->total - size) % c->cap;
  uint64_t grid = (n + (uint64_t)kPermThreads - 1) / kPermThreads;
  if (grid > 4ull * c->coop_sms) grid = 4ull * c->coop_sms;
  uint32_t per_cta = (uint32_t)((uint64_t)rank_want(n) * nb / n);
  if (per_cta < 1) per_cta = 1;
  if (per_cta > kRankBuckets) per_cta = kRankBuckets;
  const dim3 g((unsigned)grid), blk(kPermThreads);
  cudaError_t e = launch_pdl(k_perm_keys, g, blk, s, n, seed, round, lg, sc);
  if (e == cudaSuccess) e = launch_pdl(k_perm_scatter, g, blk, s, n, lg, sc);
  if (e == cudaSuccess)
    e = launch_pdl(k_perm_rank, dim3((nb + per_cta - 1) / per_cta), blk, s, n, lg, per_cta, sc,
                   oldest, c->cap, idx);
  return e;
}

}  // namespace edp
