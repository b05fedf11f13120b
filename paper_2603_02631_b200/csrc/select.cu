// Chunk pooling, top-k chunk selection and span compaction (Appendix A.1.2, Section 3.2).
// These steps touch a few hundred KB at most; they are latency-bound and each is a single launch.
#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace spf {
namespace {

// ------------------------------------------------------------------------------------------------
// Pooling.  The mean over a chunk of the w-wide window sums is a sum over the tokens in reach, each times the number of the
// chunk's windows that it lies in, so a chunk of 32 with w = 13 reads 44 values once instead of 13 values for each of 32
// tokens.  A warp per chunk adds up in a fixed order, so the result does not depend on scheduling.
// ------------------------------------------------------------------------------------------------
constexpr int kPoolWarps = 8;

struct PoolRule {
  int half, chunk;
  float inv_w;
  bool in_range_divisor;      // the window's divisor: always w (zeros beyond the ends), or the number of tokens it covers
};

__device__ __forceinline__ float warp_total(float x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

// Score of a chunk window by window: where windows reach beyond the prompt's ends and each has a divisor of its own, and where
// the weighted sum below, up to min(w, chunk) times larger than what the windows' means add up to, has overflowed.
__device__ __noinline__ float pool_by_windows(const float* importance, int64_t n_tokens, const PoolRule& r, int64_t lo, int64_t hi) {
  float sum = 0.f;
  for (int64_t s = lo + (threadIdx.x & 31); s < hi; s += 32) {
    const int64_t a = max(s - r.half, (int64_t)0), b = min(s + r.half, n_tokens - 1);
    float win = 0.f;
    for (int64_t t = a; t <= b; ++t) win += __ldcg(importance + t);
    sum += r.in_range_divisor ? win / (float)(b - a + 1) : win * r.inv_w;
  }
  return warp_total(sum) / (float)(hi - lo);
}

__device__ __forceinline__ bool is_finite(float x) { return fabsf(x) < INFINITY; }

// Score of chunk j, in every lane.  Int counts tokens of a chunk and its surroundings: 32 bits unless the chunk is longer than
// kShortChunk.
constexpr int kShortChunk = 1 << 26;

template <class Int>
__device__ __forceinline__ float pool_chunk(const float* __restrict__ importance, int64_t n_tokens, const PoolRule& r, int64_t j) {
  const int64_t lo = j * r.chunk, rest = n_tokens - lo;
  const float* from = importance + lo;
  const Int size = (Int)min((int64_t)r.chunk, rest);
  const Int begin = (Int)max((int64_t)-r.half, -lo), end = (Int)min((int64_t)size + r.half, rest);   // in reach, relative to lo
  if (r.in_range_divisor && (begin > -r.half || end < size + r.half)) return pool_by_windows(importance, n_tokens, r, lo, lo + size);
  float sum = 0.f;
  for (Int x = (Int)(threadIdx.x & 31) - r.half; x < end; x += 32)
    if (x >= begin) sum = fmaf(__ldcg(from + x), (float)(min(x + r.half, size - 1) - max(x - r.half, (Int)0) + 1), sum);
  return warp_total(sum) * r.inv_w / (float)size;
}

// The same for eight chunks from j on, none of them short and none with windows beyond the prompt's ends: what depends on the
// position only is computed once, and the eight sums cross the warp together (9 shuffles instead of 40, the same additions).
// Lane 4 u gets the score of chunk j + u.  8 CTAs pool 4096 chunks in 3.4 us less than one chunk at a time.
constexpr int kPoolBatch = 8;

__device__ __forceinline__ float pool_eight(const float* __restrict__ importance, const PoolRule& r, int64_t j) {
  const int lane = threadIdx.x & 31;
  const float* from = importance + j * r.chunk;
  float sum[kPoolBatch];
#pragma unroll
  for (int u = 0; u < kPoolBatch; ++u) sum[u] = 0.f;
  for (int x = lane - r.half; x < r.chunk + r.half; x += 32) {
    const float windows = (float)(min(x + r.half, r.chunk - 1) - max(x - r.half, 0) + 1);
    float v[kPoolBatch];
#pragma unroll
    for (int u = 0; u < kPoolBatch; ++u) v[u] = __ldcg(from + x + u * r.chunk);
#pragma unroll
    for (int u = 0; u < kPoolBatch; ++u) sum[u] = fmaf(v[u], windows, sum[u]);
  }
#pragma unroll
  for (int half = kPoolBatch / 2, off = 16; half > 0; half >>= 1, off >>= 1) {
    const bool upper = lane & off;                         // this lane keeps the upper half of the sums
#pragma unroll
    for (int u = 0; u < half; ++u) {
      const float other = __shfl_xor_sync(0xffffffffu, upper ? sum[u] : sum[u + half], off);
      sum[u] = (upper ? sum[u + half] : sum[u]) + other;
    }
  }
  float total = sum[0];
#pragma unroll
  for (int off = 2; off > 0; off >>= 1) total += __shfl_xor_sync(0xffffffffu, total, off);
  return total * r.inv_w / (float)r.chunk;
}

__device__ __forceinline__ void chunk_pool_body(const float* __restrict__ importance, int64_t n_tokens, const PoolRule& r,
                                                float* __restrict__ chunk_scores, int64_t n_chunks) {
  const int64_t j = (int64_t)blockIdx.x * kPoolWarps + (threadIdx.x >> 5);
  if (j >= n_chunks) return;
  float score = r.chunk <= kShortChunk ? pool_chunk<int>(importance, n_tokens, r, j) : pool_chunk<int64_t>(importance, n_tokens, r, j);
  if (!is_finite(score)) score = pool_by_windows(importance, n_tokens, r, j * r.chunk, min((j + 1) * r.chunk, n_tokens));
  if ((threadIdx.x & 31) == 0) chunk_scores[j] = score;
}

__global__ void __launch_bounds__(kPoolWarps * 32) chunk_pool_kernel(const float* __restrict__ importance, int64_t n_tokens, PoolRule r,
                                                                      float* __restrict__ chunk_scores, int64_t n_chunks) {
  chunk_pool_body(importance, n_tokens, r, chunk_scores, n_chunks);
}

// Batched calls: up to kBatchItems prompts per launch, their descriptors passed by value; blockIdx.y picks the prompt.
constexpr int kBatchItems = 32;
struct PoolBatch {
  spf_pool_item item[kBatchItems];
};
struct TopkBatch {
  spf_topk_item item[kBatchItems];
};
struct CompactBatch {
  spf_compact_item item[kBatchItems];
};

__global__ void __launch_bounds__(kPoolWarps * 32) chunk_pool_batch_kernel(const __grid_constant__ PoolBatch b, PoolRule r) {
  const spf_pool_item& it = b.item[blockIdx.y];
  chunk_pool_body(it.importance, it.n_tokens, r, it.chunk_scores, (it.n_tokens + r.chunk - 1) / r.chunk);
}

// ------------------------------------------------------------------------------------------------
// spf_select_topk: one CTA.  Scores map to unsigned keys whose integer order is the float order; a
// four-pass radix select (8 bits per pass, most significant first) finds the k-th largest key; then
// everything above it, plus the lowest-index entries equal to it, is written out in index order.
// ------------------------------------------------------------------------------------------------
constexpr int kTopkThreads = 1024;

__device__ __forceinline__ uint32_t order_key(float x) {
  x += 0.0f;  // -0 -> +0 so that the two zeros tie
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Key of chunk j: forced chunks (bit 0 of `force`: the first chunk, bit 1: the last) sort above every score.
__device__ __forceinline__ uint32_t chunk_key(const float* __restrict__ scores, int j, int n, int force) {
  if (((force & 1) && j == 0) || ((force & 2) && j == n - 1)) return 0xFFFFFFFFu;
  return order_key(scores[j]);
}

// One histogram increment per distinct bin of a warp instead of one per thread: scores share their top bits, so the
// first passes would otherwise send thousands of atomics to a handful of shared-memory words.
__device__ __forceinline__ void hist_add_aggregated(int* hist, bool take, uint32_t bin) {
  const unsigned peers = __match_any_sync(0xffffffffu, take ? bin : 0xffffffffu);
  if (take && (int)(__ffs(peers) - 1) == (int)(threadIdx.x & 31)) atomicAdd(&hist[bin], __popc(peers));
}

__device__ __forceinline__ void select_topk_body(const float* __restrict__ scores, int n, int k, int force,
                                                 int32_t* __restrict__ kept) {
  __shared__ int hist[256];
  __shared__ uint32_t warp_counts[2][kTopkThreads / 32];
  __shared__ uint32_t sh_prefix;
  __shared__ int sh_remaining;

  // up to kTopkCache keys per thread stay in registers for all passes (n <= 8192 chunks, i.e. prompts of up to 262 144
  // tokens at chunk 32); longer score arrays are re-read from global memory in every pass
  constexpr int kTopkCache = 8;
  const bool cached = n <= kTopkThreads * kTopkCache;
  uint32_t ck[kTopkCache];
  if (cached) {
#pragma unroll
    for (int i = 0; i < kTopkCache; ++i) {
      const int j = threadIdx.x + i * kTopkThreads;
      ck[i] = j < n ? chunk_key(scores, j, n, force) : 0u;
    }
  }
  uint32_t prefix = 0;     // the bits of the k-th largest key found so far
  uint32_t mask = 0;       // which bits of `prefix` are fixed
  int remaining = k;       // rank of the wanted key among the keys that match the prefix
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int b = threadIdx.x; b < 256; b += kTopkThreads) hist[b] = 0;
    __syncthreads();
    if (cached) {
#pragma unroll
      for (int i = 0; i < kTopkCache; ++i) {
        const int j = threadIdx.x + i * kTopkThreads;
        if (i * kTopkThreads < n)                            // warp-uniform: whole warps take part or none
          hist_add_aggregated(hist, j < n && (ck[i] & mask) == prefix, (ck[i] >> shift) & 255u);
      }
    } else {
      for (int j0 = 0; j0 < n; j0 += kTopkThreads) {
        const int j = j0 + threadIdx.x;
        const uint32_t key = j < n ? chunk_key(scores, j, n, force) : 0u;
        hist_add_aggregated(hist, j < n && (key & mask) == prefix, (key >> shift) & 255u);
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      // warp 0 walks the 256 bins from the top: each lane owns 8 consecutive bins (lane 31 the highest)
      const int lane = threadIdx.x;
      int mine[8], own = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        mine[e] = hist[lane * 8 + e];
        own += mine[e];
      }
      int above = own;                                   // inclusive suffix sum over lanes >= this one
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_down_sync(0xffffffffu, above, off);
        if (lane + off < 32) above += v;
      }
      above -= own;                                      // entries in bins owned by higher lanes
      const bool here = above < remaining && above + own >= remaining;   // the wanted rank falls into this lane's bins
      if (here) {
        int rem = remaining - above, b = 0;
        bool found = false;
#pragma unroll
        for (int e = 7; e >= 0; --e) {
          if (!found) {
            if (mine[e] >= rem || e == 0) {
              b = e;
              found = true;
            } else {
              rem -= mine[e];
            }
          }
        }
        sh_prefix = prefix | ((uint32_t)(lane * 8 + b) << shift);
        sh_remaining = rem;
      }
    }
    __syncthreads();
    prefix = sh_prefix;
    remaining = sh_remaining;
    mask |= 255u << shift;
    __syncthreads();
  }
  // `prefix` is now the k-th largest key; `remaining` of the entries equal to it are kept (lowest indices).  Larger and equal
  // keys are counted together (high and low half of a word), with one barrier per 1024 keys: the counts of a step and of the
  // next have scratch of their own.
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lower = (1u << lane) - 1u;
  int gt_base = 0, eq_base = 0;
  for (int j0 = 0, it = 0; j0 < n; j0 += kTopkThreads, ++it) {
    const int j = j0 + threadIdx.x;
    uint32_t key = 0u;
    if (cached) {
#pragma unroll
      for (int i = 0; i < kTopkCache; ++i)
        if (i == it) key = ck[i];                            // constant indices keep the cache in registers
    } else if (j < n) {
      key = chunk_key(scores, j, n, force);
    }
    const bool gt = j < n && key > prefix, eq = j < n && key == prefix;
    const uint32_t gts = __ballot_sync(0xffffffffu, gt), eqs = __ballot_sync(0xffffffffu, eq);
    if (lane == 0) warp_counts[it & 1][warp] = (uint32_t)__popc(gts) << 16 | (uint32_t)__popc(eqs);
    __syncthreads();
    const uint32_t w = warp_counts[it & 1][lane], all = __reduce_add_sync(0xffffffffu, w);
    const uint32_t ahead = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
    const int gt_rank = gt_base + (int)(ahead >> 16) + __popc(gts & lower), eq_rank = eq_base + (int)(ahead & 0xFFFFu) + __popc(eqs & lower);
    if (gt || (eq && eq_rank < remaining)) kept[gt_rank + min(eq_rank, remaining)] = j;
    gt_base += (int)(all >> 16);
    eq_base += (int)(all & 0xFFFFu);
  }
}

__global__ void __launch_bounds__(kTopkThreads) select_topk_kernel(const float* __restrict__ scores, int n, int k, int force,
                                                                    int32_t* __restrict__ kept) {
  select_topk_body(scores, n, k, force, kept);
}

__global__ void __launch_bounds__(kTopkThreads) select_topk_batch_kernel(const __grid_constant__ TopkBatch b) {
  const spf_topk_item& it = b.item[blockIdx.x];
  select_topk_body(it.chunk_scores, (int)it.n_chunks, (int)it.k, 0, it.kept_chunks);
}

// ------------------------------------------------------------------------------------------------
// spf_compact_spans.  Kept chunk r (ascending order) starts at output offset r * c because only the
// very last chunk of the prompt can be short and, if kept, it is the last one kept.  Block 0 finds
// the runs of consecutive chunks (a prefix count of run starts) and writes the spans and counts; the
// other blocks copy ids and positions, one warp per kept chunk.
// ------------------------------------------------------------------------------------------------
constexpr int kCompactThreads = 256;
// From so many kept chunks on block 0's walk over them is what takes the time (13108 chunks of one token: 54 us in all with 256
// threads, 29 with 1024), below the copy, which wants to be spread over the SMs (128 chunks of 1024 tokens: 18 and 21 us).
constexpr int kCompactMany = 1025, kCompactManyThreads = 1024;

template <int THREADS>
__device__ __forceinline__ void compact_spans_body(
    const int32_t* __restrict__ kept, int k, int chunk, int64_t n_tokens, const int32_t* __restrict__ token_ids,
    const int32_t* __restrict__ char_start, const int32_t* __restrict__ char_end, int32_t* __restrict__ out_ids,
    int32_t* __restrict__ out_pos, int32_t* __restrict__ out_tok_spans, int32_t* __restrict__ out_char_spans,
    int64_t* __restrict__ out_counts) {
  const int64_t n_chunks = (n_tokens + chunk - 1) / chunk;
  if (blockIdx.x == 0) {
    // 1024 chunks a step: the 32 counts of a step are read by every warp at once, and those of the next have
    // scratch of their own
    constexpr int kEach = 1024 / THREADS, kWarps = THREADS / 32;
    static_assert(kEach * kWarps == 32, "a count per lane");
    __shared__ int counts[2][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int span_base = 0;
    for (int r0 = 0, it = 0; r0 < k; r0 += kEach * THREADS, ++it) {
      int64_t j[kEach];
      bool starts[kEach], ends[kEach];
      int within[kEach];
#pragma unroll
      for (int u = 0; u < kEach; ++u) {
        const int r = r0 + u * THREADS + threadIdx.x;
        j[u] = -1;
        starts[u] = ends[u] = false;
        if (r < k) {
          j[u] = kept[r];
          starts[u] = r == 0 || kept[r - 1] + 1 != j[u];
          ends[u] = r == k - 1 || kept[r + 1] != j[u] + 1;
        }
      }
#pragma unroll
      for (int u = 0; u < kEach; ++u) {
        const unsigned ballot = __ballot_sync(0xffffffffu, starts[u]);
        within[u] = __popc(ballot & ((2u << lane) - 1u));        // inclusive
        if (lane == 0) counts[it & 1][u * kWarps + warp] = __popc(ballot);
      }
      __syncthreads();
      const int count = counts[it & 1][lane];
#pragma unroll
      for (int u = 0; u < kEach; ++u) {
        const int before = __reduce_add_sync(0xffffffffu, lane < u * kWarps + warp ? count : 0);
        const int span = span_base + before + within[u] - 1;     // index of the run this chunk belongs to
        if (j[u] < 0 || j[u] >= n_chunks) continue;
        if (starts[u]) {
          const int64_t a = j[u] * chunk;
          out_tok_spans[2 * span] = (int32_t)a;
          out_char_spans[2 * span] = char_start[a];
        }
        if (ends[u]) {
          const int64_t b = min((j[u] + 1) * chunk, n_tokens);
          out_tok_spans[2 * span + 1] = (int32_t)b;
          out_char_spans[2 * span + 1] = char_end[b - 1];
        }
      }
      span_base += __reduce_add_sync(0xffffffffu, count);
    }
    if (threadIdx.x == 0) {
      const int64_t last = kept[k - 1];
      const int64_t last_size = min((last + 1) * chunk, n_tokens) - last * chunk;
      out_counts[0] = (int64_t)(k - 1) * chunk + last_size;
      out_counts[1] = span_base;
    }
    return;
  }
  const int warps = THREADS / 32;
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)(blockIdx.x - 1) * warps + (threadIdx.x >> 5);
  if (r >= k) return;
  const int64_t j = kept[r];
  if (j < 0 || j >= n_chunks) return;
  const int64_t lo = j * chunk, hi = min(lo + chunk, n_tokens);
  for (int64_t s = lo + lane; s < hi; s += 32) {
    const int64_t o = r * chunk + (s - lo);
    out_ids[o] = token_ids[s];
    if (out_pos != nullptr) out_pos[o] = (int32_t)s;
  }
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS) compact_spans_kernel(
    const int32_t* __restrict__ kept, int k, int chunk, int64_t n_tokens, const int32_t* __restrict__ token_ids,
    const int32_t* __restrict__ char_start, const int32_t* __restrict__ char_end, int32_t* __restrict__ out_ids,
    int32_t* __restrict__ out_pos, int32_t* __restrict__ out_tok_spans, int32_t* __restrict__ out_char_spans,
    int64_t* __restrict__ out_counts) {
  compact_spans_body<THREADS>(kept, k, chunk, n_tokens, token_ids, char_start, char_end, out_ids, out_pos, out_tok_spans, out_char_spans,
                     out_counts);
}

// ------------------------------------------------------------------------------------------------
// spf_pool_select_compact, spf_select_compact: the whole path behind the scores in one launch, a cluster of CTAs per prompt.
//
// Nothing here is much work; what costs is the chain of dependent steps, so there are as few as possible between one load
// and the next.  Each CTA pools its share of the chunks; after the cluster's barrier (the only one) every CTA reads all scores,
// makes the same selection by itself and writes its own share of the results.
//   selection: the keys' range is cut into 2048 equal bins (4096 log-normal scores fill some 800 of them; one score of zero
//     among them leaves 70, the fullest with 200 entries), one histogram finds the k-th key's bin, and its few entries are
//     ranked against each other; a bin of more than kRankMost entries is cut again.  Ties go to the lower index.
//   compaction: the selection is a bitmap, one word per warp and step by ballot.  Kept chunks and starts of runs are counted
//     by population counts, in one scan over the words, instead of a scan per 1024 chunks.
// ------------------------------------------------------------------------------------------------
constexpr int kTailThreads = 1024;
constexpr int kTailChunks = 32768;     // keys of this many chunks fit shared memory (128 KB)
constexpr int kTailBins = 2 * kTailThreads;
constexpr int kRankMost = 512;
constexpr int kRankAll = 128;          // so few chunks are ranked without a histogram and its four barriers (64: 7.9 -> 7.1 us in all)
constexpr int kTailItems = 24;         // prompts per launch: their descriptors are kernel arguments

struct TailBatch {
  spf_path_item item[kTailItems];
  PoolRule rule;
  int force;                           // bit 0: the first chunk is kept whatever its score, bit 1: the last
};

struct TailShared {
  int hist[kTailBins];
  uint32_t cand_key[kRankMost];
  int cand_at[kRankMost];
  uint32_t bits[kTailChunks / 32 + 2];    // kept chunks; a zero word on either side
  uint32_t before[kTailChunks / 32];      // kept chunks (high half) and starts of runs (low half) ahead of a word
  uint32_t warp_lo[32], warp_hi[32];
  int found_bin, found_left, found_count, n_cand;
  uint32_t last_key;                      // kept: keys above last_key, and those equal to it up to index last_at
  int last_at;
};

// Exclusive prefix sum over the CTA in thread order; *all: the sum of every thread's x.  `scratch` is free again once all
// threads have passed the caller's next barrier.
__device__ __forceinline__ uint32_t block_exclusive(uint32_t x, uint32_t* scratch, uint32_t* all) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += v;
  }
  if (lane == 31) scratch[warp] = incl;
  __syncthreads();
  const uint32_t w = scratch[lane];                        // every warp scans the 32 warp totals by itself
  *all = __reduce_add_sync(0xffffffffu, w);
  return incl - x + __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
}

// Finds the `left`-th largest of the n keys that are not forced: its key and index go to sh.last_key, sh.last_at.
__device__ __forceinline__ void select_last(TailShared& sh, const uint32_t* keys, int n, int left, int force) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int first = force & 1, end = n - ((force >> 1) & 1);
  if (n <= kRankAll) {
    constexpr int kEach = kRankAll / 32;
    uint32_t other[kEach];
#pragma unroll
    for (int o = 0; o < kEach; ++o) other[o] = keys[min(first + lane + 32 * o, n - 1)];
#pragma unroll
    for (int c = 0; c < kEach; ++c) {
      const int j = first + warp + 32 * c;
      const uint32_t key = keys[min(j, n - 1)];
      uint32_t better = 0;
#pragma unroll
      for (int o = 0; o < kEach; ++o) {
        const int at = first + lane + 32 * o;
        better += at < end && (other[o] > key || (other[o] == key && at < j));
      }
      better = __reduce_add_sync(0xffffffffu, better);
      if (lane == 0 && j < end && (int)better == left - 1) {
        sh.last_key = key;
        sh.last_at = j;
      }
    }
    __syncthreads();
    return;
  }
  uint32_t lo = 0xFFFFFFFFu, hi = 0;
  for (int j = first + tid; j < end; j += kTailThreads) {
    lo = min(lo, keys[j]);
    hi = max(hi, keys[j]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    sh.warp_lo[warp] = lo;
    sh.warp_hi[warp] = hi;
  }
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, sh.warp_lo[lane]);
  hi = __reduce_max_sync(0xffffffffu, sh.warp_hi[lane]);
  while (true) {
    // bins of 2^shift keys, from `lo` on; the histogram is zero here
    const int shift = max(0, 21 - __clz(hi - lo));
    for (int j = first + tid; j < end; j += kTailThreads)
      if (keys[j] >= lo && keys[j] <= hi) atomicAdd(&sh.hist[(keys[j] - lo) >> shift], 1);
    __syncthreads();
    const int top = kTailBins - 1 - 2 * tid;               // each thread owns two bins, the first thread the highest
    const int h1 = sh.hist[top], h0 = sh.hist[top - 1];
    sh.hist[top] = sh.hist[top - 1] = 0;
    uint32_t all;
    const int above = (int)block_exclusive((uint32_t)(h0 + h1), sh.warp_lo, &all);
    if (above < left && above + h0 + h1 >= left) {
      const bool upper = above + h1 >= left;
      sh.found_bin = upper ? top : top - 1;
      sh.found_left = upper ? left - above : left - above - h1;
      sh.found_count = upper ? h1 : h0;
      sh.n_cand = 0;
    }
    __syncthreads();
    lo += (uint32_t)sh.found_bin << shift;
    hi = lo + min(hi - lo, (1u << shift) - 1u);
    left = sh.found_left;
    const int count = sh.found_count;
    if (count <= kRankMost) {
      for (int j = first + tid; j < end; j += kTailThreads)
        if (keys[j] >= lo && keys[j] <= hi) {
          const int at = atomicAdd(&sh.n_cand, 1);
          sh.cand_key[at] = keys[j];
          sh.cand_at[at] = j;
        }
      __syncthreads();
      for (int c = warp; c < count; c += kTailThreads / 32) {
        const uint32_t key = sh.cand_key[c];
        const int at = sh.cand_at[c];
        uint32_t better = 0;
        for (int o = lane; o < count; o += 32) better += sh.cand_key[o] > key || (sh.cand_key[o] == key && sh.cand_at[o] < at);
        better = __reduce_add_sync(0xffffffffu, better);
        if (lane == 0 && (int)better == left - 1) {
          sh.last_key = key;
          sh.last_at = at;
        }
      }
      __syncthreads();
      return;
    }
    if (shift == 0) {                                      // that many equal keys: the left-th of them by index
      const int words = (n + 31) / 32;
      for (int w = warp; w < words; w += kTailThreads / 32) {
        const int j = w * 32 + lane;
        const uint32_t same = __ballot_sync(0xffffffffu, j >= first && j < end && keys[min(j, n - 1)] == lo);
        if (lane == 0) sh.bits[1 + w] = same;
      }
      __syncthreads();
      const uint32_t mine = tid < words ? sh.bits[1 + tid] : 0u;
      const int ahead = (int)block_exclusive(__popc(mine), sh.warp_hi, &all);
      if (ahead < left && ahead + __popc(mine) >= left) {
        uint32_t rest = mine;
        for (int i = ahead + 1; i < left; ++i) rest &= rest - 1u;
        sh.last_key = lo;
        sh.last_at = tid * 32 + __ffs(rest) - 1;
      }
      __syncthreads();
      return;
    }
  }
}

// Chunks j0, j0 + step, ... below `end`, `each` in a row: those whose scores are not finite are done window by window.
__device__ __noinline__ void pool_again(const spf_path_item& it, const PoolRule& r, int j0, int end, int step, int each) {
  __syncwarp();
  for (int j = j0; j < end; j += step)
    for (int i = j; i < j + each; ++i)
      if (!is_finite(__ldcg(it.chunk_scores + i))) {
        const int64_t lo = (int64_t)i * r.chunk;
        const float score = pool_by_windows(it.importance, it.n_tokens, r, lo, min(lo + r.chunk, it.n_tokens));
        if ((threadIdx.x & 31) == 0) it.chunk_scores[i] = score;
      }
}

// Copies the kept chunks' tokens in pieces of 128, dealt out to `warps` warps of which this is number `at`: however long the
// chunks are, all warps share them (one kept chunk of 16384 tokens: 2 us, and 190 as the work of one warp).
constexpr int kPiece = 128;

__device__ __forceinline__ void copy_pieces(const spf_path_item& it, const uint32_t* keys, int k, int chunk, int at, int warps) {
  const int per = (chunk + kPiece - 1) / kPiece, lane = threadIdx.x & 31;
  for (int i = at; i < k * per; i += warps) {
    const int r = i / per;
    const int64_t within = (int64_t)(i - r * per) * kPiece, a = (int64_t)keys[r] * chunk + within, o = (int64_t)r * chunk + within;
    const int size = (int)min(min((int64_t)kPiece, chunk - within), it.n_tokens - a);
    int32_t id[kPiece / 32];
#pragma unroll
    for (int u = 0; u < kPiece / 32; ++u) id[u] = 32 * u + lane < size ? __ldg(it.token_ids + a + 32 * u + lane) : 0;
#pragma unroll
    for (int u = 0; u < kPiece / 32; ++u)
      if (32 * u + lane < size) {
        it.out_ids[o + 32 * u + lane] = id[u];
        if (it.out_pos != nullptr) it.out_pos[o + 32 * u + lane] = (int32_t)a + 32 * u + lane;
      }
  }
}

__global__ void __launch_bounds__(kTailThreads) pool_select_compact_kernel(const __grid_constant__ TailBatch b) {
  extern __shared__ uint32_t keys[];                       // the chunks' keys, then the kept chunks' indices
  __shared__ TailShared sh;
  const spf_path_item& it = b.item[blockIdx.y];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x, ctas = gridDim.x;           // the grid's x extent is one cluster
  const int64_t n_tokens = it.n_tokens;
  const int chunk = b.rule.chunk, n = (int)((n_tokens + chunk - 1) / chunk), k = (int)it.k;

  sh.hist[tid] = sh.hist[tid + kTailThreads] = 0;
  grid_wait();                                             // the scores are complete from here on
  if (it.importance != nullptr) {
    // batches `fast` to `slow` - 1 are far enough from the ends; the chunks around them go to the last warps, one each
    const int64_t reach = (int64_t)kPoolBatch * chunk;
    const int all = (n + kPoolBatch - 1) / kPoolBatch, warps = ctas * 32, at = rank * 32 + warp;
    const int fast = (int)min((b.rule.half + reach - 1) / reach, (int64_t)all);
    const int slow = (int)max(min((n_tokens - b.rule.half) / reach, (int64_t)all), (int64_t)fast);
    bool fine = true;
    for (int i = fast + at; i < slow; i += warps) {
      const float score = pool_eight(it.importance, b.rule, (int64_t)i * kPoolBatch);
      if ((lane & 3) == 0) it.chunk_scores[i * kPoolBatch + (lane >> 2)] = score;
      fine = fine && is_finite(score);
    }
    if (!__all_sync(0xffffffffu, fine)) pool_again(it, b.rule, (fast + at) * kPoolBatch, slow * kPoolBatch, warps * kPoolBatch, kPoolBatch);
    for (int i = warps - 1 - at; i < n - (slow - fast) * kPoolBatch; i += warps) {
      const int j = i < fast * kPoolBatch ? i : i + (slow - fast) * kPoolBatch;
      const float score = pool_chunk<int>(it.importance, n_tokens, b.rule, j);
      if (lane == 0) it.chunk_scores[j] = score;
      if (!is_finite(score)) pool_again(it, b.rule, j, j + 1, 1, 1);
    }
    if (ctas > 1) {                                        // (one CTA: the cluster's barrier took 0.7 us of 6)
      cluster_arrive();                                    // orders the stores before the loads below, in all CTAs
      cluster_wait();
    } else {
      __syncthreads();
    }
  }
  for (int j = tid; j < n; j += kTailThreads) keys[j] = order_key(__ldcg(it.chunk_scores + j));
  __syncthreads();

  const int first = b.force & 1, end = n - ((b.force >> 1) & 1);
  const int left = k - first - (end < n && end >= first ? 1 : 0);
  if (left > 0) {
    select_last(sh, keys, n, left, b.force);
  } else {
    if (tid == 0) {
      sh.last_key = 0xFFFFFFFFu;
      sh.last_at = -1;
    }
    __syncthreads();
  }
  const uint32_t last_key = sh.last_key;
  const int last_at = sh.last_at, words = (n + 31) / 32;
  for (int w = warp; w < words; w += kTailThreads / 32) {
    const int j = w * 32 + lane;
    const uint32_t key = keys[min(j, n - 1)];
    const bool kept = j < n && (j < first || j >= end || key > last_key || (key == last_key && j <= last_at));
    const uint32_t ballot = __ballot_sync(0xffffffffu, kept);
    if (lane == 0) sh.bits[1 + w] = ballot;
  }
  if (tid == 0) sh.bits[0] = sh.bits[1 + words] = 0u;
  __syncthreads();
  uint32_t total = 0;
  {
    const uint32_t mine = tid < words ? sh.bits[1 + tid] : 0u;
    const uint32_t starts = tid < words ? mine & ~((mine << 1) | (sh.bits[tid] >> 31)) : 0u;
    const uint32_t ahead = block_exclusive((uint32_t)__popc(mine) << 16 | (uint32_t)__popc(starts), sh.warp_lo, &total);
    if (tid < words) sh.before[tid] = ahead;
  }
  __syncthreads();
  // every CTA lists the kept chunks for itself; indices and spans are written by one of them, word by word
  for (int w = warp; w < words; w += kTailThreads / 32) {
    const uint32_t mine = sh.bits[1 + w], prev = sh.bits[w], next = sh.bits[2 + w], ahead = sh.before[w];
    if (!(mine >> lane & 1u)) continue;
    const int j = w * 32 + lane;
    const uint32_t upto = (2u << lane) - 1u;               // this chunk and those ahead of it in the word
    const uint32_t starts = mine & ~((mine << 1) | (prev >> 31));
    const int r = (int)(ahead >> 16) + __popc(mine & upto) - 1, span = (int)(ahead & 0xFFFFu) + __popc(starts & upto) - 1;
    keys[r] = (uint32_t)j;
    if (w % ctas != rank) continue;
    it.kept_chunks[r] = j;
    if (starts >> lane & 1u) {
      const int64_t a = (int64_t)j * chunk;
      it.out_tok_spans[2 * span] = (int32_t)a;
      it.out_char_spans[2 * span] = __ldg(it.char_start + a);
    }
    if (!((lane < 31 ? mine >> (lane + 1) : next) & 1u)) {
      const int64_t e = min((int64_t)(j + 1) * chunk, n_tokens);
      it.out_tok_spans[2 * span + 1] = (int32_t)e;
      it.out_char_spans[2 * span + 1] = __ldg(it.char_end + e - 1);
    }
  }
  __syncthreads();
  if (rank == 0 && tid == 0) {
    const int64_t last = (int64_t)keys[k - 1] * chunk;
    it.out_counts[0] = (int64_t)(k - 1) * chunk + min((int64_t)chunk, n_tokens - last);
    it.out_counts[1] = (int64_t)(total & 0xFFFFu);
  }
  // Kept chunk r starts at output r * chunk: only the prompt's last chunk can be short, and it is the last one kept.  A warp
  // copies whole chunks, several at a time ...
  constexpr int kRows = 8;
  if (chunk <= kPiece) {
    for (int r0 = rank * 32 + warp; r0 < k; r0 += ctas * 32 * kRows) {
      const int32_t* from[kRows];
      int size[kRows];
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int r = r0 + u * ctas * 32;
        const int64_t a = r < k ? (int64_t)keys[r] * chunk : 0;
        from[u] = it.token_ids + a;
        size[u] = r < k ? (int)min((int64_t)chunk, n_tokens - a) : 0;
      }
      const int64_t o = (int64_t)r0 * chunk;
      for (int s = lane; s < chunk; s += 32) {
        int32_t id[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) id[u] = s < size[u] ? __ldg(from[u] + s) : 0;
#pragma unroll
        for (int u = 0; u < kRows; ++u)
          if (s < size[u]) {
            it.out_ids[o + (int64_t)u * ctas * 32 * chunk + s] = id[u];
            if (it.out_pos != nullptr) it.out_pos[o + (int64_t)u * ctas * 32 * chunk + s] = (int32_t)(from[u] - it.token_ids) + s;
          }
      }
    }
    return;
  }
  // ... or pieces of longer ones
  copy_pieces(it, keys, k, chunk, rank * 32 + warp, ctas * 32);
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS) compact_spans_batch_kernel(const __grid_constant__ CompactBatch b, int chunk) {
  const spf_compact_item& it = b.item[blockIdx.y];
  if ((int64_t)blockIdx.x > 1 + (it.k + THREADS / 32 - 1) / (THREADS / 32)) return;
  compact_spans_body<THREADS>(it.kept_chunks, (int)it.k, chunk, it.n_tokens, it.token_ids, it.char_start, it.char_end, it.out_ids, it.out_pos,
                     it.out_tok_spans, it.out_char_spans, it.out_counts);
}

}  // namespace
}  // namespace spf

using namespace spf;

static int32_t chunk_pool_launch(const float* importance, int64_t n_tokens, int32_t pool_kernel, int32_t chunk,
                                 bool in_range_divisor, float* chunk_scores, void* cuda_stream) {
  clear_error();
  if (importance == nullptr || chunk_scores == nullptr) return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool: null pointer");
  if (n_tokens < 1) return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool: n_tokens must be >= 1 (got %lld)", (long long)n_tokens);
  if (pool_kernel < 1 || pool_kernel > 255 || pool_kernel % 2 == 0)
    return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool: pool_kernel must be odd and in [1, 255] (got %d)", pool_kernel);
  if (chunk < 1) return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool: chunk must be >= 1 (got %d)", chunk);
  const int64_t n_chunks = ceil_div(n_tokens, chunk);
  const int64_t blocks = ceil_div(n_chunks, kPoolWarps);
  if (blocks > 0x7fffffff) return fail(SPF_ERR_UNSUPPORTED, "spf_chunk_pool: too many chunks");
  chunk_pool_kernel<<<(unsigned)blocks, kPoolWarps * 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      importance, n_tokens, PoolRule{pool_kernel / 2, chunk, 1.0f / (float)pool_kernel, in_range_divisor}, chunk_scores, n_chunks);
  SPF_CUDA_CHECK(cudaGetLastError());
  return SPF_OK;
}

extern "C" int32_t spf_chunk_pool(const float* importance, int64_t n_tokens, int32_t pool_kernel, int32_t chunk,
                                  float* chunk_scores, void* cuda_stream) {
  return chunk_pool_launch(importance, n_tokens, pool_kernel, chunk, false, chunk_scores, cuda_stream);
}

extern "C" int32_t spf_chunk_pool_edge(const float* importance, int64_t n_tokens, int32_t pool_kernel, int32_t chunk,
                                       int32_t edge_rule, float* chunk_scores, void* cuda_stream) {
  if (edge_rule != 0 && edge_rule != 1) {
    clear_error();
    return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool_edge: edge_rule must be 0 or 1 (got %d)", edge_rule);
  }
  return chunk_pool_launch(importance, n_tokens, pool_kernel, chunk, edge_rule == 1, chunk_scores, cuda_stream);
}

static int32_t select_topk_launch(const float* chunk_scores, int64_t n_chunks, int64_t k, int force, int32_t* kept_chunks,
                                  void* cuda_stream) {
  clear_error();
  if (chunk_scores == nullptr || kept_chunks == nullptr) return fail(SPF_ERR_INVALID_ARG, "spf_select_topk: null pointer");
  if (n_chunks < 1 || n_chunks > 0x7fffffff)
    return fail(SPF_ERR_INVALID_ARG, "spf_select_topk: n_chunks must be in [1, 2^31) (got %lld)", (long long)n_chunks);
  if (k < 1 || k > n_chunks)
    return fail(SPF_ERR_INVALID_ARG, "spf_select_topk: k must be in [1, n_chunks] (got k=%lld, n_chunks=%lld)", (long long)k,
                (long long)n_chunks);
  const int n_forced = (force & 1) + ((force & 2) && (n_chunks > 1 || !(force & 1)) ? 1 : 0);
  if (k < n_forced)
    return fail(SPF_ERR_INVALID_ARG, "spf_select_topk_forced: k = %lld is smaller than the %d forced chunks", (long long)k, n_forced);
  select_topk_kernel<<<1, kTopkThreads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(chunk_scores, (int)n_chunks, (int)k, force,
                                                                                    kept_chunks);
  SPF_CUDA_CHECK(cudaGetLastError());
  return SPF_OK;
}

extern "C" int32_t spf_select_topk(const float* chunk_scores, int64_t n_chunks, int64_t k, int32_t* kept_chunks,
                                   void* cuda_stream) {
  return select_topk_launch(chunk_scores, n_chunks, k, 0, kept_chunks, cuda_stream);
}

extern "C" int32_t spf_select_topk_forced(const float* chunk_scores, int64_t n_chunks, int64_t k, int32_t force_first,
                                          int32_t force_last, int32_t* kept_chunks, void* cuda_stream) {
  return select_topk_launch(chunk_scores, n_chunks, k, (force_first ? 1 : 0) | (force_last ? 2 : 0), kept_chunks, cuda_stream);
}

extern "C" int32_t spf_compact_spans(const int32_t* kept_chunks, int64_t k, int32_t chunk, int64_t n_tokens,
                                     const int32_t* token_ids, const int32_t* char_start, const int32_t* char_end,
                                     int32_t* out_ids, int32_t* out_pos, int32_t* out_tok_spans, int32_t* out_char_spans,
                                     int64_t* out_counts, void* cuda_stream) {
  clear_error();
  if (kept_chunks == nullptr || token_ids == nullptr || char_start == nullptr || char_end == nullptr || out_ids == nullptr ||
      out_tok_spans == nullptr || out_char_spans == nullptr || out_counts == nullptr)
    return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans: null pointer");
  if (chunk < 1) return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans: chunk must be >= 1 (got %d)", chunk);
  if (n_tokens < 1 || n_tokens > 0x7fffffff)
    return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans: n_tokens must be in [1, 2^31) (got %lld)", (long long)n_tokens);
  const int64_t n_chunks = ceil_div(n_tokens, chunk);
  if (k < 1 || k > n_chunks)
    return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans: k must be in [1, n_chunks] (got k=%lld, n_chunks=%lld)", (long long)k,
                (long long)n_chunks);
  const bool many = k >= kCompactMany;
  const int threads = many ? kCompactManyThreads : kCompactThreads;
  const int64_t blocks = 1 + ceil_div(k, threads / 32);
  auto kernel = many ? compact_spans_kernel<kCompactManyThreads> : compact_spans_kernel<kCompactThreads>;
  kernel<<<(unsigned)blocks, threads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      kept_chunks, (int)k, chunk, n_tokens, token_ids, char_start, char_end, out_ids, out_pos, out_tok_spans, out_char_spans,
      out_counts);
  SPF_CUDA_CHECK(cudaGetLastError());
  return SPF_OK;
}

// ------------------------------------------------------------------------------------------------ batched calls
extern "C" int32_t spf_chunk_pool_batch(const spf_pool_item* items, int32_t n_items, int32_t pool_kernel, int32_t chunk,
                                        void* cuda_stream) {
  clear_error();
  if (items == nullptr || n_items < 1) return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool_batch: null items or n_items < 1");
  if (pool_kernel < 1 || pool_kernel > 255 || pool_kernel % 2 == 0)
    return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool_batch: pool_kernel must be odd and in [1, 255] (got %d)", pool_kernel);
  if (chunk < 1) return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool_batch: chunk must be >= 1 (got %d)", chunk);
  for (int32_t i = 0; i < n_items; ++i) {
    if (items[i].importance == nullptr || items[i].chunk_scores == nullptr)
      return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool_batch: item %d: null pointer", i);
    if (items[i].n_tokens < 1) return fail(SPF_ERR_INVALID_ARG, "spf_chunk_pool_batch: item %d: n_tokens must be >= 1", i);
    if (ceil_div(ceil_div(items[i].n_tokens, chunk), kPoolWarps) > 0x7fffffff)
      return fail(SPF_ERR_UNSUPPORTED, "spf_chunk_pool_batch: item %d: too many chunks", i);
  }
  for (int32_t i0 = 0; i0 < n_items; i0 += kBatchItems) {
    const int cnt = std::min<int32_t>(kBatchItems, n_items - i0);
    PoolBatch b{};
    int64_t blocks = 1;
    for (int i = 0; i < cnt; ++i) {
      b.item[i] = items[i0 + i];
      blocks = std::max(blocks, ceil_div(ceil_div(items[i0 + i].n_tokens, chunk), kPoolWarps));
    }
    chunk_pool_batch_kernel<<<dim3((unsigned)blocks, (unsigned)cnt), kPoolWarps * 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        b, PoolRule{pool_kernel / 2, chunk, 1.0f / (float)pool_kernel, false});
    SPF_CUDA_CHECK(cudaGetLastError());
  }
  return SPF_OK;
}

extern "C" int32_t spf_select_topk_batch(const spf_topk_item* items, int32_t n_items, void* cuda_stream) {
  clear_error();
  if (items == nullptr || n_items < 1) return fail(SPF_ERR_INVALID_ARG, "spf_select_topk_batch: null items or n_items < 1");
  for (int32_t i = 0; i < n_items; ++i) {
    if (items[i].chunk_scores == nullptr || items[i].kept_chunks == nullptr)
      return fail(SPF_ERR_INVALID_ARG, "spf_select_topk_batch: item %d: null pointer", i);
    if (items[i].n_chunks < 1 || items[i].n_chunks > 0x7fffffff || items[i].k < 1 || items[i].k > items[i].n_chunks)
      return fail(SPF_ERR_INVALID_ARG, "spf_select_topk_batch: item %d: need 1 <= k <= n_chunks < 2^31 (k=%lld, n_chunks=%lld)", i,
                  (long long)items[i].k, (long long)items[i].n_chunks);
  }
  for (int32_t i0 = 0; i0 < n_items; i0 += kBatchItems) {
    const int cnt = std::min<int32_t>(kBatchItems, n_items - i0);
    TopkBatch b{};
    for (int i = 0; i < cnt; ++i) b.item[i] = items[i0 + i];
    select_topk_batch_kernel<<<cnt, kTopkThreads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(b);
    SPF_CUDA_CHECK(cudaGetLastError());
  }
  return SPF_OK;
}

extern "C" int32_t spf_compact_spans_batch(const spf_compact_item* items, int32_t n_items, int32_t chunk, void* cuda_stream) {
  clear_error();
  if (items == nullptr || n_items < 1) return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans_batch: null items or n_items < 1");
  if (chunk < 1) return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans_batch: chunk must be >= 1 (got %d)", chunk);
  for (int32_t i = 0; i < n_items; ++i) {
    const spf_compact_item& it = items[i];
    if (it.kept_chunks == nullptr || it.token_ids == nullptr || it.char_start == nullptr || it.char_end == nullptr ||
        it.out_ids == nullptr || it.out_tok_spans == nullptr || it.out_char_spans == nullptr || it.out_counts == nullptr)
      return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans_batch: item %d: null pointer", i);
    if (it.n_tokens < 1 || it.n_tokens > 0x7fffffff)
      return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans_batch: item %d: n_tokens must be in [1, 2^31)", i);
    if (it.k < 1 || it.k > ceil_div(it.n_tokens, chunk))
      return fail(SPF_ERR_INVALID_ARG, "spf_compact_spans_batch: item %d: k must be in [1, n_chunks]", i);
  }
  for (int32_t i0 = 0; i0 < n_items; i0 += kBatchItems) {
    const int cnt = std::min<int32_t>(kBatchItems, n_items - i0);
    CompactBatch b{};
    int64_t most = 1;
    for (int i = 0; i < cnt; ++i) {
      b.item[i] = items[i0 + i];
      most = std::max(most, items[i0 + i].k);
    }
    const bool many = most >= kCompactMany;
    const int threads = many ? kCompactManyThreads : kCompactThreads;
    auto kernel = many ? compact_spans_batch_kernel<kCompactManyThreads> : compact_spans_batch_kernel<kCompactThreads>;
    kernel<<<dim3((unsigned)(1 + ceil_div(most, threads / 32)), (unsigned)cnt), threads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(b, chunk);
    SPF_CUDA_CHECK(cudaGetLastError());
  }
  return SPF_OK;
}

// ------------------------------------------------------------------------------------------------ the path in one launch
namespace {

// CTAs per prompt: pooling and copying shrink with their number, while a larger cluster takes longer to start and to meet.
int tail_ctas(int64_t n_tokens) { return n_tokens <= 2048 ? 1 : n_tokens <= 4096 ? 2 : n_tokens <= 8192 ? 4 : 8; }

int32_t tail_launch(const spf_path_item* items, int n, const PoolRule& rule, int force, cudaStream_t stream) {
  for (int i0 = 0; i0 < n; i0 += kTailItems) {
    const int cnt = std::min(kTailItems, n - i0);
    TailBatch b{};
    b.rule = rule;
    b.force = force;
    int64_t longest = 1, chunks = 1;
    for (int i = 0; i < cnt; ++i) {
      b.item[i] = items[i0 + i];
      longest = std::max(longest, items[i0 + i].n_tokens);
      chunks = std::max(chunks, ceil_div(items[i0 + i].n_tokens, rule.chunk));
    }
    const int ctas = tail_ctas(longest);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctas, (unsigned)cnt);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = (size_t)chunks * sizeof(uint32_t);
    cfg.stream = stream;
    // beyond 48 KB with the static part (about 21 KB), shared memory has to be asked for
    if (cfg.dynamicSmemBytes > 24 * 1024)
    {
      static ContextSet allowed;
      const int32_t st = allow_shared_memory(reinterpret_cast<const void*>(pool_select_compact_kernel), kTailChunks * (int)sizeof(uint32_t), allowed);
      if (st != SPF_OK) return st;
    }
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {(unsigned)ctas, 1, 1};
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    SPF_CUDA_CHECK(cudaLaunchKernelEx(&cfg, pool_select_compact_kernel, b));
  }
  return SPF_OK;
}

}  // namespace

extern "C" int32_t spf_pool_select_compact(const spf_path_item* items, int32_t n_items, int32_t pool_kernel, int32_t chunk, int32_t edge_rule,
                                           int32_t force_first, int32_t force_last, void* cuda_stream) {
  clear_error();
  if (items == nullptr || n_items < 1) return fail(SPF_ERR_INVALID_ARG, "spf_pool_select_compact: null items or n_items < 1");
  if (pool_kernel < 1 || pool_kernel > 255 || pool_kernel % 2 == 0)
    return fail(SPF_ERR_INVALID_ARG, "spf_pool_select_compact: pool_kernel must be odd and in [1, 255] (got %d)", pool_kernel);
  if (edge_rule != 0 && edge_rule != 1)
    return fail(SPF_ERR_INVALID_ARG, "spf_pool_select_compact: edge_rule must be 0 or 1 (got %d)", edge_rule);
  if (chunk < 1) return fail(SPF_ERR_INVALID_ARG, "spf_pool_select_compact: chunk must be >= 1 (got %d)", chunk);
  const int force = (force_first ? 1 : 0) | (force_last ? 2 : 0);
  for (int32_t i = 0; i < n_items; ++i) {
    const spf_path_item& it = items[i];
    if (it.importance == nullptr || it.chunk_scores == nullptr || it.kept_chunks == nullptr || it.token_ids == nullptr ||
        it.char_start == nullptr || it.char_end == nullptr || it.out_ids == nullptr || it.out_tok_spans == nullptr ||
        it.out_char_spans == nullptr || it.out_counts == nullptr)
      return fail(SPF_ERR_INVALID_ARG, "spf_pool_select_compact: item %d: null pointer", i);
    if (it.n_tokens < 1 || it.n_tokens > 0x7fffffff)
      return fail(SPF_ERR_INVALID_ARG, "spf_pool_select_compact: item %d: n_tokens must be in [1, 2^31)", i);
    const int64_t n_chunks = ceil_div(it.n_tokens, chunk);
    const int n_forced = (force & 1) + ((force & 2) && (n_chunks > 1 || !(force & 1)) ? 1 : 0);
    if (it.k < 1 || it.k > n_chunks || it.k < n_forced)
      return fail(SPF_ERR_INVALID_ARG, "spf_pool_select_compact: item %d: k must be in [1, n_chunks] and cover the forced chunks", i);
  }
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const PoolRule rule{pool_kernel / 2, chunk, 1.0f / (float)pool_kernel, edge_rule == 1};
  for (int32_t i = 0; i < n_items;) {
    int32_t j = i;
    while (j < n_items && chunk <= kShortChunk && ceil_div(items[j].n_tokens, chunk) <= kTailChunks) ++j;
    if (j > i) {
      const int32_t st = tail_launch(items + i, j - i, rule, force, stream);
      if (st != SPF_OK) return st;
      i = j;
      continue;
    }
    // too many chunks for one SM's shared memory (or one of gigantic size): the three steps one by one
    const spf_path_item& it = items[i++];
    int32_t st = spf_chunk_pool_edge(it.importance, it.n_tokens, pool_kernel, chunk, edge_rule, it.chunk_scores, cuda_stream);
    if (st == SPF_OK)
      st = spf_select_topk_forced(it.chunk_scores, ceil_div(it.n_tokens, chunk), it.k, force_first, force_last, it.kept_chunks, cuda_stream);
    if (st == SPF_OK)
      st = spf_compact_spans(it.kept_chunks, it.k, chunk, it.n_tokens, it.token_ids, it.char_start, it.char_end, it.out_ids, it.out_pos,
                             it.out_tok_spans, it.out_char_spans, it.out_counts, cuda_stream);
    if (st != SPF_OK) return st;
  }
  return SPF_OK;
}

extern "C" int32_t spf_select_compact(const float* chunk_scores, int64_t n_chunks, int64_t k, int32_t chunk, int64_t n_tokens,
                                      const int32_t* token_ids, const int32_t* char_start, const int32_t* char_end,
                                      int32_t* kept_chunks, int32_t* out_ids, int32_t* out_pos, int32_t* out_tok_spans,
                                      int32_t* out_char_spans, int64_t* out_counts, void* cuda_stream) {
  clear_error();
  if (chunk_scores == nullptr || kept_chunks == nullptr || token_ids == nullptr || char_start == nullptr || char_end == nullptr ||
      out_ids == nullptr || out_tok_spans == nullptr || out_char_spans == nullptr || out_counts == nullptr)
    return fail(SPF_ERR_INVALID_ARG, "spf_select_compact: null pointer");
  if (chunk < 1) return fail(SPF_ERR_INVALID_ARG, "spf_select_compact: chunk must be >= 1 (got %d)", chunk);
  if (n_tokens < 1 || n_tokens > 0x7fffffff)
    return fail(SPF_ERR_INVALID_ARG, "spf_select_compact: n_tokens must be in [1, 2^31) (got %lld)", (long long)n_tokens);
  if (n_chunks != ceil_div(n_tokens, chunk))
    return fail(SPF_ERR_INVALID_ARG, "spf_select_compact: n_chunks must be ceil(n_tokens / chunk) (got %lld for %lld tokens)",
                (long long)n_chunks, (long long)n_tokens);
  if (k < 1 || k > n_chunks)
    return fail(SPF_ERR_INVALID_ARG, "spf_select_compact: k must be in [1, n_chunks] (got k=%lld, n_chunks=%lld)", (long long)k,
                (long long)n_chunks);
  if (n_chunks > kTailChunks || chunk > kShortChunk) {
    const int32_t st = spf_select_topk(chunk_scores, n_chunks, k, kept_chunks, cuda_stream);
    return st != SPF_OK ? st
                        : spf_compact_spans(kept_chunks, k, chunk, n_tokens, token_ids, char_start, char_end, out_ids, out_pos,
                                            out_tok_spans, out_char_spans, out_counts, cuda_stream);
  }
  spf_path_item it{};
  it.n_tokens = n_tokens;
  it.chunk_scores = const_cast<float*>(chunk_scores);   // importance is null: the scores are read
  it.k = k;
  it.token_ids = token_ids;
  it.char_start = char_start;
  it.char_end = char_end;
  it.kept_chunks = kept_chunks;
  it.out_ids = out_ids;
  it.out_pos = out_pos;
  it.out_tok_spans = out_tok_spans;
  it.out_char_spans = out_char_spans;
  it.out_counts = out_counts;
  return tail_launch(&it, 1, PoolRule{0, chunk, 1.f, false}, 0, static_cast<cudaStream_t>(cuda_stream));
}
