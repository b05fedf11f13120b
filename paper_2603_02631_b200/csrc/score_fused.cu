// Host side of the fused scoring path (kernel: fused.cuh): the split of a batch over the SMs, workspace layout, tensor
// maps, and the preparing kernel that runs in front of it.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "fused.cuh"

namespace spf {
namespace {

// ---------------------------------------------------------------------------------------------- preparing kernel
// One launch per group of prompts, one block per (slab, prompt): clears what the scoring kernel accumulates into, computes
// the slab's visit-1 reference, writes the layers' tensor maps (the host encodes one per prompt; the layers differ in the
// base address only) and the slab's query operand as the tensor cores read it: the scoring kernel fetches it with one plain
// bulk copy, where a tiled copy of its (head, lookahead) rows took the TMA engine about 20 cycles a row.
//
// 8-bit keys.  The tensor cores multiply E4M3 keys only by operands of an 8-bit format, so a slab's bf16 queries are handed
// over as two E4M3 terms, q * S = hi + lo: hi = the nearest E4M3 of q * S, lo = the nearest E4M3 of the remainder.  S is a
// power of two per slab that puts the slab's largest |q| just below the format's maximum (448).  A bf16 has 8 significant
// bits and each term carries 4, so the pair is exact for every element within 2^9 of the slab's largest and off by at most
// 2^-17 of that largest value below (the remainder's last bits fall under the format's smallest step, 2^-9).  Next to
// them goes the slab's factor from accumulated dot product to base-2 logit: softmax scale * log2(e) * key scale / S.
constexpr int kPrepThreads = 256;

struct PrepPrompt {
  CUtensorMap k_map;
  const void* k_layers[kFusedMaxLayers];
  const __nv_bfloat16* q;
  CUtensorMap* k_maps_out;
  uint4* clear[2];                 // two ranges to zero, clear_words[i] 16-byte words each
  int64_t clear_words[2];
  float *refs, *slab_c;
  unsigned char* q_tiles;
  const float* key_scale;          // 8-bit keys
  const int32_t* block_table;
  int64_t n_tokens, stride_head, stride_tok, stride_block, n_pool_blocks;
  int block_tokens;
};

template <int N>
struct PrepArgs {
  PrepPrompt prompt[N];
  int n_kv_heads, group, padded_group, n_lookahead, ncols;
  float c;
};

template <int D, bool FP8, int N>
__global__ void __launch_bounds__(kPrepThreads) fused_prep_kernel(const __grid_constant__ PrepArgs<N> a) {
  const PrepPrompt& p = a.prompt[blockIdx.y];
  const int slab = blockIdx.x, n_slabs = gridDim.x;
  const int layer = slab / a.n_kv_heads, hk = slab - layer * a.n_kv_heads;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ float red[kPrepThreads / 32];
  __shared__ float s_scale;

  grid_launch_dependents();                                         // the scoring kernel may set itself up meanwhile
  for (int i = 0; i < 2; ++i)
    for (int64_t w = (int64_t)slab * kPrepThreads + threadIdx.x; w < p.clear_words[i]; w += (int64_t)n_slabs * kPrepThreads)
      p.clear[i][w] = make_uint4(0, 0, 0, 0);

  // What follows is a chain of trips to memory that the scoring kernel waits for, so independent ones go first and none waits for
  // another's (tensor maps behind a fence and the query operand behind the reference: 41.0 instead of 39.9 us for 16 layers x 8
  // heads at 4001 tokens, 24.7 instead of 22.7 for one of the shortest prompts).
  //
  // tensor maps: the first slab of a layer writes the layer's
  // (one thread, whose stores are in order)
  if (hk == 0 && threadIdx.x == kPrepThreads - 32) {
#pragma unroll
    for (int i = 0; i < 8; ++i) reinterpret_cast<uint4*>(p.k_maps_out + layer)[i] = reinterpret_cast<const uint4*>(&p.k_map)[i];
    map_set_address(p.k_maps_out + layer, p.k_layers[layer]);
    map_release();
  }

  // the slab's query operand, 16 bytes of the swizzled image per thread and step: sub-tiles of `rows_stored` rows x one
  // swizzle span, the 16-byte chunks of a row permuted by the row's index (mod 8; 64-byte rows: by half of it, mod 4)
  const __nv_bfloat16* q = p.q + (int64_t)slab * (a.group * a.n_lookahead) * D;
  auto write_image = [&](float S) {
    constexpr int ROWB = row_bytes(D, FP8), SUBROW = sub_row_bytes(ROWB), CH = SUBROW / 16, KSUB = ROWB / SUBROW, EL = FP8 ? 16 : 8;
    const int rows_stored = image_rows(a.ncols), chunks = KSUB * rows_stored * CH;
    uint4* image = reinterpret_cast<uint4*>(p.q_tiles) + (int64_t)slab * (FP8 ? 2 : 1) * chunks;
    for (int idx = threadIdx.x; idx < chunks; idx += kPrepThreads) {
      const int h = idx / (rows_stored * CH), j = idx / CH % rows_stored, pos = idx % CH;
      const int chunk = pos ^ (CH == 8 ? j & 7 : (j >> 1) & 3);
      const QueryRow r = query_row(j, a.ncols, a.padded_group);
      const bool real = r.g < a.group && r.i < a.n_lookahead;
      const uint4* src = reinterpret_cast<const uint4*>(q + (int64_t)(r.g * a.n_lookahead + r.i) * D + h * (SUBROW / (FP8 ? 1 : 2)) + chunk * EL);
      if constexpr (!FP8) {
        image[idx] = real ? __ldg(src) : make_uint4(0, 0, 0, 0);
      } else {
        uint32_t hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
        if (real) {
  #pragma unroll
          for (int half = 0; half < 2; ++half) {
            const uint4 v = __ldg(src + half);
            const __nv_bfloat162* v2 = reinterpret_cast<const __nv_bfloat162*>(&v);
  #pragma unroll
            for (int x = 0; x < 8; ++x) {
              const float2 f = __bfloat1622float2(v2[x >> 1]);
              const float s = ((x & 1) ? f.y : f.x) * S;
              const uint32_t t = float_to_e4m3(s);
              hi[2 * half + (x >> 2)] |= t << (8 * (x & 3));
              lo[2 * half + (x >> 2)] |= float_to_e4m3(s - e4m3_to_float(t)) << (8 * (x & 3));
            }
          }
        }
        image[idx] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        image[chunks + idx] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      }
    }
  };
  if constexpr (!FP8) write_image(1.f);                             // (8-bit keys: the scale comes first)

  // reference: the smallest logit of the slab's rows against one fixed sample key, plus a margin (see fused.cuh).  A bad
  // block-table entry is clamped: this is a plain load, not a bounds-checked TMA copy
  const int64_t sample_key = p.n_tokens / 2;
  int64_t sample_block = 0, sample_row = sample_key;
  if (p.block_tokens > 0) {
    sample_block = min(max((int64_t)__ldg(p.block_table + sample_key / p.block_tokens), (int64_t)0), p.n_pool_blocks - 1);
    sample_row = sample_key % p.block_tokens;
  }
  constexpr int LPR = D / 8;                                        // lanes per row: 8 elements of it each
  const int rows = a.group * a.n_lookahead;
  const int64_t k_off = sample_block * p.stride_block + hk * p.stride_head + sample_row * p.stride_tok;
  float kf[8];
  if constexpr (FP8) {
    // strides count bytes; a lane's 8 elements are 8 bytes
    const uint2 kv = __ldg(reinterpret_cast<const uint2*>(static_cast<const unsigned char*>(p.k_layers[layer]) + k_off) + lane % LPR);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      kf[e] = e4m3_to_float(kv.x >> (8 * e));
      kf[4 + e] = e4m3_to_float(kv.y >> (8 * e));
    }
  } else {
    const uint4 kv = __ldg(reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(p.k_layers[layer]) + k_off) + lane % LPR);
    const __nv_bfloat162* k2 = reinterpret_cast<const __nv_bfloat162*>(&kv);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 f = __bfloat1622float2(k2[e]);
      kf[2 * e] = f.x;
      kf[2 * e + 1] = f.y;
    }
  }
  float ref = INFINITY, top = 0.f;                                  // smallest logit; largest |q| (8-bit keys)
  for (int r0 = warp * (32 / LPR); r0 < rows; r0 += (kPrepThreads / 32) * (32 / LPR)) {
    const int row = min(r0 + lane / LPR, rows - 1);                 // padding repeats a real row
    const uint4 qv = __ldg(reinterpret_cast<const uint4*>(q + (int64_t)row * D) + lane % LPR);
    const __nv_bfloat162* q2 = reinterpret_cast<const __nv_bfloat162*>(&qv);
    float dot = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 qf = __bfloat1622float2(q2[e]);
      dot = fmaf(kf[2 * e], qf.x, fmaf(kf[2 * e + 1], qf.y, dot));
      if constexpr (FP8) top = fmaxf(top, fmaxf(fabsf(qf.x), fabsf(qf.y)));
    }
#pragma unroll
    for (int off = LPR / 2; off >= 1; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    ref = fminf(ref, dot);
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    ref = fminf(ref, __shfl_xor_sync(0xffffffffu, ref, off));
    if constexpr (FP8) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
  }
  if (lane == 0) red[warp] = ref;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kPrepThreads / 32; ++w) ref = fminf(ref, red[w]);
    // a softmax scale (and a key scale) is positive, so the smallest q.k is the smallest logit
    p.refs[slab] = fmaf(ref, FP8 ? a.c * __ldg(p.key_scale + slab) : a.c, kRefMargin);
  }
  if constexpr (FP8) {
    __syncthreads();
    if (lane == 0) red[warp] = top;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kPrepThreads / 32; ++w) top = fmaxf(top, red[w]);
      // largest power of two S with top * S <= 448 (top = 0 or not finite: S = 1)
      float S = 1.f;
      if (top > 0.f && top < INFINITY) {
        int ex;
        (void)frexpf(448.f / top, &ex);                             // 448 / top = f * 2^ex, f in [0.5, 1)
        S = ldexpf(1.f, max(-100, min(ex - 1, 100)));
      }
      s_scale = S;
      p.slab_c[slab] = a.c * __ldg(p.key_scale + slab) / S;
    }
    __syncthreads();
  }
  if constexpr (FP8) write_image(s_scale);
}

template <int N>
int32_t launch_prep(const PrepArgs<N>& args, int d, bool fp8, int n_slabs, int n_prompts, cudaStream_t stream) {
  const dim3 grid((unsigned)n_slabs, (unsigned)n_prompts);
  if (fp8) {
    if (d == 64) fused_prep_kernel<64, true, N><<<grid, kPrepThreads, 0, stream>>>(args);
    else fused_prep_kernel<128, true, N><<<grid, kPrepThreads, 0, stream>>>(args);
  } else {
    if (d == 64) fused_prep_kernel<64, false, N><<<grid, kPrepThreads, 0, stream>>>(args);
    else fused_prep_kernel<128, false, N><<<grid, kPrepThreads, 0, stream>>>(args);
  }
  SPF_CUDA_CHECK(cudaGetLastError());
  return SPF_OK;
}

// ---------------------------------------------------------------------------------------------- the split over the SMs
constexpr int kSmemBudget = kFusedSmemMost - 1024;   // minus alignment slack
// Key bytes between the first and the second read of a tile (two-pass): what still sits in L2 (126 MB, in two halves).  A
// slab of more than kLongSlab tiles for every SM of the chip is far enough ahead with less, and more of it is still there
// (sustained, 64 rows at 131072 tokens 627 -> 605 us, 32 rows at 262000 507 -> 471); with 4 tiles less lead costs 3 %.
constexpr double kL2KeyBytes = 80e6, kL2KeyBytesLong = 60e6;
constexpr int kLongSlab = 5;
// What an SM's share of the memory bandwidth brings in a microsecond: at the rate of a copy (6.5 TB/s over 148 SMs), and at that of
// a kernel that only reads (7.2 TB/s), which the resident form comes close to.
constexpr double kSmBytesPerUs = 44e3, kReadBytesPerUs = 49e3;
// Resident, fitted to 93 splits of 29 prompts, 1500 to 250003 tokens, timed under a sustained load (mean error 5.5 %; the split that
// it picks is 0.8 % slower than the best of those measured): microseconds from a slab's last key to its log-sum-exps being back,
// what a tile of the next slab takes when its keys are there already, what the sums of a slab take on top of their tiles and for
// two tiles of 32 rows, and what it costs groups to meet in global memory.
constexpr double kHandoverUs = 2.5, kBurstUs = 0.35, kSlabUs = 0.5, kTwoTilesUs = 0.45, kMeetUs = 4.0;
// What a tile of the next slab takes more where the max warps load and store its maxima in tensor memory, a slot of a key.  Without it
// 12 layers x 4 heads of 64 dimensions, 2 x 16 rows, went over 382 tiles as two groups of 64 CTAs with six tiles each: 101 us, and 83 as
// one group of 128 with three.  Of 456 prompts of 5 to 1016 tiles, 4 to 128 slabs, it changes the split of 11, none for the worse; 90
// others whose split it changes take 0.95 of the time on average (0.71 to 1.11).
constexpr double kFoldUs = 0.0125;
// 32 rows: the resident form wants room for the keys of so many microseconds beside a slab's tiles.  Sustained, 64 dimensions, bf16:
// with 10 tiles a CTA and room for 13 a pass over 180000 tokens takes 761 us and 622 in two passes, with 7 and 12 (16 slots a
// key) 577 and 457, with 7 and 16 441 and 456.  8-bit keys, 128 slabs: with 9 and 13 622 and 483, with 7 and 12 527 and 399, with 6
// and 16 334 and 336, with 8 and 16 424 and 433 (48 slabs: the two-pass form is 6 to 9 % quicker); 128 dimensions, with 9 and 13
// 704 and 726, with 8 and 12 670 and 668.
constexpr double kSpareUs = 2.0;
// 16 rows: a slab's keys take longer than their sums, and the resident form is the quicker one with any room to speak of: 128
// dimensions, bf16, with 18 tiles and room for 23 480 us and 790 in two passes, 8-bit keys 569 and 641.  With 64 dimensions, where
// products cost half as much, this ends at 8 slots a key (bf16: with 16 and 24 262 and 254; with 4 slots, 17 and 27, 1.03 times as
// long in two passes; 8-bit keys: 338 and 368) or at 16 (bf16: with 13 and 19 232 and 211; 8-bit keys: 330 and 309): the max warps
// move as many columns of maxima as of logits, and where tensor memory does not hold two slabs the next one waits for them.
constexpr int kSpareTiles = 3;

struct Geometry {
  bool ok = false, fp8 = false, once = false;
  int ncols = 0, padded_group = 0, n_slabs = 0, tile_bytes = 0;
  int max_tiles = 0;      // tiles per CTA whose running maxima fit tensor memory next to the least number of stages
  int lead = 0;           // two-pass: tiles of lead over visit 2 that L2 holds
  int handover = 0;       // two-pass: tiles that arrive while a slab's sums travel to the other SMs and come back
  // Resident form: tiles whose logits fit tensor memory next to the running maxima of `tiles` tiles.
  int resident(int tiles) const {
    return std::min(kMaxResident, (kTmemColsAll - (max_in_regs(tiles) ? 0 : tiles * (ncols / padded_group))) / ncols);
  }
  bool max_in_regs(int tiles) const { return tiles <= kRegTiles && ncols / padded_group <= kRegSlots; }
  bool holds(int64_t tiles) const { return tiles <= max_tiles && (!once || resident((int)tiles) > tiles); }   // of a CTA and slab
  int most_tiles() const {
    int t = 1;
    while (holds(t + 1)) ++t;
    return t;
  }
  // Most tiles a CTA and slab that leave the two visits room to overlap.
  int comfortable_tiles() const {
    if (!once) return std::max(1, (lead - handover) / 2);           // visit 2 takes as long as visit 1
    int t = 1;
    while (2 * resident(t + 1) >= 3 * (t + 1)) ++t;
    return t;
  }
};

Geometry geometry(const ScoreProblem& p, int sm_count) {
  Geometry g;
  g.fp8 = p.k_scale != nullptr;
  // 8-bit key caches: contiguous only, and the TMA wants 16-byte aligned layer pointers and strides (the general path reads
  // them 8 bytes at a time and takes what this refuses)
  if (g.fp8) {
    if (p.block_tokens > 0 || p.stride_tok % 16 != 0 || p.stride_head % 16 != 0) return g;
    for (int l = 0; l < p.n_layers; ++l)
      if (reinterpret_cast<uintptr_t>(p.k.p[l]) % 16 != 0) return g;
  }
  if (reinterpret_cast<uintptr_t>(p.q) % 16 != 0) return g;
  if (p.group > 8 || p.n_layers > kFusedMaxLayers || p.n_tokens > (int64_t)1 << 30) return g;
  g.padded_group = p.group <= 2 ? p.group : p.group <= 4 ? 4 : 8;
  const int rows = g.padded_group * p.n_lookahead;
  if (rows > 64) return g;
  g.ncols = rows <= 16 ? 16 : rows <= 32 ? 32 : 64;
  g.n_slabs = p.n_layers * p.n_kv_heads;
  g.tile_bytes = kTileKeys * row_bytes(p.head_dim, g.fp8);
  g.handover = std::max(2, (int)(3.0 * kSmBytesPerUs / g.tile_bytes));
  const int tiles = (int)std::min<int64_t>(ceil_div(ceil_div(p.n_tokens, kTileKeys), std::min(sm_count, kFusedMaxCtas)), 1 << 20);
  g.lead = std::max(2, (int)((tiles > kLongSlab ? kL2KeyBytesLong : kL2KeyBytes) / ((double)sm_count * g.tile_bytes)));
  const int spare = g.resident(tiles) - tiles, slots = g.ncols / g.padded_group;
  if (g.ncols == 32) g.once = spare >= std::max(kSpareTiles, (int)std::ceil(kSpareUs * kSmBytesPerUs / g.tile_bytes));
  if (g.ncols == 16) g.once = spare >= (p.head_dim == 64 && slots >= (g.fp8 ? 16 : 8) ? std::max(kSpareTiles, tiles) : kSpareTiles);
  g.max_tiles = (kTmemColsAll - 4 * g.ncols) / (g.ncols / g.padded_group);
  g.ok = tiles <= g.max_tiles;
  return g;
}

struct Split {
  int parts = 1, per_part = 1, tiles = 1;   // `tiles` per CTA of a group
  double cost = 0;                          // time, in tiles that an SM's share of the memory bandwidth brings
};

// Time of a prompt of T tiles x S slabs as `parts` groups of `per_part` CTAs, fitted to measurements at 1.5k to 250k tokens.
// Three things can bound it, and near a tie they add up:
//   memory: the average, not the CTA with the most tiles (one with more than its share gets more bandwidth);
//   latency (resident): a tile's place is taken until its slab's log-sum-exps are back, and there is room for `held` slabs;
//   the sum warps, which every slab costs something on top of its tiles.
// Two-pass: the tiles, stretched where L2 does not hold the lead that the hand-over takes.
double split_cost(const Geometry& g, int64_t n_tiles, int tiles, int parts, int share) {
  const int slabs = (g.n_slabs + parts - 1) / parts;
  const double units = (double)tiles * slabs, fair = (double)n_tiles * g.n_slabs / share;
  if (!g.once) {
    const double stretch = units > g.lead ? std::max(1.0, (double)(2 * tiles + g.handover) / g.lead) : 1.0;
    return units * stretch + 0.1 * slabs + 2.0 * tiles;
  }
  const double us = g.tile_bytes / kReadBytesPerUs, per_tile = (double)g.resident(tiles) / tiles;
  const double held = std::max(1.0, 0.5 * (per_tile + std::floor(per_tile)));
  const double burst = kBurstUs + (g.max_in_regs(tiles) ? 0.0 : kFoldUs * g.ncols / g.padded_group);
  const double latency = std::max(kHandoverUs / us + tiles, slabs / held * (kHandoverUs + tiles * burst) / us);
  const double sums = slabs * (kSlabUs + kTwoTilesUs * g.ncols / 32 * ((tiles + 1) / 2)) / us;
  return std::cbrt(fair * fair * fair + latency * latency * latency + sums * sums * sums) + 2.5 * tiles + (parts > 1 ? kMeetUs / us : 0.0);
}

// The best split over at most `ctas` CTAs; cost < 0 if there is none.  `share`: CTAs among which the memory bandwidth is
// divided, for this prompt's part of it.
Split best_split(const Geometry& g, int64_t n_tiles, int ctas, int share) {
  Split best;
  best.cost = -1;
  for (int parts = 1; parts <= std::min(ctas, g.n_slabs); ++parts) {
    const int most = (int)std::min<int64_t>(ctas / parts, n_tiles);
    const int64_t tiles = ceil_div(n_tiles, most);
    if (!g.holds(tiles)) break;
    const int per_part = (int)ceil_div(n_tiles, tiles);              // no more CTAs than these tiles need
    const double cost = split_cost(g, n_tiles, (int)tiles, parts, share);
    if (best.cost < 0 || cost < best.cost * 0.999) {
      best.parts = parts;
      best.per_part = per_part;
      best.tiles = (int)tiles;
      best.cost = cost;
    }
  }
  return best;
}

// Splits a group of prompts, as group_size made it, over the SMs, each on CTAs of its own: CTAs in proportion to the tiles, but
// as many as hold them (what that hands out too many comes from the prompts with the most to spare), then a few moves from
// the prompt that would be done first to the one that would be done last.
bool split_group(const Geometry* g, const int64_t* n_tiles, int n, int sm_count, Split* out) {
  if (n == 1) {
    out[0] = best_split(g[0], n_tiles[0], sm_count, sm_count);
    return out[0].cost >= 0;
  }
  const int most = g[0].most_tiles();                                // the same for all: they differ in lead alone
  int64_t total = 0;
  for (int i = 0; i < n; ++i) total += n_tiles[i];
  int least[kFusedMaxBatch], ctas[kFusedMaxBatch], left = sm_count;
  for (int i = 0; i < n; ++i) {
    least[i] = (int)ceil_div(n_tiles[i], most);
    left -= ctas[i] = std::max(least[i], (int)(n_tiles[i] * sm_count / total));
  }
  for (; left < 0; ++left) {
    int rich = 0;
    for (int i = 1; i < n; ++i)
      if (ctas[i] - least[i] > ctas[rich] - least[rich]) rich = i;
    --ctas[rich];
  }
  for (int i = 0; i < n; ++i) out[i] = best_split(g[i], n_tiles[i], ctas[i], ctas[i]);
  for (int step = 0; step < 32; ++step) {
    int slow = 0, quick = -1;
    for (int i = 1; i < n; ++i)
      if (out[i].cost > out[slow].cost) slow = i;
    if (left == 0) {
      for (int i = 0; i < n; ++i)
        if (i != slow && ctas[i] > least[i] && (quick < 0 || out[i].cost < out[quick].cost)) quick = i;
      if (quick < 0 || out[quick].cost > 0.9 * out[slow].cost) break;
    }
    const Split slow_was = out[slow], quick_was = quick >= 0 ? out[quick] : Split{};
    if (quick >= 0) {
      --ctas[quick];
      out[quick] = best_split(g[quick], n_tiles[quick], ctas[quick], ctas[quick]);
    } else {
      --left;
    }
    ++ctas[slow];
    out[slow] = best_split(g[slow], n_tiles[slow], ctas[slow], ctas[slow]);
    if (quick >= 0 && out[quick].cost >= slow_was.cost) {            // no better: take the move back and stop
      out[quick] = quick_was;
      out[slow] = slow_was;
      break;
    }
  }
  for (int i = 0; i < n; ++i)
    if (out[i].cost < 0) return false;
  return true;
}

// How many prompts, from the first on, go into one launch: while their tiles leave the visits room to overlap, and while there
// are CTAs that hold them.
int group_size(const Geometry* g, const int64_t* n_tiles, int n, int sm_count) {
  const int held = g[0].most_tiles();
  double tiles = 0, most = 1e30;
  int64_t ctas = 0;
  int count = 0;
  while (count < n) {
    tiles += (double)n_tiles[count];
    most = std::min(most, (double)g[count].comfortable_tiles() * sm_count);
    ctas += ceil_div(n_tiles[count], held);
    if (count > 0 && (tiles > most || ctas > sm_count)) break;
    ++count;
  }
  return count;
}

// Shared-memory and tensor-memory stages for CTAs that hold the running maxima of `tiles` tiles.
bool pick_stages(const Geometry& g, int d, int tiles, bool paged, FusedArgs* a, int* smem_bytes) {
  a->table_tiles = paged ? tiles : 0;
  if (g.once) {
    a->max_in_regs = g.max_in_regs(tiles);
    a->t_stages[0] = g.resident(tiles);
    a->t_stages[1] = 0;
    for (int ks = kMaxKeyStages; ks >= 2; --ks) {
      a->k_stages[0] = ks;
      a->k_stages[1] = 0;
      const FusedSmem lay = fused_smem(d, g.fp8, g.ncols, true, a->table_tiles, a->k_stages);
      if ((int)lay.total <= kSmemBudget) {
        *smem_bytes = (int)lay.total + 1024;
        return a->t_stages[0] > tiles;
      }
    }
    return false;
  }
  // as many accumulator stages as fit, visit 1 first (its epilogue is the longer one)
  const int stages = std::min(2 * kMaxTmemStages, (kTmemColsAll - tiles * (g.ncols / g.padded_group)) / g.ncols);
  if (stages < 4) return false;                                      // two for each visit (see fused_multiply)
  a->t_stages[0] = (stages + 1) / 2;
  a->t_stages[1] = stages / 2;
  for (int ks = 20; ks >= 4; --ks) {
    a->k_stages[0] = (ks + 1) / 2;
    a->k_stages[1] = ks / 2;
    const FusedSmem lay = fused_smem(d, g.fp8, g.ncols, false, a->table_tiles, a->k_stages);
    if ((int)lay.total <= kSmemBudget) {
      *smem_bytes = (int)lay.total + 1024;
      return true;
    }
  }
  return false;
}

// ---------------------------------------------------------------------------------------------- workspace
struct FusedWorkspace {
  size_t k_maps, refs, slab_c, q_tiles;              // written by the preparing kernel
  size_t row_sums, lse;                              // cleared by it, the sums as far as used
  size_t finished, amax;                             // cleared by it where groups meet
  size_t total;
};

FusedWorkspace fused_workspace(const ScoreProblem& p) {
  const size_t n_slabs = (size_t)p.n_layers * p.n_kv_heads, n_tiles = (size_t)ceil_div(p.n_tokens, kTileKeys);
  const int ncols = 64;                              // whatever the padding of the group makes of the rows
  FusedWorkspace w;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align_up(o + bytes, 256);
    return at;
  };
  w.k_maps = take((size_t)p.n_layers * sizeof(CUtensorMap));
  w.refs = take(n_slabs * sizeof(float));
  w.slab_c = take(p.k_scale != nullptr ? n_slabs * sizeof(float) : 0);
  w.q_tiles = take(n_slabs * 2 * ncols * (size_t)p.head_dim);     // bf16, or two 8-bit terms
  w.row_sums = take(n_slabs * std::min<size_t>(n_tiles, kFusedMaxCtas) * ncols * sizeof(float));
  w.lse = take(n_slabs * ncols * sizeof(unsigned long long));
  w.finished = take(n_tiles * 4 * sizeof(unsigned));
  w.amax = take((size_t)p.n_lookahead * n_tiles * kTileKeys * sizeof(unsigned));
  w.total = o;
  return w;
}

// ---------------------------------------------------------------------------------------------- tensor maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static std::once_flag once;
  static EncodeTiledFn fn = nullptr;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult res;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &res) == cudaSuccess &&
        res == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// The prompt's key map.  A key tile is ONE copy of (sub-row, 128 keys, sub-tiles): a row longer than the swizzle span is
// seen as several sub-rows, one span apart.
int32_t encode_key_map(const ScoreProblem& p, const Geometry& g, CUtensorMap* map) {
  EncodeTiledFn encode = encode_fn();
  if (encode == nullptr) return fail(SPF_ERR_CUDA, "spf_score: cuTensorMapEncodeTiled is not available from the driver");
  const int d = p.head_dim, es = g.fp8 ? 1 : 2;
  const int subrow = sub_row_bytes(row_bytes(d, g.fp8)), ksub = row_bytes(d, g.fp8) / subrow;
  const cuuint64_t x = (cuuint64_t)(subrow / es), hkv = (cuuint64_t)p.n_kv_heads;
  const bool paged = p.block_tokens > 0;
  // paged: a table entry outside the pool reads as zeros instead of faulting
  const cuuint64_t tokens = paged ? (cuuint64_t)p.block_tokens : (cuuint64_t)p.n_tokens;
  const cuuint64_t tok_stride = paged ? (cuuint64_t)d : (cuuint64_t)p.stride_tok;
  const cuuint64_t head_stride = paged || p.n_kv_heads == 1 ? tok_stride * tokens : (cuuint64_t)p.stride_head;
  const cuuint64_t dims[5] = {x, tokens, (cuuint64_t)ksub, hkv, (cuuint64_t)p.n_pool_blocks};
  const cuuint64_t strides[4] = {tok_stride * es, (cuuint64_t)subrow, head_stride * es, hkv * head_stride * es};
  const cuuint32_t box[5] = {(cuuint32_t)x, (cuuint32_t)kTileKeys, (cuuint32_t)ksub, 1, 1};
  const cuuint32_t ones[5] = {1, 1, 1, 1, 1};
  const CUresult r = encode(map, g.fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, paged ? 5 : 4,
                            const_cast<__nv_bfloat16*>(p.k.p[0]), dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            subrow == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(SPF_ERR_CUDA, "spf_score: encoding the key tensor map failed (CUresult %d)", (int)r);
  return SPF_OK;
}

template <int N>
int32_t launch_group(const ScoreProblem* p, int n, const Geometry* geometries, const Split* split, char* base, int sm_count, int32_t* dev_status,
                     cudaStream_t stream, int mode, const float* lse_in) {
  PrepArgs<N> prep{};
  FusedArgs args{};
  const ScoreProblem& p0 = p[0];
  const Geometry& g = geometries[0];                                 // the prompts' differ in lead alone
  prep.n_kv_heads = args.n_kv_heads = p0.n_kv_heads;
  prep.group = args.group = p0.group;
  prep.padded_group = g.padded_group;
  prep.n_lookahead = args.n_lookahead = p0.n_lookahead;
  prep.ncols = g.ncols;
  prep.c = args.c = p0.c_log2;
  args.n_prompts = n;
  args.n_layers = p0.n_layers;
  args.mode = mode;
  args.dev_status = dev_status;
  FusedLaunch l{g.ncols, g.padded_group, 0, 0, g.once};
  int most_tiles = 1;
  for (int i = 0; i < n; ++i) {
    const ScoreProblem& q = p[i];
    const FusedWorkspace w = fused_workspace(q);
    PrepPrompt& pp = prep.prompt[i];
    FusedPrompt& fp = args.prompt[i];
    const int32_t st = encode_key_map(q, g, &pp.k_map);
    if (st != SPF_OK) return st;
    const bool meet = split[i].parts > 1;
    for (int layer = 0; layer < q.n_layers; ++layer) pp.k_layers[layer] = q.k.p[layer];
    pp.q = q.q;
    pp.k_maps_out = reinterpret_cast<CUtensorMap*>(base + w.k_maps);
    // the sums of a narrower geometry, or of fewer CTAs, use (and clear) the front of their region
    pp.clear[0] = reinterpret_cast<uint4*>(base + w.row_sums);
    pp.clear_words[0] = (int64_t)g.n_slabs * split[i].per_part * g.ncols * (int64_t)sizeof(float) / 16;
    pp.clear[1] = reinterpret_cast<uint4*>(base + w.lse);
    pp.clear_words[1] = (int64_t)(((meet ? w.total : w.finished) - w.lse) / 16);
    pp.refs = reinterpret_cast<float*>(base + w.refs);
    pp.slab_c = reinterpret_cast<float*>(base + w.slab_c);
    pp.q_tiles = reinterpret_cast<unsigned char*>(base + w.q_tiles);
    pp.key_scale = q.k_scale;
    pp.block_table = q.block_table;
    pp.n_tokens = q.n_tokens;
    pp.stride_head = q.stride_head;
    pp.stride_tok = q.stride_tok;
    pp.stride_block = (int64_t)q.n_kv_heads * q.block_tokens * q.head_dim;
    pp.n_pool_blocks = q.n_pool_blocks;
    pp.block_tokens = q.block_tokens;

    fp.k_maps = pp.k_maps_out;
    fp.q_tiles = pp.q_tiles;
    fp.row_sums = reinterpret_cast<float4*>(base + w.row_sums);
    fp.lse = reinterpret_cast<unsigned long long*>(base + w.lse);
    fp.refs = pp.refs;
    fp.slab_c = g.fp8 ? pp.slab_c : nullptr;
    fp.amax = reinterpret_cast<unsigned*>(base + w.amax);
    fp.finished = reinterpret_cast<unsigned*>(base + w.finished);
    fp.importance = q.importance;
    fp.lse_out = q.lse_out;
    fp.extra_lse = q.extra_lse;
    fp.lse_in = lse_in;
    fp.block_table = q.block_table;
    fp.n_tokens = q.n_tokens;
    fp.block_tokens = q.block_tokens;
    fp.n_tiles = (int)ceil_div(q.n_tokens, kTileKeys);
    fp.cta0 = l.n_cta;
    fp.parts = split[i].parts;
    fp.per_part = split[i].per_part;
    fp.lead = std::max(geometries[i].lead, split[i].tiles + g.handover);
    l.n_cta += split[i].parts * split[i].per_part;
    if ((int64_t)split[i].tiles * split[i].per_part < fp.n_tiles || l.n_cta > sm_count)
      return fail(SPF_ERR_UNSUPPORTED, "spf_score: no split of %d key tiles over the SMs", fp.n_tiles);
    most_tiles = std::max(most_tiles, split[i].tiles);
    base += w.total;
  }
  if (!pick_stages(g, p0.head_dim, most_tiles, p0.block_tokens > 0, &args, &l.smem_bytes))
    return fail(SPF_ERR_UNSUPPORTED, "spf_score: shape not covered by the fused path");
  const int32_t st = launch_prep<N>(prep, p0.head_dim, g.fp8, g.n_slabs, n, stream);
  if (st != SPF_OK) return st;
  if (p0.head_dim == 64) return g.fp8 ? fused_launch_d64_fp8(args, l, stream) : fused_launch_d64(args, l, stream);
  return g.fp8 ? fused_launch_d128_fp8(args, l, stream) : fused_launch_d128(args, l, stream);
}

// One CTA waits on an mbarrier that nothing ever arrives on, with the kernels' own bounded wait and a 20 ms limit: the wait
// must give up, record SPF_ERR_TIMEOUT and let the kernel return normally.
__global__ void bounded_wait_selftest_kernel(int32_t* dev_status) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const Abort ab{&abort_flag, dev_status, 20000000ull};
  mbar_wait_warp(smem_u32(&bar), 0u, ab);
  __syncthreads();
}

}  // namespace

int32_t bounded_wait_selftest_launch(int32_t* dev_status, cudaStream_t stream) {
  bounded_wait_selftest_kernel<<<1, 64, 0, stream>>>(dev_status);
  SPF_CUDA_CHECK(cudaGetLastError());
  return SPF_OK;
}

bool score_fused_supported(const ScoreProblem& p, int sm_count) { return geometry(p, sm_count).ok; }

size_t score_fused_workspace_bytes(const ScoreProblem& p) { return fused_workspace(p).total; }

int32_t score_fused_launch(const ScoreProblem* p, int n_prompts, void* workspace, int sm_count, int32_t* dev_status, cudaStream_t stream,
                           int* done, int mode, const float* lse_in) {
  sm_count = std::min(sm_count, kFusedMaxCtas);
  Geometry g[kFusedMaxBatch];
  int64_t n_tiles[kFusedMaxBatch];
  int n = 0;
  for (; n < std::min(n_prompts, kFusedMaxBatch); ++n) {
    g[n] = geometry(p[n], sm_count);
    if (n > 0 && (!g[n].ok || g[n].once != g[0].once)) break;  // refused, or scored in the other form, when its turn comes
    if (!g[n].ok) return fail(SPF_ERR_UNSUPPORTED, "spf_score: shape not covered by the fused path");
    n_tiles[n] = ceil_div(p[n].n_tokens, kTileKeys);
  }
  n = group_size(g, n_tiles, n, sm_count);
  Split split[kFusedMaxBatch];
  if (!split_group(g, n_tiles, n, sm_count, split)) return fail(SPF_ERR_UNSUPPORTED, "spf_score: shape not covered by the fused path");
  if (done != nullptr) *done = n;
  char* base = static_cast<char*>(workspace);
  return n == 1 ? launch_group<1>(p, n, g, split, base, sm_count, dev_status, stream, mode, lse_in)
                : launch_group<kFusedMaxBatch>(p, n, g, split, base, sm_count, dev_status, stream, mode, lse_in);
}

}  // namespace spf
