// Token-importance scoring, fused path: ONE persistent kernel that reads the key cache once from HBM.
//
// Why logits are looked at twice.  The max over (layer, head) is taken over softmax PROBABILITIES, so a logit can only be
// compared across heads after its row's log-sum-exp is known, and that needs all N keys of the row.  Each (layer, kv-head)
// slab of keys is therefore visited twice:
//   visit 1 ("sum")  accumulates  sum_s exp2(c * q.k - ref)  per query row;
//   visit 2 ("max")  folds  max_{l,h} (c * q.k - lse)  into a running maximum per (lookahead i, key s).
//
// Two forms of the kernel, by what lies between the visits.
//   Resident (template ONCE): the logits wait in tensor memory.  A tile's 128 x NCOLS accumulators are summed by the sum
//   warps and stay where they are until the slab's log-sum-exps arrive; then the max warps fold them and free the columns.
//   Keys are copied and multiplied once.  This needs room for a CTA's tiles of one slab plus those that arrive during the
//   hand-over: up to 32 query rows, and prompts of up to a few hundred thousand tokens (see Geometry::resident).
//   Two-pass: the logits are recomputed.  The two visits are two independent pipelines (TMA warp -> key ring -> MMA warp ->
//   tensor-memory ring -> epilogue warps) that share the SM and meet only in the log-sum-exps.  Visit 2 follows visit 1 over
//   the same list of tiles as soon as a slab's log-sum-exps are there; visit 1 may be at most `lead` tiles ahead of it, so
//   that the second read still finds its tiles in L2.  For 64 query rows, where tensor memory holds six tiles' logits.
//
// Work split.  A prompt has T tiles of 128 keys and S slabs.  Its CTAs form `parts` groups; group p takes the slabs s with
// s % parts == p and its CTAs deal the T tiles out among themselves.  One group (parts = 1) is the plain split for long
// prompts: a CTA owns its tiles for all slabs and writes their importance alone.  More groups are what keeps the chip busy
// when there are fewer tiles than SMs, and what evens out a last round of tiles that would leave most SMs idle; the groups'
// running maxima then meet in global memory (integer max on order-preserving bits, exact and independent of order), and the
// last group to finish 32 keys turns them into importance.  Several prompts share one launch, each with CTAs of its own.
//
// Tensor-core tiles.  The operands in shared memory are 128 keys x d (TMA) and the slab's query rows x d (query_row: row j
// is lookahead i and head g of the GQA group, the group padded to a power of two).  Resident, and visit 2 of the two-pass form:
// keys are the tensor-memory lanes.  A thread has four keys of every fourth column, and the rows are dealt to the columns so that
// these are all heads of a lookahead: the max over them is in-thread, a thread needs a quarter of the log-sum-exps, and the sum
// over keys ends every slab with a reduction over eight lanes of up to 8 columns.  Visit 1 of the two-pass form, 32 rows and more: query rows are the lanes
// (weight-stationary instructions, which fill all 128 lanes with 32 or 64 rows), so the sum over keys stays inside a thread
// too; with 64 columns the reduction cost 1000 to 2900 cycles per slab and CTA.  With 16 rows half of those lanes would be
// padding, and twice the tensor memory: keys are the lanes there.  The running maxima live in tensor memory next to the
// accumulators.
//
// Warps.  0 / 1: TMA producers of visit 1 / visit 2.  2 / 3: MMA issuers (resident: 0 and 2 alone).  4: fetches log-sum-exps for
// visit 2.  5..7: publishers (store this CTA's row sums of a slab; add up all CTAs' sums of the rows this CTA owns).  In groups of
// few CTAs one warp stores and others add up all rows instead: resident, 1 and 4..7; two-pass, 6 and 4..5.  8..15: "sum" warps.  16..23:
// "max" warps.  Of the eight warps of a visit, warp % 4 picks the TMEM lane quadrant and the next bit the `set`: the two sets
// take turns at the tiles, so that one set's tensor-memory loads and waits run while the other set computes.  (Splitting every tile's columns between the sets kept all eight warps in step,
// all waiting or all computing.)
//
// Reference.  Visit 1 subtracts one reference per slab inside the exp2 argument: the SMALLEST logit of the slab's rows
// against one fixed sample key, plus a margin of 60 (base-2 units).  Every row's largest logit is at least its own sample
// logit, hence at least reference - 60, and ex2.approx.ftz only flushes terms below reference - 126, i.e. terms more than
// 2^66 times smaller than the row's largest: no row can lose anything that matters, whatever the spread between the heads
// of a group.  What can still go wrong is overflow: a row sum reaches 2^128 when some logit lies about 188 - log2(keys at
// that level) base-2 units (157 at the very least, about 109 nats) above the slab's smallest sample logit.  That is
// detected (the sum is inf) and reported as SPF_ERR_RANGE; the caller can then use the general path.
//
// Cross-CTA step.  All CTAs use the same reference for a slab, so their partial sums can simply be added.  Each CTA stores
// its sums as plain words, [slab][CTA of the group][four rows], zero meaning "not there yet".  In a group of few CTAs
// everybody reads everybody's words and adds them up; in a larger one every four rows of a slab have an owner, which does
// that and stores the log-sum-exps as 64-bit words {value, 1} that every CTA polls.  Sums are taken in double and in a fixed
// order, so every run arrives at the same bits.  No atomics, no fences, no counters: 2 or 3 us from a slab's last sum to its
// log-sum-exps everywhere, where exact atomic sums with an arrival counter took 5.4.  This latency is what the split over
// the SMs is built around: how far visit 2 trails visit 1 is what has to fit in tensor memory (or in L2).  Visit 1 waits for
// other CTAs only through that room, which covers at least one whole slab, so every slab's sums complete and the words
// always arrive.
//
// Every wait on a barrier, word or flag in this file is bounded: on expiry the kernel records SPF_ERR_TIMEOUT, drains and
// returns normally.  The one wait that has no limit is the hardware's own: tcgen05.alloc blocks while another resident CTA
// on the SM holds tensor memory (this kernel asks for all of it), i.e. until that CTA exits.
#pragma once

#include "score.cuh"
#include "tc_ptx.cuh"

namespace spf {

constexpr int kFusedThreads = 768;
constexpr int kFusedSmemMost = 227 * 1024;   // dynamic shared memory of a CTA
constexpr int kVisitWarps = 8;         // epilogue warps per visit
constexpr int kSumWarp0 = 8, kMaxWarp0 = 16;
// Groups of up to this many CTAs add up everybody's row sums in every CTA (see fused_gather): one hop instead of two, for reading
// up to 7 KB a slab and CTA.  Up to 56, which are seven words of 128 bits a lane with 32 rows: three groups of 49 CTAs with 32 rows
// each take 178 us for 16 layers x 8 heads at 50000 tokens, in two hops 200; one prompt of 2 to 56 tiles and 16 or 128 slabs is up to
// 16 % faster and never more than 2 % slower; two groups of 74 gained nothing.  64 rows have one pair of warps for it, to which a slab
// of many CTAs is more work than its tiles: over 128 slabs, 8 CTAs to a group take 0.99 of the time in two hops, 12 1.01, 16 1.09, 28
// 1.20 (71.7 us for 8 heads x 8 of 64 dimensions at 3554 tokens, 58.2 in two hops; 54.6 and 68.8 with the keys in L2).
__host__ __device__ constexpr int gather_ctas(int ncols) { return ncols == 64 ? 12 : 56; }
__host__ __device__ constexpr bool gather_alone(int ncols, int n_ctas) { return n_ctas <= gather_ctas(ncols); }
constexpr int kFetchWarp = 4, kPublisherWarp0 = 5, kPublisherWarps = 3;
constexpr int kGatherWarp0 = 4, kTeamWarps = 2;
__host__ __device__ constexpr int gather_teams(bool once) { return once ? 2 : 1; }
__host__ __device__ constexpr int store_warp(bool once) { return once ? 1 : kGatherWarp0 + kTeamWarps; }   // one that has nothing else to do
constexpr int kMaxQStages = 4;         // query tiles in flight per visit (two-pass: 2)
constexpr int kMaxKeyStages = 16;      // key tiles in flight per visit
// Two-pass: accumulator stages per visit.  64 rows at 131072 tokens have three for each visit; with two for each set of visit 1
// and one for each of visit 2 (as many in all) a pass took 559 instead of 519 us, with 8-bit keys 581 instead of 530.
constexpr int kMaxTmemStages = 16;
constexpr int kMaxResident = 32;       // resident: tiles in tensor memory
constexpr int kRegTiles = 8, kRegSlots = 8;   // running maxima stay in registers up to this many tiles a CTA and lookahead slots a key
constexpr int kTmemColsAll = 512;      // the CTA takes all of its SM's tensor memory
constexpr int kOffSlots = 4;           // slabs whose log-sum-exps may be in shared memory at once
constexpr int kSumSlots = 4;           // slabs whose row sums may be on their way to the publishers at once
constexpr float kRefMargin = 60.f;     // base-2 units added to the sampled reference logit

// Key rows are d bf16 (128 or 256 bytes) or d E4M3 bytes (64 or 128).  A tile is stored as sub-tiles of 128 keys x one
// swizzle span: 128 bytes of the row (128-byte swizzle), or the whole row where it has only 64 bytes (64-byte swizzle).
__host__ __device__ constexpr int row_bytes(int d, bool fp8) { return fp8 ? d : 2 * d; }
__host__ __device__ constexpr int sub_row_bytes(int rowb) { return rowb > 128 ? 128 : rowb; }
// Rows of a slab's query operand in shared memory.  16 rows are stored as 32, of which the upper half is zero and not read: with
// the room that this leaves, keys of 128 dimensions have five stages.  With a sixth, 28 layers at 250003 tokens took 2160
// instead of 2126 us.
__host__ __device__ constexpr int image_rows(int ncols) { return ncols < 32 ? 32 : ncols; }
// Two-pass, visit 1: query rows are the accumulator's lanes, 32 rows x 32 columns or 64 x 64 a tile.  Else keys x query rows;
// either way a tile has as many columns as query rows.
__host__ __device__ constexpr bool sums_by_rows(bool once, int ncols) { return !once && ncols >= 32; }

// Which query row is column j of the logits (row j of the slab's query operand): lookahead i, head g of the GQA group, padded to a
// power of two.  A thread that has every fourth column of a key has all heads of a lookahead (of two columns' distance where there
// are only 16 columns for 8 heads).
struct QueryRow {
  int i, g;
};
__host__ __device__ constexpr QueryRow query_row(int j, int ncols, int padded_group) {
  const int t = j & 3, c = j >> 2;
  return ncols == 16 && padded_group == 8 ? QueryRow{t >> 1, 2 * c + (t & 1)} : QueryRow{c / padded_group * 4 + t, c % padded_group};
}

// Log-sum-exps in shared memory: what a thread of visit 2 needs is in one piece, the four pieces on banks of their own.
constexpr int kOffFloats = 4 * (64 / 4 + 4);   // per slab
__host__ __device__ constexpr int off_stride(int ncols) { return ncols / 4 + 4; }
__device__ __forceinline__ void store_off(float* off, int ncols, int j, float v) { off[(j & 3) * off_stride(ncols) + (j >> 2)] = v; }

struct FusedPrompt {
  const CUtensorMap* k_maps;   // [n_layers] (element of a sub-row, key, sub-tile, kv-head[, pool block])
  const unsigned char* q_tiles;   // [slab] query operands as the tensor cores read them (swizzled, padding rows zero)
  float4* row_sums;            // [slab][per_part][NCOLS / 4] each CTA's sums of exp2(c*q.k - ref) for four rows; 0: not there yet
  unsigned long long* lse;     // [slab][NCOLS] {log-sum-exp in base-2 units, 1} once known
  const float* refs;           // [slab] reference of visit 1
  const float* slab_c;         // [slab] 8-bit keys: accumulated dot product -> base-2 logit; null: FusedArgs::c for all
  unsigned* amax;              // [m][n_tiles * 128] order-preserving bits of the running maxima (parts > 1)
  unsigned* finished;          // [n_tiles][4] arrivals at `amax` (parts > 1)
  float* importance;           // [N]
  float* lse_out;              // optional [L][Hq][m], natural log
  const float* extra_lse;      // optional [L][Hq][m], natural log: what each row's denominator holds besides the prompt keys
  const float* lse_in;         // visit 2 alone: row log-sum-exps supplied by the caller, natural log, [L][Hq][m]
  const int32_t* block_table;  // paged key cache (block_tokens > 0): pool block of each logical block
  int64_t n_tokens;
  int block_tokens, n_tiles;
  int cta0, parts, per_part;   // CTAs cta0 .. cta0 + parts * per_part - 1
  int lead;                    // tiles that visit 1 may be ahead of visit 2
};

struct FusedArgs {
  FusedPrompt prompt[kFusedMaxBatch];
  int n_prompts, n_layers, n_kv_heads, group, n_lookahead;
  int table_tiles;             // tiles per CTA for which there is a table (paged key cache), else 0
  int mode;                    // 0: the whole computation; 1: visit 1 alone (row log-sum-exps of these keys); 2: visit 2 alone
  int k_stages[2], t_stages[2];   // per visit: key tiles in shared memory, tiles' logits in tensor memory (resident: [0] alone)
  int max_in_regs;             // resident: no CTA has more than kRegTiles tiles
  float c;                     // softmax scale * log2(e)
  int32_t* dev_status;         // optional
};

// Barrier addresses (8 bytes each): two visits' rings, the log-sum-exp slots, the row-sum slots.
struct FusedBars {
  uint32_t base;
  static constexpr int kVisit = 2 * (kMaxKeyStages + kMaxQStages), kTmem = 2 * kVisit, kShared = kTmem + 2 * kMaxResident;
  static constexpr int kOffReady = kShared, kOffFree = kOffReady + kOffSlots, kSumsReady = kOffFree + kOffSlots;
  static constexpr int kSumsFree = kSumsReady + kSumSlots, kMmaDone = kSumsFree + kSumSlots, kCount = kMmaDone + 2;
  __device__ uint32_t k_full(int v, int s) const { return base + 8u * (v * kVisit + s); }
  __device__ uint32_t k_empty(int v, int s) const { return base + 8u * (v * kVisit + kMaxKeyStages + s); }
  __device__ uint32_t q_full(int v, int s) const { return base + 8u * (v * kVisit + 2 * kMaxKeyStages + s); }
  __device__ uint32_t q_empty(int v, int s) const { return base + 8u * (v * kVisit + 2 * kMaxKeyStages + kMaxQStages + s); }
  __device__ uint32_t t_full(int v, int s) const { return base + 8u * (kTmem + v * kMaxTmemStages + s); }   // resident: v = 0 alone
  __device__ uint32_t t_empty(int v, int s) const { return t_full(v, s) + 8u * kMaxResident; }
  __device__ uint32_t off_ready(int x) const { return base + 8u * (kOffReady + x); }
  __device__ uint32_t off_free(int x) const { return base + 8u * (kOffFree + x); }
  __device__ uint32_t sums_ready(int x) const { return base + 8u * (kSumsReady + x); }
  __device__ uint32_t sums_free(int x) const { return base + 8u * (kSumsFree + x); }
  __device__ uint32_t mma_done(int v) const { return base + 8u * (kMmaDone + v); }
};
static_assert(2 * kMaxTmemStages <= kMaxResident, "the two-pass stages use the same barriers");

struct FusedSmem {
  uint32_t k_off[2], q_off[2], sums_off, off_off, offc_off, bar_off, misc_off, tile_off, total;
};

__host__ __device__ inline FusedSmem fused_smem(int d, bool fp8, int ncols, bool once, int tiles, const int k_stages[2]) {
  FusedSmem s;
  uint32_t o = 0;
  const uint32_t rowb = (uint32_t)row_bytes(d, fp8), q_rows = (uint32_t)image_rows(ncols);
  for (int v = 0; v < 2; ++v) { s.k_off[v] = o; o += (uint32_t)k_stages[v] * kTileKeys * rowb; }
  for (int v = 0; v < 2; ++v) { s.q_off[v] = o; o += (uint32_t)(once ? (v == 0 ? kMaxQStages : 0) : 2) * (fp8 ? 2 : 1) * q_rows * rowb; }
  s.sums_off = o;  o += kSumSlots * 256 * 4;            // [slot][set][quadrant][lane]
  s.off_off = o;   o += kOffSlots * kOffFloats * 4;
  s.offc_off = o;  o += kOffSlots * 4;
  s.bar_off = o;   o += FusedBars::kCount * 8;
  s.misc_off = o;  o += 64;
  s.tile_off = o;  o += tiles * 8;                      // paged key cache: row in the block and pool block of each tile
  s.total = o;
  return s;
}

struct Ring {
  int stage = 0;
  uint32_t phase = 0;
  int n;
  __device__ explicit Ring(int n_) : n(n_) {}
  __device__ void advance() {
    if (++stage == n) {
      stage = 0;
      phase ^= 1u;
    }
  }
  __device__ void advance(int by) {
    for (stage += by; stage >= n; stage -= n) phase ^= 1u;
  }
};

// Reads what the preparing kernel writes.  This kernel may be started while that one still runs (it asks for that; a cooperative
// launch was not seen to overlap, but nothing here relies on it), so these are not read-only for its lifetime: __ldg may be moved
// ahead of the wait for the other kernel, a volatile load stays behind it.  (Through L1, which has nothing of them before: the loads
// of neighbouring slabs share a line.)
__device__ __forceinline__ float produced(const float* at) {
  float x;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(at));
  return x;
}

// fp32 <-> unsigned bits whose integer order is the float order (0 is below every float).
__device__ __forceinline__ unsigned order_bits(float x) {
  const unsigned b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_order_bits(unsigned u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

template <int D, int NCOLS, int G, bool FP8, bool ONCE>
struct FusedTraits {
  static constexpr int QS = ONCE ? kMaxQStages : 2;                // query tiles in flight per visit
  static constexpr int CW = NCOLS < 32 ? NCOLS : 32;               // visit 2: accumulators per tensor-memory load
  static constexpr int NCH = NCOLS / CW;                           // loads per tile: 1 or 2
  static constexpr int NI = NCOLS / G;                             // lookahead slots per key in the running-max columns
  static constexpr int NIW = CW / G;                               // of which one load's accumulators hold
  static constexpr int CT = CW / 4;                                // a thread's columns of a load, each for four keys
  static constexpr bool PAIRS = G > CT;                            // 8 heads in 16 columns: two lanes share a lookahead's heads
  static constexpr int ROWB = row_bytes(D, FP8);                   // bytes per key row: 64, 128 or 256
  static constexpr int SUBROW = sub_row_bytes(ROWB);               // the swizzle span: 128 bytes, or the whole 64-byte row
  static constexpr int KSUB = ROWB / SUBROW;                       // sub-tiles per key tile
  static constexpr int KSTEPS = SUBROW / 32;                       // tensor-core instructions per sub-tile (32 bytes of the row each)
  static constexpr int XSUB = SUBROW / (FP8 ? 1 : 2);              // elements per sub-tile row
  static constexpr int kSubTileBytes = kTileKeys * SUBROW;
  static constexpr int kTileBytes = KSUB * kSubTileBytes;
  static constexpr int QPARTS = FP8 ? 2 : 1;                       // 8-bit keys: the queries come as two E4M3 terms
  static constexpr int kQSub = image_rows(NCOLS) * SUBROW;
  static constexpr int kQBytes = QPARTS * KSUB * kQSub;
};

// What every warp of a CTA knows about its share of the work.
struct FusedShare {
  const FusedPrompt* p;
  int part, parts, first, step;   // this CTA's slabs are part, part + parts, ...; its tiles first, first + step, ...
  int n_slabs, n_tiles;           // how many of each
  __device__ int slab(int n) const { return part + n * parts; }
  __device__ int tile(int lt) const { return first + lt * step; }
};

// ---------------------------------------------------------------------------------------------- TMA producer of one visit
template <class T, bool ONCE>
__device__ __forceinline__ void fused_produce(const FusedArgs& a, const FusedShare& sh, int v, unsigned char* k_tiles, unsigned char* q_tiles,
                                              const int2* tile_at, const FusedBars& bars, volatile int* visit2_issued, const Abort& ab) {
  const FusedPrompt& p = *sh.p;
  Ring kr(a.k_stages[v]), qr(T::QS);
  const uint64_t policy = !ONCE && v == 0 ? l2_policy_keep() : l2_policy_drop();
  const uint32_t k_smem = smem_u32(k_tiles), q_smem = smem_u32(q_tiles);
  const CUtensorMap* const maps = p.k_maps;
  const unsigned char* const q_src = p.q_tiles;
  const bool paged = p.block_tokens > 0;
  const int n_kv_heads = a.n_kv_heads;
  const int lead = !ONCE && a.mode == 0 ? p.lead : 0x7fffffff;
  // slab n is (layer, hk); from one slab of the CTA to the next both advance by a fixed step
  int layer = sh.part / n_kv_heads, hk = sh.part - layer * n_kv_heads, issued = 0;
  const int layer_step = sh.parts / n_kv_heads, hk_step = sh.parts - layer_step * n_kv_heads;
  map_acquire(maps + layer);
#pragma unroll 1
  for (int n = 0; n < sh.n_slabs; ++n) {
    const CUtensorMap* map = maps + layer;
    if (!mbar_wait(bars.q_empty(v, qr.stage), qr.phase ^ 1u, ab)) return;
    mbar_expect_tx(bars.q_full(v, qr.stage), (uint32_t)T::kQBytes);
    bulk_load(q_smem + (uint32_t)(qr.stage * T::kQBytes), q_src + (int64_t)sh.slab(n) * T::kQBytes, (uint32_t)T::kQBytes,
              bars.q_full(v, qr.stage));
    qr.advance();
#pragma unroll 1
    for (int lt = 0; lt < sh.n_tiles; ++lt, ++issued) {
      if (!ONCE && v == 0) {
        // never more than `lead` tiles ahead of visit 2
        unsigned long long t0 = 0;
        for (uint32_t it = 1; issued - *visit2_issued >= lead; ++it) {
          if (give_up(it, t0, ab)) return;
          __nanosleep(40);
        }
      }
      if (!mbar_wait(bars.k_empty(v, kr.stage), kr.phase ^ 1u, ab)) return;
      const uint32_t dst = k_smem + (uint32_t)(kr.stage * T::kTileBytes), bar = bars.k_full(v, kr.stage);
      mbar_expect_tx(bar, (uint32_t)T::kTileBytes);
      if (paged) {
        const int2 at = tile_at[lt];
        tma_load_5d(dst, map, 0, at.x, 0, hk, at.y, bar, policy);
      } else {
        tma_load_4d(dst, map, 0, sh.tile(lt) * kTileKeys, 0, hk, bar, policy);
      }
      kr.advance();
      if (v == 1) *visit2_issued = issued + 1;
    }
    const int before = layer;
    hk += hk_step;
    layer += layer_step;
    if (hk >= n_kv_heads) {
      hk -= n_kv_heads;
      ++layer;
    }
    if (layer != before && n + 1 < sh.n_slabs) map_acquire(maps + layer);
  }
}

// ---------------------------------------------------------------------------------------------- MMA issuer of one visit
// Tile k of the CTA (k counts over slabs and tiles) has its logits in stage k mod stages.  One thread walks the
// loop.  (The whole warp in step, with votes on the barriers and an elected lane at each tile, took 460 cycles to issue a tile's
// four instructions and 120 for its barriers, 0.34 us a tile in all: more than the sums of 32 rows take.  One thread's loop takes 150,
// traced at 32768 tokens with 32 rows of 64 dimensions.)
// It commits tile after tile, so whoever has seen a tile's barrier complete knows those of the tiles before it to be, too.  The
// warps of visit 1 rely on that: a set asks for every other tile, the ring of stages is common to both sets, and with three stages
// the barrier's phase before was another set's tile (a parity tells one round from the next only).  It takes at least two stages.
// ROWS: query rows are the accumulator's lanes (weight-stationary instructions), else the keys.  SETS: a ring of stages for
// each of the two sets of epilogue warps, the odd tiles' behind the even tiles': a tile's maxima belong to one set, so with an
// odd number of tiles a set skips two, and in a common ring of two stages it could take the tile before the one that it
// skipped for its own (a barrier's parity tells one round from the next only).
template <class T, int NCOLS, bool FP8, bool ROWS, bool SETS>
__device__ __forceinline__ void fused_multiply(const FusedArgs& a, const FusedShare& sh, int v, const unsigned char* k_tiles,
                                               const unsigned char* q_tiles, uint32_t tmem, const FusedBars& bars, const Abort& ab) {
  if (!elect_one()) return;
  constexpr uint32_t idesc = ROWS ? instr_desc(NCOLS, kTileKeys, FP8) : instr_desc(kTileKeys, NCOLS, FP8);
  const uint64_t k_desc0 = smem_desc<T::SUBROW>(smem_u32(k_tiles));
  const uint64_t q_desc0 = smem_desc<T::SUBROW>(smem_u32(q_tiles));
  Ring kr(a.k_stages[v]), qr(T::QS), even(SETS ? (a.t_stages[v] + 1) / 2 : a.t_stages[v]), odd(a.t_stages[v] / 2);
  const int n_slabs = sh.n_slabs, n_tiles = sh.n_tiles;
#pragma unroll 1
  for (int n = 0; n < n_slabs; ++n) {
    if (!mbar_wait(bars.q_full(v, qr.stage), qr.phase, ab)) return;
    const uint64_t qd0 = q_desc0 + (uint64_t)((qr.stage * T::kQBytes) >> 4);
    auto tile = [&](Ring& tr, int stage0) -> bool {
      const int stage = stage0 + tr.stage;
      if (!mbar_wait2(bars.k_full(v, kr.stage), kr.phase, bars.t_empty(v, stage), tr.phase ^ 1u, ab)) return false;
      tc_fence_after();
      const uint32_t d_tmem = tmem + (uint32_t)(stage * NCOLS);
      const uint64_t kd0 = k_desc0 + (uint64_t)((kr.stage * T::kTileBytes) >> 4);
#pragma unroll
      for (int part = 0; part < T::QPARTS; ++part)                 // 8-bit keys: the two query terms accumulate into the same columns
#pragma unroll
        for (int h = 0; h < T::KSUB; ++h)
#pragma unroll
          for (int ks = 0; ks < T::KSTEPS; ++ks) {
            const uint64_t kd = kd0 + (uint64_t)((h * T::kSubTileBytes) >> 4) + 2u * ks;
            const uint64_t qd = qd0 + (uint64_t)(((part * T::KSUB + h) * T::kQSub) >> 4) + 2u * ks;
            tc_mma<FP8, ROWS>(d_tmem, ROWS ? qd : kd, ROWS ? kd : qd, idesc, (uint32_t)((part | h | ks) != 0));
          }
      tc_commit(bars.k_empty(v, kr.stage));
      tc_commit(bars.t_full(v, stage));
      kr.advance();
      tr.advance();
      return true;
    };
#pragma unroll 1
    for (int lt = 0; lt < n_tiles; ++lt)
      if (!(SETS && (lt & 1) ? tile(odd, even.n) : tile(even, 0))) return;
    tc_commit(bars.q_empty(v, qr.stage));
    qr.advance();
  }
  // leave only after everything issued has completed and signalled its barriers
  tc_commit(bars.mma_done(v));
  mbar_wait(bars.mma_done(v), 0u, ab);
}

// ---------------------------------------------------------------------------------------------- visit 1: sums
// A thread has one query row and, per tile, 32 or 64 of its keys (64 rows: lanes 64.. repeat the rows for the tile's second
// half; 32 rows: a quarter of the keys per quadrant).  Bound by the exp2 unit (16 results a cycle and SM: 512 cycles per
// tile of 64 rows; the loop alone with its MMAs takes 645).  One load of 32 columns at a time, computed before the next is
// asked for: the other set's warps fill the gap, and keeping a load in flight across the arithmetic measured 8 to 15 % slower.
template <class T, int NCOLS, bool FP8>
__device__ __forceinline__ void sum_by_rows(const FusedArgs& a, const FusedShare& sh, int warp, int lane, uint32_t tmem, float* sums,
                                          const FusedBars& bars, const Abort& ab) {
  constexpr int NL = NCOLS / 32;                                   // tensor-memory loads of 32 columns per tile
  const FusedPrompt& p = *sh.p;
  const int quad = warp & 3, set = (warp - kSumWarp0) >> 2;
  const int n_slabs = sh.n_slabs, n_tiles = sh.n_tiles;
  const float* const refs = p.refs;
  const float* const slab_c = p.slab_c;
  const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16) ;
  const int full_tiles = (int)(p.n_tokens / kTileKeys);            // tiles below this index have 128 real keys
  const int tail_keys = (int)(p.n_tokens - (int64_t)full_tiles * kTileKeys) - (NCOLS == 64 ? (quad >> 1) * 64 : quad * 32);
  Ring tr(a.t_stages[0]);
  tr.advance(set);
  int lt = set;                                                    // this set's next tile, counted from the slab's first
  bool ready = false;                                              // that tile's logits are there: asked before this one's arithmetic
  float next_ref = produced(refs + sh.slab(0)), next_c = FP8 ? produced(slab_c + sh.slab(0)) : a.c;
#pragma unroll 1
  for (int n = 0; n < n_slabs; ++n) {
    const uint64_t nref = pack2(-next_ref, -next_ref), cc = pack2(next_c, next_c);
    if (n + 1 < n_slabs) {
      next_ref = produced(refs + sh.slab(n + 1));
      if constexpr (FP8) next_c = produced(slab_c + sh.slab(n + 1));
    }
    uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 1
    for (; lt < n_tiles; lt += 2) {
      if (!__all_sync(0xffffffffu, ready) && !mbar_wait_warp(bars.t_full(0, tr.stage), tr.phase, ab)) return;
      tc_fence_after();
      const uint32_t taddr = lane_addr + (uint32_t)(tr.stage * NCOLS);
      const uint32_t empty = bars.t_empty(0, tr.stage);
      tr.advance(2);
#pragma unroll
      for (int load = 0; load < NL; ++load) {
        uint32_t r[32];
        tmem_issue<32>(taddr + (uint32_t)(32 * load), r);
        tmem_load_wait();
        tmem_ready<32>(r);
        if (load + 1 == NL) {
          // the stage can be overwritten: its last accumulators are in registers
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(empty);
          ready = mbar_test_wait(bars.t_full(0, tr.stage), tr.phase);
        }
        if (sh.tile(lt) < full_tiles) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float x, y;
            unpack2(fma2(pack2(r[2 * j], r[2 * j + 1]), cc, nref), x, y);
            acc[j & 3] = add2(acc[j & 3], pack2(fast_exp2(x), fast_exp2(y)));
          }
        } else {
          // the prompt's last, partial tile: keys beyond the end count nothing
          const int left = tail_keys - load * 32;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float x, y;
            unpack2(fma2(pack2(r[2 * j], r[2 * j + 1]), cc, nref), x, y);
            acc[j & 3] = add2(acc[j & 3], pack2(2 * j < left ? fast_exp2(x) : 0.f, 2 * j + 1 < left ? fast_exp2(y) : 0.f));
          }
        }
      }
    }
    lt -= n_tiles;
    const int slot = n % kSumSlots;
    if (n >= kSumSlots)
      if (!mbar_wait_warp(bars.sums_free(slot), (uint32_t)(n / kSumSlots - 1) & 1u, ab)) return;
    float x, y;
    unpack2(add2(add2(acc[0], acc[1]), add2(acc[2], acc[3])), x, y);
    sums[((slot * 2 + set) * 4 + quad) * 32 + lane] = x + y;
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.sums_ready(slot));
  }
}

// The sums where keys are the lanes.  Tiles k with k mod 2 == set; a thread has four keys of a tile and sums of a quarter of the
// rows, which the warp's eight groups of lanes share out at the end of a slab (7 shuffles for 32 rows; with one key and all rows
// to a thread there were 31, and that step took 0.38 us).  (The two-pass form with 64 or 32 rows has query rows as lanes instead.
// With 16 rows keys are the quicker ones, 960 -> 910 us for 16 layers x 8 heads at 340942 tokens, and its columns are half as many:
// 28 tiles a CTA at 16 slots a key instead of 26, where the general path takes 152 us for two layers at 511438 tokens and this one
// 105.)
template <class T, int NCOLS, bool FP8, bool ONCE>
__device__ __forceinline__ void sum_by_keys(const FusedArgs& a, const FusedShare& sh, int warp, int lane, uint32_t tmem, float* sums,
                                             const FusedBars& bars, const Abort& ab) {
  constexpr int CT = NCOLS / 4;
  const FusedPrompt& p = *sh.p;
  const int quad = warp & 3, set = (warp - kSumWarp0) >> 2;
  const int n_slabs = sh.n_slabs, n_tiles = sh.n_tiles;
  const float* const refs = p.refs;
  const float* const slab_c = p.slab_c;
  const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16);
  const int full_tiles = (int)(p.n_tokens / kTileKeys);            // tiles below this index have 128 real keys
  // of the last, partial tile: real keys from this thread's first on
  const int tail_keys = (int)(p.n_tokens - (int64_t)full_tiles * kTileKeys) - quad * 32 - (lane >> 2);
  const bool frees = !ONCE || a.mode == 1;                // else the max warps do (whose loads come after these: see Stored)
  Ring tr(a.t_stages[0]);
  tr.advance(set);
  int lt = set;                                                    // this set's next tile, counted from the slab's first
  float next_ref = produced(refs + sh.slab(0)), next_c = FP8 ? produced(slab_c + sh.slab(0)) : a.c;
#pragma unroll 1
  for (int n = 0; n < n_slabs; ++n) {
    const uint64_t nref = pack2(-next_ref, -next_ref), cc = pack2(next_c, next_c);
    if (n + 1 < n_slabs) {
      next_ref = produced(refs + sh.slab(n + 1));
      if constexpr (FP8) next_c = produced(slab_c + sh.slab(n + 1));
    }
    uint64_t acc[CT];                                              // two keys each
#pragma unroll
    for (int j = 0; j < CT; ++j) acc[j] = 0ull;
#pragma unroll 1
    for (; lt < n_tiles; lt += 2) {
      if (!mbar_wait_warp(bars.t_full(0, tr.stage), tr.phase, ab)) return;
      tc_fence_after();
      uint32_t r[NCOLS];
      tmem_issue_quarters<NCOLS>(lane_addr + (uint32_t)(tr.stage * NCOLS), r);
      tmem_load_wait();
      tmem_ready<NCOLS>(r);
      if (frees) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.t_empty(0, tr.stage));
      }
      tr.advance(2);
      if (sh.tile(lt) < full_tiles) {
#pragma unroll
        for (int j = 0; j < NCOLS / 2; ++j) {
          float x, y;
          unpack2(fma2(pack2(r[2 * j], r[2 * j + 1]), cc, nref), x, y);
          acc[j % CT] = add2(acc[j % CT], pack2(fast_exp2(x), fast_exp2(y)));
        }
      } else {
        // keys beyond the prompt's end count nothing
#pragma unroll
        for (int j = 0; j < NCOLS / 2; ++j) {
          const int key = j / CT * 16;
          float x, y;
          unpack2(fma2(pack2(r[2 * j], r[2 * j + 1]), cc, nref), x, y);
          acc[j % CT] = add2(acc[j % CT], pack2(key < tail_keys ? fast_exp2(x) : 0.f, key + 8 < tail_keys ? fast_exp2(y) : 0.f));
        }
      }
    }
    lt -= n_tiles;
    // Transposing butterfly steps over the eight groups of lanes, each of which halves the columns a lane holds, then (16 columns)
    // one plain step.  The publishers add up quadrants and sets.
    float s[CT];
#pragma unroll
    for (int j = 0; j < CT; ++j) {
      float x, y;
      unpack2(acc[j], x, y);
      s[j] = x + y;
    }
    int width = CT;
#pragma unroll
    for (int off = 16; off >= 4; off >>= 1) {
      if (width > 1) {
        width >>= 1;
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int j = 0; j < CT / 2; ++j) {
          if (j < width) {
            const float send = upper ? s[j] : s[j + width];
            const float keep = upper ? s[j + width] : s[j];
            s[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
          }
        }
      } else {
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], off);
      }
    }
    const int slot = n % kSumSlots;
    if (n >= kSumSlots)
      if (!mbar_wait_warp(bars.sums_free(slot), (uint32_t)(n / kSumSlots - 1) & 1u, ab)) return;
    float* out = sums + ((slot * 2 + set) * 4 + quad) * 32;
    if constexpr (NCOLS == 32) {
      out[lane] = s[0];
    } else {
      if ((lane & 4) == 0) out[(lane >> 3) * 4 + (lane & 3)] = s[0];
    }
    tc_fence_before();                                             // the slab's loads from tensor memory are done (see Stored)
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.sums_ready(slot));
  }
}

// ---------------------------------------------------------------------------------------------- publishers
// Everybody's row sums of a slab, as they come in: LANES quads (float4 of rows) q0 .. q0 + LANES - 1, lane mod LANES being the
// quad, lane / LANES the first CTA.  Whatever is not there yet is asked for again.  A quad is stored and loaded as one 128-bit word.
template <int NCOLS, int LANES, int MAXW>
struct RowSums {
  static constexpr int Q = NCOLS / 4, STEP = 32 / LANES;           // CTAs per load of the warp
  uint64_t lo[MAXW], hi[MAXW];                                     // rows 0 and 1, 2 and 3 of the quad
  const float4* in;
  int left;                                                        // CTAs from this lane's first on
  __device__ __forceinline__ void begin(const FusedPrompt& p, int slab, int q0, int n_ctas, int lane) {
    in = p.row_sums + ((int64_t)slab * p.per_part + lane / LANES) * Q + q0 + lane % LANES;
    left = n_ctas - lane / LANES;
#pragma unroll
    for (int i = 0; i < MAXW; ++i) lo[i] = hi[i] = 0ull;
  }
  __device__ __forceinline__ bool missing(int i) const { return STEP * i < left && (uint32_t)lo[i] == 0u; }
  __device__ __forceinline__ void ask() {
#pragma unroll
    for (int i = 0; i < MAXW; ++i)
      if (missing(i))
        asm volatile("{\n.reg .b128 w;\nld.relaxed.gpu.global.b128 w, [%2];\nmov.b128 {%0, %1}, w;\n}"
                     : "=l"(lo[i]), "=l"(hi[i])
                     : "l"(in + (int64_t)STEP * i * Q)
                     : "memory");
  }
  __device__ __forceinline__ bool there() const {
    bool all = true;
#pragma unroll
    for (int i = 0; i < MAXW; ++i) all = all && !missing(i);
    return __all_sync(0xffffffffu, all);
  }
};

// The log-sum-exp, in base-2 units, of one row from its total: reported where it is to be.
static __device__ __noinline__ float lse_of(double total, float ref, const float* extra, float* out, int32_t* status) {
  // log2 of the total: its binary exponent plus the log2 of its mantissa in single precision; an empty (below every
  // normal number) or overflowed row sum has none
  const long long tb = __double_as_longlong(total);
  const float mant = (float)__longlong_as_double((tb & 0x000fffffffffffffll) | 0x3ff0000000000000ll);
  float lse2 = ref + ((float)((int)((tb >> 52) & 0x7ff) - 1023) + log2f(mant));
  if (!(total > 1.2e-38 && total < (double)INFINITY)) lse2 = INFINITY;
  if (extra != nullptr) {
    // the denominator also holds exp(extra): log2-add, in the order that cannot overflow
    const float e = __ldg(extra) * kLog2e;
    const float hi = fmaxf(lse2, e), lo = fminf(lse2, e);
    lse2 = hi + log2f(1.f + exp2f(lo - hi));
  }
  if (status != nullptr && !(lse2 > -INFINITY && lse2 < INFINITY)) atomicCAS(status, 0, (int32_t)SPF_ERR_RANGE);
  if (out != nullptr) *out = lse2 * kLn2;
  return lse2;
}

// The log-sum-exps, in base-2 units, from a complete set of sums: lane (with lane mod 8 < LANES) gets that of row
// 4 * (q0 + lane mod LANES) + lane / 8.
template <int NCOLS, int G, int LANES, int MAXW>
__device__ __forceinline__ float row_lse(const FusedArgs& a, const FusedPrompt& p, const RowSums<NCOLS, LANES, MAXW>& w, int n_ctas, int slab,
                                         float ref, int q0, int lane, bool report) {
  double t[4] = {0.0, 0.0, 0.0, 0.0};                              // the CTAs' shares are fp32: exact to 2^-53
#pragma unroll
  for (int i = 0; i < MAXW; ++i) {
    if (i > 0 && RowSums<NCOLS, LANES, MAXW>::STEP * i >= n_ctas) break;
    float x[4];
    unpack2(w.lo[i], x[0], x[1]);
    unpack2(w.hi[i], x[2], x[3]);
#pragma unroll
    for (int e = 0; e < 4; ++e) t[e] += (double)x[e];
  }
  // two transposing steps leave one row per lane: lanes 8.. have t[1], 16.. t[2], 24.. t[3]
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const double send = (lane & 16) ? t[e] : t[e + 2], keep = (lane & 16) ? t[e + 2] : t[e];
    t[e] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
  {
    const double send = (lane & 8) ? t[0] : t[1], keep = (lane & 8) ? t[1] : t[0];
    t[0] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int off = 4; off >= LANES; off >>= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], off);
  const QueryRow r = query_row(4 * (q0 + lane % LANES) + (lane >> 3), NCOLS, G);
  if (!((lane & 7) < LANES && r.g < a.group && r.i < a.n_lookahead)) return INFINITY;   // rows that do not exist: exp2(x - lse2) = 0
  const int64_t at = ((int64_t)slab * a.group + r.g) * a.n_lookahead + r.i;
  return lse_of(t[0], ref, p.extra_lse != nullptr ? p.extra_lse + at : nullptr, report && p.lse_out != nullptr ? p.lse_out + at : nullptr,
                report ? a.dev_status : nullptr);
}

// How many slabs' row sums a warp has stored: what the gathering and the fetching warps wait for before they ask for anybody's.
// Released and acquired, it carries an order that the words in global memory do not: the sum warps' loads of a slab's logits come
// before the max warps' work on that slab, hence before the products (or the maxima at the end) that overwrite them.  (An arrival of
// the sum warps at every tile's barrier instead costs up to 2 %: 16 rows of 64 dimensions, 8-bit keys, 12 layers x 4 heads at 89720
// tokens 91.1 -> 92.8 us, this way 91.4.)
struct Stored {
  uint32_t at;                                                     // one word for each warp that stores
  __device__ __forceinline__ void release(int which, int n) const {
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(at + 4u * which), "r"(n) : "memory");
  }
  __device__ __forceinline__ int acquire(int which) const {
    int n;
    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(n) : "r"(at + 4u * which) : "memory");
    return n;
  }
  // Until more than n are stored; all lanes of the warp agree.
  __device__ __forceinline__ bool wait(int which, int n, const Abort& ab) const {
    unsigned long long t0 = 0;
#pragma unroll 1
    for (uint32_t it = 1; __any_sync(0xffffffffu, acquire(which) <= n); ++it) {
      if (__any_sync(0xffffffffu, give_up(it, t0, ab))) return false;
      __nanosleep(20);
    }
    return true;
  }
};

// Stores this CTA's sums of quads q0 .. q0 + LANES - 1 of its n-th slab for all to read (a row that does not exist gets its
// meaningless sum stored too: everybody waits for every word).
template <int NCOLS, int LANES>
__device__ __forceinline__ void store_sums(const FusedPrompt& p, const FusedShare& sh, int n, int q0, int lane, const float* sums,
                                           const FusedBars& bars) {
  constexpr int Q = NCOLS / 4;
  const int slot = n % kSumSlots, q = q0 + lane;
  float t[4] = {0.f, 0.f, 0.f, 0.f};
  if (lane < LANES) {
    // [set][quadrant][lane]: 64 rows: quadrants 0 and 2 have rows 0..31, 1 and 3 rows 32..63; else every quadrant all rows
    const float* in = sums + slot * 256 + (NCOLS == 64 ? (q >> 3) * 32 + (q & 7) * 4 : q * 4);
#pragma unroll
    for (int set = 0; set < 2; ++set)
#pragma unroll
      for (int quad = 0; quad < (NCOLS == 64 ? 2 : 4); ++quad) {
        const float4 v = *reinterpret_cast<const float4*>(in + set * 128 + quad * (NCOLS == 64 ? 64 : 32));
        t[0] += v.x;
        t[1] += v.y;
        t[2] += v.z;
        t[3] += v.w;
      }
    unsigned w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) w[e] = max(__float_as_uint(t[e]), 1u);   // never "not there yet"; 2^-149 is nothing to a row's sum
    asm volatile("{\n.reg .b128 w;\n.reg .b64 lo, hi;\nmov.b64 lo, {%1, %2};\nmov.b64 hi, {%3, %4};\nmov.b128 w, {lo, hi};\n"
                 "st.relaxed.gpu.global.b128 [%0], w;\n}"
                 ::"l"(p.row_sums + ((int64_t)sh.slab(n) * p.per_part + sh.first) * Q + q), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                 : "memory");
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(bars.sums_free(slot));
}

// Few CTAs to a group: every CTA adds up everybody's sums.  One warp stores the CTA's own, slab after slab; two warps (resident:
// two teams of two that take the slabs in turn) wait for everybody's, half the rows each.  (With the same warps storing and
// waiting, sums went out up to 2.3 us late: 32 rows at 4001 tokens.)
template <int NCOLS>
__device__ __forceinline__ void fused_store(const FusedShare& sh, int lane, const float* sums, const Stored& stored, const FusedBars& bars,
                                            const Abort& ab) {
#pragma unroll 1
  for (int n = 0; n < sh.n_slabs; ++n) {
    if (!mbar_wait_warp(bars.sums_ready(n % kSumSlots), (uint32_t)(n / kSumSlots) & 1u, ab)) return;
    store_sums<NCOLS, NCOLS / 4>(*sh.p, sh, n, 0, lane, sums, bars);
    if (lane == 0) stored.release(0, n + 1);
  }
}

template <class T, int NCOLS, int G, bool FP8, int TEAMS>
__device__ __forceinline__ void fused_gather(const FusedArgs& a, const FusedShare& sh, int which, int lane, const Stored& stored, float* off,
                                             float* off_c, const FusedBars& bars, const Abort& ab) {
  constexpr int LANES = NCOLS / 4 / kTeamWarps;                    // quads of this warp
  constexpr int MAXW = (gather_ctas(NCOLS) * LANES + 31) / 32;
  const FusedPrompt& p = *sh.p;
  const int n_ctas = min(p.per_part, p.n_tiles), q0 = which % kTeamWarps * LANES;
  if (a.mode == 1 && sh.first != 0) return;                        // visit 1 alone: nobody but the one that reports needs the sums
  RowSums<NCOLS, LANES, MAXW> w;
#pragma unroll 1
  for (int n = which / kTeamWarps; n < sh.n_slabs; n += TEAMS) {
    const int slab = sh.slab(n);
    w.begin(p, slab, q0, n_ctas, lane);
    const float ref = produced(p.refs + slab);                     // its way to L2 and back passes during the waits below
    const float c = FP8 ? produced(p.slab_c + slab) : 0.f;
    // not before the own sums are out: polling for words that cannot be there yet slows the key copies down
    if (!stored.wait(0, n, ab)) return;
    unsigned long long t0 = 0;
#pragma unroll 1
    for (uint32_t it = 1;; ++it) {
      w.ask();
      if (w.there()) break;
      if (__any_sync(0xffffffffu, give_up(it, t0, ab))) return;
      if (it > 4) __nanosleep(100);                                // CTAs far apart: then there is also time
    }
    const float lse2 = row_lse<NCOLS, G, LANES, MAXW>(a, p, w, n_ctas, slab, ref, q0, lane, sh.first == 0);
    if (a.mode == 1) continue;
    const int x = n % kOffSlots;
    if (n >= kOffSlots)
      if (!mbar_wait_warp(bars.off_free(x), (uint32_t)(n / kOffSlots - 1) & 1u, ab)) return;
    if ((lane & 7) < LANES) store_off(off + x * kOffFloats, NCOLS, 4 * (q0 + lane % LANES) + (lane >> 3), -lse2);
    if constexpr (FP8) {
      if (q0 == 0 && lane == 0) off_c[x] = c;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.off_ready(x));
  }
}

// Many: publisher w takes slabs w, w + 3, ...: stores this CTA's row sums, then adds up those of the rows that it owns -- item
// n * Q + q, rows 4q .. 4q + 3 of the group's n-th slab, belongs to CTA (item mod CTAs) -- and stores their log-sum-exps for all.
// Not before its own sums are out: polling for words that cannot be there yet slowed the key copies down.
template <class T, int NCOLS, int G>
__device__ __forceinline__ void fused_publish(const FusedArgs& a, const FusedShare& sh, int which, int lane, const float* sums, const Stored& stored,
                                              const FusedBars& bars, const Abort& ab) {
  constexpr int Q = NCOLS / 4, MAXW = (kFusedMaxCtas + 31) / 32;   // lane q has rows 4q .. 4q + 3
  const FusedPrompt& p = *sh.p;
  const int n_ctas = min(p.per_part, p.n_tiles);
#pragma unroll 1
  for (int n = which; n < sh.n_slabs; n += kPublisherWarps) {
    const int slab = sh.slab(n);
    if (!mbar_wait_warp(bars.sums_ready(n % kSumSlots), (uint32_t)(n / kSumSlots) & 1u, ab)) return;
    store_sums<NCOLS, Q>(p, sh, n, 0, lane, sums, bars);
    if (lane == 0) stored.release(which, n + 1);
#pragma unroll 1
    for (int q = (int)(((unsigned)(n + 1) * (unsigned)n_ctas * Q + sh.first - n * Q) % (unsigned)n_ctas); q < Q; q += n_ctas) {
      RowSums<NCOLS, 1, MAXW> w;
      w.begin(p, slab, q, n_ctas, lane);
      const float ref = produced(p.refs + slab);
      unsigned long long t0 = 0;
#pragma unroll 1
      for (uint32_t it = 1;; ++it) {
        w.ask();
        if (w.there()) break;
        if (__any_sync(0xffffffffu, give_up(it, t0, ab))) return;
        __nanosleep(100);
      }
      const float lse2 = row_lse<NCOLS, G, 1, MAXW>(a, p, w, n_ctas, slab, ref, q, lane, true);
      if ((lane & 7) == 0) {
        const unsigned long long word = (1ull << 32) | __float_as_uint(lse2);
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p.lse + (int64_t)slab * NCOLS + 4 * q + (lane >> 3)), "l"(word) : "memory");
      }
      __syncwarp();
    }
  }
}

// ---------------------------------------------------------------------------------------------- log-sum-exps for visit 2
// Fetches each slab's log-sum-exps in turn and hands them to the max warps through shared memory (negated: what visit 2 adds).
template <class T, int NCOLS, int G, bool FP8>
__device__ __forceinline__ void fused_fetch_lse(const FusedArgs& a, const FusedShare& sh, int lane, const Stored& stored, float* off, float* off_c,
                                                const FusedBars& bars, const Abort& ab) {
  const FusedPrompt& p = *sh.p;
  constexpr int RPL = NCOLS == 64 ? 2 : 1;
  const bool there_already = a.mode == 2;                          // supplied by the caller
#pragma unroll 1
  for (int n = 0; n < sh.n_slabs; ++n) {
    const int slab = sh.slab(n);
    const float c = FP8 ? produced(p.slab_c + slab) : 0.f;
    float v[RPL];
    if (there_already) {
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        const QueryRow q = query_row(min(lane + 32 * r, NCOLS - 1), NCOLS, G);
        v[r] = q.g < a.group && q.i < a.n_lookahead ? -__ldg(p.lse_in + ((int64_t)slab * a.group + q.g) * a.n_lookahead + q.i) * kLog2e : -INFINITY;
      }
    } else {
      if (!stored.wait(n % kPublisherWarps, n, ab)) return;
      unsigned long long w[RPL], t0 = 0;
#pragma unroll 1
      for (uint32_t it = 1;; ++it) {
        bool there = true;
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
          asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w[r]) : "l"(p.lse + (int64_t)slab * NCOLS + min(lane + 32 * r, NCOLS - 1)) : "memory");
          there = there && (w[r] >> 32) != 0ull;
        }
        if (__all_sync(0xffffffffu, there)) break;
        if (__any_sync(0xffffffffu, give_up(it, t0, ab))) return;
      }
#pragma unroll
      for (int r = 0; r < RPL; ++r) v[r] = -__uint_as_float((unsigned)w[r]);
    }
    const int slot = n % kOffSlots;
    if (n >= kOffSlots)
      if (!mbar_wait_warp(bars.off_free(slot), (uint32_t)(n / kOffSlots - 1) & 1u, ab)) return;
#pragma unroll
    for (int r = 0; r < RPL; ++r)
      if (lane + 32 * r < NCOLS) store_off(off + slot * kOffFloats, NCOLS, lane + 32 * r, v[r]);
    if constexpr (FP8) {
      if (lane == 0) off_c[slot] = c;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.off_ready(slot));
  }
}

// ---------------------------------------------------------------------------------------------- importance
// Mean over the lookahead of exp2(running max) for a tile's keys.  One group of CTAs (parts = 1): straight from the maxima.
// Several: the groups' maxima meet in global memory, and whichever warp brings the last contribution for 32 keys reads the
// result.  v[x] belongs to key 8 * key_of(x) + lane / 4 of the quadrant and lookahead i_of(x).
template <int NI, bool PAIRS>
__device__ __forceinline__ void finish_tile(const FusedArgs& a, const FusedPrompt& p, int tile, int quad, int lane, const uint32_t (&v)[NI]) {
  const float inv_m = 1.f / (float)a.n_lookahead;
  const int64_t key0 = (int64_t)tile * kTileKeys + quad * 32;
  const int t = lane & 3;
  auto key_of = [&](int x) { return PAIRS ? 2 * (t & 1) + x : x & 3; };
  auto i_of = [&](int x) { return PAIRS ? t >> 1 : (x >> 2) * 4 + t; };
  int64_t key;
  float sum = 0.f;
  if (p.parts == 1) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};                             // of the thread's keys, over its lookahead slots
#pragma unroll
    for (int x = 0; x < NI; ++x) {
      const float e = i_of(x) < a.n_lookahead ? fast_exp2(__uint_as_float(v[x])) : 0.f;
      if constexpr (PAIRS) {
        s[x] += (t & 1) == 0 ? e : 0.f;
        s[2 + x] += (t & 1) != 0 ? e : 0.f;
      } else {
        s[x & 3] += e;
      }
    }
    // the four lanes of a key's lookahead slots; lane t keeps key 8 * t + lane / 4
#pragma unroll
    for (int u = 0; u < 2; ++u) s[u] = ((t & 2) ? s[u + 2] : s[u]) + __shfl_xor_sync(0xffffffffu, (t & 2) ? s[u] : s[u + 2], 2);
    sum = ((t & 1) ? s[1] : s[0]) + __shfl_xor_sync(0xffffffffu, (t & 1) ? s[0] : s[1], 1);
    key = key0 + 8 * t + (lane >> 2);
  } else {
    const int64_t n_pad = (int64_t)p.n_tiles * kTileKeys;
#pragma unroll
    for (int x = 0; x < NI; ++x)
      if (i_of(x) < a.n_lookahead)
        atomicMax(p.amax + (int64_t)i_of(x) * n_pad + key0 + 8 * key_of(x) + (lane >> 2), order_bits(__uint_as_float(v[x])));
    __threadfence();
    __syncwarp();
    unsigned before = 0;
    if (lane == 0) before = atomicAdd(p.finished + tile * 4 + quad, 1u);
    if (__shfl_sync(0xffffffffu, before, 0) + 1u != (unsigned)p.parts) return;
    __threadfence();
    key = key0 + lane;
#pragma unroll 4
    for (int i = 0; i < a.n_lookahead; ++i) sum += fast_exp2(from_order_bits(__ldcg(p.amax + (int64_t)i * n_pad + key)));
  }
  if (key < p.n_tokens) p.importance[key] = sum * inv_m;
}

// The tiles of a max warp's set, from the maxima in tensor memory: tile lt's in stage (first + lt) mod stages, `cols` columns each.
template <class T>
__device__ __forceinline__ void fused_finish(const FusedArgs& a, const FusedShare& sh, int warp, int lane, uint32_t lane_addr, Ring first, int cols) {
  const int quad = warp & 3, set = (warp - kMaxWarp0) >> 2;
  first.advance(set);
#pragma unroll 1
  for (int lt = set; lt < sh.n_tiles; lt += 2) {
    constexpr int LD = T::NI < 32 ? T::NI : 32;                    // columns per load
    uint32_t v[T::NI];
#pragma unroll
    for (int i = 0; i < T::NI; i += LD)
      tmem_issue<LD>(lane_addr + (uint32_t)(first.stage * cols + i), *reinterpret_cast<uint32_t(*)[LD]>(v + i));
    tmem_load_wait();
    tmem_ready<T::NI>(v);
    finish_tile<T::NI, T::PAIRS>(a, *sh.p, sh.tile(lt), quad, lane, v);
    first.advance(2);
  }
}

// ---------------------------------------------------------------------------------------------- visit 2: maxima
// Folds one load's accumulators into the running maxima over (layer, head) of the base-2 logits less their rows'
// log-sum-exps (slots past n_lookahead hold padding and are never read).  Maximum 4 * ih + k is that of the thread's key k and
// lookahead 4 * ih + lane % 4; PAIRS: the two lanes of a lookahead's heads keep two keys each.
template <class T, int G>
__device__ __forceinline__ void fold_maxima(const uint32_t (&r)[T::CW], uint32_t (&am)[T::NIW], const float* off, float scale, int lane) {
  float z[4][T::CT];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < T::CT; ++c) {
      const int at = h * (T::CW / 2) + 2 * c;
      z[2 * h][c] = fmaf(__uint_as_float(r[at]), scale, off[c]);
      z[2 * h + 1][c] = fmaf(__uint_as_float(r[at + 1]), scale, off[c]);
    }
  if constexpr (T::PAIRS) {
    float top[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) top[k] = fmaxf(max3(z[k][0], z[k][1], z[k][2]), z[k][3]);
    const bool odd = lane & 1;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float other = __shfl_xor_sync(0xffffffffu, odd ? top[u] : top[2 + u], 1);
      am[u] = __float_as_uint(max3(__uint_as_float(am[u]), odd ? top[2 + u] : top[u], other));
    }
  } else {
#pragma unroll
    for (int ih = 0; ih < T::CT / G; ++ih)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float m = __uint_as_float(am[4 * ih + k]);
        if constexpr (G == 1) {
          m = fmaxf(m, z[k][ih]);
        } else {
#pragma unroll
          for (int g = 0; g < G; g += 2) m = max3(m, z[k][ih * G + g], z[k][ih * G + g + 1]);
        }
        am[4 * ih + k] = __float_as_uint(m);
      }
  }
}

// -inf in the running maxima of a set's tiles.
template <class T>
__device__ __forceinline__ void clear_maxima(uint32_t amax_addr, int set, int n_tiles) {
  uint32_t ninf[T::NIW];
#pragma unroll
  for (int j = 0; j < T::NIW; ++j) ninf[j] = 0xff800000u;
#pragma unroll 1
  for (int lt = set; lt < n_tiles; lt += 2)
#pragma unroll
    for (int ch = 0; ch < T::NCH; ++ch) tmem_store<T::NIW>(amax_addr + (uint32_t)(lt * T::NI + ch * T::NIW), ninf);
}

// ---------------------------------------------------------------------------------------------- visit 2: maxima of the tiles
// Begins a slab once its log-sum-exps are there.  A tile's maxima always belong to the same warps (lt mod 2 == set).  REGS: up
// to kRegTiles tiles, whose maxima stay in registers and leave all of tensor memory to the logits.
template <class T, int NCOLS, int G, bool FP8, bool ONCE, bool REGS>
__device__ __forceinline__ void fused_max(const FusedArgs& a, const FusedShare& sh, int warp, int lane, uint32_t tmem, uint32_t amax_tmem,
                                          const float* off, const float* off_c, const FusedBars& bars, const Abort& ab) {
  constexpr int V = ONCE ? 0 : 1;                                  // whose logits: resident: those that were summed
  constexpr int CW = T::CW, NCH = T::NCH, NIW = T::NIW, MINE = REGS ? kRegTiles / 2 : 1;
  static_assert(!REGS || NCH == 1, "one load per tile");
  const int quad = warp & 3, set = (warp - kMaxWarp0) >> 2;
  const int n_tiles = sh.n_tiles;
  const uint32_t lane_bits = (uint32_t)(quad * 32) << 16;
  const uint32_t lane_addr = tmem + lane_bits, amax_addr = amax_tmem + lane_bits;
  uint32_t am[MINE][NIW];
  if constexpr (REGS) {
#pragma unroll
    for (int u = 0; u < MINE; ++u)
#pragma unroll
      for (int j = 0; j < NIW; ++j) am[u][j] = 0xff800000u;        // -inf
  } else {
    clear_maxima<T>(amax_addr, set, n_tiles);
  }
  // resident: the stage of the slab's first tile; two-pass: a ring per set, this one's first stage and the next to be read
  Ring first(ONCE ? a.t_stages[V] : (a.t_stages[V] + 1 - set) / 2);
  Ring last = first, end = first;                                  // resident: that of the slab before, and the slab's last tile's
  bool ready = false;
  const int stage0 = ONCE ? 0 : set * ((a.t_stages[V] + 1) / 2);
#pragma unroll 1
  for (int n = 0; n < sh.n_slabs; ++n) {
    const int slot = n % kOffSlots;
    if (ONCE) {
      // That the log-sum-exps contain these logits orders nothing (they come by way of relaxed words in global memory).  For the
      // products, the barrier of the slab's last tile does, whose commit tracks everything issued before it: asked ahead of the
      // log-sum-exps, whose wait hides it.  For the sum warps' loads: see Stored.
      end = first;
      end.advance(n_tiles - 1);
      if (!mbar_wait_warp(bars.t_full(V, end.stage), end.phase, ab)) return;
    }
    if (!mbar_wait_warp(bars.off_ready(slot), (uint32_t)(n / kOffSlots) & 1u, ab)) return;
    const float4* my_off = reinterpret_cast<const float4*>(off + slot * kOffFloats + (lane & 3) * off_stride(NCOLS));
    float o[T::CT];                                                // one load a tile: the same for all tiles
    auto load_off = [&](int ch) {
#pragma unroll
      for (int j = 0; j < T::CT / 4; ++j) *reinterpret_cast<float4*>(o + 4 * j) = my_off[ch * (T::CT / 4) + j];
    };
    if (NCH == 1) load_off(0);
    const float c = FP8 ? off_c[slot] : a.c;
    Ring tr = first;
    if (ONCE) {
      tr.advance(set);
      tc_fence_after();
    }
    auto fold = [&](int lt, uint32_t (&m)[NIW]) -> bool {
      if constexpr (!ONCE) {
        if (!__all_sync(0xffffffffu, ready) && !mbar_wait_warp(bars.t_full(V, stage0 + tr.stage), tr.phase, ab)) return false;
        tc_fence_after();
      }
      if (!REGS) tmem_store_wait();                                // the maxima read below may be this warp's last stores
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) {
        const uint32_t m_addr = amax_addr + (uint32_t)(lt * T::NI + ch * NIW);
        uint32_t r[CW];
        tmem_issue_quarters<CW>(lane_addr + (uint32_t)((stage0 + tr.stage) * NCOLS + ch * CW), r);
        if (!REGS) tmem_issue<NIW>(m_addr, m);
        tmem_load_wait();
        tmem_ready<CW>(r);
        if (!REGS) tmem_ready<NIW>(m);
        if (ch + 1 == NCH) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bars.t_empty(V, stage0 + tr.stage));
          tr.advance(ONCE ? 2 : 1);
          if (!ONCE) ready = mbar_test_wait(bars.t_full(V, stage0 + tr.stage), tr.phase);   // the next tile's, before this one's arithmetic
        }
        if (NCH > 1) load_off(ch);
        fold_maxima<T, G>(r, m, o, c, lane);
        if (!REGS) tmem_store<NIW>(m_addr, m);
      }
      return true;
    };
    if constexpr (REGS) {
#pragma unroll
      for (int u = 0; u < MINE; ++u)
        if (set + 2 * u < n_tiles)
          if (!fold(set + 2 * u, am[u])) return;
    } else {
#pragma unroll 1
      for (int lt = set; lt < n_tiles; lt += 2)
        if (!fold(lt, am[0])) return;
    }
    if (ONCE) {
      last = first;
      first = end;
      first.advance();
    } else {
      first = tr;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.off_free(slot));
  }
  if constexpr (REGS) {
    // to the columns of the last slab's logits, which only this warp would still read
    Ring to = last;
    to.advance(set);
#pragma unroll
    for (int u = 0; u < MINE; ++u) {
      if (set + 2 * u < n_tiles) tmem_store<NIW>(lane_addr + (uint32_t)(to.stage * NCOLS), am[u]);
      to.advance(2);
    }
    tmem_store_wait();
    fused_finish<T>(a, sh, warp, lane, lane_addr, last, NCOLS);
  } else {
    tmem_store_wait();
    fused_finish<T>(a, sh, warp, lane, amax_addr, Ring(1 << 30), T::NI);
  }
}

// ---------------------------------------------------------------------------------------------- kernel
template <int D, int NCOLS, int G, bool FP8, bool ONCE>
__global__ void __launch_bounds__(kFusedThreads, 1) score_fused_kernel(const __grid_constant__ FusedArgs a) {
  using T = FusedTraits<D, NCOLS, G, FP8, ONCE>;
  static_assert(T::CW % G == 0, "a load's accumulators must hold whole GQA groups");
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment by offsetting the shared array itself, so that the compiler still knows these are shared-memory
  // addresses (a round trip through an integer would turn every access into a generic one)
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const FusedSmem lay = fused_smem(D, FP8, NCOLS, ONCE, a.table_tiles, a.k_stages);
  float* sums = reinterpret_cast<float*>(smem + lay.sums_off);
  float* off = reinterpret_cast<float*>(smem + lay.off_off);
  float* off_c = reinterpret_cast<float*>(smem + lay.offc_off);
  volatile int* misc = reinterpret_cast<volatile int*>(smem + lay.misc_off);  // [0] abort, [1] tensor-memory base, [2] tiles visit 2 has issued, [3..] slabs whose sums are stored
  const FusedBars bars{smem_u32(smem + lay.bar_off)};
  const Abort ab{misc, a.dev_status};
  const Stored stored{smem_u32(smem + lay.misc_off) + 12u};
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // ------------------------------------------------------------------ this CTA's share
  FusedShare sh;
  {
    int pi = 0;
    while (pi + 1 < a.n_prompts && (int)blockIdx.x >= a.prompt[pi + 1].cta0) ++pi;
    const FusedPrompt& p = a.prompt[pi];
    const int local = (int)blockIdx.x - p.cta0;
    sh.p = &p;
    sh.parts = p.parts;
    sh.part = local % p.parts;
    sh.first = local / p.parts;
    sh.step = p.per_part;
    const int slabs = a.n_layers * a.n_kv_heads;
    sh.n_slabs = (slabs - sh.part + p.parts - 1) / p.parts;
    sh.n_tiles = sh.first < min(p.per_part, p.n_tiles) ? (p.n_tiles - sh.first + sh.step - 1) / sh.step : 0;
  }
  if (sh.n_tiles == 0) return;
  const bool visit1 = a.mode != 2, visit2 = a.mode != 1;
  const bool gathers = visit1 && gather_alone(NCOLS, min(sh.p->per_part, sh.p->n_tiles));

  // ------------------------------------------------------------------ set-up
  if (threadIdx.x < 3 + kPublisherWarps) misc[threadIdx.x] = 0;
  for (int x = (int)threadIdx.x - 32; x >= 0 && x < FusedBars::kCount; x += kFusedThreads) {
    uint32_t count = 1;
    if (x >= FusedBars::kTmem + kMaxResident && x < FusedBars::kShared) count = kVisitWarps / 2;   // t_empty
    else if (x >= FusedBars::kOffReady && x < FusedBars::kOffFree) count = gathers ? kTeamWarps : 1;
    else if (x >= FusedBars::kOffFree && x < FusedBars::kSumsFree) count = kVisitWarps;            // off_free, sums_ready
    mbar_init(bars.base + 8u * x, count);
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  int2* const tile_at = reinterpret_cast<int2*>(smem + lay.tile_off);
  if (sh.p->block_tokens > 0) {
    grid_wait();
    for (int lt = threadIdx.x; lt < sh.n_tiles; lt += kFusedThreads) {
      const int key0 = sh.tile(lt) * kTileKeys;
      tile_at[lt] = make_int2(key0 % sh.p->block_tokens, __ldg(sh.p->block_table + key0 / sh.p->block_tokens));
    }
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)&misc[1])),
                 "r"(kTmemColsAll)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = (uint32_t)misc[1];
  // tensor memory: the accumulator stages, then the running maxima, [local tile][NI] columns (a lane has four keys of a quarter of the lookahead slots, as fold_maxima has them)
  const uint32_t tmem_v2 = tmem_base + (uint32_t)(a.t_stages[0] * NCOLS);
  const uint32_t amax_tmem = tmem_v2 + (uint32_t)(ONCE ? 0 : a.t_stages[1] * NCOLS);
  grid_wait();                                                     // what the preparing kernel wrote is visible from here on
  grid_launch_dependents();                                        // the next kernel starts where SMs are free, and waits there

  // ------------------------------------------------------------------ roles
  // resident, 32 rows: 768 threads start with 80 registers each; 256 x 64 + 512 x 88 is the same sum
  constexpr bool kMoveRegs = ONCE && NCOLS == 32;
  if (warp < 4) {
    if constexpr (kMoveRegs) reg_dec<64>();
    const int v = warp & 1;
    unsigned char *k_tiles = smem + lay.k_off[v], *q_tiles = smem + lay.q_off[v];
    if (ONCE && v == 1) {
      if (gathers && warp == store_warp(ONCE)) fused_store<NCOLS>(sh, lane, sums, stored, bars, ab);
    } else if (ONCE || (v == 0 ? visit1 : visit2)) {
      if (warp < 2) {
        if (lane == 0) fused_produce<T, ONCE>(a, sh, v, k_tiles, q_tiles, tile_at, bars, misc + 2, ab);
      } else if (v == 0) {
        fused_multiply<T, NCOLS, FP8, sums_by_rows(ONCE, NCOLS), false>(a, sh, 0, k_tiles, q_tiles, tmem_base, bars, ab);
      } else {
        fused_multiply<T, NCOLS, FP8, false, true>(a, sh, 1, k_tiles, q_tiles, tmem_v2, bars, ab);
      }
    }
  } else if (warp < kSumWarp0) {
    if constexpr (kMoveRegs) reg_dec<64>();
    if (gathers) {
      if (warp < kGatherWarp0 + gather_teams(ONCE) * kTeamWarps)
        fused_gather<T, NCOLS, G, FP8, gather_teams(ONCE)>(a, sh, warp - kGatherWarp0, lane, stored, off, off_c, bars, ab);
      else if (warp == store_warp(ONCE))
        fused_store<NCOLS>(sh, lane, sums, stored, bars, ab);
    } else if (warp == kFetchWarp) {
      if (visit2) fused_fetch_lse<T, NCOLS, G, FP8>(a, sh, lane, stored, off, off_c, bars, ab);
    } else if (visit1) {
      fused_publish<T, NCOLS, G>(a, sh, warp - kPublisherWarp0, lane, sums, stored, bars, ab);
    }
  } else if (warp < kMaxWarp0) {
    if constexpr (kMoveRegs) reg_inc<88>();
    if (visit1) {
      if constexpr (sums_by_rows(ONCE, NCOLS)) sum_by_rows<T, NCOLS, FP8>(a, sh, warp, lane, tmem_base, sums, bars, ab);
      else sum_by_keys<T, NCOLS, FP8, ONCE>(a, sh, warp, lane, tmem_base, sums, bars, ab);
    }
  } else {
    if constexpr (kMoveRegs) reg_inc<88>();
    const uint32_t logits = ONCE ? tmem_base : tmem_v2;
    if (!visit2) {
    } else if constexpr (ONCE && T::NI <= kRegSlots) {
      if (a.max_in_regs) fused_max<T, NCOLS, G, FP8, ONCE, true>(a, sh, warp, lane, logits, amax_tmem, off, off_c, bars, ab);
      else fused_max<T, NCOLS, G, FP8, ONCE, false>(a, sh, warp, lane, logits, amax_tmem, off, off_c, bars, ab);
    } else {
      fused_max<T, NCOLS, G, FP8, ONCE, false>(a, sh, warp, lane, logits, amax_tmem, off, off_c, bars, ab);
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (misc[0] != 0) {
    // a wait ran out somewhere: give copies and MMAs still in flight time to land before TMEM goes away
    const unsigned long long t0 = global_timer();
    while (global_timer() - t0 < 2000000ull) __nanosleep(1000);
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemColsAll) : "memory");
  }
}

// Launches the instantiation for this geometry (one translation unit per head dimension and key format).
struct FusedLaunch {
  int ncols, padded_group, n_cta, smem_bytes;
  bool once;
};
int32_t fused_launch_d64(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream);
int32_t fused_launch_d128(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream);
int32_t fused_launch_d64_fp8(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream);
int32_t fused_launch_d128_fp8(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream);

// The kernel's cross-CTA hand-over needs every CTA of the grid on an SM at the same time.  The launch therefore asks the
// runtime for exactly that guarantee (a cooperative launch; no grid-wide barrier is used): a grid that cannot be
// co-resident -- fewer SMs available than the device reports, e.g. under MPS with a limited SM share -- is refused here
// instead of spinning into the bounded waits.  SMs that are merely busy with other kernels delay the launch; they do not
// break it.
template <int D, int NCOLS, int G, bool FP8, bool ONCE>
int32_t fused_launch_one(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream) {
  auto kern = score_fused_kernel<D, NCOLS, G, FP8, ONCE>;
  static ContextSet allowed;
  const int32_t st = allow_shared_memory(reinterpret_cast<const void*>(kern), kFusedSmemMost, allowed);
  if (st != SPF_OK) return st;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)l.n_cta);
  cfg.blockDim = dim3(kFusedThreads);
  cfg.dynamicSmemBytes = (size_t)l.smem_bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  // The launch may overlap the preparing kernel; grid_wait() orders what reads its results.  (Cooperative, it was seen to start 1.8 to
  // 2 us after that kernel's end all the same.)
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, args);
  if (err == cudaErrorCooperativeLaunchTooLarge) {
    (void)cudaGetLastError();
    return fail(SPF_ERR_UNSUPPORTED, "spf_score: the %d CTAs of the fused kernel cannot all be resident on this device; use the general path",
                l.n_cta);
  }
  SPF_CUDA_CHECK(err);
  return SPF_OK;
}

template <int D, int NCOLS, bool FP8, bool ONCE>
int32_t fused_launch_group(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream) {
  if constexpr (NCOLS <= 32) {                                     // one head per group: at most 32 lookahead queries
    if (l.padded_group == 1) return fused_launch_one<D, NCOLS, 1, FP8, ONCE>(args, l, stream);
  }
  switch (l.padded_group) {
    case 2: return fused_launch_one<D, NCOLS, 2, FP8, ONCE>(args, l, stream);
    case 4: return fused_launch_one<D, NCOLS, 4, FP8, ONCE>(args, l, stream);
    default: return fused_launch_one<D, NCOLS, 8, FP8, ONCE>(args, l, stream);
  }
}

template <int D, bool FP8>
int32_t fused_launch(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream) {
  switch (l.ncols) {
    case 16: return l.once ? fused_launch_group<D, 16, FP8, true>(args, l, stream) : fused_launch_group<D, 16, FP8, false>(args, l, stream);
    case 32: return l.once ? fused_launch_group<D, 32, FP8, true>(args, l, stream) : fused_launch_group<D, 32, FP8, false>(args, l, stream);
    default: return fused_launch_group<D, 64, FP8, false>(args, l, stream);
  }
}

}  // namespace spf
