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
// Tensor-core tiles.  The operands in shared memory are 128 keys x d (TMA) and the slab's query rows x d (row j = i * G + g:
// lookahead i, head g of the GQA group, the group padded to a power of two).  Resident, and visit 2 of the two-pass form:
// keys are the tensor-memory lanes, so the max over the heads of a group is in-thread; the sum over keys ends every slab
// with a 32-lane reduction of up to 32 columns.  Visit 1 of the two-pass form, 32 rows and more: query rows are the lanes
// (weight-stationary instructions, which fill all 128 lanes with 32 or 64 rows), so the sum over keys stays inside a thread
// too; with 64 columns the reduction cost 1000 to 2900 cycles per slab and CTA.  With 16 rows half of those lanes would be
// padding, and twice the tensor memory: keys are the lanes there.  The running maxima live in tensor memory next to the
// accumulators.
//
// Warps.  0 / 1: TMA producers of visit 1 / visit 2.  2 / 3: MMA issuers (resident: one of each).  4: fetches log-sum-exps
// for visit 2.  5..7: publishers (store this CTA's row sums of a slab; add up all CTAs' sums of the rows this CTA owns).  8..15: "sum" warps.  16..23: "max" warps.  Of the eight warps of a visit, warp % 4 picks the TMEM
// lane quadrant and the next bit the `set`: the two sets take turns at the tiles, so that one set's tensor-memory loads and
// waits run while the other set computes.  (Splitting every tile's columns between the sets kept all eight warps in step,
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
// Groups of up to this many CTAs add up everybody's row sums in every CTA (see fused_publish): one hop instead of two, about
// 2 us instead of 3, for reading 16 * CTAs * NCOLS / 4 bytes a slab and CTA.
constexpr int kGatherCtas = 40;
__host__ __device__ constexpr bool gather_alone(int ncols, int n_ctas) { return ncols <= 32 && n_ctas <= kGatherCtas; }
constexpr int kFetchWarp = 4, kPublisherWarp0 = 5, kPublisherWarps = 3;
constexpr int kMaxQStages = 4;         // query tiles in flight per visit (two-pass: 2)
constexpr int kMaxKeyStages = 16;      // key tiles in flight per visit
// Two-pass: accumulator stages per visit.  64 rows at 131072 tokens have three for each visit; with two for each set of visit 1
// and one for each of visit 2 (as many in all) a pass took 559 instead of 519 us, with 8-bit keys 581 instead of 530.
constexpr int kMaxTmemStages = 16;
constexpr int kMaxResident = 32;       // resident: tiles in tensor memory
constexpr int kRegTiles = 8, kRegSlots = 8;   // running maxima stay in registers up to this many tiles a CTA and lookahead slots a key
constexpr int kTmemColsAll = 512;      // the CTA takes all of its SM's tensor memory
constexpr int kOffSlots = 4;           // slabs whose log-sum-exps may be in shared memory at once
constexpr int kSumSlots = 8;           // slabs whose row sums may be on their way to the publishers at once
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
  static constexpr int kCount = kShared + 2 * kOffSlots + 2 * kSumSlots + 2;
  __device__ uint32_t k_full(int v, int s) const { return base + 8u * (v * kVisit + s); }
  __device__ uint32_t k_empty(int v, int s) const { return base + 8u * (v * kVisit + kMaxKeyStages + s); }
  __device__ uint32_t q_full(int v, int s) const { return base + 8u * (v * kVisit + 2 * kMaxKeyStages + s); }
  __device__ uint32_t q_empty(int v, int s) const { return base + 8u * (v * kVisit + 2 * kMaxKeyStages + kMaxQStages + s); }
  __device__ uint32_t t_full(int v, int s) const { return base + 8u * (kTmem + v * kMaxTmemStages + s); }   // resident: v = 0 alone
  __device__ uint32_t t_empty(int v, int s) const { return t_full(v, s) + 8u * kMaxResident; }
  __device__ uint32_t off_ready(int x) const { return base + 8u * (kShared + x); }
  __device__ uint32_t off_free(int x) const { return base + 8u * (kShared + kOffSlots + x); }
  __device__ uint32_t sums_ready(int x) const { return base + 8u * (kShared + 2 * kOffSlots + x); }
  __device__ uint32_t sums_free(int x) const { return base + 8u * (kShared + 2 * kOffSlots + kSumSlots + x); }
  __device__ uint32_t mma_done(int v) const { return base + 8u * (kShared + 2 * kOffSlots + 2 * kSumSlots + v); }
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
  s.off_off = o;   o += kOffSlots * 64 * 4;
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

// Reads what the preparing kernel writes.  This kernel is started while that one still runs, so these are not read-only for its
// lifetime: __ldg may be moved ahead of the wait for the other kernel, a volatile load stays behind it.  (Through L1, which
// has nothing of them before: the loads of neighbouring slabs share a line.)
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
  for (int n = 0; n < sh.n_slabs; ++n) {
    const CUtensorMap* map = maps + layer;
    if (!mbar_wait(bars.q_empty(v, qr.stage), qr.phase ^ 1u, ab)) return;
    mbar_expect_tx(bars.q_full(v, qr.stage), (uint32_t)T::kQBytes);
    bulk_load(q_smem + (uint32_t)(qr.stage * T::kQBytes), q_src + (int64_t)sh.slab(n) * T::kQBytes, (uint32_t)T::kQBytes,
              bars.q_full(v, qr.stage));
    qr.advance();
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
// Tile k of the CTA (k counts over slabs and tiles) has its logits in stage k mod stages.  The whole warp walks the loop
// (addresses and descriptors stay warp-uniform); one elected lane issues.
// ROWS: query rows are the accumulator's lanes (weight-stationary instructions), else the keys.  SETS: a ring of stages for
// each of the two sets of epilogue warps, the odd tiles' behind the even tiles': a tile's maxima belong to one set, so with an
// odd number of tiles a set skips two, and in a common ring of two stages it could take the tile before the one that it
// skipped for its own (a barrier's parity tells one round from the next only).
template <class T, int NCOLS, bool FP8, bool ROWS, bool SETS>
__device__ __forceinline__ void fused_multiply(const FusedArgs& a, const FusedShare& sh, int v, const unsigned char* k_tiles,
                                               const unsigned char* q_tiles, uint32_t tmem, const FusedBars& bars, const Abort& ab) {
  constexpr uint32_t idesc = ROWS ? instr_desc(NCOLS, kTileKeys, FP8) : instr_desc(kTileKeys, NCOLS, FP8);
  const uint64_t k_desc0 = smem_desc<T::SUBROW>(smem_u32(k_tiles));
  const uint64_t q_desc0 = smem_desc<T::SUBROW>(smem_u32(q_tiles));
  Ring kr(a.k_stages[v]), qr(T::QS), even(SETS ? (a.t_stages[v] + 1) / 2 : a.t_stages[v]), odd(a.t_stages[v] / 2);
  const int n_slabs = sh.n_slabs, n_tiles = sh.n_tiles;
  for (int n = 0; n < n_slabs; ++n) {
    if (!mbar_wait_warp(bars.q_full(v, qr.stage), qr.phase, ab)) return;
    const uint64_t qd0 = q_desc0 + (uint64_t)((qr.stage * T::kQBytes) >> 4);
    auto tile = [&](Ring& tr, int stage0) -> bool {
      const int stage = stage0 + tr.stage;
      if (!mbar_wait2_warp(bars.k_full(v, kr.stage), kr.phase, bars.t_empty(v, stage), tr.phase ^ 1u, ab)) return false;
      tc_fence_after();
      const uint32_t d_tmem = tmem + (uint32_t)(stage * NCOLS);
      const uint64_t kd0 = k_desc0 + (uint64_t)((kr.stage * T::kTileBytes) >> 4);
      if (elect_one()) {
#pragma unroll
        for (int part = 0; part < T::QPARTS; ++part)               // 8-bit keys: the two query terms accumulate into the same columns
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
      }
      __syncwarp();
      kr.advance();
      tr.advance();
      return true;
    };
    for (int lt = 0; lt < n_tiles; ++lt)
      if (!(SETS && (lt & 1) ? tile(odd, even.n) : tile(even, 0))) return;
    if (elect_one()) tc_commit(bars.q_empty(v, qr.stage));
    __syncwarp();
    qr.advance();
  }
  // leave only after everything issued has completed and signalled its barriers
  if (elect_one()) tc_commit(bars.mma_done(v));
  __syncwarp();
  mbar_wait_warp(bars.mma_done(v), 0u, ab);
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
  float next_ref = produced(refs + sh.slab(0)), next_c = FP8 ? produced(slab_c + sh.slab(0)) : a.c;
  for (int n = 0; n < n_slabs; ++n) {
    const uint64_t nref = pack2(-next_ref, -next_ref), cc = pack2(next_c, next_c);
    if (n + 1 < n_slabs) {
      next_ref = produced(refs + sh.slab(n + 1));
      if constexpr (FP8) next_c = produced(slab_c + sh.slab(n + 1));
    }
    uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
    for (; lt < n_tiles; lt += 2) {
      if (!mbar_wait_warp(bars.t_full(0, tr.stage), tr.phase, ab)) return;
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

// The sums where keys are the lanes.  Tiles k with k mod 2 == set; a thread has one key per tile and sums of all rows, which it
// shares out over the warp at the end of a slab.  (The two-pass form with its 64 rows took 10 to 20 % longer this way, whether
// a warp had all rows of every other tile or half the rows of each.  With 16 rows it is the quicker one, 960 -> 910 us for
// 16 layers x 8 heads at 340942 tokens, and its columns are half as many: 28 tiles a CTA at 16 slots a key instead of 26, where
// the general path takes 152 us for two layers at 511438 tokens and this one 105.)
template <class T, int NCOLS, bool FP8, bool ONCE>
__device__ __forceinline__ void sum_by_keys(const FusedArgs& a, const FusedShare& sh, int warp, int lane, uint32_t tmem, float* sums,
                                             const FusedBars& bars, const Abort& ab) {
  const FusedPrompt& p = *sh.p;
  const int quad = warp & 3, set = (warp - kSumWarp0) >> 2;
  const int n_slabs = sh.n_slabs, n_tiles = sh.n_tiles;
  const float* const refs = p.refs;
  const float* const slab_c = p.slab_c;
  const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16);
  const int full_tiles = (int)(p.n_tokens / kTileKeys);            // tiles below this index have 128 real keys
  const int tail_lanes = (int)(p.n_tokens - (int64_t)full_tiles * kTileKeys) - quad * 32;   // real keys of this quadrant in the last tile
  const bool frees = !ONCE || a.mode == 1;                // the accumulators wait for no visit 2
  Ring tr(a.t_stages[0]);
  tr.advance(set);
  int lt = set;                                                    // this set's next tile, counted from the slab's first
  float next_ref = produced(refs + sh.slab(0)), next_c = FP8 ? produced(slab_c + sh.slab(0)) : a.c;
  for (int n = 0; n < n_slabs; ++n) {
    const uint64_t nref = pack2(-next_ref, -next_ref), cc = pack2(next_c, next_c);
    if (n + 1 < n_slabs) {
      next_ref = produced(refs + sh.slab(n + 1));
      if constexpr (FP8) next_c = produced(slab_c + sh.slab(n + 1));
    }
    uint64_t acc[NCOLS / 2];
#pragma unroll
    for (int j = 0; j < NCOLS / 2; ++j) acc[j] = 0ull;
    const bool any = lt < n_tiles;
    for (; lt < n_tiles; lt += 2) {
      if (!mbar_wait_warp(bars.t_full(0, tr.stage), tr.phase, ab)) return;
      tc_fence_after();
      uint32_t r[NCOLS];
      tmem_issue<NCOLS>(lane_addr + (uint32_t)(tr.stage * NCOLS), r);
      tmem_load_wait();
      tmem_ready<NCOLS>(r);
      if (frees) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.t_empty(0, tr.stage));
      }
      tr.advance(2);
      if (sh.tile(lt) < full_tiles || lane < tail_lanes) {
#pragma unroll
        for (int j = 0; j < NCOLS / 2; ++j) {
          float x, y;
          unpack2(fma2(pack2(r[2 * j], r[2 * j + 1]), cc, nref), x, y);
          acc[j] = add2(acc[j], pack2(fast_exp2(x), fast_exp2(y)));
        }
      }
    }
    lt -= n_tiles;
    // Sum over the warp's 32 keys: transposing butterfly steps, each of which halves the columns a lane holds, then (16
    // columns) one plain step.  The publishers add up quadrants and sets.
    float s[NCOLS];
    s[0] = 0.f;
    if (any) {
#pragma unroll
      for (int j = 0; j < NCOLS / 2; ++j) unpack2(acc[j], s[2 * j], s[2 * j + 1]);
      int width = NCOLS;
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) {
        if (width > 1) {
          width >>= 1;
          const bool upper = (lane & off) != 0;
#pragma unroll
          for (int j = 0; j < NCOLS / 2; ++j) {
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
    }
    const int slot = n % kSumSlots;
    if (n >= kSumSlots)
      if (!mbar_wait_warp(bars.sums_free(slot), (uint32_t)(n / kSumSlots - 1) & 1u, ab)) return;
    float* out = sums + ((slot * 2 + set) * 4 + quad) * 32;
    if constexpr (NCOLS == 32) {
      out[lane] = s[0];
    } else {
      if ((lane & 1) == 0) out[lane >> 1] = s[0];
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.sums_ready(slot));
  }
}

// ---------------------------------------------------------------------------------------------- publishers
// Waits for and adds up CTAs' row sums of a slab.  LANES = 1: the four rows of quad `q`, a CTA per lane; LANES = NCOLS / 4:
// all rows, lane mod LANES being the quad.  On return lane (with lane mod 8 < LANES) has the log-sum-exp, in base-2 units,
// of row 4 * quad + lane / 8 in `lse2`; false if the wait was given up.
template <int NCOLS, int G, int LANES, int MAXW>
__device__ __forceinline__ bool sum_rows_of(const FusedArgs& a, const FusedPrompt& p, int slab, int q, int n_ctas, int lane, bool report,
                                            float& lse2, const Abort& ab) {
  constexpr int Q = NCOLS / 4, STEP = 32 / LANES;                  // CTAs per load of the warp
  if (LANES > 1) q = lane % Q;
  const int first = lane / LANES;
  const float4* in = p.row_sums + ((int64_t)slab * p.per_part + first) * Q + q;
  const float ref = produced(p.refs + slab);                        // its way to L2 and back passes during the wait below
  float4 v[MAXW];
#pragma unroll
  for (int i = 0; i < MAXW; ++i) v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto missing = [&](int i) {
    return first + STEP * i < n_ctas && (v[i].x == 0.f || v[i].y == 0.f || v[i].z == 0.f || v[i].w == 0.f);
  };
  unsigned long long t0 = 0;
  for (uint32_t it = 1;; ++it) {
    // whatever is not there yet is asked for again (a word may also be caught half written)
#pragma unroll
    for (int i = 0; i < MAXW; ++i)
      if (missing(i))
        asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[i].x), "=f"(v[i].y), "=f"(v[i].z), "=f"(v[i].w)
                     : "l"(in + (int64_t)STEP * i * Q)
                     : "memory");
    bool there = true;
#pragma unroll
    for (int i = 0; i < MAXW; ++i) there = there && !missing(i);
    if (__all_sync(0xffffffffu, there)) break;
    if (__any_sync(0xffffffffu, give_up(it, t0, ab))) return false;
    if (LANES == 1) __nanosleep(100);
  }
  double t[4] = {0.0, 0.0, 0.0, 0.0};                              // the CTAs' shares are fp32: exact to 2^-53
#pragma unroll
  for (int i = 0; i < MAXW; ++i) {
    t[0] += (double)v[i].x;
    t[1] += (double)v[i].y;
    t[2] += (double)v[i].z;
    t[3] += (double)v[i].w;
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
  const int row = 4 * q + (lane >> 3);
  lse2 = INFINITY;                                                 // rows that do not exist: exp2(x - lse2) = 0
  if ((lane & 7) < LANES && row % G < a.group && row / G < a.n_lookahead) {
    // log2 of the total: its binary exponent plus the log2 of its mantissa in single precision; an empty (below every
    // normal number) or overflowed row sum has none
    const long long tb = __double_as_longlong(t[0]);
    const float mant = (float)__longlong_as_double((tb & 0x000fffffffffffffll) | 0x3ff0000000000000ll);
    lse2 = ref + ((float)((int)((tb >> 52) & 0x7ff) - 1023) + log2f(mant));
    if (!(t[0] > 1.2e-38 && t[0] < (double)INFINITY)) lse2 = INFINITY;
    const int64_t out_idx = ((int64_t)slab * a.group + row % G) * a.n_lookahead + row / G;
    if (p.extra_lse != nullptr) {
      // the denominator also holds exp(extra): log2-add, in the order that cannot overflow
      const float e = __ldg(p.extra_lse + out_idx) * kLog2e;
      const float hi = fmaxf(lse2, e), lo = fminf(lse2, e);
      lse2 = hi + log2f(1.f + exp2f(lo - hi));
    }
    if (report) {
      if (!(lse2 > -INFINITY && lse2 < INFINITY) && a.dev_status != nullptr) atomicCAS(a.dev_status, 0, (int32_t)SPF_ERR_RANGE);
      if (p.lse_out != nullptr) p.lse_out[out_idx] = lse2 * kLn2;
    }
  }
  return true;
}

// Publisher w takes slabs w, w + 3, ...: stores this CTA's row sums (a row that does not exist gets its meaningless sum
// stored too: everybody waits for every word).  Then either this CTA adds up everybody's sums for itself (few CTAs to a
// group: one hop), or only those of the rows that it owns -- item n * Q + q, rows 4q .. 4q + 3 of the group's n-th slab,
// belongs to CTA (item mod CTAs) -- and stores their log-sum-exps for all.  Not before its own sums are out: polling for
// words that cannot be there yet slowed the key copies down.
template <class T, int NCOLS, int G, bool FP8>
__device__ __forceinline__ void fused_publish(const FusedArgs& a, const FusedShare& sh, int which, int lane, const float* sums, float* off,
                                              float* off_c, const FusedBars& bars, const Abort& ab) {
  constexpr int Q = NCOLS / 4;                                     // lane q has rows 4q .. 4q + 3
  const FusedPrompt& p = *sh.p;
  const int per_part = p.per_part, n_ctas = min(per_part, p.n_tiles);
  const bool alone = gather_alone(NCOLS, n_ctas);
  for (int n = which; n < sh.n_slabs; n += kPublisherWarps) {
    const int slot = n % kSumSlots, slab = sh.slab(n);
    if (!mbar_wait_warp(bars.sums_ready(slot), (uint32_t)(n / kSumSlots) & 1u, ab)) return;
    float t[4] = {0.f, 0.f, 0.f, 0.f};
    if (lane < Q) {
      // [set][quadrant][lane]: 64 rows: quadrants 0 and 2 have rows 0..31, 1 and 3 rows 32..63; else every quadrant all rows
      const float* in = sums + slot * 256 + (NCOLS == 64 ? (lane >> 3) * 32 + (lane & 7) * 4 : lane * 4);
#pragma unroll
      for (int set = 0; set < 2; ++set)
#pragma unroll
        for (int q = 0; q < (NCOLS == 64 ? 2 : 4); ++q) {
          const float4 v = *reinterpret_cast<const float4*>(in + set * 128 + q * (NCOLS == 64 ? 64 : 32));
          t[0] += v.x;
          t[1] += v.y;
          t[2] += v.z;
          t[3] += v.w;
        }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.sums_free(slot));
    if (lane < Q) {
      unsigned w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) w[e] = max(__float_as_uint(t[e]), 1u);   // never "not there yet"; 2^-149 is nothing to a row's sum
      asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};"
                   ::"l"(p.row_sums + ((int64_t)slab * per_part + sh.first) * Q + lane), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                   : "memory");
    }
    float lse2;
    if constexpr (NCOLS <= 32) {
      if (alone) {
        if (a.mode == 1 && sh.first != 0) continue;                // nobody reads the offsets
        const float c = FP8 ? produced(p.slab_c + slab) : 0.f;
        if (!sum_rows_of<NCOLS, G, Q, kGatherCtas * Q / 32>(a, p, slab, 0, n_ctas, lane, sh.first == 0, lse2, ab)) return;
        if (a.mode == 1) continue;
        const int x = n % kOffSlots;
        if (n >= kOffSlots)
          if (!mbar_wait_warp(bars.off_free(x), (uint32_t)(n / kOffSlots - 1) & 1u, ab)) return;
        if ((lane & 7) < Q) off[x * 64 + 4 * (lane % Q) + (lane >> 3)] = -lse2;
        if constexpr (FP8) {
          if (lane == 0) off_c[x] = c;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.off_ready(x));
        continue;
      }
    }
    for (int q = (int)(((unsigned)(n + 1) * (unsigned)n_ctas * Q + sh.first - n * Q) % (unsigned)n_ctas); q < Q; q += n_ctas) {
      if (!sum_rows_of<NCOLS, G, 1, (kFusedMaxCtas + 31) / 32>(a, p, slab, q, n_ctas, lane, true, lse2, ab)) return;
      if ((lane & 7) == 0) {
        const unsigned long long word = (1ull << 32) | __float_as_uint(lse2);
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p.lse + (int64_t)slab * NCOLS + 4 * q + (lane >> 3)), "l"(word) : "memory");
      }
      __syncwarp();
    }
  }
}

// ---------------------------------------------------------------------------------------------- log-sum-exps for visit 2
// Fetches each slab's log-sum-exps in turn, kAhead slabs' words in flight, and hands them to the max warps through shared
// memory (negated: what visit 2 adds).
template <class T, int NCOLS, int G, bool FP8>
__device__ __forceinline__ void fused_fetch_lse(const FusedArgs& a, const FusedShare& sh, int lane, float* off, float* off_c,
                                                const FusedBars& bars, const Abort& ab) {
  const FusedPrompt& p = *sh.p;
  constexpr int RPL = NCOLS == 64 ? 2 : 1;
  constexpr int kAhead = 4;
  unsigned long long w[kAhead][RPL];
  auto load = [&](unsigned long long (&dst)[RPL], int n) {
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
      const int row = min(lane + 32 * r, NCOLS - 1);
      if (a.mode == 2) {
        const bool real = row % G < a.group && row / G < a.n_lookahead;
        const float v = real ? __ldg(p.lse_in + ((int64_t)sh.slab(n) * a.group + row % G) * a.n_lookahead + row / G) * kLog2e : INFINITY;
        dst[r] = (1ull << 32) | __float_as_uint(v);
      } else {
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(dst[r]) : "l"(p.lse + (int64_t)sh.slab(n) * NCOLS + row) : "memory");
      }
    }
  };
#pragma unroll
  for (int i = 0; i < kAhead; ++i)
    if (i < sh.n_slabs) load(w[i], i);
  for (int n0 = 0; n0 < sh.n_slabs; n0 += kAhead) {
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      const int n = n0 + i;
      if (n < sh.n_slabs) {
        const float c = FP8 ? produced(p.slab_c + sh.slab(n)) : 0.f;
        unsigned long long t0 = 0;
        for (uint32_t it = 1;; ++it) {
          bool there = true;
#pragma unroll
          for (int r = 0; r < RPL; ++r) there = there && (w[i][r] >> 32) != 0ull;
          if (__all_sync(0xffffffffu, there)) break;
          if (__any_sync(0xffffffffu, give_up(it, t0, ab))) return;
          load(w[i], n);
        }
        float v[RPL];
#pragma unroll
        for (int r = 0; r < RPL; ++r) v[r] = -__uint_as_float((unsigned)w[i][r]);
        if (n + kAhead < sh.n_slabs) load(w[i], n + kAhead);
        const int slot = n % kOffSlots;
        if (n >= kOffSlots)
          if (!mbar_wait_warp(bars.off_free(slot), (uint32_t)(n / kOffSlots - 1) & 1u, ab)) return;
#pragma unroll
        for (int r = 0; r < RPL; ++r)
          if (lane + 32 * r < NCOLS) off[slot * 64 + lane + 32 * r] = v[r];
        if constexpr (FP8) {
          if (lane == 0) off_c[slot] = c;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.off_ready(slot));
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------- importance
// Mean over the lookahead of exp2(running max) for a tile's keys.  One group of CTAs (parts = 1): straight from the maxima.
// Several: the groups' maxima meet in global memory, and whichever warp brings the last contribution for 32 keys reads the
// result.
template <int NI>
__device__ __forceinline__ void finish_tile(const FusedArgs& a, const FusedPrompt& p, int tile, int quad, int lane, const uint32_t (&v)[NI]) {
  const float inv_m = 1.f / (float)a.n_lookahead;
  const int64_t key = (int64_t)tile * kTileKeys + quad * 32 + lane;
  float sum = 0.f;
  if (p.parts == 1) {
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (i < a.n_lookahead) sum += fast_exp2(__uint_as_float(v[i]));
  } else {
    const int64_t n_pad = (int64_t)p.n_tiles * kTileKeys;
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (i < a.n_lookahead) atomicMax(p.amax + (int64_t)i * n_pad + key, order_bits(__uint_as_float(v[i])));
    __threadfence();
    __syncwarp();
    unsigned before = 0;
    if (lane == 0) before = atomicAdd(p.finished + tile * 4 + quad, 1u);
    if (__shfl_sync(0xffffffffu, before, 0) + 1u != (unsigned)p.parts) return;
    __threadfence();
#pragma unroll 8
    for (int i = 0; i < a.n_lookahead; ++i) sum += fast_exp2(from_order_bits(__ldcg(p.amax + (int64_t)i * n_pad + key)));
  }
  if (key < p.n_tokens) p.importance[key] = sum * inv_m;
}

// The tiles of a max warp's set, from the maxima in tensor memory.
template <class T>
__device__ __forceinline__ void fused_finish(const FusedArgs& a, const FusedShare& sh, int warp, int lane, uint32_t amax_tmem) {
  const int quad = warp & 3, set = (warp - kMaxWarp0) >> 2;
  const uint32_t lane_addr = amax_tmem + ((uint32_t)(quad * 32) << 16);
  for (int lt = set; lt < sh.n_tiles; lt += 2) {
    constexpr int LD = T::NI < 32 ? T::NI : 32;                    // columns per load
    uint32_t v[T::NI];
#pragma unroll
    for (int i = 0; i < T::NI; i += LD)
      tmem_issue<LD>(lane_addr + (uint32_t)(lt * T::NI + i), *reinterpret_cast<uint32_t(*)[LD]>(v + i));
    tmem_load_wait();
    tmem_ready<T::NI>(v);
    finish_tile<T::NI>(a, *sh.p, sh.tile(lt), quad, lane, v);
  }
}

// ---------------------------------------------------------------------------------------------- visit 2: maxima
// Folds one load's accumulators into the running maxima over (layer, head) of the base-2 logits less their rows'
// log-sum-exps (slots past n_lookahead hold padding and are never read).
template <class T, int G>
__device__ __forceinline__ void fold_maxima(const uint32_t (&r)[T::CW], uint32_t (&am)[T::NIW], const ulonglong2* off2, uint64_t cc) {
  float z[T::CW];
#pragma unroll
  for (int j = 0; j < T::CW / 4; ++j) {
    const ulonglong2 o = off2[j];
    unpack2(fma2(pack2(r[4 * j], r[4 * j + 1]), cc, o.x), z[4 * j], z[4 * j + 1]);
    unpack2(fma2(pack2(r[4 * j + 2], r[4 * j + 3]), cc, o.y), z[4 * j + 2], z[4 * j + 3]);
  }
#pragma unroll
  for (int i = 0; i < T::NIW; ++i) {
    float m = __uint_as_float(am[i]);
    if constexpr (G == 1) {
      m = fmaxf(m, z[i]);
    } else {
#pragma unroll
      for (int g = 0; g < G; g += 2) m = max3(m, z[i * G + g], z[i * G + g + 1]);
    }
    am[i] = __float_as_uint(m);
  }
}

// -inf in the running maxima of a set's tiles.
template <class T>
__device__ __forceinline__ void clear_maxima(uint32_t amax_addr, int set, int n_tiles) {
  uint32_t ninf[T::NIW];
#pragma unroll
  for (int j = 0; j < T::NIW; ++j) ninf[j] = 0xff800000u;
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
  const int stage0 = ONCE ? 0 : set * ((a.t_stages[V] + 1) / 2);
  for (int n = 0; n < sh.n_slabs; ++n) {
    const int slot = n % kOffSlots;
    if (!mbar_wait_warp(bars.off_ready(slot), (uint32_t)(n / kOffSlots) & 1u, ab)) return;
    const ulonglong2* off2 = reinterpret_cast<const ulonglong2*>(off + slot * 64);
    const float c = FP8 ? off_c[slot] : a.c;
    const uint64_t cc = pack2(c, c);
    Ring tr = first;
    if (ONCE) tr.advance(set);
    auto fold = [&](int lt, uint32_t (&m)[NIW]) -> bool {
      // resident: complete long since (the log-sum-exps contain it), except where visit 2 runs alone
      if (!mbar_wait_warp(bars.t_full(V, stage0 + tr.stage), tr.phase, ab)) return false;
      tc_fence_after();
      if (!REGS) tmem_store_wait();                                // the maxima read below may be this warp's last stores
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) {
        const uint32_t m_addr = amax_addr + (uint32_t)(lt * T::NI + ch * NIW);
        uint32_t r[CW];
        tmem_issue<CW>(lane_addr + (uint32_t)((stage0 + tr.stage) * NCOLS + ch * CW), r);
        if (!REGS) tmem_issue<NIW>(m_addr, m);
        tmem_load_wait();
        tmem_ready<CW>(r);
        if (!REGS) tmem_ready<NIW>(m);
        if (ch + 1 == NCH) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bars.t_empty(V, stage0 + tr.stage));
        }
        fold_maxima<T, G>(r, m, off2 + ch * (CW / 4), cc);
        if (!REGS) tmem_store<NIW>(m_addr, m);
      }
      tr.advance(ONCE ? 2 : 1);
      return true;
    };
    if constexpr (REGS) {
#pragma unroll
      for (int u = 0; u < MINE; ++u)
        if (set + 2 * u < n_tiles)
          if (!fold(set + 2 * u, am[u])) return;
    } else {
      for (int lt = set; lt < n_tiles; lt += 2)
        if (!fold(lt, am[0])) return;
    }
    if (ONCE) first.advance(n_tiles);
    else first = tr;
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.off_free(slot));
  }
  if constexpr (REGS) {
#pragma unroll
    for (int u = 0; u < MINE; ++u)
      if (set + 2 * u < n_tiles) finish_tile<NIW>(a, *sh.p, sh.tile(set + 2 * u), quad, lane, am[u]);
  } else {
    tmem_store_wait();
    fused_finish<T>(a, sh, warp, lane, amax_tmem);
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
  volatile int* misc = reinterpret_cast<volatile int*>(smem + lay.misc_off);  // [0] abort, [1] tensor-memory base, [2] tiles visit 2 has issued
  const FusedBars bars{smem_u32(smem + lay.bar_off)};
  const Abort ab{misc, a.dev_status};
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

  // ------------------------------------------------------------------ set-up
  if (threadIdx.x == 0) {
    misc[0] = 0;
    misc[1] = 0;
    misc[2] = 0;
    for (int v = 0; v < (ONCE ? 1 : 2); ++v) {
      for (int s = 0; s < a.k_stages[v]; ++s) {
        mbar_init(bars.k_full(v, s), 1);
        mbar_init(bars.k_empty(v, s), 1);
      }
      for (int s = 0; s < T::QS; ++s) {
        mbar_init(bars.q_full(v, s), 1);
        mbar_init(bars.q_empty(v, s), 1);
      }
      for (int s = 0; s < a.t_stages[v]; ++s) {
        mbar_init(bars.t_full(v, s), 1);
        mbar_init(bars.t_empty(v, s), kVisitWarps / 2);
      }
      mbar_init(bars.mma_done(v), 1);
    }
    for (int x = 0; x < kOffSlots; ++x) {
      mbar_init(bars.off_ready(x), 1);
      mbar_init(bars.off_free(x), kVisitWarps);
    }
    for (int x = 0; x < kSumSlots; ++x) {
      mbar_init(bars.sums_ready(x), kVisitWarps);
      mbar_init(bars.sums_free(x), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // paged key cache: a tile never straddles a block (blocks are multiples of 128 tokens): one lookup per tile for the whole kernel
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
  // tensor memory: the accumulator stages, then the running maxima, [local tile][NI] columns (lane = key)
  const uint32_t tmem_v2 = tmem_base + (uint32_t)(a.t_stages[0] * NCOLS);
  const uint32_t amax_tmem = tmem_v2 + (uint32_t)(ONCE ? 0 : a.t_stages[1] * NCOLS);
  grid_wait();                                                     // what the preparing kernel wrote is visible from here on
  grid_launch_dependents();                                        // the next kernel starts where SMs are free, and waits there

  // ------------------------------------------------------------------ roles
  // resident, 32 rows: 768 threads start with 80 registers each; 256 x 64 + 512 x 88 is the same sum
  constexpr bool kMoveRegs = ONCE && NCOLS == 32;
  const bool visit1 = a.mode != 2, visit2 = a.mode != 1;
  if (warp < 4) {
    if constexpr (kMoveRegs) reg_dec<64>();
    const int v = warp & 1;
    if (ONCE ? v == 0 : (v == 0 ? visit1 : visit2)) {
      unsigned char *k_tiles = smem + lay.k_off[v], *q_tiles = smem + lay.q_off[v];
      if (warp < 2) {
        if (lane == 0) fused_produce<T, ONCE>(a, sh, v, k_tiles, q_tiles, tile_at, bars, misc + 2, ab);
      } else {
        if (v == 0) fused_multiply<T, NCOLS, FP8, sums_by_rows(ONCE, NCOLS), false>(a, sh, 0, k_tiles, q_tiles, tmem_base, bars, ab);
        else fused_multiply<T, NCOLS, FP8, false, true>(a, sh, 1, k_tiles, q_tiles, tmem_v2, bars, ab);
      }
    }
  } else if (warp < kSumWarp0) {
    if constexpr (kMoveRegs) reg_dec<64>();
    if (warp == kFetchWarp) {
      if (visit2 && !(visit1 && gather_alone(NCOLS, min(sh.p->per_part, sh.p->n_tiles)))) fused_fetch_lse<T, NCOLS, G, FP8>(a, sh, lane, off, off_c, bars, ab);
    } else if (visit1) {
      fused_publish<T, NCOLS, G, FP8>(a, sh, warp - kPublisherWarp0, lane, sums, off, off_c, bars, ab);
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
  // the launch overlaps the preparing kernel; grid_wait() orders what reads its results
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
