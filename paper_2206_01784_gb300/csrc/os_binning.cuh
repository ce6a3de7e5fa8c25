// Phase 3 of Onesweep (arXiv 2206.01784, Section 3, "Chained scan
// digit-binning kernel"; Figures 6-8): one single-pass digit-binning
// iteration, ~2n global words moved per pass.
//
// One block per tile of T = NT * IPT keys. Per tile:
//  1. tile id from a global atomic counter, so tiles run in order whatever the
//     hardware's block schedule (the look-back then always makes progress);
//  2. the tile's keys (and values) are staged into shared memory by bulk
//     copies on the TMA engine (one elected thread, an mbarrier completes).
//     The copy covers the 16-byte-aligned span around the tile, so tiles that
//     start anywhere (segments of a batch) still use it; plain loads are the
//     fallback when that span would leave the array;
//  3. early counts: each warp counts the digits of its part of the tile with
//     shared-memory atomics (the paper's privatised, atomically updated
//     histograms of the upfront kernel, here per warp and per tile);
//  4. thread i publishes (L, count of digit i) in the tile's status counter
//     and sends the first round of its look-back over the preceding tiles'
//     counters of digit i (Section 3, decoupled look-back); a block scan of
//     the counts gives the tile-relative bin starts. Homogeneous-tile
//     short-circuit: if every key has the same digit, ranking and local
//     reorganisation are skipped and the tile is written straight to its
//     bin (Section 3, last paragraph of the kernel description);
//  5. each warp's per-digit counters start at the local position of its
//     first key of that digit (tile bin start plus the lower warps' counts);
//  6. warp-level multi-split ranking: each warp walks its keys in 32-wide
//     batches and ranks each among the warp's equal digits, either as in the
//     paper with one ballot per digit bit ANDed together and the lowest lane
//     of each group bumping the warp's counter (Section 3, WLMS paragraph), or
//     with counting atomics whose undefined order among equal lanes is
//     replaced by lane order (rank_atomic). With counters that start at local
//     positions, the rank is the key's place in the tile's shared-memory
//     bins, and the key is written there at once.
//     Every few batches the look-back's round in flight is folded in
//     and the next one sent, so its L2 round trips ride along the ranking. A
//     __match_any_sync per key measured 1.7x slower than the ballots on
//     GB300 (the match instruction saturates the ADU pipe) and is not used;
//     the values follow the keys' positions;
//  7. the look-back ends (bounded wait) and publishes (G, inclusive prefix),
//     and runs of keys (and values) are copied from the shared-memory bins to
//     their global bins, consecutive threads writing consecutive addresses.
//
// The paper's block publishes its counts after ranking; counting first
// publishes them a ranking earlier, so a tile's predecessors' counts are
// there by the time its ranking ends, and the separate reorganisation loop
// (re-reading each key's digit offset) disappears.
//
// In segmented mode (os_sort_batch) every segment is a sort of its own: its
// tiles form one look-back chain that starts at the segment's first tile, and
// it has its own bin offsets.
//
// There are no per-key bounds checks: a chain's ragged last tile is filled up
// with keys that sort behind it and are never stored. A second body for it
// would be fetched cold by one block at the very end of every pass, which
// costs a pass about 25 us (8.0M u32 pairs: 78 us a pass, 2^23 pairs: 49).
#pragma once

#include "os_common.cuh"
#include "os_internal.h"
#include "os_places.h"

namespace onesweep {

// Tile geometries (threads per block, keys per thread, resident blocks per
// SM). Index = the geometry part of the launcher's tile configuration.
// Geometry 0, the default, has the largest tile of which three blocks still
// fit an SM by registers (80 a thread) and shared memory (76 KB for 32-bit
// pairs, 72 KB for 64-bit pairs): the look-back's reads, its wait and the
// per-tile scans are paid per tile, and longer runs write fewer partial lines,
// while fewer than 24 warps leave the shared-memory pipe idle. Measured at
// 2^28 u32, ms per pass, pairs / keys only: 256 x 24 x 3 blocks 1.13 / 0.836,
// 256 x 32 x 3 1.01 / 0.723, 256 x 36 x 3 - / 0.721, 384 x 32 x 2 1.03 /
// 0.730, 512 x 24 x 2 1.34 / 0.742, 256 x 40 x 2 1.07 / 0.799, 512 x 32 x 1
// 1.20 / 0.868; at 2^27 u64: 256 x 12 x 3 0.905 / 0.741, 256 x 16 x 3 0.788 /
// 0.630, 256 x 20 x 3 0.714 / 0.566, 256 x 24 x 2 0.765 / 0.606. The smaller
// tiles are faster only where the largest one makes little more than one wave
// of blocks (4.2M u32 pairs: 124 us a sort with geometry 1 against 133, 6.5M
// 176 against 174).
template <int KBITS, int CFG> struct TileShape;
template <> struct TileShape<32, 0> { static constexpr int NT = 256, IPT = 32, MINB = 3; };
template <> struct TileShape<32, 1> { static constexpr int NT = 256, IPT = 24, MINB = 3; };
template <> struct TileShape<32, 2> { static constexpr int NT = 256, IPT = 16, MINB = 4; };
template <> struct TileShape<64, 0> { static constexpr int NT = 256, IPT = 20, MINB = 3; };
template <> struct TileShape<64, 1> { static constexpr int NT = 256, IPT = 16, MINB = 3; };
template <> struct TileShape<64, 2> { static constexpr int NT = 256, IPT = 8, MINB = 4; };

// Digit-ranking variants of step 6. Two methods find a key's rank among the
// equal digits of its warp: ballots (one per digit bit, the paper's WLMS; ALU
// work, insensitive to the key distribution) and counting atomics (every lane
// adds one to its digit's counter and reads it back; shared-memory work that
// slows down when many lanes share a digit).
constexpr int kRankBallot = 0;    // ballots only
constexpr int kRankAdaptive = 1;  // atomics, one digit apart, or ballots, by the place's ranking word
constexpr int kRankAtomic = 2;    // counting atomics only
constexpr int kRankDominant = 3;  // (one digit apart: a body of the adaptive variant, not a variant)

// Batches whose counting atomics are in flight together: they do not depend
// on one another, so a chunk pays one shared-memory round trip. Pairs keep
// their positions in registers beside the keys and take two (2^28 u32 pairs:
// 1.003 ms per pass against 1.017 with four; keys only 0.727 with two, 0.723
// with four, 0.716 with eight).
__host__ __device__ constexpr int rank_chunk(bool pairs, int ipt) { return pairs || ipt % 4 != 0 ? 2 : 4; }

template <int KBITS, bool PAIRS, int CFG = 0>
struct BinningConfig {
  static constexpr int NT = TileShape<KBITS, CFG>::NT;            // threads per block
  static constexpr int IPT = TileShape<KBITS, CFG>::IPT;          // keys per thread
  static constexpr int MIN_BLOCKS = TileShape<KBITS, CFG>::MINB;  // resident blocks per SM
  static constexpr int T = NT * IPT;                              // keys per tile
  static constexpr int NW = NT / 32;
  using K = typename KeyWord<KBITS>::type;
  // staging buffers hold a tile plus the slack of a 16-byte-aligned span
  static constexpr size_t kbuf_bytes = (size_t)T * sizeof(K) + 16;
  static constexpr size_t vbuf_bytes = PAIRS ? (size_t)T * 4 + 16 : 0;
  static constexpr size_t whist_bytes = (size_t)NW * kRadix * 4;  // [NW][256] digit counts
  static constexpr size_t small_bytes = 2 * kRadix * 4 + 64 * 4 + 2 * 8;
  static constexpr size_t smem_bytes = kbuf_bytes + vbuf_bytes + whist_bytes + small_bytes;
};

// Lanes of the warp whose digit equals this lane's (valid lanes only): one
// vote per digit bit (Section 3, WLMS), keeping the lanes that agree on it.
// RB: bits per digit.
template <int RB = kRadixBits>
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, bool valid, uint32_t valid_mask) {
  uint32_t peers = valid_mask;
#pragma unroll
  for (int b = 0; b < RB; ++b) {
    const bool bit = (d >> b) & 1u;
    const uint32_t v = __ballot_sync(0xFFFFFFFFu, bit);
    peers &= bit ? v : ~v;
  }
  return valid ? peers : 0u;
}

// Float keys: FLIP bit 0 applies the sign-flip to loaded keys (first pass),
// bit 1 undoes it on stored keys (last pass).
template <int FLIP, typename K>
__device__ __forceinline__ K load_transform(K k) {
  return (FLIP & 1) ? flip_to_ordered(k) : k;
}
template <int FLIP, typename K>
__device__ __forceinline__ K store_transform(K k) {
  return (FLIP & 2) ? flip_from_ordered(k) : k;
}

// Where a tile sits: set up by the kernel's front-end, read by the body.
struct TileCtx {
  uint32_t tile;         // row of the tile in the status slabs
  uint32_t chain_first;  // first tile of its look-back chain
  uint32_t start;        // array index of the tile's first key
  uint32_t count;        // keys in the tile (0: no tile for this block)
  uint32_t koff, voff;   // staging offsets (elements) of the tile in kbuf / vbuf
  uint32_t out_base;     // array index of the chain's (segment's) first key
  uint32_t out_len;      // keys in the chain's segment
  uint32_t bulk;         // staged by bulk copies (wait on the mbarriers)
  uint32_t rank_word;    // how this place (of this segment) is ranked (finish_place in os_common.cuh)
  const uint32_t* bin_offsets;  // this place's 256 bin offsets (segment-relative)
};

__device__ __forceinline__ uint32_t lanemask_ge() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_ge;" : "=r"(m));
  return m;
}

// Warp-level multi-split ranking of one 32-key batch with ballots. Returns the
// value the warp's running counter of the key's digit has just before the key
// (its rank among the warp's equal digits, or its local position when the
// counters start at local positions). cnt: this warp's 256 running counters.
template <bool FULL, int RB = kRadixBits>
__device__ __forceinline__ uint32_t rank_ballot(uint32_t* cnt, uint32_t d, bool valid) {
  // the running count first: its shared-memory round trip overlaps the votes
  // (the previous batch's update is already visible)
  const uint32_t old = valid ? cnt[d] : 0u;
  const uint32_t valid_mask = FULL ? 0xFFFFFFFFu : __ballot_sync(0xFFFFFFFFu, valid);
  const uint32_t peers = digit_peers<RB>(d, valid, valid_mask);
  const uint32_t below = __popc(peers & lanemask_lt());
  __syncwarp();
  if (valid && below == 0) cnt[d] = old + __popc(peers);
  __syncwarp();
  return old + below;
}

// The same for U batches with counting atomics. Every lane adds 1 to the low
// half of its digit's counter and its lane number to the high half; the old
// low half is then the key's rank if lanes sharing a digit were served in lane
// order. That order is not defined, so it is checked: after a warp barrier
// every lane reads its counter again, and the difference to its old value
// holds how many sharers were served from this lane on and the sum of their
// lane numbers. A lane that finds itself last, or followed by exactly one
// sharer in a higher lane, is in order; the digits of all other lanes (three
// or more sharers, or a pair served in reverse) are settled one by one with a
// vote on the digit and the lane numbers. Uniform 8-bit digits need that in
// one batch of thirteen when pairs are served in lane order, and in most
// batches otherwise. The batches' atomics and reads do not depend on the
// checks, so a chunk's shared-memory round trips overlap. The running counts
// stay below 2^16 (a tile's keys), so the halves do not mix.
//
// The ranking is bound by the L1 data pipe, which moves one wavefront a cycle
// and takes 3.4 for 32 random digits' counters. A batch costs two such
// accesses here, and no chain runs from one batch to the next; lane masks in
// shared memory (OR, read, clear) beside a counter's read and update cost five
// and a chain of round trips. The keys-only kernel went from 29.9 to 23.5
// wavefronts and from 78 to 66 instructions per 32 keys, and a 2^28 pass of
// the same 6144-key tiles from 0.944 to 0.838 ms (pairs 1.232 to 1.128).
// Settling every shared digit with votes, without the lane sums, took 1.04 ms.
template <bool FULL, int U>
__device__ __forceinline__ void rank_atomic(uint32_t* cnt, const uint32_t (&d)[U], const bool (&valid)[U],
                                            uint32_t (&rank)[U]) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t inc = (lane << 16) + 1u;
  uint32_t old[U], after[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    old[u] = (FULL || valid[u]) ? atomicAdd(cnt + d[u], inc) : 0u;
    __syncwarp();
    after[u] = (FULL || valid[u]) ? *const_cast<volatile uint32_t*>(cnt + d[u]) : inc;
    __syncwarp();
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    rank[u] = old[u] & 0xFFFFu;
    const uint32_t later = after[u] - old[u] - inc;  // sharers served after this lane: count, sum of lanes
    uint32_t open = __ballot_sync(0xFFFFFFFFu, (later & 0xFFFEu) != 0u || later - 1u < (lane << 16));
    while (open) {
      const uint32_t dl = __shfl_sync(0xFFFFFFFFu, d[u], 31 - __clz(open));
      const bool same = d[u] == dl && (FULL || valid[u]);
      const uint32_t peers = __ballot_sync(0xFFFFFFFFu, same);
      if (same) rank[u] = (after[u] & 0xFFFFu) - __popc(peers & lanemask_ge());
      open &= ~peers;
    }
  }
}

// Counting atomics with one digit set apart, for a place where many keys share
// it: their lanes would meet in one counter, one after another, but they are
// ranked by a single vote, with the digit's running position in a register
// (`position`, the same in every lane). The other digits then collide little
// (kRestShares says where that pays).
template <int U>
__device__ __forceinline__ void rank_dominant(uint32_t* cnt, uint32_t dominant, uint32_t& position,
                                              const uint32_t (&d)[U], uint32_t (&rank)[U]) {
  bool other[U];
#pragma unroll
  for (int u = 0; u < U; ++u) other[u] = d[u] != dominant;
  rank_atomic<false, U>(cnt, d, other, rank);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const uint32_t same = __ballot_sync(0xFFFFFFFFu, !other[u]);
    if (!other[u]) rank[u] = position + __popc(same & lanemask_lt());
    position += __popc(same);
  }
}

// Decoupled look-back of one digit in rounds: issue() reads the counters of
// up to W preceding tiles (one L2 round trip), consume() folds in what came
// back - stopping at a counter not yet published, which the next round reads
// again - until a G counter or the chain's first tile is reached, and then
// publishes this tile's (G, inclusive prefix). A round may stay in flight
// while the block does other work between issue() and consume().
//
// Beyond the paper's N/L/G protocol, a walk that has passed m preceding tiles
// but not yet reached a G counter publishes (A, m + 1, sum of the m + 1
// counts through this tile) in place of its L: a later walk that reads it adds
// the whole span's count and continues below it, instead of reading the m + 1
// tiles one by one. Each value a walk adds is the exact sum of a contiguous
// span ending where it reads, and the spans it adds are disjoint and
// adjacent, so the prefix is the paper's; a word only ever goes N -> L ->
// A... -> G, written by its own tile's walker.
template <int W>
struct Lookback {
  uint32_t s[W];       // counters of the round in flight
  uint32_t left;       // preceding tiles of the chain not yet accumulated
  uint32_t total;      // preceding tiles of the chain
  uint32_t exclusive;  // sum of the accumulated counters
  uint32_t own;        // this tile's count of the digit
  uint32_t* mine;      // this tile's counter of the digit (null: publish nothing)
  bool done;

  __device__ __forceinline__ void start(uint32_t tile, uint32_t chain_first) {
    left = tile - chain_first;
    total = left;
    exclusive = 0u;
    done = left == 0u;
  }
  // (G, exclusive + own): the inclusive prefix of the digit through this tile
  __device__ __forceinline__ void publish_global() {
    if (mine) st_relaxed_gpu(mine, (kFlagGlobal << kStatusShift) | (exclusive + own));
  }
  // (A, span, sum): this tile and the total - left predecessors passed so far
  __device__ __forceinline__ void publish_aggregate() {
    const uint32_t span = total - left + 1u;
    const uint32_t sum = exclusive + own;
    if (mine && span <= kAggMaxSpan && sum <= kAggValueMask)
      st_relaxed_gpu(mine, (kFlagAggregate << kStatusShift) | ((span - 1u) << kAggSpanShift) | sum);
  }
  // reads tiles chain_first + left - 1, chain_first + left - 2, ...
  __device__ __forceinline__ void issue(const uint32_t* status, uint32_t chain_first, int digit) {
#pragma unroll
    for (int w = 0; w < W; ++w)
      s[w] = (uint32_t)w < left ? ld_relaxed_gpu(status + (size_t)(chain_first + left - 1u - w) * kRadix + digit)
                                : (kFlagGlobal << kStatusShift);
  }
  __device__ __forceinline__ void consume() {
    const uint32_t left0 = left;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (done) break;
      const uint32_t flag = s[w] >> kStatusShift;
      if (flag == kFlagNotReady) break;  // read this tile again next round
      if (flag == kFlagAggregate) {
        // a whole span ending at this tile; the round's next rows lie inside it
        exclusive += s[w] & kAggValueMask;
        left -= ((s[w] >> kAggSpanShift) & (kAggMaxSpan - 1u)) + 1u;
        if (left == 0u) done = true;
        break;
      }
      exclusive += s[w] & kValueMask;
      --left;
      if (flag == kFlagGlobal || left == 0u) done = true;
    }
    if (done)
      publish_global();
    else if (left != left0)
      publish_aggregate();
  }
  // rounds until the walk ends, each waiting for its reads; a wait past the
  // poll limit records a timeout and still publishes (the successors' walks
  // then end instead of timing out one after another)
  __device__ __forceinline__ void finish(const PassArgs& a, uint32_t chain_first, int digit) {
    uint32_t spins = 0;
    while (!done) {
      issue(a.status, chain_first, digit);
      consume();
      if (done) break;
      if (++spins >= a.spin_limit) {
        atomicOr(a.error, kErrTimeout);
        break;
      }
      if ((spins & 255u) == 0 && (ld_relaxed_gpu(a.error) & kErrTimeout)) break;
    }
    if (!done) publish_global();
  }
};
// Counters read per look-back round. A walk is rarely long - a tile's
// predecessors have mostly published spans or prefixes - and every further
// counter of a round costs registers, issue slots and L2 reads in all 256
// walkers. 2^28 u32 pairs / keys only, us a sort, with 8, 6, 4, 3, 2 and 1
// counters (8, 6 and 3 in a build 1.5 / 3 % slower): 4432 / 3285, 4348 / 3223,
// 4212 / 3077, 4231 / 3121, 4104 / 3007, 4102 / 2998.
constexpr int kLookbackWindow = 1;
// Tiles ahead whose keys (and values) a starting block prefetches into L2
// (measured at 2^28 keys on GB300: 48, 144 and 384 tiles ahead all shorten a
// pass by about 1 %; the tile's own staging copy then waits less).
constexpr uint32_t kPrefetchTiles = 48;
// Keys a thread writes per step of the write-out. Nothing there has to stay in
// registers, and a body unrolled whole spends its time on instruction fetches
// (ncu: 12 % of the warps' stalls). us a sort, unrolled by 32 / 4 / 2 / 1: 2^28
// u32 pairs 4100 / 4064 / 4004 / 4112, keys only 2940 / 2907 / 2953 / 3128; 2^26
// u64 pairs 2964 / 2938 / 2945 / 3038; 2^26 pairs of 2-word keys 1344 / 1298 /
// 1275 / 1319; 3.3M u32 pairs 87.3 / 85.2 / 87.2 / 87.4.
constexpr int kWriteUnroll = 4;
// Ranking batches between two look-back rounds: about one L2 round trip of
// ranking work, so a round's reads have come back when it is consumed. With one
// counter a round, keys only rank fast enough for a round every 4 batches (2^28
// u32 keys 2949 us a sort, every 8 2998; 2^26 u64 keys 2338, 2361); pairs and
// the other ranking methods do not (2^28 u32 pairs 4100, 4102; 2^26 pairs of 3-
// word keys 1398, 1361, 5-word keys 1143, 1114).
__host__ __device__ constexpr int round_every(bool pairs, int rank) {
  return !pairs && rank == kRankAtomic ? 4 : 8;
}

template <int KBITS, bool PAIRS, int CFG, int RANK, int FLIP, int RB>
__device__ __forceinline__ void binning_tile(const PassArgs& a, unsigned char* smem, const TileCtx& c) {
  using C = BinningConfig<KBITS, PAIRS, CFG>;
  using K = typename C::K;
  constexpr int NT = C::NT, IPT = C::IPT, NW = C::NW;
  constexpr int R = 1 << RB;  // bins of this pass's digits (the tables keep rows of kRadix)
  static_assert(R <= kRadix && R <= NT, "one thread per digit");

  K* kt = reinterpret_cast<K*>(smem) + c.koff;
  uint32_t* vt = reinterpret_cast<uint32_t*>(smem + C::kbuf_bytes) + c.voff;
  // [NW][256] digit counts (turned into running local positions before the
  // ranking)
  uint32_t* wcnt = reinterpret_cast<uint32_t*>(smem + C::kbuf_bytes + C::vbuf_bytes);
  uint32_t* dstart = wcnt + NW * kRadix;       // [256] tile-local start of each digit's bin
  uint32_t* gbase = dstart + kRadix;           // [256] segment index of local position 0 of each bin
  uint32_t* misc = gbase + kRadix;             // [64] scan scratch
  uint64_t* mbar = reinterpret_cast<uint64_t*>(misc + 64);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int shift = a.shift;
  const uint32_t mask = a.mask;
  const uint32_t dxor = a.digit_xor;
  const uint32_t tile = c.tile;
  const uint32_t pads = (uint32_t)C::T - c.count;  // of a ragged tile

  // the next pass's status counters of this tile start at N
  if (a.status_clear && tid < kRadix)
    for (size_t row = tile; row < a.status_clear_rows; row += a.num_tiles) a.status_clear[row * kRadix + tid] = 0u;
  const uint32_t bin_offset = tid < R ? c.bin_offsets[tid] : 0u;
  uint32_t* status = a.status + (size_t)tile * kRadix;
  const bool publish = (int64_t)tile != a.fault_tile;
  const bool chain_head = tile == c.chain_first;

  // this warp's counts start at zero
  uint32_t* wc = wcnt + warp * kRadix;
#pragma unroll
  for (int i = lane; i < R; i += 32) wc[i] = 0u;

  if (c.bulk) {
    if (!mbar_wait_bounded(&mbar[0], 0, kBulkWaitLimit)) atomicOr(a.error, kErrTimeout);
  } else {
    __syncthreads();
  }
  if (pads) {
    // a ragged tile (the last of its chain) is filled up with keys of the
    // pass's highest digit: they sort behind every key of the tile, are left
    // out of the published counts, and the write-out ends before them
    const K ordered = (K)(mask ^ dxor) << shift;
    const K pad = (FLIP & 1) ? flip_from_ordered(ordered) : ordered;
    for (uint32_t i = c.count + tid; i < (uint32_t)C::T; i += NT) kt[i] = pad;
    __syncthreads();
  }
  __syncwarp();

  // keys of this thread: warp-striped, batch i of warp w covers tile positions
  // [w*IPT*32 + i*32, +32), so batch order and lane order are input order
  K key[IPT];
  const uint32_t wbase = (uint32_t)warp * IPT * 32 + lane;
#pragma unroll
  for (int i = 0; i < IPT; ++i) key[i] = load_transform<FLIP>(kt[wbase + i * 32]);

  // 3. early counts: each warp's digit histogram of its part of the tile
#pragma unroll
  for (int i = 0; i < IPT; ++i) atomicAdd(wc + digit_of(key[i], shift, mask, dxor), 1u);
  const uint32_t d0 = digit_of(load_transform<FLIP>(kt[0]), shift, mask, dxor);
  if (tid == 0) misc[NW] = 0u;  // set below by the digit that holds every key, if one does
  __syncthreads();

  // 4. tile digit counts: publish L now, and start the look-back (step 6),
  //    whose rounds then ride along the ranking; a tile whose keys share one
  //    digit skips ranking and reorganisation (homogeneous-tile short-circuit)
  uint32_t filled = 0;       // thread d < 256: keys of digit d in this tile, the pads included ...
  uint32_t digit_count = 0;  // ... and without
  if (tid < R) {
#pragma unroll
    for (int w = 0; w < NW; ++w) filled += wcnt[w * kRadix + tid];
    digit_count = filled - ((uint32_t)tid == mask ? pads : 0u);
    if (publish)
      st_relaxed_gpu(status + tid, ((chain_head ? kFlagGlobal : kFlagLocal) << kStatusShift) | digit_count);
  }
  const bool walker = tid < R && !chain_head;
  Lookback<kLookbackWindow> lb;
  bool issued = false;
  if (walker) {
    lb.start(tile, c.chain_first);
    lb.mine = publish ? status + tid : nullptr;
    lb.own = digit_count;
    lb.issue(a.status, c.chain_first, tid);
    issued = true;
  }
  // block scan of the counts (a warp scan, one barrier, the lower warps'
  // totals), which also tells whether every key has the same digit
  static_assert(NW < 64, "scan scratch");
  uint32_t incl = filled;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) misc[warp] = incl;
  // (without the pads: all-equal keys would otherwise rank one tile, the last,
  // in every pass; 4.0M u32 pairs 95 us a sort so, 70 as it is)
  if (digit_count == c.count) misc[NW] = 1u;
  __syncthreads();
  const bool homogeneous = misc[NW] != 0u;

  if (homogeneous) {
    if (PAIRS && c.bulk && !mbar_wait_bounded(&mbar[1], 0, kBulkWaitLimit)) atomicOr(a.error, kErrTimeout);
    if (tid < R) dstart[tid] = 0u;
  } else {
    // 5. tile-local bin starts, and each warp's counters set to where its
    //    first key of each digit goes
    uint32_t excl = incl - filled;
    for (int w = 0; w < NW; ++w)
      if (w < warp) excl += misc[w];
    if (tid < R) {
      uint32_t run = excl;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const uint32_t cw = wcnt[w * kRadix + tid];
        wcnt[w * kRadix + tid] = run;
        run += cw;
      }
      dstart[tid] = excl;
    }
    __syncthreads();

    // 6a. warp-level multi-split ranking straight to local positions: each
    //     key is written into its shared-memory bin as soon as it is ranked
    //     (every key is in registers since the barrier above); for pairs the
    //     positions are kept, two 16-bit positions per register
    uint32_t pos2[PAIRS ? IPT / 2 + 1 : 1];
    const uint32_t dominant = c.rank_word - 1u;
    uint32_t dominant_position = RANK == kRankDominant ? wc[dominant] : 0u;
    constexpr int U = RANK == kRankBallot ? 1 : rank_chunk(PAIRS, IPT);
    constexpr int kRound = round_every(PAIRS, RANK);
    static_assert(IPT % U == 0 && kRound % U == 0, "whole chunks of batches");
#pragma unroll
    for (int i0 = 0; i0 < IPT; i0 += U) {
      uint32_t d[U], p[U];
      const bool valid[U] = {};
#pragma unroll
      for (int u = 0; u < U; ++u) d[u] = digit_of(key[i0 + u], shift, mask, dxor);
      if constexpr (RANK == kRankBallot)
        p[0] = rank_ballot<true, RB>(wc, d[0], true);
      else if constexpr (RANK == kRankDominant)
        rank_dominant<U>(wc, dominant, dominant_position, d, p);
      else
        rank_atomic<true, U>(wc, d, valid, p);  // (every lane is valid)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u;
        kt[p[u]] = key[i];
        if (PAIRS) {
          if (i & 1)
            pos2[i / 2] |= p[u] << 16;
          else
            pos2[i / 2] = p[u];
        }
      }
      // a look-back round: fold in the last one's reads, send the next
      if ((i0 + U) % kRound == 0 && i0 + U < IPT && walker) {
        if (issued) lb.consume();
        issued = !lb.done;
        if (issued) lb.issue(a.status, c.chain_first, tid);
      }
    }
    if (PAIRS) {
      // values: read this thread's values, wait for every read, then scatter
      if (c.bulk && !mbar_wait_bounded(&mbar[1], 0, kBulkWaitLimit)) atomicOr(a.error, kErrTimeout);
      uint32_t val[IPT];
#pragma unroll
      for (int i = 0; i < IPT; ++i) val[i] = vt[wbase + i * 32];
      __syncthreads();
#pragma unroll
      for (int i = 0; i < IPT; ++i) vt[(i & 1) ? (pos2[i / 2] >> 16) : (pos2[i / 2] & 0xFFFFu)] = val[i];
    }
  }

  // 6b. the rest of the decoupled look-back: thread d walks back over the
  //     counters of digit d in the preceding tiles of the chain until it
  //     reaches a G counter; then it publishes (G, inclusive prefix)
  uint32_t exclusive = 0;
  if (walker) {
    if (issued) lb.consume();
    lb.finish(a, c.chain_first, tid);
    exclusive = lb.exclusive;
  }
  if (tid < R) {
    gbase[tid] = bin_offset + exclusive - dstart[tid];
    // the strip's last tile: where the next strip's keys of this digit start
    if (a.carry_out && tile == a.num_tiles - 1) a.carry_out[tid] = bin_offset + exclusive + digit_count;
  }
  __syncthreads();

  // 7. coalesced scatter of each local bin run to its global bin
  K* keys_out = static_cast<K*>(a.keys_out) + c.out_base;
  uint32_t* vals_out = PAIRS ? a.vals_out + c.out_base : nullptr;
  const uint32_t out_len = c.out_len;
  // (the range check is for a place made from counts that never came: a
  // look-back that ran past its limit)
  if (homogeneous) {
    const uint32_t g0 = gbase[d0];
    for_each_key<NT, kWriteUnroll>(tid, c.count, [&](uint32_t j) {
      const K k = store_transform<FLIP>(load_transform<FLIP>(kt[j]));
      const uint32_t g = g0 + j;
      if (g < out_len) {
        keys_out[g] = k;
        if (PAIRS) vals_out[g] = vt[j];
      }
    });
  } else {
    for_each_key<NT, kWriteUnroll>(tid, c.count, [&](uint32_t j) {
      const K k = kt[j];
      const uint32_t g = gbase[digit_of(k, shift, mask, dxor)] + j;
      if (g < out_len) {
        keys_out[g] = store_transform<FLIP>(k);
        if (PAIRS) vals_out[g] = vt[j];
      }
    });
  }
}

// Kernel front-end: tile id, where the tile sits, staging. SEG selects the
// segmented (batch) mode, where a.n is the length of the whole key array.
template <int KBITS, bool PAIRS, int CFG, int RANK, int FLIP, bool SEG, int RB = kRadixBits>
__global__ void __launch_bounds__(BinningConfig<KBITS, PAIRS, CFG>::NT, BinningConfig<KBITS, PAIRS, CFG>::MIN_BLOCKS)
    binning_kernel(PassArgs a) {
  using C = BinningConfig<KBITS, PAIRS, CFG>;
  using K = typename C::K;
  constexpr int NT = C::NT, T = C::T, NW = C::NW;
  constexpr uint32_t kKeysPer16B = 16 / sizeof(K);

  extern __shared__ __align__(128) unsigned char smem[];
  K* kbuf = reinterpret_cast<K*>(smem);
  uint32_t* vbuf = reinterpret_cast<uint32_t*>(smem + C::kbuf_bytes);
  uint32_t* whist = reinterpret_cast<uint32_t*>(smem + C::kbuf_bytes + C::vbuf_bytes);
  uint32_t* misc = whist + NW * kRadix + 2 * kRadix;
  uint64_t* mbar = reinterpret_cast<uint64_t*>(misc + 64);
  __shared__ TileCtx s_ctx;
  const int tid = threadIdx.x;

  // 1. tile id and where the tile sits. The launch may start while the one
  // before it ends (programmatic dependent launch): only the tile id, from a
  // counter that no other launch touches, is taken before the wait for it.
  uint32_t tile = 0;
  if (tid == 0) tile = atomicAdd(a.tile_counter, 1u);
  pdl_wait();
  if (tid == 0) {
    TileCtx c{};
    c.tile = tile;
    if (SEG) {
      // (the descriptor and the number of tiles are read together)
      const uint4 d = tile < a.num_tiles ? a.tile_desc[tile] : make_uint4(0, 0, 0, 0);
      if (tile < min(*a.total_tiles, a.num_tiles)) {
        c.chain_first = d.z;
        const uint32_t local = (tile - d.z) * (uint32_t)T;
        if (local < d.y) {
          c.start = d.x;
          c.count = min((uint32_t)T, d.y - local);
          c.out_base = d.x - local;
          c.out_len = d.y;
          c.bin_offsets = a.bin_offsets + (size_t)d.w * a.offsets_stride;
          if (RANK == kRankAdaptive && a.rank_words) c.rank_word = a.rank_words[(size_t)d.w * a.rank_stride];
        }
      }
    } else if (tile < a.num_tiles) {
      c.start = tile * (uint32_t)T;
      c.count = min((uint32_t)T, a.n - c.start);
      c.chain_first = 0;
      c.out_base = 0;
      c.out_len = a.out_total;
      c.bin_offsets = a.bin_offsets;
      if (RANK == kRankAdaptive && a.rank_words) c.rank_word = a.rank_words[0];
    }
    if (c.count > 0 && a.use_bulk) {
      // the 16-byte-aligned span covering the tile, if it stays in the array
      const uint32_t ks = c.start & ~(kKeysPer16B - 1u);
      const uint32_t vs = c.start & ~3u;
      const uint32_t koff = c.start - ks, voff = c.start - vs;
      const uint32_t kbytes = ((koff + c.count) * (uint32_t)sizeof(K) + 15u) & ~15u;
      const uint32_t vbytes = ((voff + c.count) * 4u + 15u) & ~15u;
      c.bulk = (uint64_t)ks * sizeof(K) + kbytes <= (uint64_t)a.n * sizeof(K) &&
               (!PAIRS || (uint64_t)vs * 4u + vbytes <= (uint64_t)a.n * 4u);
      if (c.bulk) {
        c.koff = koff;
        c.voff = voff;
        mbar_init(&mbar[0], 1);
        mbar_init(&mbar[1], 1);
        fence_mbar_init();
        mbar_arrive_expect_tx(&mbar[0], kbytes);
        bulk_copy_g2s(kbuf, static_cast<const K*>(a.keys_in) + ks, kbytes, &mbar[0]);
        if (PAIRS) {
          mbar_arrive_expect_tx(&mbar[1], vbytes);
          bulk_copy_g2s(vbuf, a.vals_in + vs, vbytes, &mbar[1]);
        }
      }
    }
    // the tile kPrefetchTiles ahead starts well within one block lifetime:
    // bring it into L2 now, so its staging copy reads L2 instead of DRAM
    const uint32_t ahead = tile + kPrefetchTiles;
    if (SEG && a.use_bulk && c.count > 0 && ahead < min(*a.total_tiles, a.num_tiles)) {
      // whole 16-byte words from the one holding the tile's first key
      const uint4 d = a.tile_desc[ahead];
      const uint32_t end = d.x + min((uint32_t)T, d.y - (ahead - d.z) * (uint32_t)T);
      const uint32_t ks = d.x & ~(kKeysPer16B - 1u), vs = d.x & ~3u;
      const uint32_t kbytes = ((end - ks) * (uint32_t)sizeof(K)) & ~15u, vbytes = ((end - vs) * 4u) & ~15u;
      if (kbytes) bulk_prefetch_l2(static_cast<const K*>(a.keys_in) + ks, kbytes);
      if (PAIRS && vbytes) bulk_prefetch_l2(a.vals_in + vs, vbytes);
    }
    if (!SEG && a.use_bulk && ahead < a.num_tiles && (uint64_t)(ahead + 1) * T <= a.n) {
      const size_t first = (size_t)ahead * T;
      bulk_prefetch_l2(static_cast<const K*>(a.keys_in) + first, (uint32_t)(T * sizeof(K)));
      if (PAIRS) bulk_prefetch_l2(a.vals_in + first, (uint32_t)T * 4u);
    }
    s_ctx = c;
  }
  __syncthreads();
  const TileCtx c = s_ctx;
  pdl_launch_dependents();  // the next launch's blocks may take the slots that this one's last blocks leave
  if (c.count == 0) return;  // no tile left (or the workspace's counters were not reset)

  // 2. plain staging when the bulk copy does not apply
  if (!c.bulk) {
    const K* keys_in = static_cast<const K*>(a.keys_in) + c.start;
    for (uint32_t i = tid; i < c.count; i += NT) kbuf[i] = keys_in[i];
    if (PAIRS)
      for (uint32_t i = tid; i < c.count; i += NT) vbuf[i] = a.vals_in[c.start + i];
  }

  // adaptive ranking: one uniform branch per tile between whole bodies
  constexpr int R0 = RANK == kRankAdaptive ? kRankAtomic : RANK;
  if (RANK == kRankAdaptive && c.rank_word == kRankWordBallots)
    binning_tile<KBITS, PAIRS, CFG, kRankBallot, FLIP, RB>(a, smem, c);
  else if (RANK == kRankAdaptive && c.rank_word != 0u)
    binning_tile<KBITS, PAIRS, CFG, kRankDominant, FLIP, RB>(a, smem, c);
  else
    binning_tile<KBITS, PAIRS, CFG, R0, FLIP, RB>(a, smem, c);
}

}  // namespace onesweep
