// One block's part of a sort whose keys stay on the chip (os_small.cu, and the
// short segments of a batch in os_batch.cu): a stable digit-binning pass of up
// to NT * IPT keys held in registers, into digit order in shared memory.
#pragma once

#include "os_binning.cuh"

namespace onesweep {

// SPREAD: the tile's keys are spread evenly over the block's threads (ceil(n /
// NT) each) rather than filling the first warps with IPT a thread, so that a
// tile takes time by its length; for tiles that are whole sorts. APART (whole
// sorts of keys of any kind): a digit that many keys of a warp share is ranked
// apart, and places that all keys share are passed over.
template <int KBITS, bool PAIRS, int NT_, int IPT_, bool SPREAD = false, bool APART = false>
struct SmallTile {
  using K = typename KeyWord<KBITS>::type;
  static constexpr uint32_t kDominantLanes = 6;  // lanes of the first batch that make a digit dominant
  static constexpr int NT = NT_, IPT = IPT_, NW = NT / 32;
  static constexpr int T = NT * IPT;        // keys per tile
  static constexpr int Q = NT / kRadix;     // parts of 8 warps, whose counts of a digit one thread adds up
  static constexpr int WPP = NW / Q;
  // with few keys a thread, the first pass's values are loaded beside its keys:
  // both come from DRAM, and there are registers for both
  static constexpr bool kValuesFirst = IPT <= 4;
  static_assert(NT % kRadix == 0 && Q <= 4 && T < (1 << 16), "tile shape (the counters' halves are 16 bits wide)");
  // shared memory (bytes)
  static constexpr size_t kbuf = 0;                                   // the tile in digit order
  static constexpr size_t vbuf = kbuf + (size_t)T * sizeof(K);
  static constexpr size_t wcnt = vbuf + (PAIRS ? (size_t)T * 4 : 0);  // [NW][256] running counts of each warp
  static constexpr size_t psum = wcnt + (size_t)NW * kRadix * 4;      // [Q][256] digit counts of a part
  static constexpr size_t gsum = psum + (size_t)Q * kRadix * 4;       // [Q][8] ... of 32 digits
  static constexpr size_t dsum = gsum + 32 * 4;  // APART: [NW] bits that differ in a warp, [NW] its first key
  static constexpr size_t smem_bytes = dsum + (APART ? 2 * NW * sizeof(K) : 0);

  K key[IPT];
  uint32_t val[PAIRS ? IPT : 1];
  uint32_t count;   // keys in the tile
  uint32_t wbase;   // tile position of this thread's first key
  int ipt;          // keys of a thread (SPREAD)
  uint32_t total;   // threads 0..255, after bin(): the tile's count of digit tid ...
  uint32_t excl;    // ... and of the digits below it

  // This thread's keys: warp-striped, batch i of warp w covers positions
  // [w*keys()*32 + i*32, +32), so batch order and lane order are tile order.
  __device__ __forceinline__ void init(unsigned char* smem, uint32_t n) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    count = n;
    ipt = SPREAD ? (int)((n + NT - 1) / NT) : IPT;
    wbase = (uint32_t)warp * keys() * 32 + lane;
    clear_counts(smem);
  }
  __device__ __forceinline__ int keys() const { return SPREAD ? ipt : IPT; }
  __device__ __forceinline__ bool valid(int i) const {
    return (!SPREAD || i < ipt) && wbase + i * 32 < count;
  }
  __device__ __forceinline__ void clear_counts(unsigned char* smem) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint4* row = reinterpret_cast<uint4*>(smem + wcnt) + warp * (kRadix / 4);
    row[lane] = make_uint4(0, 0, 0, 0);
    row[lane + 32] = make_uint4(0, 0, 0, 0);
  }
  // kL2: read past L1 (which may hold what the buffer held two passes ago)
  template <bool kL2 = false>
  __device__ __forceinline__ void load_keys(const K* keys, int flip = 0) {
#pragma unroll
    for (int i = 0; i < IPT; ++i)
      key[i] = !valid(i) ? K(0) : kL2 ? __ldcg(keys + wbase + i * 32) : keys[wbase + i * 32];
    if (flip) {
#pragma unroll
      for (int i = 0; i < IPT; ++i) key[i] = flip_to_ordered(key[i]);
    }
  }
  template <bool kL2 = false>
  __device__ __forceinline__ void load_values(const uint32_t* vals) {
    if constexpr (PAIRS) {
#pragma unroll
      for (int i = 0; i < IPT; ++i)
        val[i] = !valid(i) ? 0u : kL2 ? __ldcg(vals + wbase + i * 32) : vals[wbase + i * 32];
    }
  }

  // One binning pass: on return kbuf (and vbuf) hold the tile in stable digit
  // order, visible to the block, and total / excl are set. values() loads
  // this thread's values: it is called once the keys are ranked, so the values
  // take no registers before and their way here is covered by the scan.
  // publish(total) is called by threads 0..255 as soon as the counts are known.
  //
  // Four barriers; what bounds a tile of a few thousand keys is their latency
  // and that of the shared-memory round trips between them. So the scan over
  // 256 digits takes no barrier of its own: each warp adds the sums of the
  // lower groups of 32 digits itself (one load, one warp reduction).
  // note (APART): each warp leaves the bits in which its keys differ, for
  // differing_bits().
  template <typename Values, typename Publish>
  __device__ __forceinline__ void bin(unsigned char* smem, int shift, uint32_t mask, uint32_t dxor, Values values,
                                      Publish publish, bool note = false) {
    constexpr int U = IPT % 4 == 0 ? 4 : 2;
    K* kb = reinterpret_cast<K*>(smem + kbuf);
    uint32_t* vb = reinterpret_cast<uint32_t*>(smem + vbuf);
    uint32_t* wcnt_all = reinterpret_cast<uint32_t*>(smem + wcnt);
    uint32_t* ps = reinterpret_cast<uint32_t*>(smem + psum);
    uint32_t* gs = reinterpret_cast<uint32_t*>(smem + gsum);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t* wc = wcnt_all + warp * kRadix;

    // rank each key among its warp's equal digits. A warp whose keys share one
    // digit has nothing to rank. APART: a digit that many of the warp's first
    // keys share (the most frequent of four sampled lanes') is ranked by votes,
    // for its atomics would all meet in one counter
    uint32_t rank2[IPT / 2];  // two 16-bit ranks to a register
    uint32_t d0;
    bool differ = false;
    if constexpr (APART) {
      // whole keys are compared, at one operation each, and only as many as
      // there are: by digits, all IPT of them, 2048 segments of a median of 1500
      // u32 pairs took 140 us and take 130 (64-bit keys cost two operations a
      // compare, so theirs go by digits after the first pass: 274 / 271)
      const K first = __shfl_sync(0xFFFFFFFFu, key[0], 0);
      d0 = digit_of(first, shift, mask, dxor);
      if (KBITS == 32 || note) {
        K bits = 0;
#pragma unroll
        for (int i0 = 0; i0 < IPT; i0 += U) {
          if (SPREAD && i0 >= ipt) break;
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (valid(i0 + u)) bits |= key[i0 + u] ^ first;
        }
        differ = ((uint32_t)(bits >> shift) & mask) != 0u;
        if (note) {
          bits = warp_or(bits);
          if (lane == 0) {
            reinterpret_cast<K*>(smem + dsum)[warp] = bits;
            reinterpret_cast<K*>(smem + dsum)[NW + warp] = first;
          }
        }
      } else {
#pragma unroll
        for (int i0 = 0; i0 < IPT; i0 += U) {
          if (SPREAD && i0 >= ipt) break;
#pragma unroll
          for (int u = 0; u < U; ++u) differ |= valid(i0 + u) && digit_of(key[i0 + u], shift, mask, dxor) != d0;
        }
      }
    } else {
      d0 = __shfl_sync(0xFFFFFFFFu, digit_of(key[0], shift, mask, dxor), 0);
#pragma unroll
      for (int i = 0; i < IPT; ++i) differ |= valid(i) && digit_of(key[i], shift, mask, dxor) != d0;
    }
    if (__any_sync(0xFFFFFFFFu, differ)) {
      uint32_t dominant = kRadix, most = kDominantLanes - 1, position = 0;
      if constexpr (APART) {
        const uint32_t mine = valid(0) ? digit_of(key[0], shift, mask, dxor) : kRadix;
#pragma unroll
        for (int l = 0; l < 32; l += 8) {
          const uint32_t dl = __shfl_sync(0xFFFFFFFFu, mine, l);
          const uint32_t lanes = __popc(__ballot_sync(0xFFFFFFFFu, mine == dl));
          if (dl < kRadix && lanes > most) {
            most = lanes;
            dominant = dl;
          }
        }
      }
#pragma unroll
      for (int i0 = 0; i0 < IPT; i0 += U) {
        if (SPREAD && i0 >= ipt) break;
        uint32_t d[U], r[U];
        bool v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          d[u] = digit_of(key[i0 + u], shift, mask, dxor);
          v[u] = valid(i0 + u) && (!APART || d[u] != dominant);
        }
        rank_atomic<false, U>(wc, d, v, r);
        if (APART && dominant < kRadix) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const bool same = valid(i0 + u) && d[u] == dominant;
            const uint32_t lanes = __ballot_sync(0xFFFFFFFFu, same);
            if (same) r[u] = position + __popc(lanes & lanemask_lt());
            position += __popc(lanes);
          }
        }
#pragma unroll
        for (int u = 0; u < U; u += 2) rank2[(i0 + u) / 2] = r[u] | r[u + 1] << 16;
      }
      if (APART && dominant < kRadix && lane == 0) wc[dominant] = position;
    } else {
#pragma unroll
      for (int i = 0; i < IPT; i += 2) rank2[i / 2] = (i * 32 + lane) | ((i + 1) * 32 + lane) << 16;
      const uint32_t first = (uint32_t)warp * keys() * 32;
      if (lane == 0 && count > first) wc[d0] = min((uint32_t)keys() * 32, count - first);
    }
    values();
    __syncthreads();

    // thread (q, d): digit d's counts in the 8 warps of part q
    const int d = tid & (kRadix - 1), q = tid >> kRadixBits;
    uint32_t part[WPP], sum = 0;
#pragma unroll
    for (int w = 0; w < WPP; ++w) {
      part[w] = wcnt_all[(q * WPP + w) * kRadix + d] & 0xFFFFu;  // (the high halves hold lane sums)
      sum += part[w];
    }
    if (Q > 1) ps[tid] = sum;
    const uint32_t group = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0) gs[warp] = group;  // warp = q * 8 + d / 32
    __syncthreads();
    uint32_t all = sum, lower = 0;  // digit d in the whole tile, and in the parts below q
    if (Q > 1) {
      all = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const uint32_t p = ps[i * kRadix + d];
        all += p;
        if (i < q) lower += p;
      }
    }
    if (tid < kRadix) publish(all);
    const uint32_t below = __reduce_add_sync(0xFFFFFFFFu, lane < NW && (lane & 7) < (warp & 7) ? gs[lane] : 0u);
    uint32_t incl = all;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    total = all;
    excl = below + incl - all;
    uint32_t run = excl + lower;
#pragma unroll
    for (int w = 0; w < WPP; ++w) {
      wcnt_all[(q * WPP + w) * kRadix + d] = run;
      run += part[w];
    }
    __syncthreads();

#pragma unroll
    for (int i = 0; i < IPT; ++i) {
      if (valid(i)) {
        const uint32_t rank = (i & 1) ? rank2[i / 2] >> 16 : rank2[i / 2] & 0xFFFFu;
        const uint32_t p = wc[digit_of(key[i], shift, mask, dxor)] + rank;
        kb[p] = key[i];
        if (PAIRS) vb[p] = val[i];
      }
    }
    __syncwarp();
    clear_counts(smem);
    __syncthreads();
  }
  // The bits in which the tile's keys differ, as its warps noted them in a pass.
  __device__ __forceinline__ K differing_bits(const unsigned char* smem) const {
    const uint32_t lane = threadIdx.x & 31;
    const K* noted = reinterpret_cast<const K*>(smem + dsum);
    return warp_or(lane < NW && lane * keys() * 32 < count ? noted[lane] | (noted[NW + lane] ^ noted[NW]) : K(0));
  }
  __device__ __forceinline__ static K warp_or(K x) {
    if constexpr (sizeof(K) == 4) return __reduce_or_sync(0xFFFFFFFFu, x);
    return (K)__reduce_or_sync(0xFFFFFFFFu, (uint32_t)x) |
           (K)((uint64_t)__reduce_or_sync(0xFFFFFFFFu, (uint32_t)((uint64_t)x >> 32)) << 32);
  }
  // A whole sort of the tile: p passes, then the store. APART: after the first
  // pass, a place whose digit all keys share would leave them as they are and is
  // passed over (2048 segments of a median of 1500 u32 pairs: keys below 65536
  // 123 -> 90 us, all equal 105 -> 64, uniform words 130 / 130; the first pass
  // is not worth a barrier of its own: 145).
  __device__ __forceinline__ void sort(unsigned char* smem, const K* keys_in, const uint32_t* vals_in, K* keys_out,
                                       uint32_t* vals_out, int places, int begin_bit, int end_bit, uint32_t top_xor,
                                       uint32_t descending, int flip) {
    const K* kb = reinterpret_cast<const K*>(smem + kbuf);
    const uint32_t* vb = reinterpret_cast<const uint32_t*>(smem + vbuf);
    load_keys(keys_in, flip);
    if (kValuesFirst) load_values(vals_in);
    K differ = ~K(0);
    for (int pass = 0; pass < places; ++pass) {
      const int shift = begin_bit + kRadixBits * pass;
      const uint32_t mask = (1u << min(kRadixBits, end_bit - shift)) - 1u;
      if (pass > 0) {
        if (APART && ((uint32_t)(differ >> shift) & mask) == 0u) continue;
        load_keys(kb);
      }
      bin(
          smem, shift, mask, (pass == places - 1 ? top_xor : 0u) ^ (descending ? mask : 0u),
          [&] {
            if (pass > 0)
              load_values(vb);
            else if (!kValuesFirst)
              load_values(vals_in);
          },
          [](uint32_t) {}, pass == 0);
      if (APART && pass == 0) differ = differing_bits(smem);
    }
    for (uint32_t j = threadIdx.x; j < count; j += NT) {
      const K k = kb[j];
      keys_out[j] = flip ? flip_from_ordered(k) : k;
      if (PAIRS) vals_out[j] = vb[j];
    }
  }
};

}  // namespace onesweep
