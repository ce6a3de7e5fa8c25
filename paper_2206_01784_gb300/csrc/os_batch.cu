// Segmented (batched) sort: many independent arrays sorted together
// (os_sort_batch). Each segment is its own Onesweep sort (arXiv 2206.01784,
// Section 3): its own digit histograms and bin offsets, its own look-back
// chain. What this file adds around the binning kernel:
//
//  * plan: one block reads the segment boundaries on the device and lays out
//    the work. Segments of up to one block's capacity are listed by class for
//    the one-block sorts; each longer ("large") segment gets a row of its own,
//    consecutive tile ids (its look-back chain) and histogram work items.
//    Nothing is read back to the host, so a batch can be captured in a CUDA
//    graph;
//  * one-block sorts: blocks take the listed segments one after another and
//    sort each on the chip (SmallTile): one global read and one write;
//  * histograms of the large segments: work items of up to kHistChunk keys
//    count the digits of every place into their segment's histograms; the item
//    that finishes a segment last takes the exclusive sums (the segment's bin
//    offsets), as the single-array histogram kernel does for the whole array.
//    They also write a descriptor per tile for the binning passes.
//
// Grids and workspaces are bounded by what n keys can make: a large segment
// is longer than class 0's capacity, so there are at most n / (capacity + 1) of
// them whatever the number of segments.
#include "os_small.cuh"

namespace onesweep {

int device_sm_count();
int ws_grid(uint32_t num_tiles);  // min(num_tiles, SMs of the current device)

namespace {

constexpr int kPlanThreads = 1024;
constexpr int kSegHistThreads = 1024;
constexpr int kSegHistVec = 4;  // 16-byte loads in flight per thread per step of the segment histogram

// Classes of the one-block sorts: a block's threads, keys a thread, and how many
// blocks fit an SM (64 registers a thread). The smaller a class's blocks, the
// more of them share an SM and cover one another's barriers; the last class
// holds the longest segment one block can (by shared memory).
struct BatchClass {
  int threads, keys_per_thread, blocks_per_sm;
  constexpr uint32_t capacity() const { return (uint32_t)(threads * keys_per_thread); }
};
constexpr BatchClass kClass32[kBatchClasses] = {{256, 16, 4}, {512, 16, 2}, {1024, 16, 1}};
constexpr BatchClass kClass64[kBatchClasses] = {{256, 8, 4}, {512, 8, 2}, {1024, 8, 1}};

// Exclusive prefix sum of a pair of words over the block.
__device__ __forceinline__ uint2 block_exclusive_sum2(uint2 v, uint2* tmp, uint2* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint2 x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y0 = __shfl_up_sync(0xFFFFFFFFu, x.x, o), y1 = __shfl_up_sync(0xFFFFFFFFu, x.y, o);
    if (lane >= o) {
      x.x += y0;
      x.y += y1;
    }
  }
  if (lane == 31) tmp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const uint2 w = tmp[lane];
    uint2 s = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y0 = __shfl_up_sync(0xFFFFFFFFu, s.x, o), y1 = __shfl_up_sync(0xFFFFFFFFu, s.y, o);
      if (lane >= o) {
        s.x += y0;
        s.y += y1;
      }
    }
    tmp[lane] = make_uint2(s.x - w.x, s.y - w.y);
    if (lane == 31) tmp[32] = s;
  }
  __syncthreads();
  *total = tmp[32];
  return make_uint2(tmp[warp].x + x.x - v.x, tmp[warp].y + x.y - v.y);
}

__global__ void __launch_bounds__(kPlanThreads) batch_plan_kernel(BatchArgs b) {
  __shared__ uint2 tmp[2][33];
  const int tid = threadIdx.x;
  // invalid segments, and the longest one
  bool bad = false, longest = false;
  for (uint32_t s = tid; s < b.num_segments; s += kPlanThreads) {
    const uint64_t lo = b.seg_offsets[s], hi = b.seg_offsets[s + 1];
    bad |= hi < lo || hi > b.n_total || hi - lo >= (1ull << 30);
    longest |= hi - lo > b.class_max[kBatchClasses - 1];
  }
  bad = __syncthreads_or(bad);
  // when there are binning passes to run, the segments above class 0 join them:
  // they add little to passes whose time is mostly fixed, while the longest of
  // them takes tens of microseconds in one block
  const uint32_t small_max = __syncthreads_or(longest) ? b.class_max[0] : b.class_max[kBatchClasses - 1];
  uint32_t tiles = 0, items = 0, large = 0, listed[kBatchClasses] = {0, 0, 0};
  for (uint32_t base = 0; base < b.num_segments && !bad; base += kPlanThreads) {
    const uint32_t s = base + tid;
    uint32_t nt = 0, nh = 0, start = 0, len = 0;
    if (s < b.num_segments) {
      start = (uint32_t)b.seg_offsets[s];
      len = (uint32_t)(b.seg_offsets[s + 1] - b.seg_offsets[s]);
      if (len > small_max) {
        nt = (len + b.tile_keys - 1) / b.tile_keys;
        nh = (len + b.hist_chunk - 1) / b.hist_chunk;
      }
    }
    const int cls = len == 0 || nt ? -1 : len <= b.class_max[0] ? 0 : len <= b.class_max[1] ? 1 : 2;
    // exclusive sums of tiles, items, and (at most 1024 a step, 16 bits each)
    // of large segments and of each class
    uint2 work_total, low_total;
    const uint2 work = block_exclusive_sum2(make_uint2(nt, nh), tmp[0], &work_total);
    const uint2 rank = block_exclusive_sum2(
        make_uint2((nt ? 1u : 0u) | (cls == 0 ? 1u << 16 : 0u), (cls == 1 ? 1u : 0u) | (cls == 2 ? 1u << 16 : 0u)),
        tmp[1], &low_total);
    if (nt) {
      const uint32_t li = large + (rank.x & 0xFFFFu), tb = tiles + work.x, hb = items + work.y;
      if (li < b.max_large && (uint64_t)hb + nh <= b.max_items) {
        b.large_range[li] = make_uint2(start, len);
        b.tile_base[li] = tb;
        b.hist_base[li] = hb;
        for (uint32_t h = 0; h < nh; ++h) b.hist_large[hb + h] = li;
      }
    }
    if (cls == 0) b.class_list[listed[0] + (rank.x >> 16)] = s;
    if (cls == 1) b.class_list[b.num_segments + listed[1] + (rank.y & 0xFFFFu)] = s;
    if (cls == 2) b.class_list[2 * (size_t)b.num_segments + listed[2] + (rank.y >> 16)] = s;
    tiles += work_total.x;
    items += work_total.y;
    large += low_total.x & 0xFFFFu;
    listed[0] += low_total.x >> 16;
    listed[1] += low_total.y & 0xFFFFu;
    listed[2] += low_total.y >> 16;
    __syncthreads();
  }
  if (tid == 0) {
    bad = bad || tiles > b.max_tiles || items > b.max_items || large > b.max_large;
    if (!bad) {
      b.tile_base[large] = tiles;
      b.hist_base[large] = items;
    }
    b.totals[0] = bad ? 0u : tiles;
    b.totals[1] = bad ? 0u : items;
#pragma unroll
    for (int c = 0; c < kBatchClasses; ++c) b.class_count[c] = bad ? 0u : listed[c];
    if (bad) atomicOr(b.error, kErrBadSegments);
  }
}

// Per-segment digit histograms of every place (Section 3, "Upfront histogram
// kernel", per segment). One persistent 1024-thread block per SM takes a
// contiguous range of the batch's work items (chunks of hist_chunk keys, a
// segment's items consecutive), so a block mostly meets whole runs of one
// segment's items: it counts them into block-private histograms and flushes
// them to the segment's global histograms with global atomics once per run.
// As in the single-array histogram kernel, each lane owns its own copy of the
// counters, laid out in its own shared-memory bank (counter e of copy c at
// word e * C + c), so every warp-wide atomic is one conflict-free wavefront
// and skewed keys cost no more than uniform ones; keys are read with 128-bit
// streaming loads (the unaligned head and tail of a chunk one key per
// thread). The flush that completes a segment's items takes the segment's
// exclusive sums (its bin offsets) and ranking words.
template <int KBITS>
struct BatchHistLayout {
  static constexpr int P = KBITS / 8;                 // places of 8-bit digits
  static constexpr int C = KBITS == 32 ? 32 : 16;     // counter copies (lanes per copy: 32 / C)
  static constexpr size_t smem_bytes = (size_t)P * kRadix * C * 4;  // 128 KiB
};

template <int KBITS>
__global__ void __launch_bounds__(kSegHistThreads, 1) batch_histogram_kernel(BatchArgs b) {
  using K = typename KeyWord<KBITS>::type;
  using BL = BatchHistLayout<KBITS>;
  constexpr int P = BL::P, C = BL::C;
  constexpr int PER_VEC = 16 / (int)sizeof(K);  // keys per 16-byte vector
  extern __shared__ __align__(16) uint32_t sh[];  // [P * 256][C]
  __shared__ uint32_t s_last;
  const int tid = threadIdx.x, lane = tid & 31;
  pdl_launch_dependents();

  {
    uint4* s4 = reinterpret_cast<uint4*>(sh);
    for (int i = tid; i < P * kRadix * C / 4; i += kSegHistThreads) s4[i] = make_uint4(0, 0, 0, 0);
  }
  // zero the first pass's status rows on the way (grid-stride, 16-byte stores)
  {
    uint4* c = reinterpret_cast<uint4*>(b.clear);
    const uint64_t nv = (uint64_t)__ldcg(b.totals) * (kRadix / 4);
    for (uint64_t i = (uint64_t)blockIdx.x * kSegHistThreads + tid; i < nv; i += (uint64_t)gridDim.x * kSegHistThreads)
      c[i] = make_uint4(0, 0, 0, 0);
  }
  __syncthreads();

  const int p = b.num_places;
  const uint32_t last_mask = (1u << (b.end_bit - (b.begin_bit + 8 * (p - 1)))) - 1u;
  const bool flip = b.flip != 0;
  uint32_t* mine = sh + (lane % C);
  auto count_key = [&](K k) {
    const K o = flip ? flip_to_ordered(k) : k;
#pragma unroll
    for (int pl = 0; pl < P; ++pl) {
      if (pl < p) {
        const uint32_t d =
            digit_of(o, b.begin_bit + 8 * pl, pl == p - 1 ? last_mask : 0xFFu, pl == p - 1 ? b.top_xor : 0u);
        atomicAdd(mine + (pl * kRadix + d) * C, 1u);
      }
    }
  };

  // add this block's copies of every counter into the segment's histograms
  // (each lane starts at a different copy, so a warp's reads and the zeroing
  // stores hit distinct banks); the flush that completes the segment's work
  // items takes its exclusive sums
  auto flush = [&](uint32_t seg, uint32_t nitems) {  // seg: row of a large segment
    __syncthreads();
    uint32_t* gh = b.seg_hist + (size_t)seg * p * kRadix;
    for (int e = tid; e < p * kRadix; e += kSegHistThreads) {
      uint32_t sum = 0;
#pragma unroll 8
      for (int c = 0; c < C; ++c) {
        uint32_t* w = sh + e * C + ((c + lane) % C);
        sum += *w;
        *w = 0u;
      }
      if (sum) atomicAdd(gh + e, sum);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      const uint32_t items = __ldcg(b.hist_base + seg + 1) - __ldcg(b.hist_base + seg);
      s_last = (atomicAdd(b.seg_done + seg, nitems) + nitems == items) ? 1u : 0u;
    }
    __syncthreads();
    if (s_last) {
      __threadfence();
      const uint32_t len = __ldcg(b.large_range + seg).y;
      uint32_t* go = b.seg_bin_offsets + (size_t)seg * p * kRadix;
      if (const int pl = tid >> 5; pl < p) {
        const uint32_t word = finish_place(gh + pl * kRadix, go + pl * kRadix, pl == p - 1 ? last_mask : 0xFFu,
                                           b.descending, len);
        if (lane == 0) b.seg_rank_words[(size_t)seg * p + pl] = word;
      }
    }
    __syncthreads();
  };

  // this block's contiguous range of work items
  // (the plan's words are read from L2, as in the class sorts)
  const uint32_t total_items = __ldcg(b.totals + 1);
  const uint32_t per_block = (total_items + gridDim.x - 1) / gridDim.x;
  const uint32_t it0 = min(blockIdx.x * per_block, total_items);
  const uint32_t it1 = min(it0 + per_block, total_items);
  uint32_t cur = 0xFFFFFFFFu, run = 0;
  for (uint32_t item = it0; item < it1; ++item) {
    const uint32_t seg = __ldcg(b.hist_large + item);
    if (seg != cur) {
      if (run) flush(cur, run);
      cur = seg;
      run = 0;
    }
    const uint2 range = __ldcg(b.large_range + seg);
    const uint32_t s0 = range.x, len = range.y;
    const uint32_t lo = (item - __ldcg(b.hist_base + seg)) * b.hist_chunk;
    const uint32_t cnt = min(b.hist_chunk, len - lo);
    // descriptors of the tiles that start in this chunk
    const uint32_t chain = __ldcg(b.tile_base + seg);
    for (uint32_t t = (lo + b.tile_keys - 1) / b.tile_keys + tid; t * b.tile_keys < lo + cnt; t += kSegHistThreads)
      b.tile_desc[chain + t] = make_uint4(s0 + t * b.tile_keys, len, chain, seg);
    const K* keys = static_cast<const K*>(b.keys_in) + s0 + lo;
    // 16-byte vectors between an unaligned head and a tail of fewer than PER_VEC keys
    const uintptr_t addr = reinterpret_cast<uintptr_t>(keys);
    uint32_t head = (uint32_t)(((16u - (addr & 15u)) & 15u) / sizeof(K));
    if (head > cnt) head = cnt;
    const uint32_t nvec = (cnt - head) / PER_VEC;
    const uint32_t tail_start = head + nvec * PER_VEC;
    const uint4* vkeys = reinterpret_cast<const uint4*>(keys + head);
    for (uint32_t base = 0; base < nvec; base += kSegHistThreads * kSegHistVec) {
      uint4 v[kSegHistVec];
#pragma unroll
      for (int u = 0; u < kSegHistVec; ++u) {
        const uint32_t idx = base + u * kSegHistThreads + tid;
        v[u] = idx < nvec ? __ldcs(vkeys + idx) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < kSegHistVec; ++u) {
        if (base + u * kSegHistThreads + tid < nvec) {
          const K* kk = reinterpret_cast<const K*>(&v[u]);
#pragma unroll
          for (int j = 0; j < PER_VEC; ++j) count_key(kk[j]);
        }
      }
    }
    const uint32_t extra = head + (cnt - tail_start);
    if ((uint32_t)tid < extra) count_key(keys[(uint32_t)tid < head ? tid : tail_start + (tid - head)]);
    ++run;
  }
  if (run) flush(cur, run);
  if (blockIdx.x == 0) pdl_wait();  // the class sorts before this kernel have ended when it ends
}

// One-block sorts of one class's segments: resident blocks take them one after
// another. The classes and the histogram kernel after them work on different
// segments, so each is launched to start when the one before has started
// (programmatic dependent launch) and fills the SMs that it leaves idle. Block 0
// waits for the kernel before to complete before it ends itself: what the
// stream runs after the last of them then follows them all.
template <int KBITS, bool PAIRS, int CLS, bool WIDE>
struct ClassTile {
  static constexpr BatchClass kShape = KBITS == 32 ? kClass32[CLS] : kClass64[CLS];
  static constexpr BatchClass kClass = WIDE ? BatchClass{1024, (int)kShape.capacity() / 1024, 1} : kShape;
  using Tile = SmallTile<KBITS, PAIRS, kClass.threads, kClass.keys_per_thread, true, true>;
  static_assert(kClass.blocks_per_sm * (Tile::smem_bytes + 1024) <= 228 * 1024, "blocks of a class on an SM");
};

template <int KBITS, bool PAIRS, int CLS, bool WIDE>
__global__ void __launch_bounds__(ClassTile<KBITS, PAIRS, CLS, WIDE>::kClass.threads,
                                  ClassTile<KBITS, PAIRS, CLS, WIDE>::kClass.blocks_per_sm)
    batch_class_sort_kernel(BatchArgs b) {
  using Tile = typename ClassTile<KBITS, PAIRS, CLS, WIDE>::Tile;
  using K = typename Tile::K;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ uint32_t s_item;
  pdl_launch_dependents();
  // (what the plan wrote is read from L2: this kernel may start while the one
  // before it, which the plan's completion let start, is still running)
  const uint32_t items = __ldcg(b.class_count + CLS);
  const uint32_t* list = b.class_list + (size_t)CLS * b.num_segments;
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(b.class_next + CLS, 1u);
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= items) break;
    const uint32_t seg = __ldcg(list + item);
    const uint64_t s0 = b.seg_offsets[seg];
    Tile t;
    t.init(smem, (uint32_t)(b.seg_offsets[seg + 1] - s0));
    t.sort(smem, static_cast<const K*>(b.keys_in) + s0, PAIRS ? b.vals_in + s0 : nullptr,
           static_cast<K*>(b.keys_out) + s0, PAIRS ? b.vals_out + s0 : nullptr, b.num_places, b.begin_bit, b.end_bit,
           b.top_xor, b.descending, b.flip);
    __syncthreads();  // everyone has read s_item and the sorted tile
  }
  if (blockIdx.x == 0) pdl_wait();
}

// Dynamic shared memory of which `blocks` fit an SM (228 KB, of which each
// block takes 1 KB besides) and one more does not.
constexpr size_t smem_for_blocks(int blocks) {
  return (228 * 1024 / (size_t)(blocks + 1) - 1024 + 128) / 128 * 128;
}

template <int KBITS, bool PAIRS, int CLS, bool WIDE>
cudaError_t launch_class(const BatchArgs& b, bool* after_kernel, cudaStream_t s) {
  using CT = ClassTile<KBITS, PAIRS, CLS, WIDE>;
  auto* kernel = batch_class_sort_kernel<KBITS, PAIRS, CLS, WIDE>;
  const int sms = device_sm_count();
  if (sms <= 0) return cudaErrorInvalidConfiguration;
  // at most one block per segment the class can have, by the class below's capacity
  uint64_t grid = CLS == 0 ? b.n_total : b.n_total / (b.class_max[CLS == 0 ? 0 : CLS - 1] + 1);
  if (grid > b.num_segments) grid = b.num_segments;
  if (grid > (uint64_t)sms * CT::kClass.blocks_per_sm) grid = (uint64_t)sms * CT::kClass.blocks_per_sm;
  if (grid == 0) return cudaSuccess;
  // The kernel starts while blocks of the one before still hold most SMs, and
  // its own would fill up the few that are free: a grid of fewer blocks than
  // the device holds takes more shared memory, so that no SM takes more than
  // its share. us a batch of u32 pairs without and with it: 305 segments of
  // 4096 keys 55.3 / 48.7, of 3000 49.5 / 43.4 (600 of 4096 63.4 / 63.5: four
  // blocks an SM either way); u64 pairs, 305 of 1000 51.2 / 47.1.
  constexpr size_t least = CT::Tile::smem_bytes;
  constexpr size_t most = smem_for_blocks(1) > least ? smem_for_blocks(1) : least;
  const int share = (int)((grid + sms - 1) / sms);
  size_t bytes = share < CT::kClass.blocks_per_sm ? smem_for_blocks(share) : least;
  if (bytes < least) bytes = least;
  // set on every launch, and always to the most: an idempotent host-side attribute
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e != cudaSuccess) return e;
  e = launch_kernel(kernel, (unsigned)grid, CT::kClass.threads, bytes, s, *after_kernel, b);
  *after_kernel = true;
  return e;
}

// the longest first, so that the shorter sorts fill the gaps at the end. The
// first of them waits for the plan as any kernel does.
template <int KBITS, bool PAIRS>
cudaError_t launch_classes(const BatchArgs& b, bool* after_class, cudaStream_t s) {
  // At most one segment an SM: the longest one's own time counts, so a segment
  // gets a whole block of 1024 threads, unless they are so short (128 keys on
  // the mean) that most of the threads would idle. us a batch, blocks of 256 or
  // 512 / 1024 threads: 16 segments of 4096 u32 pairs 30.7 / 28.7, 32 i32 of a
  // median of 768 34.8 / 30.7, 30 f32 of 226 24.6 / 20.5, 16 u64 of 3584, AND of 3
  // words, 76.7 / 69.8; short ones: 152 of 86 u32 pairs 18.5 / 19.9, u64 32.8 /
  // 36.9. Two segments an SM take turns: 304 of 4096 u32 pairs 45.1 / 50.7, of 86
  // 28.6 / 32.8, 304 of 1000 u64 45.0 / 56.9.
  const bool wide = b.num_segments <= (uint32_t)device_sm_count() && b.n_total >= 128ull * b.num_segments;
  cudaError_t e = launch_class<KBITS, PAIRS, 2, false>(b, after_class, s);
  if (e == cudaSuccess)
    e = wide ? launch_class<KBITS, PAIRS, 1, true>(b, after_class, s)
             : launch_class<KBITS, PAIRS, 1, false>(b, after_class, s);
  if (e == cudaSuccess)
    e = wide ? launch_class<KBITS, PAIRS, 0, true>(b, after_class, s)
             : launch_class<KBITS, PAIRS, 0, false>(b, after_class, s);
  return e;
}

}  // namespace

uint32_t batch_class_capacity(int key_bits, int cls) {
  return key_bits == 32 ? kClass32[cls].capacity() : kClass64[cls].capacity();
}

cudaError_t launch_batch_plan(const BatchArgs& b, cudaStream_t s) {
  batch_plan_kernel<<<1, kPlanThreads, 0, s>>>(b);
  return cudaGetLastError();
}

template <int KBITS>
cudaError_t launch_batch_histogram_t(const BatchArgs& b, int grid, bool after_class, cudaStream_t s) {
  constexpr size_t bytes = BatchHistLayout<KBITS>::smem_bytes;
  // set on every launch: an idempotent host-side attribute
  cudaError_t e = cudaFuncSetAttribute(batch_histogram_kernel<KBITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)bytes);
  if (e != cudaSuccess) return e;
  return launch_kernel(batch_histogram_kernel<KBITS>, (unsigned)grid, kSegHistThreads, bytes, s, after_class, b);
}

cudaError_t launch_batch_histogram(int key_bits, const BatchArgs& b, bool after_class, cudaStream_t s) {
  // one block per SM (128 KiB of shared memory each), at most one per work item
  const int grid = ws_grid(b.max_items > 0 ? b.max_items : 1u);
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  return key_bits == 32 ? launch_batch_histogram_t<32>(b, grid, after_class, s)
                        : launch_batch_histogram_t<64>(b, grid, after_class, s);
}

cudaError_t launch_batch_class_sorts(int key_bits, bool pairs, const BatchArgs& b, bool* after_class, cudaStream_t s) {
  *after_class = false;
  if (key_bits == 32)
    return pairs ? launch_classes<32, true>(b, after_class, s) : launch_classes<32, false>(b, after_class, s);
  return pairs ? launch_classes<64, true>(b, after_class, s) : launch_classes<64, false>(b, after_class, s);
}

}  // namespace onesweep
