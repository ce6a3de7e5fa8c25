// Sorts small enough to stay on the chip from the first load to the last
// store, in one launch: all p digit places of an LSD radix sort (arXiv
// 2206.01784, Section 3) over keys that live in registers and shared memory.
//
// What bounds such a sort is not bandwidth but the number of steps that wait
// on one another: a launch sequence (memset, histogram, p binning passes) pays
// a launch, a cold start and a drain per step, about 10 us each, whatever the
// size. Here the array is cut into one tile per block and every pass is:
//   1. each warp ranks its keys among its equal digits (rank_atomic) and the
//      block adds up its warps' digit counts;
//   2. the blocks exchange their 256 digit counts; every block then knows
//      where each of its digits' runs starts in the whole array (the paper's
//      exclusive sums over places and tiles, without a look-back chain: all
//      tiles are resident, so each block simply reads all counts);
//   3. the tile is put in digit order in shared memory and its runs are
//      written to the pass's destination, coalesced; after a barrier over the
//      blocks each block reads its tile of the next pass back from L2.
// A sort of one tile is the same without the exchange: its keys go from
// registers to shared memory and back.
//
// Three forms, by how the blocks wait for one another: one block
// (__syncthreads), one cluster of up to kMaxCluster blocks (the hardware's
// cluster barrier), or a cooperative grid of at most one block per SM (grid
// barrier). In the last two every block reaches every barrier on every path,
// and all blocks are resident, so no barrier can wait for a block that has not
// started. The exchange's polls are bounded: one that runs out records a
// timeout, its block goes on, and every store stays range-checked.
#include <cooperative_groups.h>

#include "os_small.cuh"

namespace onesweep {

namespace {

namespace cg = cooperative_groups;

enum SmallScope { kScopeBlock = 0, kScopeCluster = 1, kScopeGrid = 2 };
// blocks of the largest grid (a lane's rows of 14-bit counts, each at most a
// tile, then add up within 16 bits)
constexpr int kRowsPerLane = 5;
constexpr int kMaxGrid = 32 * kRowsPerLane;
constexpr uint32_t kMaxTile = 12288;
static_assert(kRowsPerLane * kMaxTile < (1u << 16), "packed sums");
// blocks of the largest cluster (above 8: non-portable, but a GPC of this chip holds 16)
constexpr int kMaxCluster = 16;

template <int KBITS, bool PAIRS, int NT, int IPT, int SCOPE>
struct SmallLayout {
  using Tile = SmallTile<KBITS, PAIRS, NT, IPT, SCOPE == kScopeBlock>;
  static_assert(Tile::T < (1 << 14), "exchanged counts are 14 bits wide");
  static constexpr bool kCluster = SCOPE == kScopeCluster;
  static constexpr size_t scan = Tile::smem_bytes;                        // [8] scan scratch
  static constexpr size_t gtot = scan + 32;                               // [256] digit totals of all blocks
  static constexpr size_t glow = gtot + kRadix * 4;                       // [256] ... of the lower blocks, then bin bases
  // cluster: [16][256] counts of each block, then the next pass's tile
  static constexpr size_t rows = glow + kRadix * 4;
  static constexpr size_t krecv = rows + (kCluster ? (size_t)kMaxCluster * kRadix * 4 : 0);
  static constexpr size_t vrecv = krecv + (kCluster ? (size_t)Tile::T * sizeof(typename Tile::K) : 0);
  static constexpr size_t smem_bytes =
      SCOPE == kScopeBlock ? Tile::smem_bytes : vrecv + (kCluster && PAIRS ? (size_t)Tile::T * 4 : 0);
};

// Four exchanged count words (eight 14-bit counts, each under a 2-bit epoch).
__device__ __forceinline__ uint4 ld_relaxed_gpu_v4(const uint4* p) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}

// Exclusive prefix of v over threads 0..255 (other threads pass through).
// Contains one __syncthreads; `tmp` holds 8 words.
__device__ __forceinline__ uint32_t exclusive_sum_256(uint32_t v, uint32_t* tmp) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t x = v;
  if (tid < kRadix) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) tmp[warp] = x;
  }
  __syncthreads();
  uint32_t below = 0;
  if (tid < kRadix) {
#pragma unroll
    for (int w = 0; w < 7; ++w)
      if (w < warp) below += tmp[w];
  }
  return below + x - v;
}

// Every block's counts of the pass, added up: a warp takes groups of 8 digits,
// one block's row per lane and kRowsPerLane rows in flight, so that the whole
// matrix costs about one L2 round trip once the last block has published.
template <int NW>
__device__ __forceinline__ void gather_counts(const SmallArgs& a, const uint4* counts, uint32_t epoch, uint32_t* gtot,
                                              uint32_t* glow) {
  constexpr int GPW = kRadix / 8 / NW;  // groups per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t blk = blockIdx.x, blocks = gridDim.x;
  const uint32_t want = epoch * 0x40004000u;
  auto ready = [want](const uint4& c) {
    return (c.x & 0xC000C000u) == want && (c.y & 0xC000C000u) == want && (c.z & 0xC000C000u) == want &&
           (c.w & 0xC000C000u) == want;
  };
  uint4 c[GPW][kRowsPerLane];
  bool all = false;
  for (uint32_t spins = 0; !all; ++spins) {
    if (spins >= a.spin_limit) {
      atomicOr(a.error, kErrTimeout);
      break;
    }
#pragma unroll
    for (int g = 0; g < GPW; ++g) {
#pragma unroll
      for (int i = 0; i < kRowsPerLane; ++i) {
        const uint32_t r = lane + 32 * i;
        if (r >= blocks)
          c[g][i] = make_uint4(want, want, want, want);
        else if (spins == 0 || !ready(c[g][i]))
          c[g][i] = ld_relaxed_gpu_v4(counts + (size_t)(warp * GPW + g) * blocks + r);
      }
    }
    all = true;
#pragma unroll
    for (int g = 0; g < GPW; ++g)
#pragma unroll
      for (int i = 0; i < kRowsPerLane; ++i) all = all && ready(c[g][i]);
  }
  __syncwarp();
#pragma unroll
  for (int g = 0; g < GPW; ++g) {
    // a lane's rows add up within 16 bits: two counts to a word
    uint32_t tot[4] = {0, 0, 0, 0}, low[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < kRowsPerLane; ++i) {
      const uint32_t w[4] = {c[g][i].x & 0x3FFF3FFFu, c[g][i].y & 0x3FFF3FFFu, c[g][i].z & 0x3FFF3FFFu,
                             c[g][i].w & 0x3FFF3FFFu};
      const bool below = lane + 32u * i < blk;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        tot[j] += w[j];
        low[j] += below ? w[j] : 0u;
      }
    }
    uint32_t mt = 0, ml = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t t = __reduce_add_sync(0xFFFFFFFFu, (tot[j >> 1] >> (16 * (j & 1))) & 0xFFFFu);
      const uint32_t l = __reduce_add_sync(0xFFFFFFFFu, (low[j >> 1] >> (16 * (j & 1))) & 0xFFFFu);
      if (lane == j) {
        mt = t;
        ml = l;
      }
    }
    if (lane < 8) {
      gtot[(warp * GPW + g) * 8 + lane] = mt;
      glow[(warp * GPW + g) * 8 + lane] = ml;
    }
  }
}

template <int KBITS, bool PAIRS, int NT, int IPT, int SCOPE>
__global__ void __launch_bounds__(NT, 1) small_sort_kernel(SmallArgs a) {
  using L = SmallLayout<KBITS, PAIRS, NT, IPT, SCOPE>;
  using Tile = typename L::Tile;
  using K = typename Tile::K;
  constexpr uint32_t T = Tile::T;
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x;
  const uint32_t blk = SCOPE == kScopeBlock ? 0u : blockIdx.x;
  const uint32_t blocks = SCOPE == kScopeBlock ? 1u : gridDim.x;
  const uint32_t start = blk * T;

  if (blk == 0 && tid == 0) *a.error = 0u;
  Tile t;
  t.init(smem, min(T, a.n - start));
  if constexpr (SCOPE == kScopeBlock) {
    t.sort(smem, static_cast<const K*>(a.keys_in), a.vals_in, static_cast<K*>(a.keys_out), a.vals_out, a.num_places,
           a.begin_bit, a.end_bit, a.top_xor, a.descending, a.flip);
    return;
  } else {
    const K* kbuf = reinterpret_cast<const K*>(smem + Tile::kbuf);
    const uint32_t* vbuf = reinterpret_cast<const uint32_t*>(smem + Tile::vbuf);
    uint32_t* scan = reinterpret_cast<uint32_t*>(smem + L::scan);
    uint32_t* gtot = reinterpret_cast<uint32_t*>(smem + L::gtot);
    uint32_t* glow = reinterpret_cast<uint32_t*>(smem + L::glow);
    uint32_t* rows = reinterpret_cast<uint32_t*>(smem + L::rows);
    K* krecv = reinterpret_cast<K*>(smem + L::krecv);
    uint32_t* vrecv = reinterpret_cast<uint32_t*>(smem + L::vrecv);
    // this block's column of both count matrices starts at epoch 0
    if (SCOPE == kScopeGrid && tid < 64)
      (tid < 32 ? a.counts_even : a.counts_odd)[(size_t)(tid & 31) * blocks + blk] = make_uint4(0, 0, 0, 0);
    t.load_keys(static_cast<const K*>(a.keys_in) + start, a.flip);
    if (Tile::kValuesFirst) t.load_values(a.vals_in + start);
    const uint32_t* vsrc = a.vals_in;  // this pass's values (grid)
    // every block is running (its shared memory may be written) and its
    // column is clear
    if constexpr (SCOPE == kScopeCluster)
      cg::this_cluster().sync();
    else
      cg::this_grid().sync();

    for (int pass = 0; pass < a.num_places; ++pass) {
      const int shift = a.begin_bit + kRadixBits * pass;
      const bool last = pass == a.num_places - 1;
      const uint32_t mask = (1u << min(kRadixBits, a.end_bit - shift)) - 1u;
      const uint32_t dxor = (last ? a.top_xor : 0u) ^ (a.descending ? mask : 0u);
      uint32_t bin;
      if constexpr (SCOPE == kScopeCluster) {
        auto cluster = cg::this_cluster();
        auto values = [&] {
          if (pass > 0)
            t.load_values(vrecv);
          else if (!Tile::kValuesFirst)
            t.load_values(a.vals_in + start);
        };
        t.bin(smem, shift, mask, dxor, values, [&](uint32_t total) {
          for (uint32_t r = 0; r < blocks; ++r) cluster.map_shared_rank(rows, r)[blk * kRadix + tid] = total;
        });
        cluster.sync();
        uint32_t tot = 0, low = 0;
        if (tid < kRadix) {
          for (uint32_t r = 0; r < blocks; ++r) {
            const uint32_t c = rows[r * kRadix + tid];
            tot += c;
            if (r < blk) low += c;
          }
        }
        bin = exclusive_sum_256(tot, scan);
        if (tid < kRadix) glow[tid] = bin + low - t.excl;
      } else {
        // 14 bits of each count under the pass's epoch (1-3 in turn on each of
        // the two matrices, so what an earlier pass left is never taken for
        // this one's)
        const uint32_t epoch = 1u + (uint32_t)(pass >> 1) % 3u;
        uint4* counts = (pass & 1) ? a.counts_odd : a.counts_even;
        auto values = [&] {
          if (pass > 0 || !Tile::kValuesFirst) t.template load_values<true>(vsrc + start);
        };
        t.bin(smem, shift, mask, dxor, values, [&](uint32_t total) {
          const uint32_t field = total | (epoch << 14);
          const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, field, 1);
          if ((tid & 1) == 0)
            st_relaxed_gpu(reinterpret_cast<uint32_t*>(counts + (size_t)(tid >> 3) * blocks + blk) + ((tid & 7) >> 1),
                           field | (next << 16));
        });
        gather_counts<NT / 32>(a, counts, epoch, gtot, glow);
        __syncthreads();
        bin = exclusive_sum_256(tid < kRadix ? gtot[tid] : 0u, scan);
        if (tid < kRadix) glow[tid] += bin - t.excl;
      }
      __syncthreads();

      // the runs to their places in the whole array
      if (SCOPE == kScopeCluster && !last) {
        auto cluster = cg::this_cluster();
        for (uint32_t j = tid; j < t.count; j += NT) {
          const K k = kbuf[j];
          const uint32_t g = glow[digit_of(k, shift, mask, dxor)] + j;
          if (g < a.n) {
            cluster.map_shared_rank(krecv, g / T)[g % T] = k;
            if (PAIRS) cluster.map_shared_rank(vrecv, g / T)[g % T] = vbuf[j];
          }
        }
        cluster.sync();
        t.load_keys(krecv);
        continue;
      }
      const bool to_out = ((a.num_places - 1 - pass) & 1) == 0;
      K* kdst = static_cast<K*>(to_out ? a.keys_out : a.alt_keys);
      uint32_t* vdst = to_out ? a.vals_out : a.alt_vals;
      for (uint32_t j = tid; j < t.count; j += NT) {
        const K k = kbuf[j];
        const uint32_t g = glow[digit_of(k, shift, mask, dxor)] + j;
        if (g < a.n) {
          kdst[g] = last && a.flip ? flip_from_ordered(k) : k;
          if (PAIRS) vdst[g] = vbuf[j];
        }
      }
      if (last) break;
      if constexpr (SCOPE == kScopeGrid) {
        cg::this_grid().sync();
        t.template load_keys<true>(kdst + start);
        vsrc = vdst;
      }
    }
  }
}

template <int KBITS, bool PAIRS, int NT, int IPT, int SCOPE>
cudaError_t launch_small_t(const SmallArgs& a, cudaStream_t s) {
  using L = SmallLayout<KBITS, PAIRS, NT, IPT, SCOPE>;
  static_assert(L::smem_bytes <= 227 * 1024, "shared memory of one block");
  auto* kernel = small_sort_kernel<KBITS, PAIRS, NT, IPT, SCOPE>;
  // set on every launch: idempotent host-side attributes, so concurrent
  // callers on any device need no shared state
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem_bytes);
  if (e != cudaSuccess) return e;
  const uint32_t blocks = SCOPE == kScopeBlock ? 1u : (a.n + L::Tile::T - 1) / L::Tile::T;
  if (SCOPE == kScopeCluster && blocks > 8) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = L::smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  if (SCOPE == kScopeCluster) {
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = blocks;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  } else if (SCOPE == kScopeGrid) {
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
  }
  cfg.attrs = &attr;
  cfg.numAttrs = SCOPE == kScopeBlock ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

// The forms: tile, how the blocks wait for one another, and the most keys.
// Measured (graph replay, us a sort of u32 pairs; the pass-by-pass kernels take
// 43 to 61 up to 2^16 keys and 53 to 70 beyond):
//   one block     1000 keys 6.2, 4096 keys 12.3 (a cluster of 4: 14.4)
//   cluster       16384 keys 16.5 (a grid of 2048-key tiles: 24.6)
//   grid          2048-key tiles: 65536 keys 24.6, 300000 26.7
//                 4096: 600000 32.8, 8192: 2^20 43.1, 12288: 1.8M 57.4
// A larger tile costs a pass more (the block's ranking and scatter are bound by
// its SM's shared memory), a smaller one needs more SMs, so each form ends
// where the device's SMs, one tile each, end. Clusters end at 16 blocks of 1024
// keys: with larger tiles the stores into other blocks' shared memory (about 32
// cycles per warp) are slower than a grid's way through L2 (65536 keys: 32.8
// against 24.6). 64-bit pairs: 1000 keys 10.3, 16384 34.9, 300000 51.3, 2^20
// 96.
// Those are uniform words. Keys whose digits repeat meet in the counters here,
// where the passes go over to votes, and gain less or lose at the top of the
// range (one launch / the passes; the AND of 3 words, of 5, all equal): 150 000
// u32 pairs 31 / 39, 29 / 39, 23 / 30; 2^20 57 / 70, 55 / 61, 35 / 41; 1.87M 76 /
// 76, 74 / 65, 43 / 45 (uniform 57 / 66); u64 pairs, 2^20 123 / 106, 121 / 99, 74 /
// 78 (uniform 96 / 104). Setting a frequent digit apart, as a batch's sorts do,
// costs uniform words about 1 us a pass; a lower limit costs them 7 to 15 %.
struct SmallForm {
  uint32_t tile;
  int scope;
  uint32_t most_keys;  // grid: keys per SM of the device
};
constexpr SmallForm kForm[] = {
    {0, 0, 0},
    {1024, kScopeBlock, 1024},
    {4096, kScopeBlock, 4096},
    {1024, kScopeCluster, 16 * 1024},
    {2048, kScopeGrid, 2048},
    {4096, kScopeGrid, 4096},
    {8192, kScopeGrid, 8192},
    {kMaxTile, kScopeGrid, kMaxTile},  // 32-bit keys
};
constexpr int kSmallForms = (int)(sizeof(kForm) / sizeof(kForm[0])) - 1;

template <int KBITS, bool PAIRS>
cudaError_t launch_small_kp(int form, const SmallArgs& a, cudaStream_t s) {
  switch (form) {
    case 1: return launch_small_t<KBITS, PAIRS, 256, 4, kScopeBlock>(a, s);
    case 2: return launch_small_t<KBITS, PAIRS, 1024, 4, kScopeBlock>(a, s);
    case 3: return launch_small_t<KBITS, PAIRS, 256, 4, kScopeCluster>(a, s);
    case 4: return launch_small_t<KBITS, PAIRS, 512, 4, kScopeGrid>(a, s);
    case 5: return launch_small_t<KBITS, PAIRS, 1024, 4, kScopeGrid>(a, s);
    case 6: return launch_small_t<KBITS, PAIRS, 1024, 8, kScopeGrid>(a, s);
    case 7:
      if constexpr (KBITS == 32) return launch_small_t<KBITS, PAIRS, 1024, 12, kScopeGrid>(a, s);
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

int small_form(int key_bits, uint64_t n, int sms) {
  if (n == 0 || sms <= 0) return 0;
  if (sms > kMaxGrid) sms = kMaxGrid;
  for (int f = 1; f <= kSmallForms; ++f) {
    if (key_bits == 64 && kForm[f].tile == kMaxTile) continue;
    const uint64_t most = (uint64_t)kForm[f].most_keys * (kForm[f].scope == kScopeGrid ? sms : 1);
    if (n <= most) return f;
  }
  return 0;
}

uint32_t small_blocks(int form, uint64_t n) {
  return form > 0 && form <= kSmallForms ? (uint32_t)((n + kForm[form].tile - 1) / kForm[form].tile) : 0u;
}

bool small_needs_matrices(int form) { return form > 0 && form <= kSmallForms && kForm[form].scope == kScopeGrid; }

cudaError_t launch_small(int key_bits, bool pairs, int form, const SmallArgs& a, cudaStream_t s) {
  if (key_bits == 32) return pairs ? launch_small_kp<32, true>(form, a, s) : launch_small_kp<32, false>(form, a, s);
  return pairs ? launch_small_kp<64, true>(form, a, s) : launch_small_kp<64, false>(form, a, s);
}

}  // namespace onesweep
