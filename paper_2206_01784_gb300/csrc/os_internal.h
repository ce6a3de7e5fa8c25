// Host-side interface between the C ABI (os_api.cu) and the kernel
// translation units. Plain structs of device pointers and sizes.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace onesweep {

// Launches a one-argument kernel; early: it may start once every block of the
// stream's last kernel has called pdl_launch_dependents or has ended. Between
// the passes of a sort that hides the launch, the first tile ids and the last
// blocks' drain: 3.3M u32 keys 78 -> 68 us, 2.0M u64 pairs 161 -> 141, 2^28 u32
// pairs 4218 -> 4180. (A proxy fence before the bulk copies, which the wait
// does not need, made every pass 5 % slower.)
template <typename Args>
cudaError_t launch_kernel(void (*kernel)(Args), unsigned grid, unsigned threads, size_t smem_bytes, cudaStream_t s,
                          bool early, const Args& args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args);
}

// Phase 1 + 2 (Section 3, "Upfront histogram kernel", "Exclusive sum kernel").
struct HistArgs {
  const void* keys;          // n keys (device)
  uint64_t n;
  int flip;                  // float keys: apply the sign-flip before taking digits
  int num_places;            // p
  int radix_bits;            // d: place i covers bits [begin_bit + d*i, min(+d, end_bit)); 5..8
  int begin_bit;
  int end_bit;
  uint32_t* hist;            // [p][256] zeroed by the caller (device); 2^d bins used per row
  uint32_t* offsets;         // [p][256] written by the last block (device)
  uint32_t* done_counter;    // zeroed by the caller (device)
  uint32_t* clear;           // words to zero on the way (status slab of pass 0), may be null
  uint64_t clear_words;
  uint32_t* rank_words;      // [p] how each place's digits are ranked (finish_place; may be null)
  uint32_t top_xor;          // signed keys: high bit of the top place's digit inverted (else 0)
  uint32_t descending;       // offsets (and the reported histograms) for complemented digits
};

// Phase 3, one digit-binning pass (Section 3, "Chained scan digit-binning kernel").
struct PassArgs {
  const void* keys_in;
  void* keys_out;
  const uint32_t* vals_in;   // null for keys only
  uint32_t* vals_out;
  uint32_t n;
  uint32_t num_tiles;
  int shift;                 // digit = (ordered key >> shift) & mask
  uint32_t mask;
  int flip_in;               // apply the float sign-flip to loaded keys
  int flip_out;              // undo it on stored keys
  int use_bulk;              // inputs 16-byte aligned: stage full tiles with bulk copies
  const uint32_t* bin_offsets;  // [256] global bin offsets of this place
  uint32_t* status;          // [num_tiles][256] status counters, zeroed
  uint32_t* status_clear;    // slab of the next launch, to zero (may be null) ...
  uint32_t status_clear_rows;  // ... rows 0 .. status_clear_rows-1 of it (>= num_tiles)
  uint32_t* tile_counter;    // zeroed; hands out tile ids in launch order
  uint32_t* error;           // device status word
  uint32_t spin_limit;       // look-back polls before giving up
  int64_t fault_tile;        // test hook: tile that never publishes (-1 = none)

  // Strips (Section 3, "Handling very large problems"): a pass over more than
  // one strip is one launch per strip. keys_in / vals_in point at the strip,
  // n is the strip's length and bin_offsets hold the strip's bin bases (where
  // its first key of each digit lands); out_total is the whole array's length
  // (the output bound). The strip's last tile writes the next strip's bases to
  // carry_out (null when there is no next strip).
  uint32_t out_total;
  uint32_t* carry_out;

  // Segmented mode (os_sort_batch); tile_desc == nullptr means one array of n
  // keys. Each large segment is its own sort: its tiles form one look-back
  // chain and it has its own bin offsets. A tile's descriptor: array index of
  // its first key, its segment's length, its chain's first tile, its segment's
  // row (bin offsets, ranking words).
  const uint4* tile_desc;        // [tiles]
  const uint32_t* total_tiles;   // device word: tiles in this pass
  uint32_t offsets_stride;       // words between two segments' bin offsets

  // Ranking words from the histogram pass (null: none); the word of segment s
  // (0 for one array) is rank_words[s * rank_stride].
  const uint32_t* rank_words;
  uint32_t rank_stride;
  uint32_t digit_xor;            // signed keys, top place: invert the digit's high bit (else 0)
  uint32_t early;                // may start while the stream's last kernel, of this library, ends
};

// A whole sort in one launch (os_small.cu).
struct SmallArgs {
  const void* keys_in;
  void* keys_out;
  const uint32_t* vals_in;   // null for keys only
  uint32_t* vals_out;
  void* alt_keys;            // n keys and values between two passes (more than one block only)
  uint32_t* alt_vals;
  uint4* counts_even;        // [32][blocks] exchanged digit counts of even / odd passes
  uint4* counts_odd;
  uint32_t* error;           // device status word
  uint32_t n;
  int flip;                  // float keys
  int num_places;
  int begin_bit;
  int end_bit;
  uint32_t top_xor;          // signed keys: high bit of the top place's digit inverted (else 0)
  uint32_t descending;       // bin by the complemented digit of every place
  uint32_t spin_limit;       // polls of one block's counts before giving up
};

// Form of the one-launch sort for n keys on a device of `sms` SMs; 0: none
// (the array is too large for it). small_blocks: its blocks.
int small_form(int key_bits, uint64_t n, int sms);
uint32_t small_blocks(int form, uint64_t n);
bool small_needs_matrices(int form);  // exchanges counts through SmallArgs::counts_*
cudaError_t launch_small(int key_bits, bool pairs, int form, const SmallArgs& a, cudaStream_t s);

// Segmented sort: the plan, the histograms of the large segments and the
// one-block sorts of the others (os_batch.cu).
constexpr int kBatchClasses = 3;  // of the one-block sorts
struct BatchArgs {
  const void* keys_in;
  void* keys_out;
  const uint32_t* vals_in;
  uint32_t* vals_out;
  const uint64_t* seg_offsets;   // [S+1]
  uint32_t num_segments;
  uint64_t n_total;
  int flip;                      // float keys
  int num_places;
  int begin_bit;
  int end_bit;
  uint32_t class_max[kBatchClasses];  // longest segment of each class of the one-block sorts
  uint32_t tile_keys;            // binning tile of the large segments
  uint32_t hist_chunk;           // keys per histogram work item
  uint32_t max_large;            // capacity of the large segments' rows
  uint32_t max_tiles;            // capacity of tile_desc
  uint32_t max_items;            // capacity of hist_large
  uint32_t* class_list;          // [kBatchClasses][S] segments of each class
  uint32_t* class_count;         // [kBatchClasses]
  uint32_t* class_next;          // [kBatchClasses] zeroed
  uint2* large_range;            // [max_large] first key, length
  uint32_t* tile_base;           // [max_large+1] first tile
  uint32_t* hist_base;           // [max_large+1] first histogram work item
  uint32_t* hist_large;          // [max_items] row of each work item's segment
  uint4* tile_desc;              // [max_tiles] (PassArgs::tile_desc)
  uint32_t* totals;              // [0] binning tiles, [1] histogram items
  uint32_t* seg_done;            // [max_large] zeroed
  uint32_t* seg_hist;            // [max_large][p][256] zeroed
  uint32_t* seg_bin_offsets;     // [max_large][p][256]
  uint32_t* seg_rank_words;      // [max_large][p]
  uint32_t top_xor;              // signed keys: high bit of the top place's digit inverted (else 0)
  uint32_t descending;           // bin by the complemented digit of every place
  uint32_t* error;
  uint32_t* clear;               // status slab of the first pass, whose rows in use are zeroed
};

constexpr uint32_t kErrBadSegments = 2u;  // device status word bit: invalid segment offsets

cudaError_t launch_batch_plan(const BatchArgs& b, cudaStream_t s);
// *after_class: whether the stream's last kernel is now a class sort (which the
// histogram kernel may overlap).
cudaError_t launch_batch_class_sorts(int key_bits, bool pairs, const BatchArgs& b, bool* after_class, cudaStream_t s);
cudaError_t launch_batch_histogram(int key_bits, const BatchArgs& b, bool after_class, cudaStream_t s);
uint32_t batch_class_capacity(int key_bits, int cls);

// Keys per tile of a binning variant.
uint32_t tile_keys_for(int key_bits, bool pairs, int cfg);

int sort_on_workspace(int key_type, const void* keys_in, void* keys_out, const uint32_t* vals_in, uint32_t* vals_out,
                      uint64_t n, int begin_bit, int end_bit, void* ws, size_t ws_bytes, void* stream);

cudaError_t launch_histogram(int key_bits, const HistArgs& a, int num_sms, cudaStream_t s);
// Launches variant cfg of the binning kernel (the variant a plan was made with).
cudaError_t launch_binning(int key_bits, bool pairs, int cfg, const PassArgs& a, cudaStream_t s,
                           int radix_bits = 8);

}  // namespace onesweep
