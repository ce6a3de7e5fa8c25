// Which positions of a sorted tile are written out. Host and device: the walk
// is checked on the CPU over the last tiles below 2^32, where a run on the
// device would take 100 GB.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define OS_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define OS_HOST_DEVICE inline
#endif

namespace onesweep {

// Calls write(j) for one thread's positions j of a sorted tile of `count` keys,
// UNROLL of them a step. A ragged tile is filled up with pads: they have the
// highest digit, binning is stable, so they lie at the positions count and
// above, and that is what keeps them out of the output. Their places - the
// chain's end and up, to the next multiple of the tile - do not: 32 bits do not
// always hold them (2^32 is not a multiple of 5120 or 6144), and past 2^32 they
// come round to the array's first places.
template <uint32_t THREADS, int UNROLL, typename Write>
OS_HOST_DEVICE void for_each_key(uint32_t thread, uint32_t count, Write write) {
#ifdef __CUDACC__
#pragma unroll UNROLL
#endif
  for (uint32_t j = thread; j < count; j += THREADS) write(j);
}

}  // namespace onesweep
