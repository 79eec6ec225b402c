// Which epilogue warp of a CTA is the last to have stored its part of a tile (GEMMs of chained problems: the others wait for the
// tile's rows).  Plain C++, so that the rule is tested on the host over every order in which the warps can come.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define QE_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define QE_HOST_DEVICE inline
#endif

namespace qe {

// Nothing keeps the warps of a CTA on the same tile.  With two accumulators, a warp starts tile n + 2 when all have handed back the
// accumulator of tile n; they hand one back before they count its tile, so one that has handed back tile n is sure to have counted
// tile n - 1 and no more.  So the tiles n, n + 1 and n + 2 can be waiting for their last warp at once, and n + 3 shares no
// counter with them.  (One counter for all took two arrivals of a fast warp for those of two, and released rows before they were
// stored.)
constexpr uint32_t kTileCounters = 4;

// This warp has stored its part of the CTA's n-th tile; add(i) adds one to counter i and says what it was.
template <class Add>
QE_HOST_DEVICE bool last_of_tile(uint32_t n, uint32_t warps, Add add) {
  return (add(n % kTileCounters) + 1) % warps == 0;
}

}  // namespace qe
