// How the radix passes cut a segment.  Plain C++, so that the CPU tests run it up
// to the longest segment (2^32 - 1 items).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define GS_RANGES_FN __host__ __device__ __forceinline__
#else
#define GS_RANGES_FN inline
#endif

namespace gs {

// A block walks its range as for (tile = begin; tile < end; tile += tile_items), with
// positions up to a tile past its end.  Where those do not fit 32 bits, the passes
// run on 64-bit positions (which cost them registers: the sort of 45M pairs 1.45
// against 1.40 ms with the checks that 32 bits would need).
inline bool positions_wrap(uint64_t len, int tile_items) { return len + (uint64_t)tile_items > 0xffffffffull; }

// The items [begin, end) of range b of a segment of len items, whose tiles are cut
// into bps contiguous ranges of equal length up to one tile.
template <class Pos>
struct Range {
  Pos begin, end;
};
template <class Pos>
GS_RANGES_FN Range<Pos> range_of(uint32_t len, uint32_t tile_items, uint32_t bps, uint32_t b) {
  const uint32_t tiles = len / tile_items + (len % tile_items != 0), per = tiles / bps, extra = tiles % bps;
  const uint32_t t0 = b * per + (b < extra ? b : extra), n = per + (b < extra);
  const Pos begin = (Pos)t0 * tile_items, end = t0 + n >= tiles ? (Pos)len : (Pos)(t0 + n) * tile_items;
  return {begin, n ? end : begin};
}

}  // namespace gs
