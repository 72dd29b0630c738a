// Which words a tile's copy to shared memory reads (stage_tile in k_verify.cu).  The tile's bytes
// start a0 bytes into a 16-byte granule and are `total` long; word w is bytes 4w .. 4w + 3 from
// that granule's start.  Whole granules are read as one, the two at the ends word by word, so
// that every 4-byte word read holds at least one byte of the tile (an empty tile: none).
#pragma once
#include <cstdint>

#ifndef POSLO_HD
#ifdef __CUDACC__
#define POSLO_HD __host__ __device__ __forceinline__
#else
#define POSLO_HD inline
#endif
#endif

namespace poslo {

// The granules that lie wholly inside the tile are lo .. hi - 1.
POSLO_HD uint32_t stage_granule_lo(uint32_t a0) { return (a0 + 15) >> 4; }
POSLO_HD uint32_t stage_granule_hi(uint32_t a0, uint32_t total) { return (a0 + total) >> 4; }

// The words of the granules at the two ends: whether the k-th of eight candidates (k < 4 the
// first granule's, then the last one's) is read, and which word it is.
POSLO_HD bool stage_end_word(uint32_t a0, uint32_t total, uint32_t k, uint32_t& w) {
  const uint32_t hi = stage_granule_hi(a0, total), end = a0 + total;
  const bool tail = k >= 4;
  w = 4 * (tail ? hi : 0u) + (k & 3u);
  const bool partial = tail ? (end & 15u) != 0 && !(hi == 0 && a0 != 0) : a0 != 0;
  return total != 0 && partial && 4 * w + 4 > a0 && 4 * w < end;
}

}  // namespace poslo
