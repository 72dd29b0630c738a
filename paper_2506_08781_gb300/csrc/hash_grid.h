// The hashing's launch shape: tiles of kHashTile entries are taken by groups of kHashThreads
// threads (group k takes tiles k, k + groups, ...), one or more groups to a block.  A batch of few
// tiles must not fill the first blocks and leave the other SMs idle, so groups are numbered across
// the blocks first: the tiles of a batch of t tiles lie on min(t, SMs) SMs.  It matters in POSLO+,
// where a block is alone on its SM and its groups share the SM's shared-memory pipe: hashing of
// 16,384 entries of U[32, 256] bytes takes 74 us, 134 with the groups of a block numbered in a row
// (64 tiles on 16 SMs); of 4,096 entries of 4 KiB 0.75 ms, 2.32 in a row; of 40,000 97 us, 143.
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

constexpr int kHashThreads = 128;
constexpr int kHashTile = 256;

// Groups for n entries, at most `cap`: a group without a tile only writes an empty partial.
POSLO_HD uint32_t hash_groups_of(uint64_t n, uint32_t cap) {
  const uint64_t tiles = (n + kHashTile - 1) / kHashTile;
  return tiles < 1 ? 1u : tiles < cap ? (uint32_t)tiles : cap;
}

// Blocks for `groups` groups of at most `per_block` to a block: one group each while there are no
// more groups than SMs, else as many blocks as keep every SM with one, or more once all are full.
// sms = 0: as few blocks as hold the groups, for a hashing that is not what its call waits for
// (kHashApart): on more SMs it takes more of what the decoding and the MSM run on.  POSLO+ Distill
// of 13,323 entries 278 us so and 301 spread over the SMs, of 26,730 entries of 64 bytes 355 and
// 372, of 60,000 504 and 523; shard records of 13,323 entries 331 and 356.
POSLO_HD uint32_t hash_blocks(uint32_t groups, uint32_t per_block, uint32_t sms) {
  const uint32_t full = (groups + per_block - 1) / per_block;
  return groups <= sms ? groups : full > sms ? full : sms;
}

// Group g of block b has number b * block_step + g * group_step: across the blocks first, or in a
// row when every place of the grid has a group.  Then all SMs have work either way, and in a row
// the last round's tiles end on some SMs before the others, where what is launched behind the
// hashing begins: POSLO+-C Distill of 2^20 entries 1.04 ms, 1.10 across, of 600,000 0.70 and 0.75
// (hashing alone of 262,144 entries is 231 us in a row and 211 across).
struct HashSteps {
  uint32_t block_step, group_step;
};
POSLO_HD HashSteps hash_steps(uint32_t groups, uint32_t blocks, uint32_t per_block) {
  return groups == blocks * per_block ? HashSteps{per_block, 1u} : HashSteps{1u, blocks};
}

}  // namespace poslo
