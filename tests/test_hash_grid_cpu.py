"""The hashing's launch shape: every group has a place of its own in the grid, and the tiles of a
batch lie on as many SMs as there are tiles (POSLO+ has several groups to a block, one block to an
SM; numbered inside a block first, 64 tiles would lie on 16 of 152 SMs).  The arithmetic is
compiled for the host from the header the kernel and its launch use.  A hashing that its call does
not wait for (no number of SMs given) takes as few blocks as hold its groups instead."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_08781_gb300", "csrc")
SMS = 152

PROBE = r"""
#include <cstdio>
#include <set>
#include "hash_grid.h"
using namespace poslo;
int main() {
  const uint64_t ns[] = {0, 1, 255, 256, 257, 1024, 16384, 38912, 38913, 40000, 77824, 77825, 116736, 150000,
                         155648, 155649, 1048576, 1048577};
  for (uint64_t n : ns)
    for (uint32_t per : {1u, 2u, 4u})
    for (uint32_t sms : {SMSu, 0u}) {
      const uint32_t groups = hash_groups_of(n, 4 * SMS), blocks = hash_blocks(groups, per, sms);
      const HashSteps steps = hash_steps(groups, blocks, per);
      std::set<uint32_t> ids, busy;
      uint32_t in_range = 0;
      for (uint32_t b = 0; b < blocks; ++b)
        for (uint32_t g = 0; g < per; ++g) {
          const uint32_t id = b * steps.block_step + g * steps.group_step;
          if (id >= groups) continue;
          ++in_range;
          ids.insert(id);
          if ((uint64_t)id * kHashTile < n) busy.insert(b);
        }
      std::printf("%llu %u %u %u %u %u %zu %zu\n", (unsigned long long)n, per, sms, groups, blocks, in_range,
                  ids.size(), busy.size());
    }
}
""".replace("SMS", str(SMS))


def test_tiles_lie_on_as_many_blocks_as_they_can(tmp_path):
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    rows = [tuple(map(int, r.split()))
            for r in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) == 18 * 3 * 2
    for n, per, sms, groups, blocks, in_range, ids, busy in rows:
        tiles = -(-n // 256)
        assert groups == min(max(tiles, 1), 4 * SMS)
        assert in_range == ids == groups, (n, per)            # each group once
        if sms:
            assert busy >= min(tiles, SMS), (n, per, busy)    # one tile to an SM before two
        assert blocks <= max(sms, -(-groups // per)), (n, per)   # no more blocks than needed
