"""Which words the hashing reads when it copies a tile's messages to shared memory: exactly those
that hold a byte of a message, for every alignment of the first byte, and none for a tile whose
messages are all empty (its pointer need not be readable).  The index arithmetic is compiled for
the host from the header the kernel uses."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_08781_gb300", "csrc")
TOTALS = 100

PROBE = r"""
#include <cstdio>
#include "stage.h"
int main() {
  for (uint32_t a0 = 0; a0 < 16; ++a0)
    for (uint32_t total = 0; total < %d; ++total) {
      std::printf("%%u %%u", a0, total);
      for (uint32_t g = poslo::stage_granule_lo(a0); g < poslo::stage_granule_hi(a0, total); ++g)
        for (uint32_t k = 0; k < 4; ++k) std::printf(" %%u", 4 * g + k);
      uint32_t w;
      for (uint32_t k = 0; k < 8; ++k)
        if (poslo::stage_end_word(a0, total, k, w)) std::printf(" %%u", w);
      std::printf("\n");
    }
}
""" % TOTALS


def test_a_tile_reads_the_words_that_hold_its_bytes(tmp_path):
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(lines) == 16 * TOTALS
    for line in lines:
        a0, total, *words = map(int, line.split())
        assert sorted(words) == sorted({(a0 + i) // 4 for i in range(total)}), (a0, total)
