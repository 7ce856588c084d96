"""Slot numbers of a frame's packed tiles (csrc/frame_slots.h), host-compiled with
g++, at the largest frames that are accepted (2^31 - 1 pixels, 1024 materials):
the last slots lie past 2^31, and the free slots of a last tile are exactly those
between a material's pixels and the next material's first tile."""
import os
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r'''
#include <cstdio>
#include <cstdint>
#include <initializer_list>
#include "frame_slots.h"
using namespace nbtc;
int main() {
  for (int64_t n = 0; n < (int64_t(1) << 31); n += n < 4096 || n > 2147479000 ? 1 : 7919 * 127) {
    const int px = (int)n;
    const int64_t tiles = (n + 127) / 128;
    if (packed_tiles(px) != tiles) { printf("tiles of %d\n", px); return 1; }
    if (n + free_slots(px) != tiles * 128) { printf("free slots of %d\n", px); return 1; }
    for (int first : {0, 1, (1 << 24) + 1023})
      if (packed_slot(first, px) != (int64_t)first * 128 + n) { printf("slot %d %d\n", first, px); return 1; }
  }
  // 1023 materials of one pixel, then the rest of the largest frame
  const int last = 2147483647 - 1023;
  if (packed_slot(1023, last - 1) != 1023ll * 128 + last - 1 || packed_slot(1023, last - 1) <= 2147483647ll) return 1;
  printf("OK\n");
  return 0;
}
'''


def test_packed_slots_of_the_largest_frames():
    with tempfile.TemporaryDirectory() as d:
        c = os.path.join(d, "t.cpp")
        open(c, "w").write(SRC)
        exe = os.path.join(d, "t")
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-I",
                               os.path.join(ROOT, "paper_2506_06040_gb300", "csrc"), c, "-o", exe])
        out = subprocess.run([exe], capture_output=True, text=True, timeout=300).stdout
    assert out.strip() == "OK", out
