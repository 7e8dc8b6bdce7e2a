"""How the radix passes cut a segment into ranges, run on the CPU.

A block walks its range as `for (tile = begin; tile < end; tile += tile_items)` on
32-bit positions, or on 64-bit ones where `positions_wrap` says so.  Every item
belongs to one tile of one range, in order, and every walk ends: up to the longest
segment that the sort accepts (2^32 - 1 items), where the position after the last
tile does not fit 32 bits."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_00395_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "ranges.cuh"

template <class Pos>
bool walk(uint32_t len, uint32_t tile, uint32_t bps) {
  uint64_t at = 0;
  for (uint32_t b = 0; b < bps; ++b) {
    const gs::Range<Pos> r = gs::range_of<Pos>(len, tile, bps, b);
    uint64_t steps = 0;
    for (Pos t = r.begin; t < r.end; t += tile) {
      if (t != at || ++steps > (1u << 22)) return false;  // out of order, or a walk without end
      at += r.end - t < tile ? r.end - t : tile;
      const Pos last = t + tile - 1;  // the tile's last place
      if ((last < r.end) != ((uint64_t)t + tile - 1 < (uint64_t)r.end)) return false;
    }
  }
  return at == len;
}

int main() {
  const uint32_t top = 0xffffffffu;
  for (uint32_t tile : {2048u, 4096u})
    for (uint32_t bps : {1u, 3u, 32u, 57u, 304u, 456u})
      for (uint32_t len : {0u, 1u, 2047u, 2048u, 2049u, 4097u, 1000003u, 456u * 2048, 0x7ffffffcu, 0x80000000u,
                           top - 8192, top - 4097, top - 4096, top - 4095, top - 2048, top - 2047, top - 100, top}) {
        const bool ok = gs::positions_wrap(len, 4096) ? walk<uint64_t>(len, tile, bps) : walk<uint32_t>(len, tile, bps);
        if (!ok) return std::printf("%u items, tiles of %u, %u ranges\n", len, tile, bps), 1;
      }
  return 0;
}
"""


def test_every_item_once_and_every_walk_ends(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "ranges.cpp", tmp_path / "ranges"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
