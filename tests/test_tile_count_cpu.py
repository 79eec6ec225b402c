"""Which epilogue warp announces a stored tile of chained GEMMs (csrc/tile_count.h), over every order in which the warps can come."""
import subprocess

import pytest

from paper_2609_23536_b200 import build

# A warp's n-th tile: it takes the tile when the tile's MMAs are done, which wait for the accumulator of tile n - 2 from every
# warp; it hands its accumulator back; it counts the tile.  Places: 2 n before it has handed back tile n, 2 n + 1 before it has
# counted it.  The counters follow from the places, so these are all there is to walk through; warps are alike, so in order.
HARNESS = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <set>
#include <vector>
#include "tile_count.h"
int main(int argc, char** argv) {
  const uint32_t warps = std::atoi(argv[1]), tiles = std::atoi(argv[2]);
  typedef std::vector<uint32_t> Places;
  std::set<Places> seen{Places(warps, 0)};
  std::vector<Places> todo(seen.begin(), seen.end());
  uint32_t furthest_apart = 0;
  while (!todo.empty()) {
    const Places at = todo.back();
    todo.pop_back();
    const auto counted = [&](uint32_t n) { return (uint32_t)std::count_if(at.begin(), at.end(), [&](uint32_t p) { return p > 2 * n + 1; }); };
    const auto back = [&](uint32_t n) { return std::all_of(at.begin(), at.end(), [&](uint32_t p) { return p > 2 * n; }); };
    for (uint32_t w = 0; w < warps; ++w) {
      const uint32_t n = at[w] / 2;
      if (n == tiles) continue;
      if (at[w] % 2 == 0) {
        if (n >= 2 && !back(n - 2)) continue;  // its MMAs have not started
      } else {
        const bool last = qe::last_of_tile(n, warps, [&](uint32_t i) {
          uint32_t v = 0;
          for (uint32_t t = i; t < tiles; t += qe::kTileCounters) v += counted(t);
          return v;
        });
        if (last != (counted(n) == warps - 1)) {
          std::printf("tile %u: said %d with %u of %u stored\n", n, (int)last, counted(n) + 1, warps);
          return 1;
        }
        furthest_apart = std::max(furthest_apart, n - *std::min_element(at.begin(), at.end()) / 2);
      }
      Places next = at;
      ++next[w];
      std::sort(next.begin(), next.end());
      if (seen.insert(next).second) todo.push_back(next);
    }
  }
  std::printf("%zu states, %u tiles apart\n", seen.size(), furthest_apart);
}
"""


@pytest.mark.parametrize("warps,tiles", [(1, 12), (2, 12), (3, 9), (8, 7)])
def test_the_last_warp_to_store_a_tile_is_the_one_that_says_so(tmp_path, warps, tiles):
    (tmp_path / "count.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", build.CSRC, "-o", str(tmp_path / "count"), str(tmp_path / "count.cpp")], check=True)
    r = subprocess.run([str(tmp_path / "count"), str(warps), str(tiles)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
    assert "%d tiles apart" % (0 if warps == 1 else 2) in r.stdout
