"""How the scan kernels deal out their work, compiled for the host: whatever segment size and grid a caller asks for, every key tile of
every row block goes to exactly one CTA, and the numbers past the last item go to nobody."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2607_11976_b200 import build

SOURCE = """
#include <algorithm>
#include <vector>
#include "lt_work_items.h"
// tiles dealt out twice, never, or outside [0, n_tiles) of blocks [0, n_blocks); what a CTA of the scan kernel does with its rounds
extern "C" long long misdealt(int n_tiles, int seg_tiles, int n_blocks, int grid, int clamp) {
  if (clamp) seg_tiles = lt::clamp_segment(seg_tiles, n_tiles);
  std::vector<int> seen(static_cast<size_t>(n_blocks) * n_tiles, 0);
  long long bad = 0;
  const unsigned int n_items = lt::count_items(n_tiles, seg_tiles, n_blocks), n_rounds = lt::count_rounds(n_items, grid);
  for (int cta = 0; cta < grid; ++cta)
    for (unsigned int round = 0; round < n_rounds; ++round) {
      int block, lo;
      if (!lt::split_item(lt::item_of_round(round, cta, grid), n_items, n_blocks, seg_tiles, block, lo)) continue;
      const long long hi = std::min<long long>(static_cast<long long>(lo) + seg_tiles, n_tiles);
      if (block < 0 || block >= n_blocks || lo < 0 || lo >= hi) {
        ++bad;
        continue;
      }
      for (long long tile = lo; tile < hi; ++tile) ++seen[static_cast<size_t>(block) * n_tiles + tile];
    }
  for (int n : seen) bad += n != 1;
  return bad;
}
"""


@pytest.fixture(scope="module")
def deal(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("items")
    (d / "items.cpp").write_text(SOURCE)
    out = os.path.join(d, "items.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", build.CSRC, "-o", out, str(d / "items.cpp")], check=True)
    lib = ctypes.CDLL(out)
    lib.misdealt.restype = ctypes.c_longlong
    return lib


@pytest.mark.parametrize("seg_tiles", [1, 3, 1000, 1 << 20, 1 << 24, 1 << 30, 2 ** 31 - 1])
@pytest.mark.parametrize("rows", [1, 64, 2405])
@pytest.mark.parametrize("grid", [1, 148, 4096, 1 << 20])
def test_every_tile_is_dealt_out_once(deal, seg_tiles, rows, grid):
    for n_tiles in (1, 2, 147, 1000, 1001, 8192):
        for clamp in (1, 0):  # (the kernels' own arithmetic holds without the host's limit too)
            assert deal.misdealt(n_tiles, seg_tiles, -(-rows // 8), grid, clamp) == 0
