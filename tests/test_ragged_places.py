"""The write-out of a ragged last tile (csrc/os_places.h), on the CPU.

The tile is filled up with pads, which the walk has to keep out of the output
at every size up to 2^32 - 1. The last tile's places are 32-bit numbers that
wrap past 2^32 where the tile does not divide it, so the sizes are those whose
last tile reaches it, for the tile of every geometry, beside small ones.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2206_01784_gb300 import build, onesweep as osw

SOURCE = r"""
#include <vector>

#include "os_places.h"
// Writes out the last tile of n keys, `count` of them taken for real: the keys
// take the places up to n, the pads those that follow, as one run of the
// highest digit does. Returns how many positions are wrongly written or left.
extern "C" uint32_t wrong_positions(uint64_t n, uint32_t tile, uint32_t count) {
  const uint32_t start = (uint32_t)((n - 1) / tile * tile);
  const uint32_t real = (uint32_t)(n - (n - 1) / tile * tile);
  std::vector<uint32_t> written(tile, 0);
  for (uint32_t thread = 0; thread < 256; ++thread)
    onesweep::for_each_key<256, 4>(thread, count, [&](uint32_t j) {
      if (start + j < (uint32_t)n) ++written[j];
    });
  uint32_t wrong = 0;
  for (uint32_t j = 0; j < tile; ++j) wrong += written[j] != (j < real ? 1u : 0u);
  return wrong;
}
"""


@pytest.fixture(scope="module")
def wrong_positions(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    folder = tmp_path_factory.mktemp("places")
    src, lib = folder / "places.cpp", folder / "libplaces.so"
    src.write_text(SOURCE)
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, str(src), "-o", str(lib)])
    fn = ctypes.CDLL(str(lib)).wrong_positions
    fn.argtypes = [ctypes.c_uint64, ctypes.c_uint32, ctypes.c_uint32]
    fn.restype = ctypes.c_uint32
    return fn


TILES = sorted({osw.os_tile_config_keys(kb, vb, cfg) for kb in (32, 64) for vb in (0, 4)
                for cfg in range(osw.os_num_tile_configs())})


@pytest.mark.parametrize("tile", TILES)
def test_only_keys_are_stored(wrong_positions, tile):
    top = (1 << 32) - 1
    last = top // tile * tile  # the first key of the last tile of the largest sort
    sizes = [1, tile - 1, tile, tile + 1, 5 * tile + 33, last - 1, last, last + 1, top - 1, top]
    sizes += [last + tile * i // 16 for i in range(1, 16)]
    for n in {n for n in sizes if 0 < n <= top}:
        real = n - (n - 1) // tile * tile
        assert wrong_positions(n, tile, real) == 0, n


def test_the_range_of_a_place_does_not_tell_pads_apart(wrong_positions):
    # 64-bit keys, 5120-key tiles: the last tile ends 1024 places past 2^32, so
    # a walk over the whole tile would store that many pads at places 0..1023
    assert wrong_positions((1 << 32) - 1, 5120, 5120) == 1024
    assert wrong_positions((1 << 32) - 1, 8192, 8192) == 0
