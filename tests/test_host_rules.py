"""Launch rules that are plain host code: compiled by themselves with g++ and checked without a GPU."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2112_05387_b200", "csrc")


def build_host(tmp_path, name, source, args=()):
    src = tmp_path / (name + ".cpp")
    src.write_text(source)
    out = tmp_path / (name + ".so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, *args, "-o", str(out), str(src)],
                   check=True)
    return ctypes.CDLL(str(out))


@pytest.fixture(scope="module")
def tile_rules(tmp_path_factory):
    lib = build_host(tmp_path_factory.mktemp("tiles"), "tiles", """
#include "conv_tiles.h"
extern "C" int alone(int cout, int m_tiles, int k_mmas, int epilogue, int wide, int* n_tiles) {
  int tile = 0;
  lp::pick_n_tile_alone(lp::ConvTileQuery{cout, m_tiles, 148, k_mmas, epilogue, wide != 0}, tile, *n_tiles);
  return tile;
}
""")

    def alone(cout, m_tiles, k_mmas, epilogue, wide):
        n = ctypes.c_int(0)
        tile = lib.alone(cout, m_tiles, k_mmas, epilogue, int(wide), ctypes.byref(n))
        return tile, n.value
    return alone


PLAIN, STATS, SHORTCUT = 0, 1, 2


# Measured microseconds of a launch alone on a B200, by channel tile: (C_out, pixel tiles, K slices, epilogue, 1x1-like)
@pytest.mark.parametrize("q,us", [
    ((320, 192, 180, STATS, False), {160: 37.0, 64: 46.0}),       # 96 images of 16x16, 3x3
    ((320, 256, 180, PLAIN, False), {160: 43.3, 64: 54.1}),       # 128 of them
    ((320, 256, 180, STATS, False), {160: 50.6, 64: 63.7}),
    ((128, 512, 72, STATS, False), {128: 20.0, 64: 21.1}),        # 64 images of 28x28
    ((192, 98, 180, PLAIN, False), {192: 19.4, 64: 29.1}),        # 49 images of 12x12
    ((288, 198, 288, STATS, False), {144: 50.4, 160: 56.1, 64: 75.5}),
    ((640, 56, 288, PLAIN, False), {160: 32.6, 128: 37.3}),
    ((256, 896, 4, SHORTCUT, True), {256: 29.2, 64: 51.0}),       # 32 images of 56x56, 1x1
    ((512, 224, 8, SHORTCUT, True), {256: 18.5, 64: 27.8}),
    ((1024, 64, 16, SHORTCUT, True), {256: 11.5, 64: 17.1}),
    ((512, 203, 64, PLAIN, True), {256: 23.8, 64: 31.9}),
    # few pixel tiles: the widest tile leaves most SMs idle
    ((256, 8, 144, STATS, False), {256: 19.0, 64: 11.3}),         # 4 images of 14x14, 3x3
    ((512, 8, 288, PLAIN, False), {256: 25.9, 64: 15.0}),
    ((1024, 8, 16, STATS, True), {256: 8.0, 64: 5.2}),
])
def test_channel_tile_of_a_launch_alone_is_a_fast_one(tile_rules, q, us):
    tile, n_tiles = tile_rules(*q)
    assert tile in us, "a tile that was not among the fast ones"
    assert us[tile] <= 1.05 * min(us.values())
    assert n_tiles == -(-q[0] // tile)


def test_channel_tiles_cover_the_channels(tile_rules):
    for cout in range(96, 2049, 32):
        for m_tiles in (1, 7, 74, 149, 1000):
            for k in (4, 36, 360):
                for epilogue in (PLAIN, STATS, SHORTCUT):
                    tile, n_tiles = tile_rules(cout, m_tiles, k, epilogue, k < 60)
                    assert 16 <= tile <= 256 and tile % 16 == 0
                    assert (n_tiles - 1) * tile < cout <= n_tiles * tile
