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
  lp::pick_n_tile_by_cost(lp::ConvTileQuery{cout, m_tiles, 148, k_mmas, epilogue, wide != 0}, 0.0, tile, *n_tiles);
  return tile;
}
extern "C" int beside(int cout, int m_tiles, int k_mmas, int epilogue, int wide, double step_flops) {
  int tile = 0, n = 0;
  lp::pick_n_tile_by_cost(lp::ConvTileQuery{cout, m_tiles, 148, k_mmas, epilogue, wide != 0}, lp::sm_time_worth(step_flops), tile, n);
  return n * tile >= cout ? tile : -1;
}
""")
    lib.beside.argtypes = [ctypes.c_int] * 5 + [ctypes.c_double]

    def alone(cout, m_tiles, k_mmas, epilogue, wide):
        n = ctypes.c_int(0)
        tile = lib.alone(cout, m_tiles, k_mmas, epilogue, int(wide), ctypes.byref(n))
        return tile, n.value
    alone.beside = lib.beside
    return alone


PLAIN, STATS, SHORTCUT = 0, 1, 2


@pytest.mark.parametrize("q,tflop,tiles", [
    ((512, 4, 288, STATS, False), 0.18, (64, 128)),       # 12 images of 6x6, a step of little work: more than 8 CTAs
    ((256, 12, 144, STATS, False), 0.18, (64, 128)),
    ((256, 896, 4, STATS, True), 0.18, (256,)),           # a launch that fills the machine as it is
    ((512, 4, 288, STATS, False), 30.0, (256,)),          # a step bound by SM time
])
def test_channel_tile_beside_other_modules(tile_rules, q, tflop, tiles):
    assert tile_rules.beside(*[int(v) for v in q], tflop * 1e12) in tiles


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


@pytest.fixture(scope="module")
def order_rules(tmp_path_factory):
    return build_host(tmp_path_factory.mktemp("order"), "order", """
#include "order_rules.h"
#include <vector>
static std::vector<lp::Span> spans(const long long* at, int n) {   // pairs (address, bytes); address 0: not given
  std::vector<lp::Span> v;
  for (int i = 0; i < n; ++i) v.push_back(lp::Span{reinterpret_cast<const void*>(at[2 * i]), (size_t)at[2 * i + 1]});
  return v;
}
extern "C" int multipliers(const long long* lambda, int n) { return lp::multipliers_apart(spans(lambda, n).data(), n); }
extern "C" int corrections(const long long* images, const long long* x, const long long* dx, const long long* x_new, int n) {
  return lp::corrections_apart(spans(images, 1)[0], spans(x, n).data(), spans(dx, n).data(), spans(x_new, n).data(), n);
}
""")


def _spans(pairs):
    flat = [v for p in pairs for v in p]
    return (ctypes.c_longlong * max(1, len(flat)))(*flat)


@pytest.mark.parametrize("spans,apart", [
    ([(64, 16), (80, 16), (96, 16)], True),       # neighbours
    ([(64, 16), (96, 16), (64, 16)], False),      # one buffer for two modules
    ([(64, 16), (79, 16)], False), ([(79, 16), (64, 16)], False), ([(64, 32), (70, 2)], False),
    ([(0, 16), (0, 16), (64, 16)], True), ([], True), ([(64, 16)], True),
])
def test_multipliers_apart(order_rules, spans, apart):
    assert bool(order_rules.multipliers(_spans(spans), len(spans))) == apart


def test_corrections_apart(order_rules):
    """Buffers drawn over one another, partially too: two AuxNets are apart if neither writes what the other one touches and no
    correction goes over the images or an x_k (one AuxNet's output is another one's input); sets of bytes, not intervals."""
    import random
    rng = random.Random(7)
    seen = set()

    def given():
        return rng.randint(1, 400), rng.choice([4, 8, 24])

    def meet(a, b):
        return bool(a[0] and b[0] and set(range(a[0], a[0] + a[1])) & set(range(b[0], b[0] + b[1])))
    for _ in range(4000):
        n = rng.randint(1, 4)
        images, x, dx = given(), [given() for _ in range(n)], [given() for _ in range(n)]
        new = [given() if rng.random() < 0.4 else (0, 8) for _ in range(n)]
        want = not any(meet(new[i], other) for i in range(n)
                       for other in [images] + x + [dx[j] for j in range(n) if j != i] + [new[j] for j in range(n) if j != i])
        seen.add((want, n))
        assert bool(order_rules.corrections(_spans([images]), _spans(x), _spans(dx), _spans(new), n)) == want
    assert len(seen) == 8
    for k in range(3):
        x, dx = [(100 * (i + 1), 96) for i in range(3)], [(2000 + 100 * i, 96) for i in range(3)]
        new = [(1000 + 100 * i, 96) for i in range(3)]
        new[k] = x[k]                             # in place
        assert not order_rules.corrections(_spans([(900, 50)]), _spans(x), _spans(dx), _spans(new), 3)
        new[k] = dx[k]                            # over its own dx: its own business
        assert order_rules.corrections(_spans([(900, 50)]), _spans(x), _spans(dx), _spans(new), 3)


@pytest.fixture(scope="module")
def f32_rules(tmp_path_factory):
    return build_host(tmp_path_factory.mktemp("f32"), "f32", """
#include "conv_f32_rules.h"
extern "C" int forward(int N, int H, int cin, int cout, int R, int s, int few) {
  const int o = (H - 1) / s + 1;
  return lp::f32_forward_on_tiles(lp::F32Conv{N, H, H, cin, o, o, cout, R, s}, few != 0);
}
extern "C" int dgrad(int N, int H, int cin, int cout, int R, int s) {
  const int o = (H - 1) / s + 1;
  return lp::f32_dgrad_on_tiles(lp::F32Conv{N, H, H, cin, o, o, cout, R, s}, 148);
}
""")


# (N, H = W, C_in, C_out, R, stride): microseconds on the tiled and on the direct kernel, measured alone on a B200
@pytest.mark.parametrize("c,tiled,direct", [
    ((64, 32, 4, 64, 3, 1), 48.4, 22.6), ((128, 32, 4, 16, 3, 1), 28.1, 14.6), ((64, 32, 4, 64, 1, 1), 29.1, 10.3),
    ((128, 32, 4, 4, 3, 1), 20.6, 11.4), ((128, 32, 8, 8, 1, 1), 15.1, 8.3), ((128, 32, 4, 64, 3, 2), 34.0, 15.4),
    ((4, 32, 4, 64, 3, 1), 7.3, 14.4), ((1, 32, 4, 64, 1, 1), 3.2, 6.2), ((32, 32, 16, 16, 3, 1), 14.0, 60.0),
    ((64, 14, 64, 256, 1, 1), 59.1, 733.0), ((64, 32, 16, 32, 1, 2), 7.8, 12.4),
])
def test_fp32_forward_takes_the_faster_kernel(f32_rules, c, tiled, direct):
    few = c[2] <= 4 and c[3] % 8 == 0
    assert bool(f32_rules.forward(*c, int(few))) == (tiled < direct)


@pytest.mark.parametrize("c,tiled,direct", [
    ((64, 28, 128, 128, 1, 1), 205.3, 133.3), ((24, 28, 128, 128, 1, 1), 80.7, 59.5), ((64, 14, 256, 64, 1, 1), 55.9, 41.0),
    ((16, 56, 256, 64, 1, 1), 165.7, 135.9), ((64, 11, 128, 128, 1, 1), 53.6, 36.2), ((128, 32, 4, 4, 1, 1), 9.1, 5.2),
    ((128, 32, 4, 4, 3, 1), 18.1, 12.4),
    ((4, 28, 128, 128, 1, 1), 19.6, 23.8), ((64, 7, 512, 512, 1, 1), 204.7, 233.7), ((16, 7, 512, 512, 1, 1), 74.3, 82.0),
    ((128, 32, 8, 64, 1, 1), 31.3, 49.2), ((64, 16, 32, 64, 1, 2), 8.9, 14.4), ((64, 32, 16, 16, 3, 1), 24.4, 53.3),
])
def test_fp32_input_gradient_takes_the_faster_kernel(f32_rules, c, tiled, direct):
    assert bool(f32_rules.dgrad(*c)) == (tiled < direct)
