"""The choice of the detection tiles (host code): the blocks of cells equal
those of the definition -- every tile of every block added up -- and a plan of
small cells takes no longer than its other tables."""
import ctypes as C
import os
import subprocess
import time

import numpy as np
import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2410_04090_gb300", "csrc")
DRIVER = r"""
#include "tile_plan.h"
using namespace jslam;
static std::vector<Geometry> geometries(const int *shape, int n, float scale)
{
    std::vector<Geometry> geo;
    for (int p = 0; p < n; ++p)
        geo.push_back(level_geometry(shape[4 * p], shape[4 * p + 1], shape[4 * p + 2], scale, shape[4 * p + 3]));
    return geo;
}
extern "C" long long plan(const int *shape, int n, float scale, int k, int border, int tw, int th, int chosen, int n_sm,
                          int *out)
{
    std::vector<LevelBlocks> blocks;
    const long long c = detect_blocks(geometries(shape, n, scale), k, border, tw, th, chosen != 0, n_sm, blocks);
    for (int p = 0; p < n; ++p)
        for (int l = 0; l < shape[4 * p + 2]; ++l) {
            out[2 * (8 * p + l)] = blocks[p][l].first;
            out[2 * (8 * p + l) + 1] = blocks[p][l].second;
        }
    return c;
}
// the definition
static int ceil_div(int a, int b) { return (a + b - 1) / b; }
static int bytes_of(int tw, int th) { return (th + 6) * (2 * 32 * (ceil_div(tw, 32) + 1) + 16 * (2 * (ceil_div(tw, 32) + 1) + 1)); }
static double cost_of(int rows, int nch)
{
    return 1000.0 * ceil_div(rows * nch, 128) + (rows ? 115.0 * ceil_div((rows + 6) * (nch + 1), 128) : 0.0) + 300.0;
}
extern "C" void define(const int *shape, int n, float scale, int k, int border, int tw, int th, int chosen, int n_sm,
                       int *out)
{
    const std::vector<Geometry> geo = geometries(shape, n, scale);
    const int chosen_h = th * 3 / 2 < 128 ? th * 3 / 2 : 128;
    const std::vector<int> heights = chosen ? std::vector<int>{ chosen_h } : std::vector<int>{ 96, 64, 48, 32, 24, 16 };
    double best = -1.0;
    for (int max_h : heights) {
        std::vector<int> pick(16 * n);
        double sum = 0.0, dearest = 0.0;
        for (int p = 0; p < n; ++p)
            for (int l = 0; l < geo[p].levels; ++l) {
                const int W = geo[p].W[l], H = geo[p].H[l], c = geo[p].c[l], cx = ceil_div(W, c), cy = ceil_div(H, c);
                double b_cost = -1.0, b_tile = 0.0;
                for (int x = 1; x <= cx && (x == 1 || x * c <= tw); ++x)
                    for (int y = 1; y <= cy && (y == 1 || y * c <= max_h); ++y) {
                        const int bw = x * c < W ? x * c : W, bh = y * c < H ? y * c : H;
                        if (x * y > 1 && (x * y * k > 2048 || bytes_of(bw, bh) > bytes_of(tw, th * 23 / 20))) break;
                        double cost = 0.0, tile = 0.0;
                        for (int y0 = 0; y0 < H; y0 += y * c)
                            for (int x0 = 0; x0 < W; x0 += x * c) {
                                const int a = y0 > border ? y0 : border, e = y0 + y * c < H - border ? y0 + y * c : H - border;
                                const double one = cost_of(e > a ? e - a : 0, ceil_div(W - x0 < x * c ? W - x0 : x * c, 32));
                                cost += one;
                                tile = one > tile ? one : tile;
                            }
                        if (b_cost < 0.0 || cost < b_cost) {
                            b_cost = cost; b_tile = tile;
                            pick[2 * (8 * p + l)] = x; pick[2 * (8 * p + l) + 1] = y;
                        }
                    }
                sum += 2.0 * b_cost;
                dearest = b_tile > dearest ? b_tile : dearest;
            }
        const double time = sum / (5.0 * n_sm) + dearest;
        if (best < 0.0 || time < best) {
            best = time;
            for (size_t i = 0; i < pick.size(); ++i) out[i] = pick[i];
        }
    }
}
"""


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    d = tmp_path_factory.mktemp("tile_plan")
    (d / "driver.cpp").write_text(DRIVER)
    so = str(d / "tile_plan.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "driver.cpp"),
                    os.path.join(CSRC, "tile_plan.cpp"), os.path.join(CSRC, "tables.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    lib.plan.restype = C.c_longlong
    return lib


def _call(fn, shapes, scale=1.2, k=1, border=19, tile=(128, 64), chosen=0, n_sm=152):
    s = np.ascontiguousarray(shapes, np.int32)
    out = np.zeros((len(shapes), 8, 2), np.int32)
    n = fn(s.ctypes.data_as(C.c_void_p), len(shapes), C.c_float(scale), k, border, *tile, chosen, n_sm,
           out.ctypes.data_as(C.c_void_p))
    return out, n


SHAPES = [
    [(320, 240, 4, 32)], [(1241, 376, 8, 32)], [(1920, 1080, 8, 32)], [(752, 480, 8, 32)], [(640, 480, 1, 32)] * 100,
    [(1241, 376, 8, 32)] * 100, [(647, 363, 5, 24)] * 24, [(800, 602, 6, 32)] * 16, [(1241, 376, 8, 16)],
    [(1920, 1080, 8, 16)], [(640, 480, 8, 8)], [(641, 479, 4, 5)], [(320, 240, 3, 3)], [(200, 150, 3, 1)],
    [(61, 4096, 2, 7)], [(4096, 61, 2, 7)], [(999, 777, 6, 128)], [(39, 39, 1, 32)], [(120, 39, 1, 64)],
    [(1920, 1080, 8, 32), (752, 480, 8, 32), (640, 480, 4, 32), (1241, 376, 8, 32)] * 4,
    [(640, 480, 4, 32), (752, 480, 4, 32)] * 8, [(640, 480, 4, 32), (640, 480, 4, 24), (640, 480, 3, 32)],
]


@pytest.mark.parametrize("shapes", SHAPES)
@pytest.mark.parametrize("options", [
    {}, dict(k=3), dict(k=8), dict(border=16), dict(border=19, scale=1.5), dict(tile=(128, 32), chosen=1),
    dict(tile=(64, 128), chosen=1, k=2), dict(tile=(128, 128), chosen=1), dict(tile=(32, 8), chosen=1),
])
def test_blocks_equal_the_definition(L, shapes, options):
    if options.get("border") == 16 and min(shapes[0][:2]) > 200:
        options = dict(options, border=(min(shapes[0][:2]) - 1) // 4)  # the border cuts tiles anywhere
    if options.get("scale") and shapes[0][2] > 4:
        shapes = [(w, h, 3, c) for w, h, _, c in shapes]
    got, _ = _call(L.plan, shapes, **options)
    want, _ = _call(L.define, shapes, **options)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("shapes", [
    [(1920, 1080, 8, 32)], [(1920, 1080, 8, 16)], [(1920, 1080, 8, 8)], [(1920, 1080, 8, 4)], [(4096, 4096, 8, 8)],
    [(4096, 4096, 8, 1)], [(1920, 1080, 8, 16), (1241, 376, 8, 16)] * 64,
])
def test_planning_is_cheap(L, shapes):
    """Blocks compared: no more than fit a tile, once for each shape of the
    batch.  10 ms is some ten times what the largest of these takes; adding up
    the tiles of every block for every height took 18 ms to 49 s."""
    distinct = set(shapes)
    most = 0
    for w, h, levels, cell in distinct:
        for l in range(levels):
            c = max(1, int(cell / 1.2 ** l))
            fit = 128 // c
            most += sum(min(96 // c, 2048 // x) for x in range(1, fit + 1)) + fit + 1
    best = 1e9
    for _ in range(3):
        t = time.perf_counter()
        _, n = _call(L.plan, shapes)
        best = min(best, time.perf_counter() - t)
    assert 0 < n <= most
    assert best < 0.010, best
    print(shapes[0], len(shapes), n, most, best * 1e3, "ms")
