"""The tiles of one axis that a window touches (csrc/lbm_tiles.hpp, compiled here as plain
C++) against a count cell by cell: every box length, window and place, on both kinds of axis."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1710_07073_gb300", "csrc")

HARNESS = r"""
#include <set>
#include "lbm_tiles.hpp"
using namespace lbm;

// Boxes, windows and places where the run is not the tiles of the cells (ascending), and
// those whose tiles exceed the bound.
template <int T> void check(int lmax, int cmax, long long out[3]) {
    for (int L = 1; L <= lmax; ++L)
        for (int p = 0; p < 2; ++p)
            for (int cells = 1; cells <= cmax; ++cells) {
                if (p && cells > L) continue;
                const int bound = axis_tile_bound(cells, L, p, T);
                // The centre lies in the box: the window reaches cells 0 .. L - 1.
                for (int lo = 1 - cells; lo < L; ++lo) {
                    std::set<int> want;
                    for (int c = lo; c < lo + cells; ++c)
                        if (p) want.insert((c % L + L) % L / T);
                        else if (c >= 0 && c < L) want.insert(c / T);
                    const AxisRun r = axis_run<T>(lo, lo + cells - 1, L, p);
                    bool same = r.n == (int)want.size();
                    int i = 0;
                    for (int t : want) same = same && i < r.n && r.tile(i++) == t;
                    ++out[0];
                    out[1] += !same;
                    out[2] += (int)want.size() > bound;
                }
            }
}
// Boxes and windows (wider ones too) whose layers are not the tiles of the cells.
extern "C" void check_layers(int lmax, int cmax, long long out[2]) {
    for (int L = 1; L <= lmax; ++L)
        for (int p = 0; p < 2; ++p)
            for (int cells = 1; cells <= cmax; ++cells)
                for (int lo = 1 - cells; lo < L; ++lo) {
                    std::set<int> want, got;
                    for (int c = lo; c < lo + cells; ++c)
                        if (p) want.insert((c % L + L) % L / 4);
                        else if (c >= 0 && c < L) want.insert(c / 4);
                    const LayerRun r = layer_run<4>(lo, lo + cells - 1, L, p);
                    for (int l = r.l0; l <= r.l1; ++l) got.insert(p ? l % ((L + 3) / 4) : l);
                    ++out[0];
                    out[1] += got != want || r.l0 < 0 || r.l1 - r.l0 >= (L + 3) / 4;
                }
}
extern "C" void check_tiles(int tile, int lmax, int cmax, long long out[3]) {
    if (tile == 4) check<4>(lmax, cmax, out);
    else check<32>(lmax, cmax, out);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiles")
    src, lib = d / "tiles.cpp", d / "tiles.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC,
                    str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib))


# Window cells: at most ceil(2 n) + 1 of n <= 9, and the lift's halo of one on each side.
@pytest.mark.parametrize("tile,lmax", [(4, 75), (32, 140)])
def test_runs_and_bound(harness, tile, lmax):
    out = (ctypes.c_longlong * 3)()
    harness.check_tiles(tile, lmax, 22, out)
    assert out[0] > 100_000
    assert (out[1], out[2]) == (0, 0)


# The guard of the overlapped step: a support widened by 4 cells on each side.
def test_layers(harness):
    out = (ctypes.c_longlong * 2)()
    harness.check_layers(75, 30, out)
    assert out[0] > 100_000
    assert out[1] == 0
