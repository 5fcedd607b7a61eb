"""Host-side rules and index arithmetic of the pixel launches, compiled as they
are: overlaps enumerated pixel by pixel against a mask, the shares of a
background's item, and when a block takes an item."""
import ctypes
import itertools
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1803_00113_gb300", "csrc")
SOURCE = """
#include "launch_rules.h"
#include "overlap.h"
using namespace celeste;
extern "C" {
void overlap(int c0, int c1, int w, int nx, int ny, int nw, int nh, int* out) {
  const Overlap o = chunk_overlap(c0, c1, w, nx, ny, nw, nh);
  out[0] = o.x; out[1] = o.y; out[2] = o.w; out[3] = o.begin; out[4] = o.end;
}
int shares(long long px, int items, int sm) { return background_shares(px, items, sm); }
int block_derivs(long long px, int items, int sm) { return block_per_item_derivs(px, items, sm); }
int block_values(long long px, int items, int sm) { return block_per_item_values(px, items, sm); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", f"-I{CSRC}", str(d / "rules.cpp"),
                    "-o", str(d / "rules.so")], check=True)
    lib = ctypes.CDLL(str(d / "rules.so"))
    for f in (lib.shares, lib.block_derivs, lib.block_values):
        f.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    return lib


@pytest.mark.parametrize("w,h", [(1, 7), (5, 4), (16, 16), (17, 9), (300, 3), (37, 20), (64, 5)])
def test_overlap_of_a_chunk(rules, w, h):
    """Every pixel of the chunk in the neighbour's patch, and no other."""
    out = (ctypes.c_int * 5)()
    area = w * h
    runs = sorted({(c, min(c + n, area)) for n in (7, 64, 256) for c in range(0, area, n)})
    sizes = sorted({1, w // 2 + 1, 2 * w}), sorted({1, h // 2 + 1, 2 * h})
    for nw, nh in itertools.product(*sizes):
        for nx in sorted({-w + 1, -w // 2, -1, 0, 1, nw // 2, nw - 1, -w, nw}):
            for ny in sorted({-h + 1, -h // 2, 0, 1, nh - 1, -h, nh}):
                # own pixel (x, y) is (x + nx, y + ny) of the neighbour
                y, x = np.mgrid[:h, :w]
                mask = ((x + nx >= 0) & (x + nx < nw) & (y + ny >= 0) & (y + ny < nh)).ravel()
                for c0, c1 in runs:
                    rules.overlap(c0, c1, w, nx, ny, nw, nh, out)
                    ox, oy, ow, b, e = out
                    q = np.arange(b, max(b, e))
                    got = (oy + q // max(ow, 1)) * w + ox + q % max(ow, 1)
                    assert np.array_equal(got, c0 + np.flatnonzero(mask[c0:c1])), (c0, c1, nx, ny, nw, nh)


def test_shares_are_a_pass_or_more(rules):
    sm = 152
    for items in (1, 37, 3040, 3041, 50000):
        for mean in (1, 32, 64, 127, 128, 255, 256, 4096):
            n = rules.shares(mean * items, items, sm)
            assert n in (1, 2, 4) and (n == 1 or mean >= 64 * n)
            assert n == 1 or items <= 20 * sm
            if items <= 20 * sm and mean >= 256:
                assert n == 4
    assert rules.shares(0, 0, sm) == 1


def test_short_items_take_a_block_only_where_they_are_resident(rules):
    sm = 152
    for items, mean, derivs, values in [(1, 1, 0, 1), (1, 32, 0, 1), (1, 33, 1, 1), (304, 64, 1, 1),
                                        (305, 95, 0, 1), (608, 96, 1, 1), (609, 256, 0, 1),
                                        (761, 191, 0, 0), (760, 25, 0, 1), (761, 25, 0, 0),
                                        (761, 192, 0, 1), (1216, 1024, 0, 1), (1217, 1024, 0, 0)]:
        assert rules.block_derivs(mean * items, items, sm) == derivs, (items, mean)
        assert rules.block_values(mean * items, items, sm) == values, (items, mean)
    assert not rules.block_derivs(0, 0, sm) and not rules.block_values(0, 0, sm)
