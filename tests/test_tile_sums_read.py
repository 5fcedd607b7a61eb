"""The epilogue reads the sums of a tile that the pass before it has written: 64
with a Hessian, 12 without (grad_kernel leaves the others as they were)."""
import os
import subprocess

import pytest

from paper_1803_00113_gb300 import build_lib

SOURCE = r"""
#include "epilogue.cuh"
using namespace celeste;
template <int kMode>
constexpr bool covers(int tiles, int written) {
  bool seen[kTileChunk * kAcc] = {};
  for (int e = 0; e < tiles * (kTileSums<kMode> / 4); ++e)
    for (int k = 0; k < 4; ++k) {
      const int at = tile_piece<kMode>(e) + k;
      if (at < 0 || at >= tiles * kAcc || seen[at]) return false;
      seen[at] = true;
    }
  for (int at = 0; at < tiles * kAcc; ++at)
    if (seen[at] != (at % kAcc < written)) return false;
  return true;
}
static_assert(covers<1>(1, kGradAcc) && covers<1>(5, kGradAcc) && covers<1>(kTileChunk, kGradAcc), "");
static_assert(covers<2>(1, kAcc) && covers<2>(5, kAcc) && covers<2>(kTileChunk, kAcc), "");
"""


def test_pieces_are_the_written_sums(tmp_path):
    nvcc = build_lib._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "pieces.cu"
    src.write_text(SOURCE)
    r = subprocess.run([nvcc, *build_lib.ARCH, "-std=c++17", f"-I{build_lib.INCLUDE}",
                        f"-I{build_lib.CSRC}", "-c", str(src), "-o", str(tmp_path / "pieces.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
