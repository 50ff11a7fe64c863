"""The rule that refines a batch's cut (csrc/batch_cut.h), compiled for the
host: work item numbers stay in range, and so do the tile table, the 8-row
floor and the threshold of 1.3 tiles per resident CTA."""
import ctypes
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2012_11075_gb300" / "csrc"
INT_MAX = 2 ** 31 - 1
PROGRAM = """
#include "batch_cut.h"
// one case of ny rows, `strips` strips wide
extern "C" int cut(int ny, int strips, int rows, long long resident, long long max_tiles,
                   long long steps) {
  return wblbe::cut_rows(rows, resident, max_tiles, steps, [&](int r) {
    const long long runs = ny / (r > 4 ? r : 4);
    return strips * (runs > 1 ? runs : 1);
  });
}
"""


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    gxx = shutil.which("g++") or pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("cut")
    (d / "cut.cpp").write_text(PROGRAM)
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", str(CSRC),
                           "-o", str(d / "cut.so"), str(d / "cut.cpp")])
    f = ctypes.CDLL(str(d / "cut.so")).cut
    f.argtypes = [ctypes.c_int] * 3 + [ctypes.c_longlong] * 3
    return f


def tiles(ny, strips, rows):
    return strips * max(1, ny // max(rows, 4))


@pytest.mark.parametrize("steps", [1, 64, 10 ** 6, 1500000, 2 * 10 ** 6, 2 ** 28, INT_MAX])
@pytest.mark.parametrize("ny,strips,rows", [(4096, 32, 128), (512, 1, 128), (128, 1, 128),
                                            (4096, 32, 16), (100, 3, 15)])
def test_work_items_of_a_refined_cut_fit_an_int(cut, ny, strips, rows, steps):
    resident = 760
    got = cut(ny, strips, rows, resident, 1 << 20, steps)
    assert got == rows or tiles(ny, strips, got) * steps + resident <= INT_MAX
    # and it is as fine as that allows
    if got >= 16 and 10 * tiles(ny, strips, got) < 13 * resident:
        assert tiles(ny, strips, got // 2) * steps + resident > INT_MAX


def test_threshold_floor_and_table(cut):
    assert cut(4096, 10, 128, 760, 1 << 20, 64) == 32       # 320, 640, 1280 tiles
    assert cut(4096, 31, 128, 760, 1 << 20, 64) == 128      # 992: 1.305 a CTA
    assert cut(4096, 30, 128, 760, 1 << 20, 64) == 64       # 960: 1.26
    assert cut(64, 1, 128, 760, 1 << 20, 64) == 8
    assert cut(64, 1, 15, 760, 1 << 20, 64) == 15
    assert cut(64, 1, 128, 760, 2, 64) == 32                # a table of two tiles
