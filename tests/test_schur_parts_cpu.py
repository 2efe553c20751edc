"""Division of a level's Schur products and of their scatter over two streams
(csrc/schur_parts.h), on the host: a scatter tile may only read product tiles of
its own part, as nothing orders the other stream's in front of it."""
from __future__ import annotations

import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1708_04539_gb300", "csrc")
SHIM = """
#include "schur_parts.h"
using namespace pselinv;
extern "C" int product(int part, long corner, long tm, long tn) {
  return schur_in_part(part, corner, tm * kProductRows, tn * kProductCols);
}
extern "C" int scatter(int part, long corner, long tp, long tq) {
  return scatter_in_part(part, corner, tp, tq);
}
extern "C" long size(int i) { return i == 0 ? kProductRows : i == 1 ? kProductCols : kScatterTile; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("parts")
    (d / "shim.cpp").write_text(SHIM)
    out = str(d / "shim.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "shim.cpp"), "-o", out], check=True)
    so = ctypes.CDLL(out)
    so.product.argtypes = so.scatter.argtypes = [ctypes.c_int] + [ctypes.c_long] * 3
    so.size.restype = ctypes.c_long
    return so


@pytest.mark.parametrize("c,cu", [(1, 1), (33, 33), (128, 128), (133, 133), (300, 300), (257, 95)])
@pytest.mark.parametrize("corner", [0, 1, 31, 32, 33, 40, 64, 65, 96, 127, 128, 129, 200, 256])
@pytest.mark.parametrize("lower", [False, True])
def test_scatter_reads_its_own_part(lib, c, cu, corner, lower):
    rows, cols, st = (lib.size(i) for i in range(3))
    for part in (1, 2):
        written = set()  # entries that this part's products write
        for tm in range(-(-c // rows)):
            for tn in range(-(-cu // cols)):
                if (not lower or (tm + 1) * rows > tn * cols) and lib.product(part, corner, tm, tn):
                    written.add((tm, tn))
        for tp in range(-(-c // st)):
            for tq in range(-(-cu // st)):
                if (lower and tp < tq) or not lib.scatter(part, corner, tp, tq):
                    continue
                # first and last entry of the tile
                for p, q in ((tp * st, tq * st),
                             (min(c, (tp + 1) * st) - 1, min(cu, (tq + 1) * st) - 1)):
                    assert (p // rows, q // cols) in written, (part, tp, tq)


@pytest.mark.parametrize("corner", [0, 1, 40, 64, 96, 128, 200])
def test_parts_cover_every_tile_once(lib, corner):
    for tp in range(10):
        for tq in range(10):
            for f in (lib.product, lib.scatter):
                assert f(1, corner, tp, tq) + f(2, corner, tp, tq) == 1
                assert f(0, corner, tp, tq) == 1
            st = lib.size(2)
            if tp * st < corner and tq * st < corner:  # the corner itself comes first
                assert lib.scatter(1, corner, tp, tq)
