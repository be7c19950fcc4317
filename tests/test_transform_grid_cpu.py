"""The rule that picks the product transform's grid (`csrc/transform_grid.h`), on the host: for lists of any extents
that the checks accept, no kept coefficient aliases on the chosen grid and no list folds two of its vectors onto one
slot, and the grid is a supported one no larger than the caller's."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1111_4429_gb300", "csrc")
SIZES = (8, 10, 12, 16, 20, 24, 30, 32, 36, 40, 48, 50, 60, 64)

SHIM = r'''
#include "transform_grid.h"
extern "C" int pick(int n, int points, int lo, int hi, int ng, const int32_t* geps, int fp32) {
  bgw::GridNeed g;
  g.points = points;
  g.lo = lo;
  g.hi = hi;
  return bgw::transform_grid(n, g, ng, geps, fp32 != 0);
}
'''


@pytest.fixture(scope="module")
def pick(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("grid")
    (d / "shim.cpp").write_text(SHIM)
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{CSRC}", str(d / "shim.cpp"), "-o",
                        str(d / "shim.so")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(str(d / "shim.so"))

    def call(n, gv, gc, ge, fp32=0):
        points = int((np.abs(gv).max(0) + np.abs(gc).max(0) + np.abs(ge).max(0)).max()) + 1
        every = np.concatenate([gv, gc, ge])
        buf = np.ascontiguousarray(ge, dtype=np.int32)
        return lib.pick(n, points, min(0, int(every.min())), max(0, int(every.max())), len(ge),
                        buf.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)), fp32)
    return call


def _list(lo, hi):
    """Points of an axis-aligned box [lo, hi] (per axis) that decide folding: its edges along each axis."""
    pts = {(0, 0, 0)}
    for d in range(3):
        for x in range(lo[d], hi[d] + 1):
            p = [0, 0, 0]
            p[d] = x
            pts.add(tuple(p))
    return np.array(sorted(pts), dtype=np.int32)


def _accepted(n, *lists):
    ok = all(x.min() >= -(n // 2) and x.max() < n - n // 2 for x in lists)
    return ok and n > int(sum(np.abs(x).max(0) for x in lists).max())


def _check(m, n, lists):
    assert m in SIZES and m <= n
    assert m > int(sum(np.abs(x).max(0) for x in lists).max())
    for x in lists:
        assert len({tuple(r) for r in x % m}) == len(x)


# an epsilon list wider than the products, and spheres of very different widths
@pytest.mark.parametrize("bands,other,eps,n", [((-1, 1), (-1, 1), (-4, 4), 20), ((-9, 9), (-1, 1), (-1, 1), 20),
                                               ((0, 0), (0, 0), (-15, 14), 32), ((-1, 1), (-14, 14), (-2, 2), 36),
                                               ((0, 14), (0, 1), (0, 1), 40), ((0, 0), (0, 0), (-8, 7), 32)])
def test_wide_lists(pick, bands, other, eps, n):
    lists = [_list([r[0]] * 3, [r[1]] * 3) for r in (bands, other, eps)]
    assert _accepted(n, *lists)
    for fp32 in (0, 1):
        _check(pick(n, *lists, fp32), n, lists)


# the next grid has the low-band lines and the smallest one has not
@pytest.mark.parametrize("w,e,n,fp64,fp32", [(11, 7, 40, 32, 32), (11, 7, 30, 30, 30), (10, 8, 40, 30, 30),
                                             (18, 12, 60, 50, 60), (18, 12, 50, 50, 50), (17, 15, 64, 50, 50),
                                             (20, 14, 64, 60, 60), (21, 15, 64, 64, 64), (21, 15, 60, 60, 60),
                                             (13, 9, 64, 36, 36), (16, 12, 64, 48, 48)])
def test_low_band_neighbours(pick, w, e, n, fp64, fp32):
    lists = [_list([-r] * 3, [r] * 3) for r in (w, w, e)]
    assert (pick(n, *lists, 0), pick(n, *lists, 1)) == (fp64, fp32)


def test_random_boxes(pick):
    rng = np.random.default_rng(5)
    done = 0
    while done < 2000:
        n = int(rng.choice(SIZES))
        lists = []
        for _ in range(3):
            w = int(rng.integers(0, n // 2 + 1))
            lists.append(_list(-rng.integers(0, w + 1, 3), rng.integers(0, w + 1, 3)))
        if not _accepted(n, *lists):
            continue
        done += 1
        _check(pick(n, *lists, done & 1), n, lists)
