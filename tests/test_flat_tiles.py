"""Tiles of the flat FP32 launch (host logic of the library; no GPU needed).

A tile of step s waits for the tiles in its list to have finished step s - 1 and may then read what
they wrote and overwrite what they read.  So every column and row that a lane of the tile pulls has
to belong to the tile itself or to one of the listed tiles: lane l holds the columns x0 - 2 + 2 l and
x0 - 1 + 2 l (lanes past the two-column halo repeat the one before) and pulls one column further on
each side, the rows run from two below the tile to two above and are pulled from one further.
Checked for wrapping and clamped geometries, with last strips of one and two columns, through the
function that plans the launch, called from a small library compiled here against the built one.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2009_05264_gb300 import build as B

PERIODIC, CHANNEL, WALLS, POOL = range(4)

PROBE = r'''
#include <cstring>
#include <vector>
#include "lbm_internal.h"
extern "C" int flat_tiles(int nx, int ny, int geometry, int rows, int cap, int* out) {
  std::vector<pplbm::FlatTile> t;
  if (!pplbm::build_flat_tiles(0, nx, ny, geometry, rows, t) || (int)t.size() > cap) return -1;
  for (size_t k = 0; k < t.size(); ++k) {
    int* o = out + k * (6 + 2 * pplbm::FLAT_MAX_DEPS);
    const int head[6] = {t[k].x0, t[k].wout, t[k].y0, t[k].rows, t[k].ntiles, t[k].ndeps};
    std::memcpy(o, head, sizeof(head));
    for (int d = 0; d < t[k].ndeps; ++d) {
      o[6 + d] = t[k].deps[d];
      o[6 + pplbm::FLAT_MAX_DEPS + d] = t[k].dep_rows[d];
    }
  }
  return (int)t.size();
}
'''
MAX_DEPS = 25


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    lib = B.build()
    d = tmp_path_factory.mktemp("flat_tiles")
    src, so = os.path.join(d, "probe.cpp"), os.path.join(d, "libprobe.so")
    open(src, "w").write(PROBE)
    subprocess.check_call([nvcc, "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-I", B.CSRC, "-I",
                           os.path.join(B.ROOT, "include"), "-o", so, src, lib, "-Xlinker", "-rpath", "-Xlinker",
                           os.path.dirname(lib)])
    P = ctypes.CDLL(so)

    def tiles(nx, ny, geometry, rows, cap=4096):
        out = np.zeros((cap, 6 + 2 * MAX_DEPS), dtype=np.int32)
        n = P.flat_tiles(nx, ny, geometry, rows, cap, out.ctypes.data_as(ctypes.c_void_p))
        return None if n < 0 else out[:n]

    return tiles


def pulled(first, last, n, wraps):
    """Indices first..last of a direction of n nodes, wrapped, or held at the ends."""
    v = np.arange(first, last + 1)
    return set(v % n) if wraps else set(np.clip(v, 0, n - 1))


WIDTHS = [1, 2, 7, 59, 60, 61, 62, 119, 121, 123, 251, 1741, 1742, 1743, 1801, 1802, 1861, 2995]


@pytest.mark.parametrize("geometry", [PERIODIC, CHANNEL, WALLS, POOL])
@pytest.mark.parametrize("ny,rows", [(3, 4), (5, 4), (33, 7), (47, 15)])
def test_a_tile_waits_for_all_that_it_pulls(plan, geometry, ny, rows):
    for nx in WIDTHS:
        t = plan(nx, ny, geometry, rows)
        assert t is not None and (t[:, 4] == len(t)).all()
        owner = np.full((ny, nx), -1)
        for k, (x0, wout, y0, nrows) in enumerate(t[:, :4]):
            assert wout % 2 == 0 and 0 < wout <= 60
            box = owner[y0:y0 + nrows, x0:min(x0 + wout, nx)]
            assert (box == -1).all()  # every node is written by one tile
            box[...] = k
        assert (owner >= 0).all()
        for k, row in enumerate(t):
            x0, wout, y0, nrows, _, ndeps = row[:6]
            deps, dep_rows = row[6:6 + ndeps], row[6 + MAX_DEPS:6 + MAX_DEPS + ndeps]
            assert (t[deps, 3] == dep_rows).all()
            xs = pulled(x0 - 3, x0 + wout + 2, nx, geometry != CHANNEL)
            ys = pulled(y0 - 3, y0 + nrows + 2, ny, geometry == PERIODIC)
            read = set(owner[np.ix_(sorted(ys), sorted(xs))].ravel()) - {k}
            assert read <= set(deps), (nx, k)
            for j in read:  # and the tile that is read from waits for its reader in turn
                assert k in t[j, 6:6 + t[j, 5]], (nx, k, j)
