"""The walk grid as the host builds it, without a GPU: from the cell that a
point of a triangle lies in, the search meets that triangle.  Points are drawn
in double and rounded to float, off the plane by far less than the margin of
the boxes (2^-19 of the largest coordinate, 32 float steps of it)."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2203_14354_gb300 import geometry as g
from tests.cuda.host import walk_grid_check

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DETECTORS = {
    "box": lambda: g.reflector_box(),                 # 12 triangles over thousands of cells
    "soup": lambda: g.random_soup(3000, seed=5, extent=60.0, size=15.0),
    "small": g.small_tpc,
}


def points(det, n, seed):
    rng = np.random.default_rng(seed)
    ids = rng.integers(0, det.n_tris, n)
    u = np.sort(rng.random((n, 2)), axis=1)
    w = np.stack([u[:, 0], u[:, 1] - u[:, 0], 1.0 - u[:, 1]], 1)
    return np.einsum("nk,nka->na", w, det.verts[det.tris[ids]].astype(np.float64)).astype(np.float32), ids


@pytest.mark.parametrize("name", DETECTORS)
@pytest.mark.parametrize("leaf_size", [1, 2, 3, 8])
def test_every_point_is_found_from_its_cell(name, leaf_size):
    det = DETECTORS[name]()
    pts, ids = points(det, 40_000, seed=leaf_size)
    status, lost, seen = walk_grid_check(det, pts, ids, leaf_size)
    assert status == 1 and seen == len(ids) and lost == 0


# a mesh of 4 mm at `offset` mm: the grid's margin grows with the coordinates, up to a quarter of a cell at 341
# times the mesh's size; beyond that there is no grid
FAR_MESH = """
import sys
sys.path.insert(0, {root!r})
from tests.test_walk_grid_host import far_sphere, points, walk_grid_check
det = far_sphere({offset})
print(walk_grid_check(det, *points(det, 20_000, seed=1)))
"""


def far_sphere(offset):
    det = g.icosphere(2.0, 2)   # 320 triangles
    det.verts = (det.verts.astype(np.float64) + [0.0, 0.0, offset]).astype(np.float32)
    return det


@pytest.mark.parametrize("offset, grid", [(0.0, 1), (-100.0, 1), (-1300.0, 1), (-2600.0, 0), (-3000.0, 0), (2e6, 0)])
def test_small_mesh_far_from_the_origin(offset, grid):
    # (in a process of its own, which can be ended: a build that splits triangles without end does not return)
    r = subprocess.run([sys.executable, "-c", FAR_MESH.format(root=ROOT, offset=offset)], capture_output=True,
                       text=True, timeout=60)
    assert r.returncode == 0, r.stderr[-2000:]
    status, lost, seen = eval(r.stdout)
    assert status == grid and lost == 0 and seen == (20_000 if grid else 0)


# no thread can be started (a default stack larger than the address space): the build does with its own
NO_THREADS = """
import ctypes, sys
sys.path.insert(0, {root!r})
from tests.test_walk_grid_host import DETECTORS, g, points, walk_grid_check
det = g.icosphere(2.0, 7)   # 327680 triangles: trees and grid are shared out over threads
pts = points(det, 20_000, seed=1)
walk_grid_check(DETECTORS["box"](), *points(DETECTORS["box"](), 10, seed=1))   # compiled before the threads go
libc, attr = ctypes.CDLL(None), ctypes.create_string_buffer(256)
assert libc.pthread_attr_init(attr) == 0
assert libc.pthread_attr_setstacksize(attr, ctypes.c_size_t(1 << 47)) == 0
assert libc.pthread_setattr_default_np(attr) == 0
print(walk_grid_check(det, *pts, n_threads=8))
"""


def test_build_without_threads():
    r = subprocess.run([sys.executable, "-c", NO_THREADS.format(root=ROOT)], capture_output=True, text=True,
                       timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]
    assert eval(r.stdout) == (1, 0, 20_000)
