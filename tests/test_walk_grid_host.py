"""The walk grid as the host builds it, without a GPU: from the cell that a
point of a triangle lies in, the search meets that triangle.  Points are drawn
in double and rounded to float, off the plane by far less than the margin of
the boxes (2^-19 of the largest coordinate, 32 float steps of it)."""
import numpy as np
import pytest

from paper_2203_14354_gb300 import geometry as g
from tests.cuda.host import walk_grid_check

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
