"""First hits of photons, found by walking the grid, against the search of the
main tree at every kind of leaf_size: of one triangle, where cells with the
same two triangles cannot share a leaf, up to the largest.  (Setup as in
test_gpu_walk: every triangle absorbs and nothing scatters.)"""
import numpy as np
import pytest

from paper_2203_14354_gb300 import geometry as g
from tests.test_gpu_walk import DETECTORS, N_OVER_C, absorbing, rays

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["box", "soup", "small"])
@pytest.mark.parametrize("leaf_size", [1, 2, 4, 8])
def test_first_hits_by_leaf_size(name, leaf_size):
    import torch
    from paper_2203_14354_gb300 import Tracker
    det = absorbing(DETECTORS[name]())
    trk = Tracker(det, leaf_size=leaf_size)
    n = 40_000
    ex = [torch.from_numpy(x).cuda() for x in rays(det, n, seed=40 + leaf_size)]
    out = trk.propagate(n, source=g.Source(g.SRC_EXPLICIT, 0), explicit=ex, per_photon=True, n_tbins=4)
    hit, t = trk.trace_rays(ex[0], out["state"][:, 3:6].contiguous())   # below the size that walks the grid
    fate, time = out["fate"].cpu().numpy(), out["time"].cpu().numpy()
    hit, t = hit.cpu().numpy(), t.cpu().numpy()
    assert (hit >= 0).sum() > n // 10
    assert np.array_equal(fate, np.where(hit >= 0, 3, 4))   # absorbed by the surface, or escaped
    assert np.array_equal(time[hit >= 0], (t * N_OVER_C)[hit >= 0])
