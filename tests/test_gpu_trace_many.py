"""Batches of rays large enough for the kernel that walks the grid (rays
cleared by empty cubes, a ring of waiting rays, layers by their cells) against
the same rays in small batches, which the other kernel answers from the main
tree: the same triangles and the same distances, bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2203_14354_gb300 import geometry as g
from tests.test_gpu_walk import DETECTORS, rays

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BATCH = 50_000


def moved(det, offset):
    det.verts = (det.verts.astype(np.float64) + offset).astype(np.float32)
    return det


MANY = {k: DETECTORS[k] for k in ("one", "box", "soup", "small", "tpc50", "layers")}
# coordinates 40 times the mesh's size (a wide margin of the cells), and 750 times (no grid)
MANY["soup_far"] = lambda: moved(DETECTORS["soup"](), [6000.0, -3000.0, 1000.0])
MANY["sphere_far"] = lambda: moved(g.icosphere(2.0, 3), [0.0, 0.0, -3000.0])


@pytest.mark.parametrize("name", MANY)
@pytest.mark.parametrize("n", [399_999, 400_000, 1_000_003])
def test_many_rays_match_small_batches(name, n):
    import torch
    from paper_2203_14354_gb300 import Tracker
    det = MANY[name]()
    trk = Tracker(det)
    org, d, _ = [torch.from_numpy(x).cuda() for x in rays(det, n, seed=n)]
    size = float(np.ptp(det.verts, axis=0).max())
    tmax = torch.from_numpy(np.random.default_rng(n).exponential(0.3 * size, n).astype(np.float32)).cuda()
    tmax[::7] = float("inf")
    tmax[::11] = 0.0

    def small(*args):
        parts = [trk.trace_rays(*(None if x is None else x[k:k + BATCH].contiguous() for x in args))
                 for k in range(0, n, BATCH)]
        return [torch.cat(x) for x in zip(*parts)]

    hit, _ = small(org, d)
    assert int((hit >= 0).sum()) > (0 if name == "one" else n // 20)
    for scale in (1.0, 0.125, 1024.0):   # directions of any length
        for skip, tm in ((None, None), (None, tmax), (hit, None), (hit, tmax)):
            args = (org, d * scale, skip, None if tm is None else tm / scale)
            a, b = trk.trace_rays(*args), small(*args)
            assert torch.equal(a[0], b[0])
            assert torch.equal(a[1], b[1])


CHECKED = r'''
import sys, numpy as np, torch
sys.path.insert(0, {root!r})
from paper_2203_14354_gb300 import Tracker, _capi
from tests.test_gpu_trace_many import MANY, rays
out = dict(checked=np.array(_capi.checked()))
for name in ("tpc50", "layers", "soup_far"):
    det = MANY[name]()
    trk = Tracker(det)
    org, d, _ = [torch.from_numpy(x).cuda() for x in rays(det, 500_001, seed=9)]
    hit, t = trk.trace_rays(org, d)
    trk.sync()   # raises on any device error bit
    out[name + "_hit"], out[name + "_t"] = hit.cpu().numpy(), t.cpu().numpy()
np.savez({path!r}, **out)
'''


def test_checked_build_of_the_walk(tmp_path):
    got = []
    for checked in ("0", "1"):
        path = str(tmp_path / f"checked{checked}.npz")
        r = subprocess.run([sys.executable, "-c", CHECKED.format(root=ROOT, path=path)],
                           env=dict(os.environ, LXO_CHECKED=checked), capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-3000:]
        got.append(np.load(path))
    assert not bool(got[0]["checked"]) and bool(got[1]["checked"])
    for k in got[0].files:
        assert k == "checked" or np.array_equal(got[0][k], got[1][k]), k
