"""Rays that start 64 times the scene's largest coordinate away, and photons that
start 32 times as far: closest hits against brute force over all triangles.
(Farther out the float triangle test itself is off by more than the boxes'
margin, 2^-19 of the largest coordinate; the photons' box tests, which are made
from the photon's place, from some 40 times on.)"""
import numpy as np
import pytest

import oracle as O
from paper_2203_14354_gb300 import geometry as g
from tests.test_gpu_walk import DETECTORS, N_OVER_C, absorbing

pytestmark = pytest.mark.gpu


def soup(offset):
    """600 triangles of 0.01 to 15 mm, as spread as they are large: small ones
    are what a box test that is off by a little misses."""
    det = g.random_soup(600, seed=11, extent=60.0, size=15.0)
    v = det.verts[det.tris].astype(np.float64)
    c = v.mean(axis=1, keepdims=True)
    k = 10.0 ** np.random.default_rng(12).uniform(-3.0, 0.0, (len(v), 1, 1))
    det.verts = (c + k * (v - c) + offset).reshape(-1, 3).astype(np.float32)
    det.tris = np.arange(3 * len(v), dtype=np.uint32).reshape(-1, 3)
    return det


SCENES = {"soup": lambda: soup(0.0), "soup_off": lambda: soup([3000.0, 2000.0, -2500.0]), "layers": DETECTORS["layers"]}


def far_rays(det, n, seed, dist):
    """Towards points of the triangles, from dist times the largest coordinate away."""
    rng = np.random.default_rng(seed)
    u = np.sort(rng.random((n, 2)), axis=1)
    w = np.stack([u[:, 0], u[:, 1] - u[:, 0], 1.0 - u[:, 1]], 1)
    aim = np.einsum("nk,nka->na", w, det.verts[det.tris[rng.integers(0, det.n_tris, n)]].astype(np.float64))
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    org = (aim - dist * float(np.abs(det.verts).max()) * d).astype(np.float32)
    d = aim - org.astype(np.float64)
    return org, (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("name, n", [("soup", 400_000), ("soup_off", 60_000), ("soup_off", 400_000), ("layers", 1500)])
def test_rays_from_far(name, n):
    import torch
    from paper_2203_14354_gb300 import Tracker
    det = SCENES[name]()
    org, d = far_rays(det, n, 5, 64.0)
    want, t_want = O.Oracle(det).trace(org, d, brute=True)
    hit, t = Tracker(det).trace_rays(torch.from_numpy(org).cuda(), torch.from_numpy(d).cuda())
    assert (want != 0xFFFFFFFF).mean() > 0.5
    assert np.array_equal(hit.cpu().numpy().view(np.uint32), want)
    assert np.array_equal(t.cpu().numpy(), t_want)


@pytest.mark.parametrize("name, n", [("soup", 200_000), ("soup_off", 60_000)])
def test_photons_from_far(name, n):
    import torch
    from paper_2203_14354_gb300 import Tracker
    det = absorbing(SCENES[name]())
    org, d = far_rays(det, n, 6, 32.0)
    pol = np.cross(d, np.eye(3)[np.abs(d).argmin(1)]).astype(np.float32)
    ex = [torch.from_numpy(x).cuda() for x in (org, d, pol)]
    out = Tracker(det).propagate(n, source=g.Source(g.SRC_EXPLICIT, 0), explicit=ex, per_photon=True, n_tbins=4)
    want, t_want = O.Oracle(det).trace(org, out["state"][:, 3:6].contiguous().cpu().numpy(), brute=True)
    hit = want != 0xFFFFFFFF
    assert np.array_equal(out["fate"].cpu().numpy(), np.where(hit, 3, 4))   # absorbed by the surface, or escaped
    assert np.array_equal(out["time"].cpu().numpy()[hit], (t_want * N_OVER_C)[hit])
