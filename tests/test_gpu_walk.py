"""The route to the closest hit (flights cleared by empty cubes, the walk
through the grid, planar layers entered by their cells) against the search of
the main tree, ray by ray, in lxo_trace_rays and in the photon kernel, and the
kernel's pool of photon slots at sizes around a lane, a warp, a CTA and the
whole GPU.

Directions 2^64 long are left to the main tree: every number of the exact
triangle test then scales by a power of two, so hits and t stay the same.

Every triangle absorbs and no medium scatters, so a photon ends at its first
hit with its direction unchanged: its time is t n / c for the t of the same
ray in lxo_trace_rays, rounded once, and it escapes where that ray misses."""
import numpy as np
import pytest

from paper_2203_14354_gb300 import geometry as g

pytestmark = pytest.mark.gpu

N_INDEX = 1.69
N_OVER_C = np.float32(float(np.float32(N_INDEX)) / 299.792458)   # the table holds n in float32


def absorbing(det):
    det.materials = [g.Material("m", N_INDEX)] * 4
    det.surfaces = [g.Surface("black", g.ABSORBER)]
    det.surface = np.zeros_like(det.surface)
    return det


DETECTORS = {
    "one": lambda: g.random_soup(1, seed=3),                       # a tree of one leaf
    "soup": lambda: g.random_soup(3000, seed=5, extent=60.0, size=15.0),
    "sphere": lambda: g.icosphere(100.0, 4),
    "box": lambda: g.reflector_box(),                              # faces along the grid's sides
    "small": g.small_tpc,
    "tpc50": g.scaled_tpc,
    "layers": lambda: g.darwin(electrodes=("cathode",), wire_um=2000.0, mesh_pitch=60.0),   # dense layers and big panels
}


def rays(det, n, seed):
    """Rays from inside and outside the mesh's box, towards everywhere, some
    along the axes and some from points on the grid's planes of symmetry."""
    rng = np.random.default_rng(seed)
    lo, hi = det.verts.min(0).astype(np.float64), det.verts.max(0).astype(np.float64)
    org = rng.uniform(lo, hi, (n, 3))
    far = rng.random(n) < 0.2
    org[far] = rng.uniform(lo - 0.3 * (hi - lo) - 1.0, hi + 0.3 * (hi - lo) + 1.0, (int(far.sum()), 3))
    mid = rng.random(n) < 0.1
    org[mid] = np.where(rng.random((int(mid.sum()), 3)) < 0.5, 0.5 * (lo + hi), org[mid])
    d = rng.normal(size=(n, 3))
    par = rng.random(n) < 0.15
    d[par] = np.eye(3)[rng.integers(0, 3, int(par.sum()))] * rng.choice([-1.0, 1.0], (int(par.sum()), 1))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    e = np.cross(d, np.eye(3)[np.abs(d).argmin(1)])
    e /= np.linalg.norm(e, axis=1, keepdims=True)
    return [x.astype(np.float32) for x in (org, d, e)]


@pytest.mark.parametrize("name", DETECTORS)
def test_first_hits_match_the_tree_search(name):
    import torch
    from paper_2203_14354_gb300 import Tracker
    det = absorbing(DETECTORS[name]())
    trk = Tracker(det)
    n = 60_000
    ex = [torch.from_numpy(x).cuda() for x in rays(det, n, seed=17)]
    out = trk.propagate(n, source=g.Source(g.SRC_EXPLICIT, 0), explicit=ex, per_photon=True, n_tbins=4)
    hit, t = trk.trace_rays(ex[0], out["state"][:, 3:6].contiguous())
    fate, time = out["fate"].cpu().numpy(), out["time"].cpu().numpy()
    hit, t = hit.cpu().numpy(), t.cpu().numpy()
    assert (hit >= 0).sum() > (0 if name == "one" else n // 10)
    assert np.array_equal(fate, np.where(hit >= 0, 3, 4))   # absorbed by the surface, or escaped
    assert np.array_equal(time[hit >= 0], (t * N_OVER_C)[hit >= 0])
    assert int(out["fates"][:7].sum()) == n


@pytest.mark.parametrize("name", DETECTORS)
@pytest.mark.parametrize("n", [1, 33, 40_000])
def test_walk_matches_the_main_tree(name, n):
    import torch
    from paper_2203_14354_gb300 import Tracker
    det = DETECTORS[name]()
    trk = Tracker(det)
    org, d, _ = [torch.from_numpy(x).cuda() for x in rays(det, n, seed=5 + n)]
    far = 2.0 ** 64
    rng = np.random.default_rng(n)
    size = float(np.ptp(det.verts, axis=0).max())
    tmax = torch.from_numpy(rng.exponential(0.3 * size, n).astype(np.float32)).cuda()
    tmax[::7] = float("inf")
    tmax[::11] = 0.0
    hit, _ = trk.trace_rays(org, d)
    for scale in (1.0, 0.125, 1024.0):   # directions of any length
        for skip, tm in ((None, None), (None, tmax), (hit, None), (hit, tmax)):
            a = trk.trace_rays(org, d * scale, skip, None if tm is None else tm / scale)
            b = trk.trace_rays(org, d * far, skip, None if tm is None else tm / far)
            assert torch.equal(a[0], b[0])
            assert torch.equal(a[1] * scale, b[1] * far)


def test_pool_sizes():
    """Runs of n photons give the first n rows of a longer run."""
    import torch
    from paper_2203_14354_gb300 import Tracker
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    trk = Tracker(g.small_tpc())
    ref = trk.propagate(2 * sms * 1024 + 7, seed=21, per_photon=True, n_tbins=8)
    for n in (1, 2, 31, 32, 33, 2 * sms - 1, 2 * sms, 2 * sms + 1, 64 * sms + 1, 2 * sms * 32 * 20 + 1,
              2 * sms * 992 - 1, 2 * sms * 992 + 1, 2 * sms * 1024):
        out = trk.propagate(n, seed=21, per_photon=True, n_tbins=8)
        for k in ("fate", "detail", "steps", "time", "state"):
            assert torch.equal(out[k], ref[k][:n]), (n, k)
        assert int(out["fates"][:7].sum()) == n
    # any launch shape and any number of ids per grab: the same photons
    for shape in ((1, 1, 128), (3, 5, 256), (32, 4096, 256)):
        trk.set_launch(*shape)
        out = trk.propagate(50_001, seed=21, per_photon=True, n_tbins=8)
        for k in ("fate", "detail", "steps", "time", "state"):
            assert torch.equal(out[k], ref[k][:50_001]), (shape, k)
