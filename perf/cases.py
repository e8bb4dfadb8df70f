"""What is timed: the work that users of this tracker have it do, through its
public entry points (Tracker, LightCollection, EventLightCollection), over the
range of detectors, sizes and options that the package, its tests and its
benchmark use.

    listed()            the cases, smallest calls first
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the detector's tracker (built once per process, as a
                        program keeps it) and the inputs made from the seed
    run(state)          one pass; returns its outputs
    work(case)          the bytes and operations that a pass cannot do without
    exact(case, seed)   the outputs in 64 bits, where they are computed numbers
"""
import math
from dataclasses import replace

import numpy as np
import torch

from paper_2203_14354_gb300 import EventLightCollection, LightCollection, Tracker
from paper_2203_14354_gb300 import geometry as g

DEVICE = "cuda:0"

# Detectors: the 14-PMT TPC of the tests, the 50 cm TPC with 61 + 61 PMTs of
# the calibration, the benchmark's DARWIN-scale mesh (hex wire meshes, 1.79e7
# triangles), and the base of the design studies (the same TPC without
# electrodes, 5.2e5 triangles, best-guess optics).
DETECTORS = {
    "small": g.small_tpc,
    "tpc50": g.scaled_tpc,
    "tpc50_dispersed": lambda: _dispersed(g.scaled_tpc()),
    "darwin": g.darwin,
    "study": lambda: g.darwin(electrodes=(), **g.PAPER_OPTICS),
}
# mean photon steps (free flights) to the fate, for work()
STEPS = {"small": 6.7, "tpc50": 19.2, "tpc50_dispersed": 19.2, "darwin": 25.8, "study": 40.7}
# radius and z range of the liquid that rays and event sources start in
VOLUME = {"small": (95.0, -99.0, -1.0), "tpc50": (480.0, -490.0, -10.0), "tpc50_dispersed": (480.0, -490.0, -10.0),
          "darwin": (1270.0, -2590.0, -10.0), "study": (1270.0, -2590.0, -10.0)}
PMTS = {"small": 14, "tpc50": 122, "tpc50_dispersed": 122, "darwin": 1778, "study": 1778}
N_FATES = 20      # fate, material and surface counters, about
OPS_STEP = 300    # random draws and interaction of one step, and the test of the triangle it meets
OPS_RAY = 90      # one box test and one triangle test

_trackers = {}


def _dispersed(det):
    """The detector with an index and a Rayleigh length of the liquid that
    change with the wavelength, lit by the LXe spectrum."""
    det.materials = list(det.materials)
    det.materials[g.LXE] = replace(det.materials[g.LXE], dn_dlambda_per_nm=-0.004, rayleigh_exp=4.0)
    det.source = det.source.with_spectrum(g.LXE_SPECTRUM)
    return det


def _tracker(name):
    if name not in _trackers:
        trk = Tracker(DETECTORS[name]())
        if name == "tpc50":   # the seven parameters of the calibration
            trk.set_adjoint([g.LXE], [0, 1, 4, 5, 6])
        _trackers[name] = trk
    return _trackers[name]


def listed():
    return [
        # a handful of rays against a small mesh: what a debugging or alignment query costs
        {"name": "trace_small_1k", "kind": "trace", "det": "small", "n": 1000, "limited": False},
        # first photon states with emission time and wavelength, for a program that has its own tracker
        {"name": "sample_4m", "kind": "sample", "det": "tpc50", "n": 4_000_001},
        # closest hits of many rays with free-flight limits in the full detector
        {"name": "trace_darwin_2m", "kind": "trace", "det": "darwin", "n": 2_000_003, "limited": True},
        # a short run with per-photon records (a unit check, an event display)
        {"name": "small_20k_records", "kind": "propagate", "det": "small", "n": 20_000, "records": True,
         "profile": False, "host": False},
        # an ordinary run of the 50 cm detector
        {"name": "tpc50_300k", "kind": "propagate", "det": "tpc50", "n": 300_007, "records": False,
         "profile": True, "host": False},
        # one gradient step: expected hits and their derivatives by seven parameters
        {"name": "tpc50_grad_1m", "kind": "grad", "det": "tpc50", "n": 1_000_000},
        # one step of a calibration: 64 sources in one launch, forward and backward
        {"name": "tpc50_calib_64x100k", "kind": "event_grad", "det": "tpc50", "events": 64, "n": 100_000},
        # the emission spectrum with dispersion
        {"name": "tpc50_spectral_3m", "kind": "propagate", "det": "tpc50_dispersed", "n": 3_000_001,
         "records": False, "profile": False, "host": False},
        # one design variant's light collection and arrival times, with the nuclear-recoil profile
        {"name": "study_2m", "kind": "propagate", "det": "study", "n": 2_000_000, "records": False,
         "profile": True, "host": False},
        # an ordinary run of the DARWIN-scale detector, results on the host
        {"name": "darwin_1m_host", "kind": "propagate", "det": "darwin", "n": 1_000_000, "records": False,
         "profile": False, "host": True},
        # batched S1 and S2 events with per-event histograms
        {"name": "darwin_events_288", "kind": "events", "det": "darwin", "events": 288, "bins": 256},
        # the benchmark's step
        {"name": "darwin_100m", "kind": "propagate", "det": "darwin", "n": 100_000_000, "records": False,
         "profile": False, "host": False},
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["trace", "sample", "propagate", "propagate", "propagate", "propagate", "grad", "event_grad",
                       "events"])
    if kind == "trace":
        return {"kind": kind, "det": rng.choice(["small", "tpc50", "study", "darwin"]),
                "n": _log_uniform(rng, 500, 4_000_000), "limited": rng.random() < 0.5}
    if kind == "sample":
        return {"kind": kind, "det": rng.choice(["small", "tpc50"]), "n": _log_uniform(rng, 1000, 8_000_000)}
    if kind == "grad":
        return {"kind": kind, "det": "tpc50", "n": _log_uniform(rng, 5000, 8_000_000)}
    if kind == "event_grad":
        return {"kind": kind, "det": "tpc50", "events": rng.randint(2, 256), "n": _log_uniform(rng, 200, 60_000)}
    if kind == "events":
        return {"kind": kind, "det": rng.choice(["darwin", "study"]), "events": rng.randint(8, 320),
                "bins": rng.choice([64, 256])}
    det = rng.choice(["small", "tpc50", "tpc50_dispersed", "study", "darwin"])
    records = rng.random() < 0.3
    n = _log_uniform(rng, 1000, 2_000_000 if records else 20_000_000)
    return {"kind": "propagate", "det": det, "n": n, "records": records, "profile": rng.random() < 0.5,
            "host": not records and rng.random() < 0.3}


def _points(det, n, rng):
    """Uniform points in the liquid, n x 3."""
    r_max, z0, z1 = VOLUME[det]
    r, a = r_max * np.sqrt(rng.random(n)), 2.0 * math.pi * rng.random(n)
    return np.stack([r * np.cos(a), r * np.sin(a), rng.uniform(z0, z1, n)], 1)


def _rays(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed))
    n = case["n"]

    def u():
        return torch.rand(n, device=DEVICE, dtype=torch.float32, generator=gen)

    r_max, z0, z1 = VOLUME[case["det"]]
    r, a = r_max * u().sqrt(), 2.0 * math.pi * u()
    org = torch.stack([r * a.cos(), r * a.sin(), z0 + (z1 - z0) * u()], 1)
    c, a = 2.0 * u() - 1.0, 2.0 * math.pi * u()
    s = (1.0 - c * c).clamp(min=0.0).sqrt()
    d = torch.stack([s * a.cos(), s * a.sin(), c], 1)
    # free-flight limits as the Rayleigh length of the liquid gives them
    tmax = -400.0 * u().clamp(min=1e-7).log() if case["limited"] else None
    return org, d, tmax


def prepare(case, seed):
    trk = _tracker(case["det"])
    st = {"case": case, "trk": trk, "seed": int(seed) & 0x7FFFFFFF}
    kind = case["kind"]
    if kind == "trace":
        st["org"], st["dir"], st["tmax"] = _rays(case, seed)
    elif kind == "sample":
        st["source"] = trk.det.source.with_profile(g.NR_PROFILE).with_spectrum(g.LXE_SPECTRUM)
    elif kind == "propagate":
        st["source"] = trk.det.source.with_profile(g.NR_PROFILE) if case["profile"] else trk.det.source
    elif kind == "grad":
        st["theta"] = trk.theta()
        rng = np.random.default_rng(seed)
        st["g"] = torch.from_numpy(rng.normal(size=trk.n_channels)).to(DEVICE)
    elif kind == "event_grad":
        rng = np.random.default_rng(seed)
        st["theta"] = trk.theta()
        st["events"] = [(g.Source(g.SRC_POINT, g.LXE, center=tuple(map(float, p))), case["n"])
                        for p in _points(case["det"], case["events"], rng)]
        st["g"] = torch.from_numpy(rng.normal(size=(case["events"], trk.n_channels))).to(DEVICE)
    elif kind == "events":
        # S1 and S2 in the proportion of darwin_events' defaults (8 to 1)
        n2 = max(1, case["events"] // 9)
        st["events"] = g.darwin_events(seed=int(seed) & 0xFFFF, n_s1=case["events"] - n2, n_s2=n2)
    return st


def run(st):
    case, trk = st["case"], st["trk"]
    kind = case["kind"]
    if kind == "trace":
        return trk.trace_rays(st["org"], st["dir"], None, st["tmax"])
    if kind == "sample":
        return trk.sample_source(case["n"], base=12345, seed=st["seed"], source=st["source"], time=True,
                                 wavelength=True)
    if kind == "propagate":
        if case["host"]:
            return trk.propagate_host(case["n"], seed=st["seed"], source=st["source"])
        return trk.propagate(case["n"], seed=st["seed"], source=st["source"], per_photon=case["records"])
    if kind == "grad":
        theta = st["theta"].clone().requires_grad_(True)
        hits = LightCollection.apply(theta, trk, case["n"], st["seed"])
        hits.backward(st["g"])
        return hits.detach(), theta.grad
    if kind == "event_grad":
        trk.upload_events(st["events"])
        theta = st["theta"].clone().requires_grad_(True)
        hits = EventLightCollection.apply(theta, trk, st["seed"])
        hits.backward(st["g"])
        return hits.detach(), theta.grad
    trk.upload_events(st["events"])
    return trk.propagate_events(seed=st["seed"], n_tbins=case["bins"])


def _event_photons(n):
    """Mean photons of n darwin_events (log-uniform counts, 8 S1 to 1 S2)."""
    n2 = max(1, n // 9)
    return (n - n2) * (1e5 - 1e2) / math.log(1e3) + n2 * (1e6 - 1e5) / math.log(10.0)


def work(case):
    kind, det = case["kind"], case["det"]
    P = PMTS[det]
    if kind == "trace":
        return {"bytes": case["n"] * (24 + 8 + (4 if case["limited"] else 0)), "flops": case["n"] * OPS_RAY}
    if kind == "sample":
        return {"bytes": case["n"] * 44, "flops": case["n"] * 400}
    if kind == "propagate":
        return {"bytes": 4 * P * 1003 + 8 * N_FATES + (52 * case["n"] if case["records"] else 0),
                "flops": case["n"] * STEPS[det] * OPS_STEP}
    if kind == "grad":
        return {"bytes": 8 * P * (1 + 7 + 2), "flops": case["n"] * STEPS[det] * OPS_STEP}
    if kind == "event_grad":
        E = case["events"]
        return {"bytes": 8 * E * P * (1 + 7 + 2), "flops": E * case["n"] * STEPS[det] * OPS_STEP}
    E = case["events"]
    return {"bytes": 4 * E * P * (case["bins"] + 3), "flops": _event_photons(E) * STEPS[det] * OPS_STEP}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _philox(seed, pid, step, draw_no):
    """Philox4x32-10 uniforms of include/lxo.h, float64 [4][n]."""
    M = np.uint64(0xFFFFFFFF)
    s32 = np.uint64(32)
    c = [pid & M, pid >> s32, np.full_like(pid, step), np.full_like(pid, draw_no)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> s32) ^ c[1] ^ np.uint64(k0), p1 & M, (p0 >> s32) ^ c[3] ^ np.uint64(k1), p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [((x >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0 ** -23 for x in c]


def _exact_sample(case, seed):
    """Polygon source with a time profile and a spectrum."""
    det = DETECTORS[case["det"]]()
    src = det.source.with_profile(g.NR_PROFILE).with_spectrum(g.LXE_SPECTRUM)
    n, sd = case["n"], int(seed) & 0x7FFFFFFF
    pid = np.uint64(12345) + np.arange(n, dtype=np.uint64)
    last = 0xFFFFFFFF
    u = _philox(sd, pid, last, 0)
    c = 2.0 * u[0] - 1.0
    s = np.sqrt(np.maximum(0.0, 1.0 - c * c))
    d = np.stack([s * np.cos(2 * math.pi * u[1]), s * np.sin(2 * math.pi * u[1]), c], 1)
    # basis perpendicular to d, and the polarisation at a uniform angle in it
    sg = np.where(d[:, 2] >= 0, 1.0, -1.0)
    a = -1.0 / (sg + d[:, 2])
    b = d[:, 0] * d[:, 1] * a
    t1 = np.stack([1.0 + sg * d[:, 0] ** 2 * a, sg * b, -sg * d[:, 0]], 1)
    t2 = np.stack([b, sg + d[:, 1] ** 2 * a, -d[:, 1]], 1)
    ang = 2 * math.pi * u[2][:, None]
    pol = np.cos(ang) * t1 + np.sin(ang) * t2
    pol /= np.linalg.norm(pol, axis=1, keepdims=True)
    pos = np.zeros((n, 3))
    pos[:, 2] = src.z_min + u[3] * (src.z_max - src.z_min)
    todo = np.arange(n)
    ap = src.radius * math.cos(math.pi / src.n_sides)
    for k in range(64):
        if not todo.size:
            break
        w = _philox(sd, pid[todo], last, 1 + k)
        done = np.zeros(todo.size, bool)
        for ur, ua in ((w[0], w[1]), (w[2], w[3])):
            r, phi = src.radius * np.sqrt(ur), 2 * math.pi * ua
            t = ua - src.phase / (2 * math.pi)
            side = np.minimum(((t - np.floor(t)) * src.n_sides).astype(np.int64), src.n_sides - 1)
            psi = src.phase + 2 * math.pi * (side + 0.5) / src.n_sides
            ok = ~done & (r * np.cos(phi) * np.cos(psi) + r * np.sin(phi) * np.sin(psi) <= ap)
            pos[todo[ok], 0], pos[todo[ok], 1] = (r * np.cos(phi))[ok], (r * np.sin(phi))[ok]
            done |= ok
        todo = todo[~done]
    w = _philox(sd, pid, last, last)
    time = src.t0 - np.where(w[0] < src.singlet_frac, src.tau_singlet_ns, src.tau_triplet_ns) * np.log(w[1])
    sigma = src.wl_fwhm_nm / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    wl = src.wl_mean_nm + sigma * np.sqrt(-2.0 * np.log(w[2])) * np.cos(2 * math.pi * w[3])
    return [torch.from_numpy(x) for x in (pos, d, pol, time, wl)]


def _exact_trace(case, seed):
    """Distances to the closest triangle (every triangle tried)."""
    det = DETECTORS[case["det"]]()
    org, d, tmax = _rays(case, seed)
    org, d = org.double(), d.double()
    v = torch.from_numpy(np.asarray(det.verts, np.float64)[np.asarray(det.tris, np.int64)]).to(DEVICE)
    v0, e1, e2 = v[:, 0], v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]
    best = torch.full((case["n"],), math.inf, dtype=torch.float64, device=DEVICE)
    lim = best.clone() if tmax is None else tmax.double()
    step = max(1, 20_000_000 // v.shape[0])
    for i in range(0, case["n"], step):
        o, dd = org[i:i + step, None], d[i:i + step, None]
        p = torch.cross(dd.expand(-1, v.shape[0], -1), e2[None].expand(dd.shape[0], -1, -1), dim=2)
        det_ = (p * e1).sum(2)
        s = o - v0
        uu = (s * p).sum(2) / det_
        q = torch.cross(s, e1[None].expand(s.shape[0], -1, -1), dim=2)
        vv = (dd * q).sum(2) / det_
        t = (e2 * q).sum(2) / det_
        eps = 1e-9
        ok = (det_ != 0) & (uu >= -eps) & (vv >= -eps) & (uu + vv <= 1 + eps) & (t > 0)
        t = torch.where(ok, t, math.inf).amin(1)
        best[i:i + step] = torch.where(t <= lim[i:i + step], t, math.inf)
    return [None, best]


def exact(case, seed):
    if case["kind"] == "sample":
        return _exact_sample(case, seed) if case["n"] <= 5_000_000 else None
    if case["kind"] == "trace" and case["det"] == "small" and case["n"] <= 20_000:
        return _exact_trace(case, seed)
    return None   # a Monte Carlo history has no 64-bit value: its counts are whole numbers
