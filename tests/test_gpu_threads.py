"""Trackers of one process used by several host threads at once."""
import ctypes as C
import threading

import pytest

from paper_2203_14354_gb300 import _capi as A
from paper_2203_14354_gb300 import geometry as g

pytestmark = pytest.mark.gpu


def test_launches_of_different_adjoint_sizes():
    """Two threads launch adjoint runs whose pools take different amounts of
    shared memory: every launch is accepted, and the sums are those of one
    thread alone."""
    import torch
    from paper_2203_14354_gb300 import Tracker
    from paper_2203_14354_gb300.tracker import make_source
    reps, n = 10_000, 8
    dets = [g.small_tpc(), g.small_tpc()]
    trks = [Tracker(d) for d in dets]
    reflectors = [i for i, s in enumerate(dets[0].surfaces) if s.type == g.REFLECTOR]
    trks[0].set_adjoint([g.LXE], [])
    trks[1].set_adjoint([m for m in range(len(dets[0].materials))][:4], reflectors[:8])
    assert trks[0].n_tallies < trks[1].n_tallies
    alone = [t.propagate(n, seed=3, n_tbins=4, adjoint=True)["fates"].clone() for t in trks]
    failed = [0, 0]
    outs = [t.alloc_results(4) for t in trks]
    streams = [torch.cuda.Stream() for _ in trks]
    for t, o in zip(trks, outs):
        o["adjoint"] = torch.zeros((t.n_channels, t.n_tallies), dtype=torch.float64, device=t.device)
    torch.cuda.synchronize()

    def work(k):
        t = trks[k]
        src, rp, res = make_source(dets[k].source), A.lxo_run_params(3, 10000, 4, 1.0, A.LXO_FLAG_ADJOINT), t._results(outs[k])
        call, ctx, st = t._L.lxo_propagate, t._ctx, C.c_void_p(streams[k].cuda_stream)
        for _ in range(reps):
            failed[k] += call(ctx, C.byref(src), n, 0, C.byref(rp), C.byref(res), st) != 0

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert failed == [0, 0]
    for k in range(2):
        assert torch.equal(outs[k]["fates"], alone[k] * reps)
