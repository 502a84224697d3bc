"""The look-back waits of the clustering and of the smallest batches, without a fault: one
FED's counts are withheld (a flag that nothing sets) under a short poll limit; the call
returns with the event flagged, other events of the batch are exact, and so is the same
call afterwards.
"""
import numpy as np
import pytest

import eventgen as eg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2101_11489_gb300 as sst  # noqa: E402
from _gpu_util import Gpu, assert_clusters_equal  # noqa: E402

N_FEDS = 24


@pytest.fixture(scope="module")
def gt():
    w = eg.WORKLOADS[0]
    calib = eg.make_calibration(N_FEDS, w.seed, w.p_bad)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    yield g, [eg.make_event(w, calib, 60 + i, n_feds=N_FEDS) for i in range(3)]
    g.close()


@pytest.mark.parametrize("amps", [False, True])
@pytest.mark.parametrize("withhold", [0, 5, N_FEDS - 2, N_FEDS - 1])
def test_clustering(gt, withhold, amps):
    g, (e, *_) = gt
    raw, fl = torch.from_numpy(e.raw).cuda(), torch.from_numpy(e.fed_len.view(np.int32)).cuda()
    d = sst.DigiBuffers.alloc(e.nbytes, N_FEDS)
    c = sst.ClusterBuffers.alloc(e.nbytes // 2 + 1, amp_capacity=4 * e.nbytes if amps else 0)
    drec = d.record()
    _, oc, ost = g.oracle(e.raw, e.fed_len, N_FEDS)
    for hold in (withhold, -1):
        sst.sst_unpack(g.ctx, raw, fl, N_FEDS, drec)
        sst.sst_testing_set_wait(g.ctx, 256 if hold >= 0 else 0, hold)
        try:
            sst.sst_cluster(g.ctx, drec, N_FEDS, c.record())  # returns: the waits give up
            torch.cuda.synchronize()
        finally:
            sst.sst_testing_set_wait(g.ctx, 0, -1)
        dh = d.to_host()
        if hold >= 0 and hold < N_FEDS - 1:
            assert dh["flags"] == ost["flags"] | sst.SST_EV_TIMEOUT
        else:  # (the last FED delays nobody)
            assert dh["flags"] == ost["flags"] and dh["n_clusters"] == ost["n_clusters"]
            assert_clusters_equal(c.to_host(0, dh["n_clusters"]), oc)


@pytest.mark.parametrize("withhold", [0, 5, N_FEDS - 2, N_FEDS - 1])
@pytest.mark.parametrize("n_events", [1, 3])
def test_smallest_batches(gt, n_events, withhold):
    g, evs = gt
    evs = evs[:n_events]
    want = [g.oracle(e.raw, e.fed_len, N_FEDS)[1:] for e in evs]
    for hold in (withhold, -1):
        sst.sst_testing_set_wait(g.ctx, 256 if hold >= 0 else 0, hold)
        try:
            got = g.batch([(e.raw, e.fed_len) for e in evs])
        finally:
            sst.sst_testing_set_wait(g.ctx, 0, -1)
        for i, ((st, cl), (oc, ost)) in enumerate(zip(got, want)):
            if i == 0 and 0 <= hold < N_FEDS - 1:
                assert st["flags"] & sst.SST_EV_TIMEOUT
            else:
                assert st == ost
                assert_clusters_equal(cl, oc)
