"""The state that the CTAs of a one-CTA-per-FED launch share, against the oracle where it
can go wrong: the unpacking of one event beside the clustering of the one before on another
stream.
"""
import numpy as np
import pytest

import eventgen as eg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2101_11489_gb300 as sst  # noqa: E402
from _gpu_util import Gpu, assert_clusters_equal, assert_digis_equal  # noqa: E402

N_FEDS = 60


def device(e):
    return torch.from_numpy(e.raw).cuda(), torch.from_numpy(e.fed_len.view(np.int32)).cuda()


@pytest.fixture()
def gt():
    w = eg.WORKLOADS[0]
    calib = eg.make_calibration(N_FEDS, w.seed, w.p_bad)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    yield w, calib, g
    g.close()


@pytest.mark.parametrize("amps", [False, True])
def test_unpacking_beside_clustering(gt, amps):
    """Event i + 1 is unpacked on one stream while event i is clustered on another, ordered event by event only."""
    w, calib, g = gt
    evs = [eg.make_event(w, calib, i, occupancy=0.005 * (1 + i % 5), n_feds=N_FEDS) for i in range(4)]
    want = [g.oracle(e.raw, e.fed_len, N_FEDS) for e in evs]
    dev = [device(e) for e in evs]
    n = 40
    d = [sst.DigiBuffers.alloc(evs[i % 4].nbytes, N_FEDS) for i in range(n)]
    c = [sst.ClusterBuffers.alloc(evs[i % 4].nbytes // 2 + 1, amp_capacity=4 * evs[i % 4].nbytes if amps else 0)
         for i in range(n)]
    rec = [x.record() for x in d]
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for i in range(n):
        with torch.cuda.stream(one):
            sst.sst_unpack(g.ctx, *dev[i % 4], N_FEDS, rec[i])
            done = one.record_event()
        with torch.cuda.stream(two):
            two.wait_event(done)
            sst.sst_cluster(g.ctx, rec[i], N_FEDS, c[i].record())
    torch.cuda.synchronize()
    for i in range(n):
        od, oc, ost = want[i % 4]
        dh = d[i].to_host()
        assert dh["flags"] == ost["flags"] and dh["n_clusters"] == ost["n_clusters"]
        assert_digis_equal(dh, od)
        assert_clusters_equal(c[i].to_host(0, dh["n_clusters"]), oc)
