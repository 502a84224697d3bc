"""Batches read in place from pinned host memory (channel streams over pieces of several
adjacent FE units) against the oracle: events of every density, FE units too large to
stage, corrupt records and records at odd offsets, in batches of every size the server
forms.
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
from test_gpu_stream import N_FEDS, PARAMS, distinct_events  # noqa: E402


@pytest.mark.parametrize("which", sorted(PARAMS))
def test_batches_read_in_place(which):
    calib = eg.make_calibration(N_FEDS, 23, 0.02)
    g = Gpu(calib.noise, calib.gain, calib.bad, PARAMS[which])
    sst.sst_server_start(g.ctx, 256 << 20, 60, 2, 512, N_FEDS, zero_copy="in_place")
    try:
        base = [(r, f) for r, f in distinct_events(calib) if r.size and r.size % 16 == 0]
        want = [g.oracle(r, f, N_FEDS)[1:] for r, f in base]
        lent = [(torch.from_numpy(r.copy()).pin_memory(), np.ascontiguousarray(f, np.uint32)) for r, f in base]
        tickets = []
        for i in range(8 * len(base)):
            code, t = sst.sst_submit(g.ctx, lent[i % len(base)][0].numpy(), lent[i % len(base)][1])
            assert code == sst.SST_OK
            tickets.append(t)
        for i, t in enumerate(tickets):
            oc, ost = want[i % len(base)]
            code, info, cl = sst.sst_poll(g.ctx, t, -1, int(base[i % len(base)][0].size))
            assert code == sst.SST_OK
            assert {k: getattr(info.status, k) for k in ost} == ost, i
            assert_clusters_equal(cl, oc)
    finally:
        sst.sst_server_stop(g.ctx)
        g.close()
