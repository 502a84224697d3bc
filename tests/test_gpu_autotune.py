"""The autotuner on batches whose kernel does not depend on the swept knobs: the context's
own tune stays, instead of whichever of equal launches was timed the fastest.
"""
import numpy as np
import pytest

import eventgen as eg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2101_11489_gb300 as sst  # noqa: E402
from _gpu_util import Gpu  # noqa: E402


def test_equal_launches_keep_the_tune():
    n_feds = 24
    w = eg.WORKLOADS[0]
    calib = eg.make_calibration(n_feds, w.seed, w.p_bad)
    e = eg.make_event(w, calib, 1, n_feds=n_feds)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    try:
        raw, fl = torch.from_numpy(e.raw).cuda(), torch.from_numpy(e.fed_len.view(np.int32)).cuda()
        off = torch.tensor([0, e.nbytes], dtype=torch.int64, device="cuda")
        room = torch.tensor([0, e.nbytes // 2 + 1], dtype=torch.int64, device="cuda")
        c, st = sst.ClusterBuffers.alloc(e.nbytes // 2 + 1), torch.zeros(4, dtype=torch.int32, device="cuda")
        keep = sst.sst_get_tune(g.ctx)
        for _ in range(8):  # one event: a block per FED record, whatever the knobs
            best, us = sst.sst_autotune(g.ctx, raw, off, fl, 1, n_feds, room, c.record(), st)
            assert best == keep and us > 0
            assert sst.sst_get_tune(g.ctx) == keep
    finally:
        g.close()
