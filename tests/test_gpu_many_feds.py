"""Detectors larger than the whole one, on either side of the lines drawn by FEDs, against the
oracle: batches (the calibration no longer fits the L2) and single events of sparse and
dense FEDs (above three FEDs an SM the clustering's tile is the smaller one).
"""
import numpy as np
import pytest

import eventgen as eg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from _gpu_util import Gpu, assert_clusters_equal, assert_digis_equal  # noqa: E402
from test_gpu_feds import patterns  # noqa: E402


@pytest.mark.parametrize("n_feds,n_events", [(640, 10), (641, 10), (641, 13), (641, 14), (641, 23), (641, 24), (1030, 3)])
def test_choice_above_the_whole_detector(n_feds, n_events):  # 8,333 | 8,974 records; 23 | 24 events
    calib = eg.make_calibration(n_feds, 29, 0.01)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    try:
        rng = np.random.default_rng(n_feds + n_events)
        evs = []
        for occ in (0.003, 0.01):
            mask = rng.random(n_feds * 96 * 256) < occ
            evs.append(eg.pack_event(np.where(mask, rng.integers(20, 256, mask.size), 0).astype(np.uint8), mask, n_feds))
        want = [g.oracle(r, f, n_feds)[1:] for r, f in evs]
        for i, (st, cl) in enumerate(g.batch([evs[k % 2] for k in range(n_events)])):
            oc, ost = want[i % 2]
            assert st == ost
            assert_clusters_equal(cl, oc)
    finally:
        g.close()


@pytest.mark.parametrize("n_feds", [456, 457])
def test_dense_and_sparse_feds_of_one_event(n_feds):
    calib = eg.make_calibration(n_feds, 31, 0.01)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    try:
        pats = patterns(n_feds, 9)
        for raw, fl in (pats["mixed"], pats["edge"]):
            dh, ch = g.event(raw, fl, n_feds)
            od, oc, _ = g.oracle(raw, fl, n_feds)
            assert_digis_equal(dh, od)
            assert_clusters_equal(ch, oc)
    finally:
        g.close()
