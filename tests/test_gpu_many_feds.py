"""Batches of detectors larger than the whole one (the calibration no longer fits the L2), on
either side of the lines between the batched kernels, against the oracle.
"""
import numpy as np
import pytest

import eventgen as eg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from _gpu_util import Gpu, assert_clusters_equal  # noqa: E402


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
