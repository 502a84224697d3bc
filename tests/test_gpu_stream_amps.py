"""Channel streams with amplitudes on every branch that forms them from the records again:
each launch shape, gains without a fixed-point multiplier (the records walked by another
routine, with other byte positions), FE units larger than the staging buffer, and corrupt
records, whose candidates are dropped; tiles and one-warp FE units.  Clusters, their
amp_first and every amplitude against the oracle.
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
from test_gpu_corrupt import corruptions  # noqa: E402
from test_gpu_feds import GAPS, amplitudes, batch, check, patterns  # noqa: E402

LOW = (0.2, 0.25, 0.2499, 1e-3)


def run(n_feds, n_events, low_gains=False, gaps=False, only=None, **tune):
    calib = eg.make_calibration(n_feds, 13, 0.03)
    gain = calib.gain.copy()
    if low_gains:
        gain[3::5] = np.resize(np.array(LOW, np.float32), gain[3::5].size)
    g = Gpu(calib.noise, gain, calib.bad, GAPS if gaps else None)
    try:
        if tune:
            sst.sst_set_tune(g.ctx, **tune)
        pats = patterns(n_feds, 8)
        events = [pats[k] for k in (only or sorted(pats))]
        events += [(r, f) for _, r, f in corruptions(*pats["sparse"])][:n_events - len(events)]
        want = [amplitudes(g, r, f, n_feds) for r, f in events]
        got = batch(g, [events[i % len(events)] for i in range(n_events)], n_feds, True)
        for i in range(n_events):
            check(got[i], want[i % len(events)], True)
    finally:
        g.close()


@pytest.mark.parametrize("gaps", [False, True])
@pytest.mark.parametrize("block", [128, 256])
@pytest.mark.parametrize("units", [1, 2])
def test_launch_shapes(block, units, gaps):
    run(4, 41, gaps=gaps, block=block, units_per_warp=units)


@pytest.mark.parametrize("block", [128, 256])
def test_tiles_with_gains_without_a_multiplier(block):
    run(4, 41, low_gains=True, block=block)


@pytest.mark.parametrize("low_gains", [False, True])
def test_units_of_one_warp(low_gains):  # 78 x 11 records: k_stream_fed, four FE units a warp
    run(78, 11, low_gains=low_gains, only=("alternating", "mixed", "non-canonical"))
