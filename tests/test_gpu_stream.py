"""The batched path's many-event kernel (one lane per channel record) against the
oracle, where it can go wrong: batches on either side of the sizes at which a warp
takes one event more, the CTA another round or the launch the other kernel; FE units
too large to stage (alternating strips); full and empty channels; corrupt and
non-canonical records; gains without a charge multiplier; hole and bad-strip limits;
every launch shape.  Integers are compared exactly, barycenters within the 1e-6
strip of the other parity tests (both sides divide in binary32).
"""
import numpy as np
import pytest

import eventgen as eg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import _fedbuild as fb  # noqa: E402
import paper_2101_11489_gb300 as sst  # noqa: E402
from _gpu_util import Gpu, assert_clusters_equal  # noqa: E402
from test_gpu_corrupt import corruptions  # noqa: E402

N_FEDS = 4
PARAMS = {"default": sst.params(), "h2b2a1": sst.params(max_seq_holes=2, max_seq_bad=2, max_adj_bad=1)}


def distinct_events(calib):
    """Events of very different density, one of alternating strips (its FE units exceed the staging buffer),
    one with every strip, one empty, one of non-canonical records, and the corrupt ones."""
    w = eg.WORKLOADS[0]
    n = N_FEDS * 96 * 256
    evs = [eg.make_event(w, calib, 90 + i, occupancy=o, n_feds=N_FEDS) for i, o in enumerate((0.005, 0.04, 0.3))]
    out = [(e.raw, e.fed_len) for e in evs]
    strips = np.arange(n)
    adc = (20 + strips * 37 % 236).astype(np.uint8)
    for mask in (strips % 2 == 0, np.ones(n, bool), np.zeros(n, bool), (strips // 256) % 5 == 0):
        out.append(eg.pack_event(np.where(mask, adc, 0).astype(np.uint8), mask, N_FEDS))
    out.append(fb.event(fb.non_canonical_feds(np.random.default_rng(3), N_FEDS)))
    return out + [(r, f) for _, r, f in corruptions(*out[1])]


def check(g, calib, n_events, tune=None):
    base = distinct_events(calib)
    want = [g.oracle(r, f, N_FEDS)[1:] for r, f in base]
    got = g.batch([base[i % len(base)] for i in range(n_events)])
    for i, (st, cl) in enumerate(got):
        oc, ost = want[i % len(base)]
        assert st == ost, i
        assert_clusters_equal(cl, oc)


@pytest.mark.parametrize("n_events", [7, 8, 9, 17, 64, 65, 255, 257])
def test_batch_sizes(n_events):
    calib = eg.make_calibration(N_FEDS, 3, 0.02)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    try:
        check(g, calib, n_events)
    finally:
        g.close()


@pytest.mark.parametrize("which", ["default", "h2b2a1"])
@pytest.mark.parametrize("block", [128, 256])
@pytest.mark.parametrize("units", [1, 2])
def test_launch_shapes(which, block, units):
    calib = eg.make_calibration(N_FEDS, 5, 0.05)
    g = Gpu(calib.noise, calib.gain, calib.bad, PARAMS[which])
    try:
        sst.sst_set_tune(g.ctx, block=block, units_per_warp=units)
        check(g, calib, 41)
    finally:
        g.close()


@pytest.mark.parametrize("gains", [(0.2, 0.25, 0.2499, 1e-3), (0.2500005, 0.2501, 0.3, 700.0), (1.0, 0.5, 2.0, 0.8)])
def test_gains_with_and_without_a_multiplier(gains):
    """Gains below 1/4 have no 32-bit multiplier: their tiles divide."""
    calib = eg.make_calibration(N_FEDS, 7, 0.01)
    gain = calib.gain.copy()
    gain[3::5] = np.resize(np.array(gains, np.float32), gain[3::5].size)
    calib = eg.Calibration(calib.noise, gain, calib.bad)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    try:
        check(g, calib, 16)
    finally:
        g.close()
