"""sst_cluster on digis that sst_unpack does not write: repeated and descending strips (each
active digi is then its own candidate, up to 256 in a channel), in a FED of many digi
chunks between two ordinary ones; and digis of other channels within a channel's range,
which take no part.  And amplitude capacities at every kind of limit.
"""
import numpy as np
import pytest

import eventgen as eg
import oracle as orc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2101_11489_gb300 as sst  # noqa: E402
from _gpu_util import Gpu, assert_clusters_equal, orc_params  # noqa: E402

CH = 96


@pytest.fixture(scope="module")
def g():
    calib = eg.make_calibration(4, 41, 0.0)  # no bad strips: every strip of a high ADC is a seed
    gpu = Gpu(calib.noise, calib.gain, calib.bad)
    yield gpu
    gpu.close()


def cluster(g, strip, adc, chan_off, amps=False):
    n_feds = (chan_off.size - 1) // CH
    d = sst.DigiBuffers.alloc(max(strip.size, 1), n_feds)
    d.strip[:strip.size] = torch.from_numpy(strip.astype(np.int32)).cuda()
    d.adc[:adc.size] = torch.from_numpy(adc.astype(np.uint8)).cuda()
    d.chan_off.copy_(torch.from_numpy(chan_off.astype(np.int32)).cuda())
    d.status.zero_()
    c = sst.ClusterBuffers.alloc(strip.size + 1, amp_capacity=2 * strip.size + 256 if amps else 0)
    sst.sst_cluster(g.ctx, d.record(), n_feds, c.record())
    torch.cuda.synchronize()
    st = d.status.cpu().numpy().view(np.uint32)
    assert st[2] == 0
    return c.to_host(0, int(st[1])), c


def ordinary(seed, n_feds=1, occ=0.3):
    """Digis of n_feds FEDs of several digi chunks each, as sst_unpack writes them."""
    rng = np.random.default_rng(seed)
    mask = rng.random(n_feds * CH * 256) < occ
    strip = np.flatnonzero(mask)
    adc = rng.integers(20, 250, strip.size).astype(np.uint8)
    off = np.concatenate([[0], np.cumsum(np.bincount(strip // 256, minlength=n_feds * CH))])
    return strip, adc, off


@pytest.mark.parametrize("amps", [False, True])
@pytest.mark.parametrize("order", ["repeated", "descending"])
@pytest.mark.parametrize("per_channel", [20, 128, 129, 256])
def test_strips_out_of_order_stay_in_their_fed(g, order, per_channel, amps):
    feds = [ordinary(1), None, ordinary(2), ordinary(3)]
    k = np.arange(per_channel)
    one = np.full(per_channel, 5) if order == "repeated" else 255 - k
    feds[1] = ((np.arange(CH)[:, None] * 256 + one).ravel(), np.full(CH * per_channel, 200),
               np.arange(CH + 1) * per_channel)
    strip = np.concatenate([s + f * CH * 256 for f, (s, _, _) in enumerate(feds)])
    adc = np.concatenate([a for _, a, _ in feds])
    off = np.concatenate([[0]] + [np.diff(o) for _, _, o in feds]).cumsum()
    got, _ = cluster(g, strip, adc, off, amps)
    fed = got["det"] // CH
    p = orc_params(g.params)
    for f in (0, 2, 3):
        cut = slice(f * CH * 256, (f + 1) * CH * 256)
        s, a, o = feds[f]
        want = orc.cluster_event({"strip": s, "adc": a, "chan_off": o}, 1, g.noise[cut],
                                 g.gain[cut.start // 128:cut.stop // 128], g.bad[cut], p)
        want["det"] = want["det"] + f * CH
        assert_clusters_equal({n: v[fed == f] for n, v in got.items() if n != "amp_first"}, want)
    mine = fed == 1
    assert mine.sum() == CH * per_channel  # each digi on its own
    assert np.array_equal(got["det"][mine], CH + np.arange(CH).repeat(per_channel))
    assert np.array_equal(got["first"][mine], np.tile(one, CH)) and np.all(got["width"][mine] == 1)


@pytest.mark.parametrize("amps", [False, True])
@pytest.mark.parametrize("occ", [0.01, 0.3])
def test_digis_of_other_channels_take_no_part(g, occ, amps):
    """Strays anywhere in a channel's range, between linked strips too, change nothing."""
    strip, adc, off = ordinary(5, 4, occ)
    want = orc.cluster_event({"strip": strip, "adc": adc, "chan_off": off}, 4, g.noise, g.gain, g.bad, orc_params(g.params))
    rng = np.random.default_rng(6)
    at = np.sort(rng.integers(0, strip.size + 1, strip.size // 3))
    chan = np.searchsorted(off, np.minimum(at, strip.size - 1), side="right") - 1  # whose range each stray is in
    other = (chan + rng.choice([-1, 1, 7, 300, -200], at.size)) % 400  # (past the last channel too)
    other = np.where(other == chan, chan + 1, other)
    out_s, out_a = np.insert(strip, at, other * 256 + rng.integers(0, 256, at.size)), np.insert(adc, at, 253)
    n = np.diff(off) + np.bincount(chan, minlength=off.size - 1)
    got, _ = cluster(g, out_s, out_a, np.concatenate([[0], np.cumsum(n)]), amps)
    assert_clusters_equal({k: v for k, v in got.items() if k != "amp_first"}, want)


@pytest.mark.parametrize("occ", [0.01, 0.3])
@pytest.mark.parametrize("short", [0, 1, 1000, -1])
def test_amplitudes_up_to_the_capacity(g, occ, short):
    """Every cluster whose amplitudes end within the capacity has them, in a single FED too."""
    for n_feds in (1, 3):
        strip, adc, off = ordinary(8, n_feds, occ)
        digis = {"strip": strip, "adc": adc, "chan_off": off}
        p = orc_params(g.params)
        want = orc.cluster_event(digis, n_feds, g.noise, g.gain, g.bad, p)
        first, amp = orc.cluster_amplitudes(digis, want, g.noise, g.gain, g.bad, p)
        cap = max(amp.size - short, 1) if short >= 0 else 1  # (a capacity of 0 is refused)
        d = sst.DigiBuffers.alloc(strip.size, n_feds)
        d.strip.copy_(torch.from_numpy(strip.astype(np.int32)).cuda())
        d.adc.copy_(torch.from_numpy(adc).cuda())
        d.chan_off.copy_(torch.from_numpy(off.astype(np.int32)).cuda())
        d.status.zero_()
        c = sst.ClusterBuffers.alloc(want["det"].size, amp_capacity=cap)
        sst.sst_cluster(g.ctx, d.record(), n_feds, c.record())
        torch.cuda.synchronize()
        assert int(d.status[2]) == (sst.SST_EV_AMP_CAPACITY if cap < amp.size else 0)
        got = c.to_host(0, int(d.status[1]))
        assert_clusters_equal({k: v for k, v in got.items() if k != "amp_first"}, want)
        fits = first + want["width"] <= cap
        assert np.array_equal(got["amp_first"], np.where(fits, first, sst.NO_AMP))
        end = int((first + want["width"])[fits].max(initial=0))
        assert np.array_equal(c.amplitudes()[:end], amp[:end])
