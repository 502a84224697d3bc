"""The one-CTA-per-FED kernels and the choice among the batched kernels against the
oracle, where they can go wrong: FED records too long to stage and FEDs of several
digi chunks (dense, alternating and full strips), empty and non-canonical ones, more
FEDs than a look-back block, batches on either side of every line of the choice, with
and without amplitudes, and launches replayed from a graph between ordinary ones.
Integers are compared exactly, barycenters within the 1e-6 strip of the other parity
tests (both sides divide in binary32).
"""
import numpy as np
import pytest

import eventgen as eg
import oracle as orc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import _fedbuild as fb  # noqa: E402
import paper_2101_11489_gb300 as sst  # noqa: E402
from _gpu_util import Gpu, assert_clusters_equal, assert_digis_equal, orc_params  # noqa: E402

GAPS = sst.params(max_seq_holes=2, max_seq_bad=2, max_adj_bad=1)


def patterns(n_feds, seed):
    """Events of ordinary and of every kind of extreme density, as (raw, fed_len)."""
    rng = np.random.default_rng(seed)
    strips = np.arange(n_feds * 96 * 256)
    fed, chan = strips // (96 * 256), strips // 256
    adc = rng.integers(4, 256, strips.size).astype(np.uint8)
    low = rng.random(strips.size)
    masks = {
        "sparse": low < 0.01,
        "chunks": low < 0.30,  # several digi chunks a FED
        "alternating": strips % 2 == 0,  # a run header per digi: the longest records
        "full": np.ones(strips.size, bool),
        "empty": np.zeros(strips.size, bool),
        "mixed": low < np.array([0.004, 0.9, 0.05, 0.0])[fed % 4] * (1 + chan % 2),  # chunks of unequal channels
        "edge": (chan % 96 < 8) | (low < 0.001),  # 2,048 digis in a FED's first channels: at a chunk's size
    }
    out = {k: eg.pack_event(np.where(m, adc, 0).astype(np.uint8), m, n_feds) for k, m in masks.items()}
    out["non-canonical"] = fb.event(fb.non_canonical_feds(rng, n_feds))
    return out


def amplitudes(g, raw, fed_len, n_feds):
    d, c, st = g.oracle(raw, fed_len, n_feds)
    af, amp = orc.cluster_amplitudes(d, c, g.noise, g.gain, g.bad, orc_params(g.params))
    return c, st, af, amp


@pytest.fixture(scope="module", params=["default", "gaps"])
def small(request):
    calib = eg.make_calibration(4, 11, 0.03)
    g = Gpu(calib.noise, calib.gain, calib.bad, GAPS if request.param == "gaps" else None)
    yield g, patterns(4, 5)
    g.close()


def batch(g, events, n_feds, amps):
    sizes = [int(r.size) for r, _ in events]
    eoff = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    coff = np.concatenate([[0], np.cumsum([s // 2 + 1 for s in sizes])]).astype(np.int64)
    aoff = np.concatenate([[0], np.cumsum([4 * s + 256 for s in sizes])]).astype(np.int64)
    raw = torch.from_numpy(np.concatenate([r for r, _ in events])).cuda()
    fl = torch.from_numpy(np.concatenate([f for _, f in events]).astype(np.uint32).view(np.int32)).cuda()
    cb = sst.ClusterBuffers.alloc(int(coff[-1]), **({"amp_capacity": int(aoff[-1])} if amps else {}))
    if amps:
        cb.amp_off = torch.from_numpy(aoff).cuda()
    st = torch.zeros(len(events) * 4, dtype=torch.int32, device="cuda")
    sst.sst_batch(g.ctx, raw, torch.from_numpy(eoff).cuda(), fl, len(events), n_feds, torch.from_numpy(coff).cuda(),
                  cb.record(), st)
    torch.cuda.synchronize()
    sth = st.cpu().numpy().view(np.uint32).reshape(-1, 4)
    amp_all = cb.amplitudes() if amps else None
    return [(sth[k], cb.to_host(int(coff[k]), int(sth[k, 1])), amp_all, int(aoff[k])) for k in range(len(events))]


def check(got, want, amps):
    st, cl, amp_all, base = got
    c, ost, af, amp = want
    assert [int(v) for v in st] == [ost[k] for k in ("n_digi", "n_clusters", "flags", "n_bad_channels")]
    assert_clusters_equal({k: cl[k] for k in ("det", "first", "width", "charge", "barycenter")}, c)
    if amps:
        assert np.array_equal(cl["amp_first"].astype(np.int64) - base, af.astype(np.int64))
        assert np.array_equal(amp_all[base:base + amp.size], amp)


def test_per_event(small):
    g, pats = small
    for name, (raw, fl) in pats.items():
        dh, ch = g.event(raw, fl, 4)
        od, oc, _ = g.oracle(raw, fl, 4)
        assert_digis_equal(dh, od)
        assert_clusters_equal(ch, oc)


@pytest.mark.parametrize("amps", [False, True])
@pytest.mark.parametrize("n_events", [1, 3, 24, 25, 60])  # 96 FED records: a CTA each; 100: channel streams
def test_few_events(small, n_events, amps):
    g, pats = small
    pats = list(pats.values())
    want = [amplitudes(g, r, f, 4) for r, f in pats]
    got = batch(g, [pats[(5 * i + 1) % len(pats)] for i in range(n_events)], 4, amps)
    for i in range(n_events):
        check(got[i], want[(5 * i + 1) % len(pats)], amps)


@pytest.mark.parametrize("n_feds,n_events,amps", [
    (1, 239, False), (1, 240, False), (1, 99, True), (2, 49, True), (2, 50, True),
    (77, 9, False), (77, 10, False), (77, 15, False), (77, 16, False),  # 693 | 770 records, 15 | 16 events
    (150, 9, False), (150, 10, False), (149, 10, False),                # 9 | 10 events, 1,500 | 1,490 records
    (77, 11, True), (86, 10, True), (150, 10, True),                    # 847 | 860 records
    (400, 9, False), (401, 9, True),                                    # 3,600 | 3,609 records
])
def test_choice_of_kernel(n_feds, n_events, amps):
    calib = eg.make_calibration(n_feds, 17, 0.02)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    try:
        pats = patterns(n_feds, 6)
        pats = [pats[k] for k in ("sparse", "mixed", "non-canonical")]
        want = [amplitudes(g, r, f, n_feds) for r, f in pats]
        got = batch(g, [pats[i % 3] for i in range(n_events)], n_feds, amps)
        for i in range(n_events):
            check(got[i], want[i % 3], amps)
    finally:
        g.close()


@pytest.mark.parametrize("n_feds", [1023, 1024, 1025, 2049])
def test_look_back_blocks(n_feds):
    calib = eg.make_calibration(n_feds, 19, 0.0)
    g = Gpu(calib.noise, calib.gain, calib.bad)
    try:
        rng = np.random.default_rng(n_feds)
        mask = rng.random(n_feds * 96 * 256) < 0.002
        raw, fl = eg.pack_event(np.where(mask, rng.integers(60, 256, mask.size), 0).astype(np.uint8), mask, n_feds)
        dh, ch = g.event(raw, fl, n_feds)
        od, oc, _ = g.oracle(raw, fl, n_feds)
        assert_digis_equal(dh, od)
        assert_clusters_equal(ch, oc)
    finally:
        g.close()


def test_replays_between_ordinary_calls(small):
    """Per-event and few-event launches captured without a warm-up, replayed between
    ordinary ones on two streams: the launches' shared state is clean for each."""
    g, pats = small
    raw, fl = pats["mixed"]
    raw_t, fl_t = torch.from_numpy(raw).cuda(), torch.from_numpy(fl.astype(np.uint32).view(np.int32)).cuda()
    d, c = sst.DigiBuffers.alloc(int(raw.size), 4), sst.ClusterBuffers.alloc(int(raw.size) // 2 + 1)
    od, oc, _ = g.oracle(raw, fl, 4)

    def launch():
        drec = d.record()
        sst.sst_unpack(g.ctx, raw_t, fl_t, 4, drec)
        sst.sst_cluster(g.ctx, drec, 4, c.record())

    def compare():
        torch.cuda.synchronize()
        dh = d.to_host()
        assert_digis_equal(dh, od)
        assert_clusters_equal(c.to_host(0, dh["n_clusters"]), oc)
        for t in (d.strip, c.det, c.barycenter):
            t.zero_()
        torch.cuda.synchronize()

    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        launch()
    for step in "griggrrgii":
        if step == "g":
            graph.replay()
        elif step == "r":
            launch()
        else:
            with torch.cuda.stream(torch.cuda.Stream()):
                launch()
        compare()
    want = amplitudes(g, raw, fl, 4)
    for n in (3, 1, 4):  # batches of other sizes keep the graph's launches whole
        for got in batch(g, [(raw, fl)] * n, 4, False):
            check(got, want, False)
        graph.replay()
        compare()
