"""The state that the CTAs of a one-CTA-per-FED launch share, against the oracle where it
can go wrong: the unpacking of one event beside the clustering of the one before on another
stream, more launches than the state has tags, and captured launches replayed after the
context has grown.
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
LAUNCHES = 2100  # twice round the 1,022 tags


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


@pytest.mark.parametrize("call", ["unpack", "noalloc", "batch"])
def test_more_launches_than_tags(gt, call):
    w, calib, g = gt
    sizes = (N_FEDS, 7, 33)
    evs = [eg.make_event(w, calib, 20 + k, n_feds=n) for k, n in enumerate(sizes)]
    dev = [device(e) for e in evs]
    bad = torch.zeros((), dtype=torch.int64, device="cuda")
    outs = []
    for e, n, (raw, fl) in zip(evs, sizes, dev):
        od, oc, ost = g.oracle(e.raw, e.fed_len, n)
        if call == "batch":
            c = sst.ClusterBuffers.alloc(e.nbytes // 2 + 1)
            st = torch.zeros(4, dtype=torch.int32, device="cuda")
            off = torch.tensor([0, e.nbytes], dtype=torch.int64, device="cuda")
            room = torch.tensor([0, e.nbytes // 2 + 1], dtype=torch.int64, device="cuda")
            status = torch.tensor([ost[k] for k in ("n_digi", "n_clusters", "flags", "n_bad_channels")],
                                  dtype=torch.int32, device="cuda")
            crec = c.record()
            outs.append((lambda raw=raw, fl=fl, n=n, st=st, off=off, room=room, crec=crec:
                         sst.sst_batch(g.ctx, raw, off, fl, 1, n, room, crec, st),
                         [(c.det, oc["det"].astype(np.int32)), (c.charge, oc["charge"].astype(np.int32)),
                          (st, status.cpu().numpy())], c))
        else:
            d = sst.DigiBuffers.alloc(e.nbytes, n)
            drec = d.record()
            f = ((lambda raw=raw, fl=fl, n=n, drec=drec: sst.sst_unpack(g.ctx, raw, fl, n, drec)) if call == "unpack" else
                 (lambda raw=raw, fl=fl, n=n, drec=drec: sst.sst_unpack_noalloc(raw, fl, n, drec)))
            outs.append((f, [(d.strip, od["strip"].astype(np.int32)), (d.adc, od["adc"]),
                             (d.chan_off, od["chan_off"].astype(np.int32))], d))
    outs = [(f, [(t.view(torch.int32) if t.dtype == torch.uint32 else t, torch.from_numpy(np.ascontiguousarray(v)).cuda())
                 for t, v in pairs], keep) for f, pairs, keep in outs]
    for i in range(LAUNCHES):
        f, pairs, _ = outs[(i * i + i // 3) % 3]
        f()
        for t, v in pairs:
            bad += (t[:v.numel()] != v).sum()
            t[:v.numel()] = -1 if t.dtype != torch.uint8 else 255
    torch.cuda.synchronize()
    assert int(bad) == 0


def test_replays_after_the_context_has_grown(gt):
    w, calib, g = gt
    e = eg.make_event(w, calib, 31, n_feds=N_FEDS)
    od, oc, _ = g.oracle(e.raw, e.fed_len, N_FEDS)
    raw, fl = device(e)
    d, c = sst.DigiBuffers.alloc(e.nbytes, N_FEDS), sst.ClusterBuffers.alloc(e.nbytes // 2 + 1)
    drec, crec = d.record(), c.record()

    def launch():
        sst.sst_unpack(g.ctx, raw, fl, N_FEDS, drec)
        sst.sst_cluster(g.ctx, drec, N_FEDS, crec)

    launch()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        launch()
    for n in (2, 9, 40):  # batches that grow the context's scratch
        for st, cl in g.batch([(e.raw, e.fed_len)] * n):
            assert_clusters_equal(cl, oc)
        for t in (d.strip, c.det):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        dh = d.to_host()
        assert_digis_equal(dh, od)
        assert_clusters_equal(c.to_host(0, dh["n_clusters"]), oc)


def test_capture_with_amplitudes_after_a_larger_batch_without(gt):
    """Once a batch with amplitudes has run, one of its size can be captured, whatever larger batches ran since."""
    w, calib, g = gt
    evs = [eg.make_event(w, calib, 40 + i, n_feds=N_FEDS) for i in range(2)]
    sizes = [e.nbytes for e in evs]
    eoff, coff, aoff = (torch.from_numpy(np.concatenate([[0], np.cumsum(v)]).astype(np.int64)).cuda()
                        for v in (sizes, [s // 2 + 1 for s in sizes], [4 * s for s in sizes]))
    raw = torch.from_numpy(np.concatenate([e.raw for e in evs])).cuda()
    fl = torch.from_numpy(np.concatenate([e.fed_len for e in evs]).view(np.int32)).cuda()
    cb = sst.ClusterBuffers.alloc(int(coff[-1]), amp_capacity=int(aoff[-1]))
    cb.amp_off = aoff
    st = torch.zeros(8, dtype=torch.int32, device="cuda")

    def launch():
        sst.sst_batch(g.ctx, raw, eoff, fl, 2, N_FEDS, coff, cb.record(), st)

    launch()
    g.batch([(e.raw, e.fed_len) for e in evs] * 20)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        launch()
    st.zero_()
    cb.det.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for i, e in enumerate(evs):
        _, oc, ost = g.oracle(e.raw, e.fed_len, N_FEDS)
        assert int(st[4 * i + 1]) == ost["n_clusters"]
        got = cb.to_host(int(coff[i]), ost["n_clusters"])
        assert_clusters_equal({k: got[k] for k in oc}, oc)


def test_a_batch_that_does_not_fit_leaves_the_context_usable(gt):
    """Scratch that could not grow (the GPU's memory is taken) is not used by the next, smaller batch."""
    w, calib, g = gt
    e = eg.make_event(w, calib, 50, n_feds=N_FEDS)
    n = 1 << 18  # needs about 4 GB of bookkeeping
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    fl = torch.zeros(1, dtype=torch.int32, device="cuda")  # (the call fails before anything is launched)
    st = torch.zeros(n * 4, dtype=torch.int32, device="cuda")
    c = sst.ClusterBuffers.alloc(16)
    for left in (2.5e9, 1.2e9, 3.5e9):  # a different array fails each time
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        taken = torch.empty(torch.cuda.mem_get_info()[0] - int(left), dtype=torch.uint8, device="cuda")
        try:
            with pytest.raises(sst.SstError) as err:
                sst.sst_batch(g.ctx, st.view(torch.uint8), off, fl, n, N_FEDS, off, c.record(), st)
            assert err.value.code == sst.SST_ERR_CUDA
        finally:
            del taken
            torch.cuda.empty_cache()
        for k in (1, 30):
            for got, cl in g.batch([(e.raw, e.fed_len)] * k):
                _, oc, ost = g.oracle(e.raw, e.fed_len, N_FEDS)
                assert got == ost
                assert_clusters_equal(cl, oc)


def test_memory_is_taken_by_the_calls_that_need_it():
    """A context that has no calibration (one that only unpacks) holds no candidate lists."""
    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    sst.sst_destroy(sst.sst_create(0, 8))  # (the library's own first use)
    before = free()
    ctx = sst.sst_create(0, 8)
    try:
        assert before - free() <= 8 << 20
    finally:
        sst.sst_destroy(ctx)
