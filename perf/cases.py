"""Performance cases of the library: what a program asks of it, through its public entry points.

A case is one pass of a program's inner loop: a detector event unpacked and clustered on its own, a batch of
events in device memory, or a batch in host memory.  The inputs are synthetic front-end records with the
geometry, noise, occupancy and cluster shapes of this repository's workloads, drawn on the GPU from the seed.

  listed()             the cases that are always measured
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs, calibration, context and output buffers: what a program has in hand
  run(state)           one pass; returns its outputs
  work(case)           bytes and operations a pass cannot do without
  exact(case, seed)    the computed numbers of run(), from plain torch in 64 bits

Fields of a case:
  api         "event" (sst_unpack + sst_cluster), "noalloc" (sst_unpack_noalloc), "batch" (sst_batch) or
              "host" (sst_batch_host)
  feds        FEDs of the detector part that is read out (96 channels of 256 strips each)
  events      events in the pass
  occ_lo/hi   fraction of strips with signal, uniform per event
  width       signal clusters are 1 .. width strips wide
  overlap     whether signal clusters may touch and overlap
  skew        FED occupancies differ by a factor log-uniform in [1/skew, skew]
  p_bad, sat  fractions of bad strips and of saturated signal strips
  holes, bad_run, adj   the clustering's hole and bad-strip limits
  amps        per-strip amplitudes of the clusters too; with positions: their local x too
  faults      fraction of FEDs absent from the readout, and of channels with a damaged record
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2101_11489_gb300 as sst

CHANNELS, STRIPS, APV = sst.CH_PER_FED, sst.STRIPS_PER_CH, sst.STRIPS_PER_APV
FE_UNITS, FE_CHANNELS, HEADER = 8, 12, 32

BASE = {"events": 1, "occ_lo": 0.015, "occ_hi": 0.015, "width": 5, "overlap": False, "skew": 1.0, "p_bad": 0.001,
        "sat": 0.0, "holes": 0, "bad_run": 1, "adj": 0, "amps": False, "positions": False, "faults": 0.0}


def listed():
    def case(name, api, feds, **kw):
        return {"name": name, "api": api, "feds": feds, **BASE, **kw}

    return [
        # a test beam or one readout crate: the smallest call, where launches and latency count
        case("event-8fed", "event", 8, occ_lo=0.01, occ_hi=0.01),
        # one partition of the detector, one event at a time
        case("event-50fed", "event", 50, occ_lo=0.01, occ_hi=0.01),
        # the whole detector, one event at a time, digis and clusters both wanted (online monitoring)
        case("event-440fed", "event", 440),
        # a data-acquisition process that may not allocate and only wants the digis
        case("noalloc-440fed", "noalloc", 440),
        # the batched entry point with a single event: a trigger that cannot wait for more
        case("batch1-440fed", "batch", 440),
        # a partition's events with damaged and absent records, holes and widening over bad strips allowed
        case("batch37-61fed-faults", "batch", 61, events=37, occ_lo=0.002, occ_hi=0.06, width=8, overlap=True,
             p_bad=0.02, sat=0.01, holes=1, bad_run=2, adj=1, faults=0.01),
        # everything a track fit wants: clusters, their amplitudes and their local positions
        case("batch16-440fed-hits", "batch", 440, events=16, occ_lo=0.005, occ_hi=0.04, amps=True, positions=True),
        # the batch that reconstruction runs on
        case("batch64-440fed", "batch", 440, events=64, occ_lo=0.005, occ_hi=0.04),
        # the same with FEDs of very different occupancy (forward and barrel modules)
        case("batch64-440fed-skew", "batch", 440, events=64, occ_lo=0.005, occ_hi=0.04, overlap=True, skew=4096.0),
        # high pile-up: dense events with wide, overlapping clusters, many bad and saturated strips
        case("batch256-440fed-dense", "batch", 440, events=256, occ_lo=0.05, occ_hi=0.05, width=12, overlap=True,
             p_bad=0.02, sat=0.03),
        # one event from pinned host memory to clusters in host memory
        case("host1-440fed", "host", 440),
        # a batch from pinned host memory to clusters in host memory
        case("host64-440fed", "host", 440, events=64, occ_lo=0.005, occ_hi=0.04),
    ]


def draw(rng: random.Random):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    c = dict(BASE)
    c["api"] = rng.choice(["event", "event", "noalloc", "batch", "batch", "batch", "batch", "host"])
    c["feds"] = max(1, min(440, round(log(1, 460))))
    most = {"event": 1, "noalloc": 1, "host": 64 * 440, "batch": 200 * 440}[c["api"]] // c["feds"]
    c["events"] = 1 if most <= 1 else round(log(1, min(256, most)))
    c["occ_lo"] = log(0.002, 0.06)
    c["occ_hi"] = min(0.06, c["occ_lo"] * rng.choice([1.0, 2.0, 8.0]))
    c["width"] = rng.randint(3, 12)
    c["overlap"] = rng.random() < 0.5
    if c["overlap"] and rng.random() < 0.3:
        c["skew"] = log(2, 4096)
    c["p_bad"] = log(0.0005, 0.02)
    c["sat"] = rng.choice([0.0, 0.0, 0.01, 0.03])
    if rng.random() < 0.3:
        c.update(holes=rng.randint(0, 2), bad_run=rng.randint(0, 3), adj=rng.randint(0, 2))
    if c["api"] in ("event", "batch") and rng.random() < 0.3:
        c["amps"] = True
        c["positions"] = rng.random() < 0.5
    if rng.random() < 0.2:
        c["faults"] = rng.uniform(0.001, 0.02)
    return c


# ---------------------------------------------------------------- inputs

def _generator(seed: int, stream: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + stream) & 0x7FFFFFFFFFFFFFFF)
    return g


def _calibration(case, seed):
    """Noise ~ U[3, 6] per strip, gain ~ U[0.8, 1.2] per APV, bad-strip flags, strip pitch per module."""
    g = _generator(seed, 0)
    n = case["feds"] * CHANNELS * STRIPS
    noise = torch.rand(n, generator=g, device="cuda") * 3.0 + 3.0
    gain = torch.rand(n // APV, generator=g, device="cuda") * 0.4 + 0.8
    bad = torch.rand(n, generator=g, device="cuda") < case["p_bad"]
    pitch = torch.rand(n // STRIPS, generator=g, device="cuda") * 125.0 + 80.0
    return noise, gain, bad, pitch


def _strips(case, seed, event, noise, gain):
    """ADC counts of one event's strips and which of them the front end records.

    Signal clusters share a Moyal-distributed charge over their strips; every strip has Gaussian noise; the
    front end keeps strips above twice their noise.  The signal is summed in fixed point, so that the same seed
    gives the same bytes."""
    g = _generator(seed, 1 + event)
    dev = "cuda"
    n_mod = case["feds"] * CHANNELS
    n = n_mod * STRIPS
    occ = random.Random(int(seed) * 7919 + event).uniform(case["occ_lo"], case["occ_hi"])
    n_cl = int(round(occ * n / (0.5 * (1 + case["width"]))))
    width = torch.randint(1, case["width"] + 1, (n_cl,), generator=g, device=dev)
    if case["skew"] > 1.0:
        fed_w = torch.exp((torch.rand(case["feds"], generator=g, device=dev, dtype=torch.float64) * 2 - 1) *
                          math.log(case["skew"]))
        edge = torch.cumsum(fed_w / fed_w.sum(), 0)
        fed = torch.searchsorted(edge, torch.rand(n_cl, generator=g, device=dev, dtype=torch.float64))
        mod = fed.clamp_(max=case["feds"] - 1) * CHANNELS + torch.randint(0, CHANNELS, (n_cl,), generator=g, device=dev)
    else:
        mod = torch.randint(0, n_mod, (n_cl,), generator=g, device=dev)
    first = (torch.rand(n_cl, generator=g, device=dev) * (STRIPS - width + 1)).long()
    first = torch.minimum(first, STRIPS - width)
    key = mod * STRIPS + first
    if not case["overlap"] and n_cl:
        key, order = torch.sort(key, stable=True)
        width = width[order]
        end = torch.cummax(key + width, 0).values
        keep = torch.ones_like(key, dtype=torch.bool)
        keep[1:] = key[1:] >= end[:-1]
        key, width = key[keep], width[keep]
    z = torch.randn(key.numel(), generator=g, device=dev, dtype=torch.float64)
    charge = (80.0 - 8.0 * torch.log((z * z).clamp_min(1e-300))).clamp_min(0.0)
    of = torch.repeat_interleave(torch.arange(key.numel(), device=dev), width)
    at = torch.arange(of.numel(), device=dev) - (torch.cumsum(width, 0) - width)[of]
    strip = key[of] + at
    weight = torch.randint(512, 1025, (of.numel(),), generator=g, device=dev)
    share = charge[of] * weight / torch.zeros_like(key).index_add_(0, of, weight)[of].clamp_min(1)
    share = share * gain[strip // APV].double()
    signal = torch.zeros(n, dtype=torch.int64, device=dev).index_add_(0, strip, (share * 65536).round().long())
    v = torch.round((signal.double() / 65536).float() + noise * torch.randn(n, generator=g, device=dev))
    adc = torch.where(v <= 253, v.clamp_min(0), torch.where(v <= 1023, 254.0, 255.0)).to(torch.uint8)
    if case["sat"] > 0:
        hit = (signal > 0) & (torch.rand(n, generator=g, device=dev) < case["sat"])
        code = 254 + (torch.rand(n, generator=g, device=dev) < 0.5).to(torch.uint8)
        adc = torch.where(hit, code, adc)
    recorded = adc.float() > 2.0 * noise
    present = torch.ones(case["feds"], dtype=torch.bool, device=dev)
    damaged = torch.zeros(n_mod, dtype=torch.bool, device=dev)
    if case["faults"] > 0:
        present = torch.rand(case["feds"], generator=g, device=dev) >= case["faults"]
        present[0] = True
        damaged = torch.rand(n_mod, generator=g, device=dev) < case["faults"]
        recorded &= present.repeat_interleave(CHANNELS * STRIPS)
    return adc, recorded, present, damaged


def _pack(case, adc, recorded, present, damaged):
    """The front end's FED records of one event (include/sst.h has the format): bytes and FED lengths."""
    dev, feds = "cuda", case["feds"]
    n_ch = feds * CHANNELS
    idx = torch.nonzero(recorded).flatten()
    brk = torch.ones_like(idx, dtype=torch.bool)
    brk[1:] = (idx[1:] != idx[:-1] + 1) | (idx[1:] % APV == 0)
    pos = torch.nonzero(brk).flatten()
    run = idx[pos]
    run_w = torch.diff(pos, append=torch.tensor([idx.numel()], device=dev))
    run_ch = run // STRIPS
    runs = torch.bincount(run_ch, minlength=n_ch)
    digis = torch.bincount(idx // STRIPS, minlength=n_ch)
    ch_len = 3 + 2 * runs + digis
    fe = ch_len.view(feds, FE_UNITS, FE_CHANNELS)
    fe_len = fe.sum(2)
    fe_pad = (fe_len + 7) // 8 * 8
    fed_len = (HEADER + fe_pad.sum(1) + 15) // 16 * 16 * present
    fed_off = torch.cumsum(fed_len, 0) - fed_len
    fe_off = fed_off[:, None] + HEADER + torch.cumsum(fe_pad, 1) - fe_pad
    ch_off = (fe_off[:, :, None] + torch.cumsum(fe, 2) - fe).reshape(-1)
    buf = torch.zeros(int(fed_len.sum()), dtype=torch.uint8, device=dev)
    head = torch.zeros((feds, HEADER), dtype=torch.uint8, device=dev)
    fed_id = torch.arange(feds, device=dev)
    for k, v in enumerate((0x53, 0x53, 0x54, 0x46)):
        head[:, k] = v
    head[:, 4], head[:, 5] = (fed_id & 255).to(torch.uint8), (fed_id >> 8).to(torch.uint8)
    head[:, 6], head[:, 7] = CHANNELS, FE_UNITS
    for k in range(4):
        head[:, 8 + k] = (fed_len >> (8 * k) & 255).to(torch.uint8)
    head[:, 16::2], head[:, 17::2] = (fe_len & 255).to(torch.uint8), (fe_len >> 8).to(torch.uint8)
    here = torch.nonzero(present).flatten()
    buf[fed_off[here, None] + torch.arange(HEADER, device=dev)] = head[here]
    ch_here = torch.nonzero(present.repeat_interleave(CHANNELS)).flatten()
    at = ch_off[ch_here]
    buf[at] = (ch_len[ch_here] & 255).to(torch.uint8)
    buf[at + 1] = (ch_len[ch_here] >> 8).to(torch.uint8)
    buf[at + 2] = torch.where(damaged[ch_here], 0, 0x5A).to(torch.uint8)
    run_end = torch.cumsum(2 + run_w, 0)
    before = torch.cat([run_end.new_zeros(1), run_end])[torch.cumsum(runs, 0) - runs]  # run bytes before the channel
    run_at = ch_off[run_ch] + 3 + run_end - (2 + run_w) - before[run_ch]
    buf[run_at] = (run & 255).to(torch.uint8)
    buf[run_at + 1] = run_w.to(torch.uint8)
    of = torch.cumsum(brk, 0) - 1
    buf[run_at[of] + 2 + torch.arange(idx.numel(), device=dev) - pos[of]] = adc[idx]
    return buf, fed_len.int()


def _events(case, seed, noise, gain):
    for e in range(case["events"]):
        adc, recorded, present, damaged = _strips(case, seed, e, noise, gain)
        yield adc, recorded, present, damaged


def _params(case):
    return sst.params(max_seq_holes=case["holes"], max_seq_bad=case["bad_run"], max_adj_bad=case["adj"])


def _capacities(case):
    """Digis, cluster records and amplitude bytes that a program reserves for one event, from the occupancy it expects
    (about 0.021 of the strips are recorded for their noise alone)."""
    strips = case["feds"] * CHANNELS * STRIPS
    digis = int(1.1 * strips * (case["occ_hi"] + 0.03)) + 512
    return digis, int(1.2 * strips * case["occ_hi"] / (0.5 * (1 + case["width"]))) + 256, digis


class Context:
    """An sst context that goes with the state that holds it."""

    def __init__(self, case, noise, gain, bad):
        self.handle = sst.sst_create(torch.cuda.current_device(), case["feds"])
        sst.sst_calib_upload(self.handle, noise.cpu().numpy(), gain.cpu().numpy(), bad.cpu().numpy().astype(np.uint8),
                             _params(case))

    def __del__(self):
        if getattr(self, "handle", None):
            sst.sst_destroy(self.handle)
            self.handle = None


def _zeroed(buffers):
    for v in vars(buffers).values():
        if isinstance(v, torch.Tensor):
            v.zero_()
        elif isinstance(v, np.ndarray):
            v.fill(0)
    return buffers


def prepare(case, seed):
    noise, gain, bad, pitch = _calibration(case, seed)
    packed = [_pack(case, *ev) for ev in _events(case, seed, noise, gain)]
    sizes = [int(r.numel()) for r, _ in packed]
    off = lambda v: np.concatenate([[0], np.cumsum(v)]).astype(np.int64)  # noqa: E731
    raw = torch.cat([r for r, _ in packed] + [torch.zeros(16, dtype=torch.uint8, device="cuda")])
    fed_len = torch.cat([f for _, f in packed])
    del packed
    s = {"case": dict(case), "raw": raw[:-16], "fed_len": fed_len}
    api, feds, events = case["api"], case["feds"], case["events"]
    digi_cap, clu_cap, amp_cap = _capacities(case)
    if api != "noalloc":
        s["ctx"] = Context(case, noise, gain, bad)
    if case["positions"]:
        sst.sst_pitch_upload(s["ctx"].handle, pitch.cpu().numpy())
    if api in ("event", "noalloc"):
        s["digis"] = _zeroed(sst.DigiBuffers.alloc(digi_cap, feds))
        s["digis_rec"] = s["digis"].record()
    if api == "host":
        def pinned(t):
            p = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            p.copy_(t)
            return p
        s["keep"] = [pinned(s.pop("raw")), pinned(s.pop("fed_len")), pinned(torch.from_numpy(off(sizes)))]
        s["raw"], s["fed_len"] = s["keep"][0].numpy(), s["keep"][1].numpy().view(np.uint32)
        s["event_off"] = s["keep"][2].numpy().view(np.uint64)
        s["clusters"] = _zeroed(sst.HostClusters.alloc(events * clu_cap, pinned=True))
        s["event_first"] = np.zeros(events + 1, np.uint64)
        s["status"] = np.zeros((events, 4), np.uint32)
        torch.cuda.synchronize()
        return s
    if api in ("event", "batch"):
        amp = events * amp_cap if case["amps"] else 0
        s["clusters"] = _zeroed(sst.ClusterBuffers.alloc(events * clu_cap, amp_capacity=amp))
        s["x"] = torch.zeros(events * clu_cap, device="cuda") if case["positions"] else None
    if api == "batch":
        s["event_off"] = torch.from_numpy(off(sizes)).cuda()
        s["clu_off"] = torch.from_numpy(off([clu_cap] * events)).cuda()
        s["status"] = torch.zeros(events * 4, dtype=torch.int32, device="cuda")
        if case["amps"]:
            s["clusters"].amp_off = torch.from_numpy(off([amp_cap] * events)).cuda()
    if api != "noalloc":
        s["clusters_rec"] = s["clusters"].record()
    return s


def run(state):
    c = state["case"]
    api, feds, events = c["api"], c["feds"], c["events"]
    if api == "host":
        o = state["clusters"]
        sst.sst_batch_host(state["ctx"].handle, state["raw"], state["event_off"], state["fed_len"], events, feds, o,
                           state["event_first"], state["status"])
        return {"det": o.det.view(np.int32), "first": o.first.view(np.int16), "width": o.width.view(np.int16),
                "charge": o.charge.view(np.int32), "barycenter": o.barycenter,
                "event_first": state["event_first"].view(np.int64), "status": state["status"].view(np.int32)}
    out = {}
    if api == "batch":
        sst.sst_batch(state["ctx"].handle, state["raw"], state["event_off"], state["fed_len"], events, feds,
                      state["clu_off"], state["clusters_rec"], state["status"])
        out["status"] = state["status"]
    else:
        d = state["digis"]
        if api == "noalloc":
            code = sst.sst_unpack_noalloc(state["raw"], state["fed_len"], feds, state["digis_rec"])
            if code != sst.SST_OK:
                raise sst.SstError(code, "sst_unpack_noalloc")
        else:
            sst.sst_unpack(state["ctx"].handle, state["raw"], state["fed_len"], feds, state["digis_rec"])
            sst.sst_cluster(state["ctx"].handle, state["digis_rec"], feds, state["clusters_rec"])
        out.update(strip=d.strip, adc=d.adc, chan_off=d.chan_off, chan_status=d.chan_status, status=d.status)
        if api == "noalloc":
            return out
    o = state["clusters"]
    out.update(det=o.det, first=o.first, width=o.width, charge=o.charge, barycenter=o.barycenter)
    if c["amps"]:
        out.update(amp=o.amp, amp_first=o.amp_first)
    if c["positions"]:
        sst.sst_local_x(state["ctx"].handle, o.det, o.barycenter, o.det.numel(), state["x"])
        out["x"] = state["x"]
    return out


# ---------------------------------------------------------------- what a pass needs

def work(case):
    """Expected bytes and operations: the records, each recorded strip's noise and bad-strip flag and each APV's
    gain once, and the outputs; about 20 operations per recorded strip (two thresholds, the gain correction, four
    sums) and 10 per cluster."""
    strips = case["feds"] * CHANNELS * STRIPS
    sigma = [3.0 + 3.0 * (k + 0.5) / 300 for k in range(300)]
    p_noise = sum(0.5 * math.erfc((math.floor(2 * s) + 0.5) / s / math.sqrt(2)) for s in sigma) / len(sigma)
    occ = 0.5 * (case["occ_lo"] + case["occ_hi"])
    clusters = occ / (0.5 * (1 + case["width"]))  # per strip
    share = [90.0 / w for w in range(1, case["width"] + 1) for _ in range(w)]  # charge of a signal strip
    p_signal = sum(0.5 * math.erfc((2 * s - q) / s / math.sqrt(2)) for s in sigma[::30] for q in share) / (10 * len(share))
    digis = 1 - math.exp(-occ) if case["overlap"] else occ
    digis = digis * p_signal + (1 - digis) * p_noise
    runs = clusters + p_noise * (1 - occ)
    keep = 1 - case["faults"]
    record = case["feds"] * (4 + HEADER + 3 * CHANNELS) + strips * (digis + 2 * runs)
    n = case["events"]
    nbytes = n * keep * record
    flops = 0.0
    if case["api"] in ("event", "noalloc"):
        nbytes += keep * 5 * strips * digis + case["feds"] * CHANNELS * 5
    if case["api"] != "noalloc":
        nbytes += strips * 5 * (1 - (1 - digis) ** n) + strips // APV * 4  # calibration, over all events once
        nbytes += n * keep * 16 * strips * clusters + n * 16
        flops = n * keep * strips * (20 * digis + 10 * clusters)
        if case["amps"]:
            nbytes += n * keep * strips * (digis + 4 * clusters)
        if case["positions"]:
            nbytes += n * keep * 4 * strips * clusters + case["feds"] * CHANNELS * 4
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same numbers in 64 bits

def _clusters64(case, adc, recorded, damaged, noise, gain, bad):
    """Kept clusters of one event in strip order: (first strip of the detector, barycenter in 64 bits).  Which strips
    and clusters pass is decided as the interface defines it (limits rounded once to 32 bits)."""
    dev = "cuda"
    idx = torch.nonzero(recorded & ~damaged.repeat_interleave(STRIPS) & ~bad).flatten()
    a = adc[idx].float()
    s = idx[a > 2.0 * noise[idx]]  # active strips
    if not s.numel():
        return s, s.double()
    a = adc[s].float()
    seed = a > 3.0 * noise[s]
    linked = torch.zeros_like(s, dtype=torch.bool)
    pair = torch.nonzero((s[1:] // STRIPS) == (s[:-1] // STRIPS)).flatten() + 1
    at, run, prev = s[pair] - 1, torch.zeros_like(pair), torch.full_like(pair, -1)
    low = s[pair - 1]
    while pair.numel():
        met = at == low
        linked[pair[met]] = True
        b = bad[at].long()
        run = torch.where(b == prev, run + 1, 1)
        go = ~met & (run <= torch.where(b == 1, case["bad_run"], case["holes"]))
        pair, at, run, prev, low = pair[go], at[go] - 1, run[go], b[go], low[go]
    of = torch.cumsum(~linked, 0) - 1  # candidate of each active strip
    begin = torch.nonzero(~linked).flatten()
    count = torch.diff(begin, append=torch.tensor([s.numel()], device=dev))
    n2 = torch.zeros(begin.numel(), device=dev)
    square = noise[s] * noise[s]
    for k in range(int(count.max())):  # summed strip by strip, in 32 bits
        more = count > k
        n2[more] = n2[more] + square[begin[more] + k]
    zero = torch.zeros(begin.numel(), dtype=torch.int64, device=dev)
    total = zero.clone().index_add_(0, of, adc[s].long())
    seeded = zero.clone().index_add_(0, of, seed.long()) > 0
    keep = seeded & (total.float() > 5.0 * torch.sqrt(n2))
    lo, hi = s[begin], s[begin + count - 1]
    for end, step in ((lo, -1), (hi, 1)):
        grow = torch.ones_like(keep)
        for _ in range(case["adj"]):
            nxt = (end + step).clamp(0, bad.numel() - 1)
            grow &= (nxt // STRIPS == end // STRIPS) & (nxt != end) & bad[nxt]
            end += step * grow.long()
    x = torch.floor(a / gain[s // APV] + 0.5).clamp_max(254).long()
    q = torch.where(a >= 254, adc[s].long(), x)
    q_sum = zero.clone().index_add_(0, of, q)
    moment = zero.clone().index_add_(0, of, (s - lo[of]) * q)
    start = (lo % STRIPS).double()
    bary = torch.where(q_sum > 0, start + 0.5 + moment.double() / q_sum.clamp_min(1).double(),
                       start + 0.5 * (hi - lo + 1).double())
    return lo[keep], bary[keep]


def exact(case, seed):
    if case["api"] == "noalloc":
        return None
    noise, gain, bad, pitch = _calibration(case, seed)
    bary, x, keep_bary = [], [], []
    for adc, recorded, present, damaged in _events(case, seed, noise, gain):
        lo, b = _clusters64(case, adc, recorded, damaged, noise, gain, bad)
        cap = _capacities(case)[1]
        slot = torch.zeros(cap, dtype=torch.float64, device="cuda")
        slot[:b.numel()] = b
        keep_bary.append(b)
        bary.append(slot)
        if case["positions"]:
            det = torch.zeros(cap, dtype=torch.int64, device="cuda")
            det[:b.numel()] = lo // STRIPS
            x.append((slot - 128.0) * pitch[det].double())
    bary = torch.cat(bary)
    if case["api"] == "host":  # the events' clusters back to back
        packed = torch.cat(keep_bary)
        bary.zero_()
        bary[:packed.numel()] = packed
    out = {"barycenter": bary}
    if case["positions"]:
        out["x"] = torch.cat(x)
    return out
