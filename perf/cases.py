"""What the trigger library is timed on: the calls that a trigger node makes,
from one short slice of one tower to a batch of 64 and the 2688-PMT array.

A case is a dict of plain values:
  via        the entry point: "batch" (trig_batch_run, all slices in one launch
             sequence), "each" (one trig_batch_run per slice), "noalloc"
             (trig_batch_run_noalloc), "events" (trig_batch_run_events),
             "towers" (trig_batch_run, then trig_array_select across the
             detectors), "engine" (trig_submit_slice / trig_poll on host
             buffers)
  detector   "nemo" (32 PMTs), "km3" (84 PMTs), "mix" (both, in turn) or
             "array" (nx * ny towers of 84 PMTs; a detector for each tower
             under "towers")
  slices     slices of a pass; slice_ns: the length of one
  khz_lo, khz_hi   hit rate of a PMT: the slices' rates are spread evenly over
             this range, in an order drawn from the seed
  muons      tracks crossing the detector in each slice; bursts: 10 ms
             bioluminescence bursts (500 kHz on 3 PMTs) in each slice
  halo       the submissions carry the halos of the neighbouring slices
  rule       "default", "level0" (N7TW1000 in front), "ladder" (N7TW1000, then
             [SC and AFC] or [FC and AFC], every seed fires) or "distinct"
             (the causal count over different PMTs)
  graph      replayed from the library's CUDA graph; tuned: the launch shape
             chosen by trig_autotune on these slices, as bench.py does, else
             the default shape

Every output is made of whole numbers (times, indexes, counts); none has a
rounding, so there are no values in 64 bits to compare them with.
"""
import math

import numpy as np
import torch

from paper_1411_3968_gb300 import _lib as trig

SLICE_NS = 200_000_000          # a time slice of the data acquisition
T_ORIGIN_NS = 1_000_000_000
PARAMS = dict(q_seed_adc=300, floor_tau_ns=20, tol_ns=20, n_num=6900, n_den=1499, corr_window_ns=3000, threshold=4,
              win_half_ns=3000, l0_hits=0, l0_window_ns=1000, l0_distinct_pmts=0, seed_rule=0, sc_window_ns=20,
              fc_window_ns=100, afc_window_ns=250, sc_dist_mm=1000, count_distinct_pmts=0)
RULES = {"default": {}, "level0": dict(l0_hits=7), "ladder": dict(l0_hits=7, seed_rule=1, threshold=1),
         "distinct": dict(count_distinct_pmts=1)}
BURST_NS, BURST_HZ, BURST_PMTS = 10_000_000, 500e3, 3


def _case(name, via, detector, slices, khz, **other):
    c = dict(name=name, via=via, detector=detector, nx=1, ny=1, slices=slices, slice_ns=SLICE_NS, khz_lo=khz[0],
             khz_hi=khz[1], muons=0, bursts=0, halo=True, rule="default", graph=False, tuned=False)
    c.update(other)
    return c


def listed():
    both = (50.0, 500.0)
    return [
        # a short slice from a real-time thread that may not allocate: launches and latency are all there is
        _case("nemo_5ms_noalloc", "noalloc", "nemo", 1, (50.0, 50.0), slice_ns=5_000_000, muons=5),
        # the NEMO Phase II tower's slice as it comes, one call
        _case("nemo_slice", "batch", "nemo", 1, (50.0, 50.0), muons=50),
        # one second of a KM3NeT-It tower with bioluminescence bursts, slice by slice
        _case("km3_5_slices", "each", "km3", 5, (55.0, 55.0), muons=40, bursts=1),
        # a node that serves several towers: a few uneven slices of odd length in one call, nothing tuned
        _case("mix_7_ragged", "batch", "mix", 7, (37.0, 411.0), slice_ns=33_333_337, muons=9),
        # the throughput workload: 64 uneven slices of both towers, replayed from a graph
        _case("mix_64", "batch", "mix", 64, both, halo=False, graph=True, tuned=True),
        # the 2688-PMT array's slice
        _case("array_2688", "batch", "array", 1, (55.0, 55.0), nx=8, ny=4, muons=1000, graph=True),
        # the Event Manager's payload of busy towers
        _case("mix_16_events", "events", "mix", 16, both, halo=False, graph=True),
        # the paper's ladder of coincidences and its distinct-PMT count
        _case("mix_16_ladder", "batch", "mix", 16, both, halo=False, rule="ladder", graph=True),
        _case("mix_16_distinct", "batch", "mix", 16, both, halo=False, rule="distinct", graph=True),
        # eight towers of one period, the selection across them and the readback of their windows
        _case("towers_8", "towers", "array", 1, (55.0, 55.0), nx=4, ny=2, muons=1000, graph=True),
        # the server: one slice from a tower's host buffers to its result, and three towers' slices together
        _case("serve_km3", "engine", "km3", 1, (55.0, 55.0), muons=10),
        _case("serve_mix_12", "engine", "mix", 12, (50.0, 55.0), muons=10),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    via = rng.choice(["batch", "batch", "batch", "each", "noalloc", "events", "towers", "engine"])
    detector = "array" if via == "towers" else rng.choice(["nemo", "km3", "mix", "mix", "array"])
    if via == "engine" and detector == "array":
        detector = "km3"
    nx, ny = (rng.randint(2, 8), rng.randint(1, 4)) if detector == "array" else (1, 1)
    if via == "towers":
        nx, ny = rng.randint(2, 4), rng.randint(1, 2)
    pmts = {"nemo": 32, "km3": 84, "mix": 58}.get(detector, 84 * nx * ny)
    lo = _log(rng, 20.0, 400.0)
    hi = min(500.0, lo * rng.choice([1.0, rng.uniform(1.0, 8.0)]))
    if detector == "array":                      # an array's PMTs run at their quiet rate
        lo = hi = rng.uniform(30.0, 60.0)
    slice_ns = rng.choice([SLICE_NS, int(_log(rng, 2e6, 2e8))])
    # no more hits than the largest listed case holds for its entry point
    most = {"batch": 2.3e8, "each": 5e7, "noalloc": 2e6, "events": 6e7, "towers": 8e6, "engine": 1.2e7}[via]
    if detector == "array":
        most = min(most, 1e6 if via == "noalloc" else 2.9e7)
    rule = rng.choice(["default", "default", "default", "level0", "ladder", "distinct"])
    if via in ("noalloc", "towers", "engine") or detector == "array":
        rule = "default"
    if rule != "default":
        most = min(most, 6e7)
    one = pmts * (lo + hi) / 2 * 1e3 * slice_ns * 1e-9
    if one > most:
        slice_ns = int(slice_ns * most / one)
        one = most
    cap = min(most / one, {"noalloc": 16, "engine": 16, "towers": 1}.get(via, 64), 8 if detector == "array" else 64)
    slices = max(1, int(_log(rng, 1.0, cap + 0.5))) if cap >= 1 else 1
    graph = via in ("batch", "events", "towers") and rng.random() < 0.6
    return dict(via=via, detector=detector, nx=nx, ny=ny, slices=slices, slice_ns=slice_ns, khz_lo=round(lo, 2),
                khz_hi=round(hi, 2), muons=rng.randint(0, 30), bursts=int(rng.random() < 0.2 and detector != "array"),
                halo=rng.random() < 0.7, rule=rule, graph=graph,
                tuned=graph and detector != "array" and rng.random() < 0.5)


# ----------------------------------------------------------------- detectors

def _tower(floors, xs, x0=0.0, y0=0.0, first_floor=0):
    """Floors 40 m apart, two PMTs at each x of the bar, odd floors turned by 90 degrees."""
    xyz, floor = [], []
    for k in range(floors):
        for x in xs:
            at = (x0 + x, y0, 40.0 * k) if k % 2 == 0 else (x0, y0 + x, 40.0 * k)
            xyz += [[round(v * 1000) for v in at]] * 2
            floor += [first_floor + k] * 2
    return xyz, floor


def _geometries(case):
    """(positions in mm, floor of each PMT, tower of each PMT) of the case's detectors."""
    nemo, km3 = _tower(8, (-3.0, 3.0)), _tower(14, (-3.0, 0.0, 3.0))
    if case["detector"] == "array":
        xyz, floor, tower = [], [], []
        for j in range(case["ny"]):
            for i in range(case["nx"]):
                t = j * case["nx"] + i
                a, b = _tower(14, (-3.0, 0.0, 3.0), 90.0 * i, 90.0 * j, 14 * t)
                xyz, floor, tower = xyz + a, floor + b, tower + [t] * len(b)
        found = [(xyz, floor, tower)]
    else:
        found = [(x, f, [0] * len(f)) for x, f in {"nemo": [nemo], "km3": [km3], "mix": [nemo, km3]}[case["detector"]]]
    return [(np.array(x, np.int32), np.array(f, np.uint32), np.array(t, np.uint32)) for x, f, t in found]


def _plan(case):
    """(detector, rate in kHz) of each slice, before the seed orders them."""
    n, kinds = case["slices"], 2 if case["detector"] == "mix" else 1
    step = (case["khz_hi"] - case["khz_lo"]) / n
    return [(k % kinds, case["khz_lo"] + (k + 0.5) * step) for k in range(n)]


# -------------------------------------------------------------------- inputs

def _muon_hits(xyz, n, lo, span, gen):
    """(PMT, time after lo, charge) of n straight downgoing tracks seen through the Cherenkov cone."""
    dev, f = "cuda", torch.float64
    pos = torch.tensor(xyz, dtype=f, device=dev) / 1000

    def uniform(*size):
        return torch.rand(size, dtype=f, device=dev, generator=gen)

    cos, phi = uniform(n, 1), 2 * math.pi * uniform(n, 1)
    sin = (1 - cos * cos).sqrt()
    along = torch.cat([sin * phi.cos(), sin * phi.sin(), -cos], 1)
    a, b = pos.min(0).values - 100, pos.max(0).values + 100
    at = a + (b - a) * uniform(n, 3)
    margin = min(10_000.0, span / 4)
    when = margin + (span - 2 * margin) * uniform(n, 1)
    v = pos[None] - at[:, None]
    reach = (v * along[:, None]).sum(2)
    d = (v - reach[..., None] * along[:, None]).norm(dim=2)
    light = torch.exp(-d / 40)
    pe = torch.poisson(3 * light, generator=gen) + 1
    theta = math.radians(41.0)
    t = when + ((reach - d / math.tan(theta)) + d / math.sin(theta) * 1.38) / 0.2998
    t = (t + 3 * torch.randn(t.shape, dtype=f, device=dev, generator=gen)).round()
    q = (100 * pe + 40 * pe.sqrt() * torch.randn(t.shape, dtype=f, device=dev, generator=gen)).round().clamp(1, 65535)
    seen = (d <= 100) & (uniform(*t.shape) < light) & (t >= 0) & (t < span)
    return seen.nonzero()[:, 1], t[seen].long(), q[seen].long()


def _hits(xyz, lo, span, khz, case, gen):
    """The hits of [lo, lo + span), grouped by PMT and in time order: records of 16 bytes as (n, 2) int64, offsets."""
    dev, f, pmts = "cuda", torch.float64, len(xyz)
    n = torch.poisson(torch.full((pmts,), khz * 1e-6 * span, dtype=f, device=dev), generator=gen).long()
    pmt = [torch.repeat_interleave(torch.arange(pmts, device=dev), n)]
    t = [(torch.rand(len(pmt[0]), dtype=f, device=dev, generator=gen) * span).long()]
    for _ in range(case["bursts"]):
        length = min(BURST_NS, span)
        begin, rows = torch.rand(2, dtype=f, device=dev, generator=gen), int(BURST_HZ * 1e-9 * length)
        some = torch.randperm(pmts, device=dev, generator=gen)[:BURST_PMTS]
        pmt.append(some.repeat(rows))
        t.append(((span - length) * begin[0] + length * torch.rand(len(pmt[-1]), dtype=f, device=dev, generator=gen)).long())
    pmt, t = torch.cat(pmt), torch.cat(t)
    q = (100 + 40 * torch.randn(len(t), device=dev, generator=gen)).round().clamp(1, 65535).long()
    if case["muons"]:
        p2, t2, q2 = _muon_hits(xyz, case["muons"], lo, float(span), gen)
        pmt, t, q = torch.cat([pmt, p2]), torch.cat([t, t2]), torch.cat([q, q2])
    key = ((pmt << 50) | (t << 16) | q).sort().values
    hits = torch.stack([((key >> 16) & ((1 << 34) - 1)) + lo, (key >> 50) | ((key & 0xffff) << 16)], 1)
    off = torch.searchsorted(key, torch.arange(pmts + 1, device=dev) << 50)
    return hits, off


def _most(case, pmts, khz, span):
    """A number of hits that a slice does not exceed."""
    n = pmts * khz * 1e-6 * span + case["bursts"] * BURST_PMTS * BURST_HZ * 1e-9 * min(BURST_NS, span)
    return int(n + 10 * math.sqrt(n)) + case["muons"] * pmts + 64


def _zeros(n):
    return torch.zeros(max(1, n), dtype=torch.int64, device="cuda")


_noalloc_stream = None          # the library's static scratch is one: its calls share a stream
_scratches = []                 # the program's scratch for its one stream, never freed: cached graphs copy into it


def _scratch(n):
    if not _scratches or _scratches[-1].numel() < n:
        _scratches.append(torch.empty(n + n // 4, dtype=torch.uint8, device="cuda"))
    return _scratches[-1]


def prepare(case, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    par = dict(PARAMS, slice_ns=case["slice_ns"], **RULES[case["rule"]])
    towers = case["via"] == "towers"
    geometries = _geometries(case)
    if towers:
        (xyz, floor, tower), = geometries
        dets = [trig.Detector(xyz[tower == b], floor[tower == b], par) for b in range(tower[-1] + 1)]
    else:
        dets = [trig.Detector(x, f, par, tower_id=w) for x, f, w in geometries]
    halo = dets[0].halo_ns if case["halo"] else 0
    plan = _plan(case)
    order = torch.randperm(len(plan), generator=torch.Generator().manual_seed(seed)).tolist()
    slices, most = [], []                         # (detector, t0, hits, offsets); the room for each one's hits
    for k, at in enumerate(order):
        kind, khz = plan[at]
        t0 = T_ORIGIN_NS + k * case["slice_ns"]
        hits, off = _hits(geometries[kind][0], t0 - halo, case["slice_ns"] + 2 * halo, khz, case, gen)
        if towers:
            for b, det in enumerate(dets):
                o = off[84 * b:84 * b + 85]
                own = hits[int(o[0]):int(o[-1])].clone()
                own[:, 1] -= 84 * b
                slices.append((det, t0, own, (o - o[0]).contiguous()))
                most.append(_most(case, 84, khz, case["slice_ns"] + 2 * halo))
        else:
            slices.append((dets[kind], t0, hits, off))
            most.append(_most(case, len(geometries[kind][0]), khz, case["slice_ns"] + 2 * halo))
    caps, win_cap = [m // 2 + 4096 for m in most], trig.win_cap_for(par)
    s = dict(case=case, dets=dets)
    if case["via"] == "engine":
        # a producer's page-locked slice buffers
        s["slices"] = [(d, t0, trig.pinned_copy(h.cpu().numpy().reshape(-1).view(trig.HIT_DTYPE)),
                        trig.pinned_copy(o.cpu().numpy().astype(np.uint64))) for d, t0, h, o in slices]
        # where the program keeps the records that it takes from the results
        s["triggers"], s["first"] = np.zeros((sum(caps), 2), np.int64), [sum(caps[:k]) for k in range(len(caps))]
        s["windows"] = np.zeros((len(caps), win_cap, 4), np.int64)
        s["counts"] = np.zeros((len(caps), 7), np.int64)
        torch.cuda.synchronize()
        return s
    # outputs: the slices' trigger lists, windows and counters, one buffer of each kind (zero past what a pass writes)
    s["inputs"] = slices
    s["triggers"], s["windows"], s["stats"] = _zeros(2 * sum(caps)), _zeros(4 * win_cap * len(slices)), _zeros(6 * len(slices))
    descs, first = [], 0
    for k, (det, t0, hits, off) in enumerate(slices):
        descs.append(trig.slice_dev(det, hits.data_ptr(), off.data_ptr(), len(hits), t0,
                                    s["triggers"].data_ptr() + 16 * first, caps[k],
                                    s["windows"].data_ptr() + 32 * win_cap * k, win_cap, s["stats"].data_ptr() + 48 * k))
        first += caps[k]
    s["descs"] = descs
    if case["tuned"]:
        for det in dets:
            mine = [d for d, one in zip(descs, slices) if one[0] is det]
            if mine:
                trig.trig_autotune(det, mine, torch.cuda.current_stream().cuda_stream)
    if case["via"] == "noalloc":
        global _noalloc_stream
        _noalloc_stream = _noalloc_stream or torch.cuda.Stream()
        torch.cuda.synchronize()
        return s
    if case["via"] == "events":
        s["events"] = _zeros(2 * sum(most))
        s["event_descs"], first = [], 0
        for n in most:
            s["event_descs"].append(trig.trig_slice_events(s["events"].data_ptr() + 16 * first, n))
            first += n
        n = trig.trig_batch_events_scratch_bytes(descs, s["event_descs"])
    else:
        n = trig.trig_batch_scratch_bytes(descs)
    s["scratch_bytes"], s["scratch"] = n, _scratch(n)
    if towers:
        s["array"] = trig.Array(dets)
        hit_cap = sum(most)
        s["seeds"], s["array_windows"], s["array_stats"] = _zeros(2 * sum(caps)), _zeros(4 * win_cap), _zeros(5)
        s["fragments"], s["readback"] = _zeros(win_cap * len(dets) + 1), _zeros(2 * hit_cap)
        s["out"] = trig.trig_array_out(s["seeds"].data_ptr(), sum(caps), s["array_windows"].data_ptr(), win_cap,
                                       s["fragments"].data_ptr(), s["readback"].data_ptr(), hit_cap,
                                       s["array_stats"].data_ptr())
        n = trig.trig_array_scratch_bytes(s["array"], descs, s["out"])
        s["array_scratch_bytes"], s["array_scratch"] = n, torch.empty(n, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------- run

def _serve(s):
    for det, t0, hits, off in s["slices"]:
        trig.trig_submit_slice(det, t0, hits, off)
    for k, (det, _, _, _) in enumerate(s["slices"]):
        r = trig.trig_poll(det, -1)
        nt, nw = len(r.triggers), len(r.windows)
        s["triggers"][s["first"][k]:s["first"][k] + nt] = r.triggers.view(np.int64).reshape(nt, 2)
        s["windows"][k, :nw] = r.windows.view(np.int64).reshape(nw, 4)
        s["counts"][k] = r.t0, r.status, r.flags, r.n_hits, r.n_seeds, nt, nw
    return dict(triggers=s["triggers"], windows=s["windows"], counts=s["counts"])


def run(s):
    via, flags = s["case"]["via"], trig.TRIG_RUN_GRAPH if s["case"]["graph"] else 0
    if via == "engine":
        return _serve(s)
    descs, out = s["descs"], dict(triggers=s["triggers"], windows=s["windows"], stats=s["stats"])
    if via == "noalloc":
        trig.trig_batch_run_noalloc(descs, _noalloc_stream.cuda_stream)
        return out
    stream, scratch, n = torch.cuda.current_stream().cuda_stream, s["scratch"].data_ptr(), s["scratch_bytes"]
    if via == "each":
        for d in descs:
            trig.trig_batch_run([d], scratch, n, stream, flags)
    elif via == "events":
        trig.trig_batch_run_events(descs, s["event_descs"], scratch, n, stream, flags)
        out["events"] = s["events"]
    else:
        trig.trig_batch_run(descs, scratch, n, stream, flags)
    if via == "towers":
        trig.trig_array_select(s["array"], descs, s["out"], s["array_scratch"].data_ptr(), s["array_scratch_bytes"], stream)
        out.update(seeds=s["seeds"], array_windows=s["array_windows"], fragments=s["fragments"],
                   readback=s["readback"], array_stats=s["array_stats"])
    return out


# ---------------------------------------------------------------------- work

def work(case):
    """Each hit and offset read once, each trigger, window and event hit written once, at the rates expected of
    Poisson hits; operations: a difference and a comparison for each pair of a seed and a hit within its causal range
    (3 us of the detector's hits)."""
    total = {"bytes": 0.0, "flops": 0.0}
    geometries = _geometries(case)
    span = case["slice_ns"] + (2 * 3000 if case["halo"] else 0)
    for kind, khz in _plan(case):
        floor = geometries[kind][1]
        pmts, mates, ghz = len(floor), int((floor == floor[0]).sum()) - 1, khz * 1e-6
        hits = pmts * ghz * span + case["bursts"] * BURST_PMTS * BURST_HZ * 1e-9 * min(BURST_NS, span)
        if case["rule"] == "ladder":
            seed = (1 - math.exp(-2 * mates * ghz * 100)) * (1 - math.exp(-4 * (mates + 1) * ghz * 250))
        else:
            seed = 1 - math.exp(-2 * mates * ghz * 20)
        fired = hits * seed
        lone = math.exp(-6000 * fired / span)     # share of the triggers that end a window, and of the time outside
        out = 16 * fired + 32 * fired * lone + 48
        if case["via"] == "events":
            out += 16 * hits * (1 - lone)
        if case["via"] == "towers":
            out += 16 * hits / 4                  # a quarter of the hits is read back at the quiet rate
        total["bytes"] += 16 * hits + 8 * (pmts + 1) + out
        total["flops"] += 2 * fired * pmts * ghz * 3000
    return total
