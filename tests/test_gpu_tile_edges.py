"""The tile pass of the default rule where its phases can go wrong: floor
cells (tau at and around powers of two, 0 and the largest), seed lists that
hold every hit, detectors at the edges of the shared-memory dt table and of
the bucketed path, equal times, and tile fills around a full tile.  Whole
numbers, equal to the oracle's."""
import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    import paper_1411_3968_gb300 as p
    from paper_1411_3968_gb300 import build
    build.build()
    p.load()
    torch.cuda.init()
    return p


def _detector(n_pmt, per_floor=6):
    k = np.arange(n_pmt)
    xyz = np.stack([1000 * (k % per_floor), np.zeros_like(k), 40_000 * (k // per_floor)], 1).astype(np.int32)
    return xyz, (k // per_floor).astype(np.uint32)


def _hits(rng, n, n_pmt, lo, hi, step=1):
    hits = np.zeros(n, workload.HIT_DTYPE)
    hits["t"] = lo + rng.integers(0, max(1, (hi - lo) // step), n) * step
    hits["pmt"] = rng.integers(0, n_pmt, n)
    hits["charge"] = rng.integers(1, 400, n)
    hits = np.sort(hits, order=["pmt", "t", "charge"], kind="stable")
    off = np.zeros(n_pmt + 1, np.uint64)
    np.cumsum(np.bincount(hits["pmt"], minlength=n_pmt), out=off[1:])
    return hits, off


@pytest.mark.parametrize("shape", [(2048, 16, 90), (1024, 4, 75), (4096, 8, 60)])
@pytest.mark.parametrize("n_pmt,n,slice_ns,step,extra", [
    (32, 6000, 300_000, 1, dict(floor_tau_ns=0)),
    (32, 6000, 300_000, 1, dict(floor_tau_ns=1)),
    (84, 9000, 300_000, 1, dict(floor_tau_ns=31)),
    (84, 9000, 300_000, 1, dict(floor_tau_ns=32)),
    (84, 500, 2_000_000, 1, dict(floor_tau_ns=60_000)),
    (84, 9000, 300_000, 1, dict(q_seed_adc=0)),
    (84, 4000, 200_000, 40, dict(q_seed_adc=150)),         # many equal times
    (1, 900, 900_000, 1, dict(q_seed_adc=300, threshold=1)),
    (96, 9000, 400_000, 1, {}),
    (97, 9000, 400_000, 1, {}),
    (128, 9000, 400_000, 1, {}),
    (129, 9000, 400_000, 1, {}),
    (129, 9000, 400_000, 1, dict(q_seed_adc=0)),
    (84, 30_000, 150_000, 1, {}),                            # hundreds of keys in each scan range
    (32, 2000, 40_000_000, 1, dict(threshold=1)),            # a few hits in the widest tiles
])
def test_tile_pass_edges(pkg, params, shape, n_pmt, n, slice_ns, step, extra):
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(n_pmt * 1000 + n))
    par = dict(params, slice_ns=slice_ns, **extra)
    halo = max(par["corr_window_ns"], par["win_half_ns"], par["floor_tau_ns"])
    t0 = 1_000_000
    xyz, floor = _detector(n_pmt)
    hits, off = _hits(rng, n, n_pmt, t0 - halo, t0 + slice_ns + halo, step)
    old = pkg.trig_get_tile_config()
    try:
        pkg.trig_set_tile_config(*shape)
        det = pkg.Detector(xyz, floor, par)
        b = DeviceBatch([SliceIn(det, t0, hits, off)])
        b.run()
        (stats, trig, win), = b.results()
    finally:
        pkg.trig_set_tile_config(*old)
    ref = oracle.run(xyz, floor, par, hits, [t0])[0]
    assert int(stats["status"]) == 0
    assert int(stats["n_seeds"]) == len(ref.seeds) and len(trig) == len(ref.triggers) and len(win) == len(ref.windows)
    for f in ("t", "pmt", "charge", "count"):
        assert np.array_equal(trig[f], ref.triggers[f]), f
    for f in ("lo", "hi", "n_hits", "n_triggers"):
        assert np.array_equal(win[f], ref.windows[f]), f
    det.close()


@pytest.mark.parametrize("n_pmt", [84, 129, 336])
@pytest.mark.parametrize("cluster_ns", [40, 4_000, 30_000])
@pytest.mark.parametrize("rule", [{}, dict(seed_rule=1, l0_hits=7, l0_window_ns=1000, threshold=1)])
def test_bursts_split_tiles(pkg, params, n_pmt, cluster_ns, rule):
    """Clusters that overfill tiles of every path, at the start, inside and at
    the end of the slice: the pieces' seeds, ranks and windows are the
    oracle's."""
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(n_pmt + cluster_ns))
    par = dict(params, slice_ns=600_000, **rule)
    t0, n = 1_000_000, 9000
    xyz, floor = _detector(n_pmt)
    hits, _ = _hits(rng, n, n_pmt, t0 - 3000, t0 + par["slice_ns"] + 3000)
    for at, share in ((t0, 0), (t0 + 250_000, 1500), (t0 + par["slice_ns"] - cluster_ns, 3000)):
        hits["t"][share:share + 1500] = at + rng.integers(0, cluster_ns, 1500)
    hits = np.sort(hits, order=["pmt", "t", "charge"], kind="stable")
    off = np.zeros(n_pmt + 1, np.uint64)
    np.cumsum(np.bincount(hits["pmt"], minlength=n_pmt), out=off[1:])
    det = pkg.Detector(xyz, floor, par)
    b = DeviceBatch([SliceIn(det, t0, hits, off)], events=True)
    old = pkg.trig_get_tile_config()
    for events, shape in ((True, (2048, 16, 90)), (False, (2048, 16, 90)), (False, (4096, 16, 95))):
        pkg.trig_set_tile_config(*shape)
        try:
            b.set_events(events)
            b.run()
            (stats, trig, win), = b.results()
        finally:
            pkg.trig_set_tile_config(*old)
        ref = oracle.run(xyz, floor, par, hits, [t0])[0]
        assert int(stats["status"]) == 0, shape
        assert int(stats["n_seeds"]) == len(ref.seeds) and len(trig) == len(ref.triggers)
        for f in ("t", "pmt", "charge", "count"):
            assert np.array_equal(trig[f], ref.triggers[f]), (shape, f)
        for f in ("lo", "hi", "n_hits", "n_triggers"):
            assert np.array_equal(win[f], ref.windows[f]), (shape, f)
        if events:
            (ev, n_ev, full), = b.event_hits()
            want = oracle.events(hits, ref.windows)
            assert not full and n_ev == len(want)
            for f in ("t", "pmt", "charge"):
                assert np.array_equal(ev[f], want[f]), (shape, f)
    det.close()


def test_more_slices_than_one_descriptor_launch_carries(pkg, params):
    """70 slices (k_put carries 64 at a time), plain and as a graph replay,
    empty ones among them: every slice the oracle's."""
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(70))
    par = dict(params, slice_ns=50_000)
    xyz, floor = _detector(84)
    det = pkg.Detector(xyz, floor, par)
    slices = []
    for k in range(70):
        t0 = 1_000_000 + k * par["slice_ns"]
        hits, off = _hits(rng, 0 if k % 23 == 5 else 300 + 20 * k, 84, t0 - 3000, t0 + par["slice_ns"] + 3000)
        slices.append(SliceIn(det, t0, hits, off))
    b = DeviceBatch(slices)
    for graph in (False, True, True):
        b.run(graph=graph)
        for s, (stats, trig, win) in zip(slices, b.results()):
            ref = oracle.run(xyz, floor, par, s.hits, [s.t0])[0]
            assert int(stats["status"]) == 0 and int(stats["n_hits"]) == len(s.hits)
            assert int(stats["n_seeds"]) == len(ref.seeds)
            for f in ("t", "pmt", "charge", "count"):
                assert np.array_equal(trig[f], ref.triggers[f]), f
            for f in ("lo", "hi", "n_hits", "n_triggers"):
                assert np.array_equal(win[f], ref.windows[f]), f
    det.close()


@pytest.mark.parametrize("n_pmt,n", [(84, 2_750_000), (336, 1_635_000)])
def test_noalloc_takes_the_largest_batches(pkg, params, n_pmt, n):
    """A slice close to what the static scratch holds (about 24 bytes a hit, 40
    above 128 PMTs) is planned with larger tiles and segments instead of
    being refused."""
    import torch
    from paper_1411_3968_gb300 import _lib
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(n))
    par = dict(params, slice_ns=200_000_000)
    xyz, floor = _detector(n_pmt)
    det = pkg.Detector(xyz, floor, par)
    hits, off = _hits(rng, n, n_pmt, 1_000_000 - 3000, 1_000_000 + par["slice_ns"] + 3000)
    b = DeviceBatch([SliceIn(det, 1_000_000, hits, off)])
    b.run()
    (stats, trig, win), = b.results()
    b.trig[0].zero_()
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    _lib.trig_batch_run_noalloc(b.descs, st.cuda_stream)
    (stats2, trig2, win2), = b.results()
    assert int(stats2["status"]) == 0 and stats2 == stats
    assert np.array_equal(trig2, trig) and np.array_equal(win2, win)
    det.close()


_OWN_SHAPE = """
import sys
sys.path[:0] = {path!r}
import numpy as np, torch
import paper_1411_3968_gb300 as pkg, workload
from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
pkg.load()
torch.cuda.init()
rng = np.random.Generator(np.random.PCG64({n}))
k = np.arange(2016)
xyz = np.stack([1000 * (k % 6), np.zeros_like(k), 40_000 * (k // 6)], 1).astype(np.int32)
par = dict({par!r}, slice_ns={slice_ns})
hits = np.zeros({n}, workload.HIT_DTYPE)
hits["t"] = 1_000_000 - 3000 + rng.integers(0, par["slice_ns"] + 6000, {n})
hits["pmt"] = rng.integers(0, 2016, {n})
hits["charge"] = rng.integers(1, 320, {n})
hits = np.sort(hits, order=["pmt", "t", "charge"], kind="stable")
off = np.zeros(2017, np.uint64)
np.cumsum(np.bincount(hits["pmt"], minlength=2016), out=off[1:])
b = DeviceBatch([SliceIn(pkg.Detector(xyz, (k // 6).astype(np.uint32), par), 1_000_000, hits, off)])
res = []
for shape in (None, (2048, 16, 90)):
    if shape:
        pkg.trig_set_tile_config(*shape)
    b.run()
    res.append(b.results()[0])
    b.trig[0].zero_()
(s0, t0, w0), (s1, t1, w1) = res
assert int(s0["status"]) == 0 and s0 == s1 and len(t0) > 1000
assert np.array_equal(t0, t1) and np.array_equal(w0, w1)
print("same")
"""


@pytest.mark.parametrize("slice_ns,n", [(32_000_000, 4_800_000), (60_000_000, 5_400_000)])
def test_own_shape_of_dense_arrays(pkg, params, slice_ns, n):
    """The library's own shape above and below the rate at which halos take a
    quarter of a tile (a process of its own: no shape is set before): what a
    set shape gives."""
    import subprocess
    import sys
    src = _OWN_SHAPE.format(path=sys.path, par=dict(params), slice_ns=slice_ns, n=n)
    r = subprocess.run([sys.executable, "-c", src], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stderr[-2000:]


@pytest.mark.parametrize("shape", [(4096, 8, 90), (2048, 16, 90)])
@pytest.mark.parametrize("n_pmt,rule", [(84, {}), (129, {}), (84, dict(count_distinct_pmts=1, threshold=1)),
                                        (84, dict(l0_hits=2, l0_window_ns=1000, l0_distinct_pmts=1, threshold=1))])
def test_tiles_of_equal_records(pkg, params, shape, n_pmt, rule):
    """Nearly a tile of hits at one time on one PMT (some charges equal too),
    and at one time and the next on the floor's other PMTs: every seed's place
    among its equals, in a time that grows with their square (12 ms for 3800
    of them) and not with their cube (0.75 s for 1750)."""
    import torch
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(shape[0] + n_pmt))
    par = dict(params, slice_ns=300_000, **rule)
    t0 = 1_000_000
    xyz, floor = _detector(n_pmt)
    hits, _ = _hits(rng, shape[0] - 600, n_pmt, t0 + 100_000, t0 + 100_001)
    hits["pmt"] = 7
    hits["charge"] = rng.integers(300, 900, len(hits))
    hits["t"][::9] += 1
    hits["pmt"][::9] = 6 + 2 * rng.integers(0, 2, len(hits[::9]))
    other, _ = _hits(rng, 600, n_pmt, t0 - 3000, t0 + par["slice_ns"] + 3000)
    hits = np.sort(np.concatenate([hits, other]), order=["pmt", "t", "charge"], kind="stable")
    off = np.zeros(n_pmt + 1, np.uint64)
    np.cumsum(np.bincount(hits["pmt"], minlength=n_pmt), out=off[1:])
    det = pkg.Detector(xyz, floor, par)
    b = DeviceBatch([SliceIn(det, t0, hits, off)])
    old = pkg.trig_get_tile_config()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    try:
        pkg.trig_set_tile_config(*shape)
        b.run()
        torch.cuda.synchronize()
        ev[0].record()
        b.run()
        ev[1].record()
        (stats, trig, win), = b.results()
    finally:
        pkg.trig_set_tile_config(*old)
    ref = oracle.run(xyz, floor, par, hits, [t0])[0]
    assert int(stats["status"]) == 0
    assert int(stats["n_seeds"]) == len(ref.seeds) and len(trig) == len(ref.triggers) and len(win) == len(ref.windows)
    for f in ("t", "pmt", "charge", "count"):
        assert np.array_equal(trig[f], ref.triggers[f]), f
    for f in ("lo", "hi", "n_hits", "n_triggers"):
        assert np.array_equal(win[f], ref.windows[f]), f
    assert ev[0].elapsed_time(ev[1]) < 100.0
    det.close()


@pytest.mark.parametrize("n_pmt", [84, 129])
@pytest.mark.parametrize("l0_hits", [2600, 1900, 1300, 40])
def test_level0_over_crowded_buckets(pkg, params, n_pmt, l0_hits):
    """Three clusters of 1200 hits in 24 ns, 700 ns apart, under a level 0 that
    none, some or all of their hits pass: each seed's windows are searched in
    a time that does not grow with the clusters' square."""
    import torch
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(l0_hits + n_pmt))
    par = dict(params, slice_ns=300_000, l0_hits=l0_hits, l0_window_ns=1000, q_seed_adc=0, threshold=1)
    t0 = 1_000_000
    xyz, floor = _detector(n_pmt)
    hits, _ = _hits(rng, 3900, n_pmt, t0 - 3000, t0 + par["slice_ns"] + 3000)
    for k in range(3):
        hits["t"][1200 * k:1200 * (k + 1)] = t0 + 100_000 + 700 * k + rng.integers(0, 24, 1200)
    hits = np.sort(hits, order=["pmt", "t", "charge"], kind="stable")
    off = np.zeros(n_pmt + 1, np.uint64)
    np.cumsum(np.bincount(hits["pmt"], minlength=n_pmt), out=off[1:])
    det = pkg.Detector(xyz, floor, par)
    b = DeviceBatch([SliceIn(det, t0, hits, off)])
    old = pkg.trig_get_tile_config()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    try:
        pkg.trig_set_tile_config(4096, 8, 90)
        b.run()
        torch.cuda.synchronize()
        ev[0].record()
        b.run()
        ev[1].record()
        (stats, trig, win), = b.results()
    finally:
        pkg.trig_set_tile_config(*old)
    ref = oracle.run(xyz, floor, par, hits, [t0])[0]
    assert int(stats["status"]) == 0
    assert int(stats["n_seeds"]) == len(ref.seeds) and len(trig) == len(ref.triggers) and len(win) == len(ref.windows)
    for f in ("t", "pmt", "charge", "count"):
        assert np.array_equal(trig[f], ref.triggers[f]), f
    for f in ("lo", "hi", "n_hits", "n_triggers"):
        assert np.array_equal(win[f], ref.windows[f]), f
    assert ev[0].elapsed_time(ev[1]) < 50.0
    det.close()


def _check_slice(pkg, det, xyz, floor, par, t0, hits, off, events):
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    b = DeviceBatch([SliceIn(det, t0, hits, off)], events=events)
    old = pkg.trig_get_tile_config()
    try:
        pkg.trig_set_tile_config(2048, 16, 90)
        b.run()
        (stats, trig, win), = b.results()
    finally:
        pkg.trig_set_tile_config(*old)
    ref = oracle.run(xyz, floor, par, hits, [t0])[0]
    assert int(stats["status"]) == 0, int(stats["flags"])
    assert int(stats["n_seeds"]) == len(ref.seeds) and len(trig) == len(ref.triggers) and len(win) == len(ref.windows)
    for f in ("t", "pmt", "charge", "count"):
        assert np.array_equal(trig[f], ref.triggers[f]), f
    for f in ("lo", "hi", "n_hits", "n_triggers"):
        assert np.array_equal(win[f], ref.windows[f]), f
    if events:
        (ev, n_ev, full), = b.event_hits()
        want = oracle.events(hits, ref.windows)
        assert not full and n_ev == len(want)
        for f in ("t", "pmt", "charge"):
            assert np.array_equal(ev[f], want[f]), f


_CROWD_RULES = [{}, dict(seed_rule=1, l0_hits=7, l0_window_ns=1000, threshold=1), dict(count_distinct_pmts=1),
                dict(l0_hits=9, l0_window_ns=400, l0_distinct_pmts=1)]


@pytest.mark.parametrize("n_pmt", [32, 84, 97, 128, 129, 336])
@pytest.mark.parametrize("slice_ns", [60_000, 1_000_000])
@pytest.mark.parametrize("rule", range(len(_CROWD_RULES)))
def test_bursts_whose_halos_crowd_a_tile(pkg, params, n_pmt, slice_ns, rule):
    """A burst of 0.6 hits/ns, 3600 within the halos of any nanosecond of it:
    2048-hit tiles take what 4096-hit tiles would.  In the short slice the
    burst sets the slice's own rate (the builds with a warp per seed)."""
    rng = np.random.Generator(np.random.PCG64(n_pmt + slice_ns + rule))
    par = dict(params, slice_ns=slice_ns, **_CROWD_RULES[rule])
    t0, n, burst = 1_000_000, 12_000, 9_000
    xyz, floor = _detector(n_pmt)
    hits, _ = _hits(rng, n, n_pmt, t0 - 3000, t0 + slice_ns + 3000)
    hits["t"][:burst] = t0 + slice_ns - 20_000 + rng.integers(0, 15_000, burst)
    hits = np.sort(hits, order=["pmt", "t", "charge"], kind="stable")
    off = np.zeros(n_pmt + 1, np.uint64)
    np.cumsum(np.bincount(hits["pmt"], minlength=n_pmt), out=off[1:])
    det = pkg.Detector(xyz, floor, par)
    for events in (False, True):
        _check_slice(pkg, det, xyz, floor, par, t0, hits, off, events)
    det.close()


@pytest.mark.parametrize("n_pmt", [84, 129])
@pytest.mark.parametrize("n", [2047, 2048, 2049, 3000, 4095, 4096, 4097])
@pytest.mark.parametrize("where", ["start", "inside", "end"])
def test_pileups_up_to_two_tiles(pkg, params, n_pmt, n, where):
    """n hits within 2 ns: up to 4096 they are processed, one more is
    reported; so too at the slice's first and last nanosecond, with half of
    them in the halo."""
    rng = np.random.Generator(np.random.PCG64(n + n_pmt))
    par = dict(params, slice_ns=300_000)
    t0 = 1_000_000
    at = {"start": t0 - 1, "inside": t0 + 100_000, "end": t0 + par["slice_ns"] - 1}[where]
    xyz, floor = _detector(n_pmt)
    hits, off = _hits(rng, n, n_pmt, at, at + 2)
    det = pkg.Detector(xyz, floor, par)
    if n <= 4096:
        _check_slice(pkg, det, xyz, floor, par, t0, hits, off, False)
    else:
        with pytest.raises(AssertionError, match="8"):
            _check_slice(pkg, det, xyz, floor, par, t0, hits, off, False)
    det.close()
