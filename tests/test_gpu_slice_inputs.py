"""Slices whose input is at the edge of what a call takes, or past it, beside
ordinary ones of the same batch: no hits at all, PMTs without hits, offsets
that are wrong where no hit is.  The neighbours' results are the oracle's,
whatever the scratch held before."""
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


def _stream(hits, n_pmt):
    hits = np.sort(hits, order=["pmt", "t", "charge"], kind="stable")
    off = np.zeros(n_pmt + 1, np.uint64)
    np.cumsum(np.bincount(hits["pmt"], minlength=n_pmt), out=off[1:])
    return hits, off


def _hits(rng, n, n_pmt, lo, hi, step=1):
    hits = np.zeros(n, workload.HIT_DTYPE)
    hits["t"] = lo + rng.integers(0, max(1, (hi - lo) // step), n) * step
    hits["pmt"] = rng.integers(0, n_pmt, n)
    hits["charge"] = rng.integers(1, 400, n)
    return _stream(hits, n_pmt)


def _assert_same(res, ref, ctx=""):
    stats, trig, win = res
    assert int(stats["status"]) == 0, ctx
    assert int(stats["n_seeds"]) == len(ref.seeds), ctx
    assert len(trig) == len(ref.triggers) and len(win) == len(ref.windows), ctx
    for f in ("t", "pmt", "charge", "count"):
        assert np.array_equal(trig[f], ref.triggers[f]), (ctx, f)
    for f in ("lo", "hi", "n_hits", "n_triggers"):
        assert np.array_equal(win[f], ref.windows[f]), (ctx, f)


def _assert_result(r, ref, ctx=""):
    assert r.status == 0 and r.n_seeds == len(ref.seeds), ctx
    for f in ("t", "pmt", "charge", "count"):
        assert np.array_equal(r.triggers[f], ref.triggers[f]), (ctx, f)
    for f in ("lo", "hi", "n_hits", "n_triggers"):
        assert np.array_equal(r.windows[f], ref.windows[f]), (ctx, f)


def _mixed(pkg, n_pmt, par, empty, n=4000):
    """Five slices, the ones in `empty` without hits, and the others' oracle results."""
    from paper_1411_3968_gb300.runner import SliceIn
    rng = np.random.Generator(np.random.PCG64(n_pmt))
    xyz, floor = _detector(n_pmt)
    det = pkg.Detector(xyz, floor, par)
    slices, refs = [], []
    for k in range(5):
        t0 = 1_000_000 + k * par["slice_ns"]
        hits, off = _hits(rng, 0 if k in empty else n + 100 * k, n_pmt, t0 - 3000, t0 + par["slice_ns"] + 3000)
        slices.append(SliceIn(det, t0, hits, off))
        refs.append(oracle.run(xyz, floor, par, hits, [t0])[0])
    return det, slices, refs


@pytest.mark.parametrize("n_pmt", [84, 129, 672, 2688])
@pytest.mark.parametrize("empty", [(0, 3), (4,), (0, 1, 2, 3, 4)])
def test_empty_slices_beside_full_ones(pkg, params, n_pmt, empty):
    import torch
    from paper_1411_3968_gb300 import _lib
    from paper_1411_3968_gb300.runner import DeviceBatch
    par = dict(params, slice_ns=300_000)
    det, slices, refs = _mixed(pkg, n_pmt, par, empty)
    b = DeviceBatch(slices)
    stream = torch.cuda.Stream()

    def noalloc():
        torch.cuda.synchronize()
        _lib.trig_batch_run_noalloc(b.descs, stream.cuda_stream)

    for name, run in (("plain", b.run), ("graph", lambda: b.run(graph=True)), ("replay", lambda: b.run(graph=True)),
                      ("noalloc", noalloc)):
        b.scratch.fill_(0x3f)
        for t in b.trig + b.win:
            t.zero_()
        run()
        for k, (res, ref) in enumerate(zip(b.results(), refs)):
            _assert_same(res, ref, (name, k))
            assert int(res[0]["n_hits"]) == len(slices[k].hits)
    det.close()


@pytest.mark.parametrize("n_pmt", [84, 672])
def test_empty_slices_with_events(pkg, params, n_pmt):
    from paper_1411_3968_gb300.runner import DeviceBatch
    par = dict(params, slice_ns=300_000)
    det, slices, refs = _mixed(pkg, n_pmt, par, (1, 4))
    b = DeviceBatch(slices, events=True)
    b.scratch.fill_(0x3f)
    b.run()
    for k, (res, ev, ref) in enumerate(zip(b.results(), b.event_hits(), refs)):
        _assert_same(res, ref, k)
        want = oracle.events(slices[k].hits, ref.windows)
        assert not ev[2] and ev[1] == len(want), k
        for f in ("t", "pmt", "charge"):
            assert np.array_equal(ev[0][f], want[f]), (k, f)
    det.close()


@pytest.mark.parametrize("n_pmt", [84, 672])
def test_empty_slices_through_the_engine(pkg, params, n_pmt):
    par = dict(params, slice_ns=300_000)
    det, slices, refs = _mixed(pkg, n_pmt, par, (0, 3))
    for _ in range(2):                      # the second time on an arena full of the first one's bytes
        pkg.trig_engine_hold(True)
        ids = [pkg.trig_submit_slice(det, s.t0, s.hits, s.pmt_off) for s in slices]
        pkg.trig_engine_hold(False)
        for k, ref in enumerate(refs):
            r = pkg.trig_poll(det, 30_000)
            assert r is not None and r.slice_id == ids[k]
            _assert_result(r, ref, k)
    det.close()


def _sparse(rng, n_pmt, used, n, lo, hi):
    """Hits of the PMTs `used` alone."""
    hits, _ = _hits(rng, n, len(used), lo, hi)
    hits["pmt"] = np.asarray(used, np.uint16)[hits["pmt"]]
    return _stream(hits, n_pmt)


def _used(n_pmt):
    """Most of the PMTs, with empty ones before the first, after the last and in runs between."""
    return [p for p in range(2, n_pmt - 3) if p % 7 not in (3, 4) and not n_pmt // 2 <= p < n_pmt // 2 + 9]


@pytest.mark.parametrize("n_pmt", [84, 128, 129, 672])
def test_runs_of_empty_pmts(pkg, params, n_pmt):
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(n_pmt + 5))
    par = dict(params, slice_ns=300_000)
    xyz, floor = _detector(n_pmt)
    det = pkg.Detector(xyz, floor, par)
    t0 = 1_000_000
    for used in (_used(n_pmt), [n_pmt - 1], [0], [0, n_pmt - 1]):
        hits, off = _sparse(rng, n_pmt, used, 3000, t0 - 3000, t0 + par["slice_ns"] + 3000)
        b = DeviceBatch([SliceIn(det, t0, hits, off)])
        b.scratch.fill_(0x3f)
        b.run()
        _assert_same(b.results()[0], oracle.run(xyz, floor, par, hits, [t0])[0], used[:3])
    det.close()


def _bad_offsets(off, n_pmt):
    """Offsets that disagree with the hits at empty PMTs only, where no hit's own run start or end shows it."""
    n = int(off[-1])
    mid = n_pmt // 2 + 4                        # inside the empty run of _used
    return {"first": (0, 1), "second": (1, n), "low": (mid, int(off[mid]) - 1), "high": (mid, int(off[mid]) + 1),
            "far": (mid, 2 ** 40), "wrapped": (mid, 2 ** 64 - 1), "after": (n_pmt - 1, n - 1), "past": (n_pmt - 2, n + 7)}


@pytest.mark.parametrize("n_pmt", [84, 129, 672])
def test_offsets_of_empty_pmts_are_checked(pkg, params, n_pmt):
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(n_pmt + 9))
    par = dict(params, slice_ns=300_000)
    xyz, floor = _detector(n_pmt)
    det = pkg.Detector(xyz, floor, par)
    t0 = 1_000_000
    hits, off = _sparse(rng, n_pmt, _used(n_pmt), 3000, t0 - 3000, t0 + par["slice_ns"] + 3000)
    ref = oracle.run(xyz, floor, par, hits, [t0])[0]
    slices = [SliceIn(det, t0, hits, off)]
    for at, value in _bad_offsets(off, n_pmt).values():
        wrong = off.copy()
        wrong[at] = value
        slices.append(SliceIn(det, t0, hits, wrong))
    # runs out of order, each at its own PMT's offset
    swapped = np.concatenate([hits[hits["pmt"] == 9], hits[hits["pmt"] == 5]])
    so = np.full(n_pmt + 1, len(swapped), np.uint64)
    n9 = int((swapped["pmt"] == 9).sum())
    so[:10], so[5], so[6], so[9], so[10] = 0, n9, len(swapped), 0, n9
    slices.append(SliceIn(det, t0, swapped, so))
    slices.append(slices[0])
    b = DeviceBatch(slices)
    b.scratch.fill_(0x3f)
    for graph in (False, True):
        b.run(graph=graph)
        res = b.results()
        for k in (0, len(slices) - 1):
            _assert_same(res[k], ref, k)
        for stats, trig, win in res[1:-1]:
            assert int(stats["status"]) == pkg.TRIG_EINVAL and int(stats["flags"]) & 0x01
            assert len(trig) == 0 and len(win) == 0 and int(stats["n_seeds"]) == 0
    assert all(len(b.rows(i)[0]) == 0 for i in range(1, len(slices) - 1))
    det.close()


# at 20 hits a microsecond a tile of 2048 hits filled to 90 % has a core of 57
# buckets of 1500 ns, and the seventh tile of these slices one of 1 to 26
LAST_TILE_SLICES = tuple(6 * 57 * 1500 + 1500 * k for k in (1, 2, 7, 26))


def _last_tile_burst(n_pmt, slice_ns, cluster_ns):
    rng = np.random.Generator(np.random.PCG64(n_pmt + slice_ns))
    t0 = 1_000_000
    hits, _ = _hits(rng, (slice_ns + 6000) // 50, n_pmt, t0 - 3000, t0 + slice_ns + 3000)
    hits["t"][:1890] = t0 + slice_ns - cluster_ns + rng.integers(0, cluster_ns, 1890)
    return _stream(hits, n_pmt)


@pytest.mark.parametrize("n_pmt", [129, 336])
@pytest.mark.parametrize("slice_ns", LAST_TILE_SLICES)
@pytest.mark.parametrize("cluster_ns", [1_200, 8_000])
def test_burst_in_a_short_last_tile(pkg, params, n_pmt, slice_ns, cluster_ns):
    """The last tile of a wide slice is overfull and its core far shorter than
    the others': its pieces end with the slice."""
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    par = dict(params, slice_ns=slice_ns)
    t0 = 1_000_000
    xyz, floor = _detector(n_pmt)
    hits, off = _last_tile_burst(n_pmt, slice_ns, cluster_ns)
    det = pkg.Detector(xyz, floor, par)
    b = DeviceBatch([SliceIn(det, t0, hits, off)])
    ref = oracle.run(xyz, floor, par, hits, [t0])[0]
    old = pkg.trig_get_tile_config()
    for shape in ((2048, 16, 90), (2048, 16, 60), (1024, 4, 90)):
        pkg.trig_set_tile_config(*shape)
        try:
            b.run()
            res, = b.results()
        finally:
            pkg.trig_set_tile_config(*old)
        if shape[0] == 1024:        # more than 1024 of the burst's hits within 3 us of any of its 1 ns cores
            assert int(res[0]["status"]) == pkg.TRIG_ECAPACITY and int(res[0]["flags"]) & 0x08
        else:
            _assert_same(res, ref, shape)
    det.close()


def test_selection_takes_hits_at_any_8_bytes(pkg, params):
    """trig_array_select reads hits by their 8-byte members: towers whose hits
    start 8 bytes past a 16-byte boundary give what aligned ones do."""
    import torch
    from paper_1411_3968_gb300 import _lib
    from paper_1411_3968_gb300.runner import ArrayBatch, SliceIn
    wl = workload.cfg_towers8()
    subs = wl.submissions[:3]
    dets = [pkg.Detector(wl.detectors[s.det_index].xyz_mm, wl.detectors[s.det_index].floor_id, params) for s in subs]
    arr = pkg.Array(dets, min_towers=1, corr_window_ns=3000, win_half_ns=3000)
    ab = ArrayBatch(arr, [SliceIn(d, s.t0, s.stream.hits, s.stream.pmt_off) for d, s in zip(dets, subs)])
    ab.run()
    want = ab.results()
    assert int(want[0]["status"]) == 0 and len(want[4]) > 10_000
    shifted = []
    for k, (d, s) in enumerate(zip(ab.batch.descs, subs)):
        nbytes = len(s.stream.hits) * 16
        buf = torch.empty(nbytes + 24, dtype=torch.uint8, device="cuda")
        buf[8:8 + nbytes].copy_(ab.batch.hits[k][:nbytes])
        assert (buf.data_ptr() + 8) % 16 == 8
        shifted.append((buf, _lib.slice_dev(dets[k], buf.data_ptr() + 8, ab.batch.offs[k].data_ptr(), len(s.stream.hits), s.t0,
                                            ab.batch.trig[k].data_ptr(), ab.batch.trig_cap[k], ab.batch.win[k].data_ptr(),
                                            ab.batch.win_cap[k], ab.batch.stats.data_ptr() + k * _lib.STATS_DTYPE.itemsize)))
    ab.hits.zero_()
    st = torch.cuda.current_stream()
    _lib.trig_array_select(arr, [x[1] for x in shifted], ab.out, ab.scratch.data_ptr(), ab.scratch_bytes, st.cuda_stream)
    got = ab.results()
    assert got[0] == want[0]
    for a, b in zip(got[1:], want[1:]):
        assert np.array_equal(a, b)
    arr.close()
    for d in dets:
        d.close()
