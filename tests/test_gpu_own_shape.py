"""The tile shape that the library chooses by itself: how it is left and given
back, and where its choice changes."""
import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu

NOMINAL = (4096, 16, 60)


@pytest.fixture(scope="module")
def pkg():
    import torch
    import paper_1411_3968_gb300 as p
    from paper_1411_3968_gb300 import build
    build.build()
    p.load()
    torch.cuda.init()
    return p


def _scratch(pkg, det, n_hits, n_slices=1):
    """Scratch bytes of a batch of such slices (its buffers are only named)."""
    from paper_1411_3968_gb300 import _lib
    d = [_lib.slice_dev(det, 4096, 4096, n_hits, 1_000_000, 4096, 1, 4096, 1, 4096) for _ in range(n_slices)]
    return pkg.trig_batch_scratch_bytes(d)


def test_the_reported_shape_gives_the_choice_back(pkg, params):
    g = workload.km3_tower()
    det = pkg.Detector(g.xyz_mm, g.floor_id, params)
    assert pkg.trig_get_tile_config() == NOMINAL
    for n in (40_000, 3_000_000):
        own = _scratch(pkg, det, n)
        pkg.trig_set_tile_config(1024, 4, 40)
        assert pkg.trig_get_tile_config() == (1024, 4, 40)
        other = _scratch(pkg, det, n)
        pkg.trig_set_tile_config(*NOMINAL)
        assert pkg.trig_get_tile_config() == NOMINAL
        assert pkg.trig_detector_tile_config(det) == dict(cap=4096, warps=16, fill_pct=60, tuned=False)
        assert _scratch(pkg, det, n) == own != other
    # the choice follows the batch: small ones are cut into more tiles a hit
    assert _scratch(pkg, det, 40_000) > _scratch(pkg, det, 3_000_000) * 40_000 / 3_000_000
    det.close()


@pytest.mark.parametrize("rate,n_slices", [(2e3, 1), (60e3, 3), (300e3, 1)])
def test_own_shape_gives_the_oracles_results(pkg, params, rate, n_slices):
    """A short batch, a few uneven slices, and one of more than eight waves of
    tiles (25 MHz of hits for 200 ms), each after another shape was set and
    taken back."""
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    g = workload.km3_tower()
    par = dict(params, slice_ns=200_000_000 if n_slices == 1 else 20_000_000)
    det = pkg.Detector(g.xyz_mm, g.floor_id, par)
    slices, refs = [], []
    for k in range(n_slices):
        t0 = workload.T_ORIGIN_NS + k * par["slice_ns"]
        st = workload.gen_stream(g, t0 - 3000, t0 + par["slice_ns"] + 3000, rate / (1 + 2 * k), n_muons=20, seed=6 + k,
                                 stream=200 + k)
        slices.append(SliceIn(det, t0, st.hits, st.pmt_off))
        refs.append(oracle.run(g.xyz_mm, g.floor_id, par, st.hits, [t0])[0])
    old = pkg.trig_get_tile_config()
    pkg.trig_set_tile_config(2048, 8, 50)
    pkg.trig_set_tile_config(*old)
    b = DeviceBatch(slices)
    b.run()
    for (stats, trig, win), ref in zip(b.results(), refs):
        assert int(stats["status"]) == 0 and int(stats["n_seeds"]) == len(ref.seeds)
        for f in ("t", "pmt", "charge", "count"):
            assert np.array_equal(trig[f], ref.triggers[f]), f
        for f in ("lo", "hi", "n_hits", "n_triggers"):
            assert np.array_equal(win[f], ref.windows[f]), f
    det.close()


@pytest.mark.parametrize("n_pmt", [1344, 2688])
@pytest.mark.parametrize("halo_hits,cap", [(300, 2048), (520, 2048), (575, 2048), (595, 4096), (900, 4096)])
def test_dense_arrays_take_larger_tiles_from_585_halo_hits(pkg, params, n_pmt, halo_hits, cap):
    """The rule counts the hits of both halos of H = 3000 ns, as wide as the
    array's dt allows: of a 200 ms slice, which tiles it is planned with."""
    k = np.arange(n_pmt)
    xyz = np.stack([1000 * (k % 6), np.zeros_like(k), 40_000 * (k // 6)], 1).astype(np.int32)
    par = dict(params, slice_ns=200_000_000)
    det = pkg.Detector(xyz, (k // 6).astype(np.uint32), par)
    assert det.halo_ns == 3000
    n = int(halo_hits * (par["slice_ns"] + 6000) / 6000)
    own = _scratch(pkg, det, n)
    try:
        pkg.trig_set_tile_config(cap, 16, 90)
        assert _scratch(pkg, det, n) == own
        pkg.trig_set_tile_config(6144 - cap, 16, 90)
        assert _scratch(pkg, det, n) != own
    finally:
        pkg.trig_set_tile_config(*NOMINAL)
    det.close()


@pytest.mark.parametrize("n_pmt,n_slices,slice_ns,n", [(2688, 16, 5_000_000, 103_952), (2688, 1, 5_000_000, 1_673_664),
                                                       (4096, 16, 2_000_000, 104_464), (128, 16, 300_000, 123_696),
                                                       (672, 16, 20_000_000, 101_456)])
def test_noalloc_takes_what_the_nominal_tables_left_room_for(pkg, params, n_pmt, n_slices, slice_ns, n):
    """Batches that fill the static scratch to within 1 KB when every slice
    has tiles of 4096 hits filled to 60 %, with two offsets a PMT, or two
    counters a bucket: they are taken, and give what trig_batch_run does."""
    import torch
    from paper_1411_3968_gb300 import _lib
    from paper_1411_3968_gb300.runner import DeviceBatch, SliceIn
    rng = np.random.Generator(np.random.PCG64(n))
    k = np.arange(n_pmt)
    xyz = np.stack([1000 * (k % 6), np.zeros_like(k), 40_000 * (k // 6)], 1).astype(np.int32)
    par = dict(params, slice_ns=slice_ns)
    det = pkg.Detector(xyz, (k // 6).astype(np.uint32), par)
    t0 = 1_000_000
    hits = np.zeros(n, workload.HIT_DTYPE)
    hits["t"] = t0 - 3000 + rng.integers(0, slice_ns + 6000, n)
    hits["pmt"] = rng.integers(0, n_pmt, n)
    hits["charge"] = rng.integers(1, 320, n)
    hits = np.sort(hits, order=["pmt", "t", "charge"], kind="stable")
    off = np.zeros(n_pmt + 1, np.uint64)
    np.cumsum(np.bincount(hits["pmt"], minlength=n_pmt), out=off[1:])
    b = DeviceBatch([SliceIn(det, t0, hits, off)] * n_slices)
    b.run()
    want = b.results()
    assert all(int(w[0]["status"]) == 0 for w in want) and len(want[0][1]) > 100
    for t in b.trig + b.win:
        t.zero_()
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    _lib.trig_batch_run_noalloc(b.descs, st.cuda_stream)
    for (s1, t1, w1), (s0, t0_, w0) in zip(b.results(), want):
        assert s1 == s0 and np.array_equal(t1, t0_) and np.array_equal(w1, w0)
    det.close()
