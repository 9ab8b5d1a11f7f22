"""Edges of the transform's accumulation (runs of FFTs, whole and short rounds,
narrowed tiles) and of the selection's block sizes, against the oracle: maps,
profile picks and counts bit for bit."""
import numpy as np
import pytest

from paper_1407_8333_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_8333_gb300 import build, fh as fhmod
    build.build()
    fhmod.load()
    return fhmod


def search(fh, inp, pp, weights=None, **shape):
    import torch
    n_dir = inp.sky.shape[0]
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda()
           for x in (inp.t, inp.offsets, inp.freq, inp.v, inp.sky)]
    plan = fh.fh_create_plan(fh.make_desc(pp, inp.t.shape[0], n_dir, inp.n_peaks, **shape))
    try:
        fh.fh_correct_doppler(plan, *dev)
        if weights is not None:
            fh.fh_set_weights(plan, weights, 4)
        maps = torch.empty((n_dir, pp["n_fdot"], pp["n_f0"]), dtype=torch.int32, device="cuda")
        fh.fh_transform(plan, 0, n_dir, maps)
        cand = fh.fh_select_candidates(plan, 0, n_dir)
        return maps.cpu().numpy(), cand.reshape(n_dir, -1, pp["top_k"])
    finally:
        fh.fh_destroy_plan(plan)


def check(fh, inp, pp, weights=None, **shape):
    import oracle
    kw = {} if weights is None else dict(weights=weights, frac_bits=4)
    want = oracle.search(inp, pp, want_maps=True, **kw)
    maps, cand = search(fh, inp, pp, weights, **shape)
    assert np.array_equal(maps, want["maps"])
    for k in ("cell", "row", "count"):
        assert np.array_equal(cand[k], want[k])


# with 4 warps a run is 3/16 of the FFTs' chunks: 5 chunks of 32 (none), 6 (one each),
# 11 and 43 (runs of 2 and 8, the last with a remainder)
@pytest.mark.parametrize("n_fft", [160, 191, 192, 193, 351, 1376])
@pytest.mark.parametrize("n_dir, n_fdot", [(1, 33), (1, 70), (2, 36), (3, 4), (2, 17)])
def test_runs_of_ffts(fh, n_fft, n_dir, n_fdot):
    for p in (0.02, 0.3):   # fewer than a round of slots per 32 FFTs, and many
        inp, pp = synth.random_case(900 + n_fft + n_fdot, n_fft=n_fft, n_bins=30, n_fdot=n_fdot,
                                    n_dir=n_dir, p=p, vmax=2e-6)
        check(fh, inp, pp, block_warps=4, tile_cells=128)


# below 43 chunks for 32 warps a warp's run is its share of the FFTs, at most 32 (a warp
# without one, the last one short, 31 and 32 to a warp, and more FFTs than 32 to each)
@pytest.mark.parametrize("n_fft", [1, 31, 33, 65, 200, 992, 993, 1023, 1025, 1300])
@pytest.mark.parametrize("n_dir, n_fdot, warps", [(1, 5, 32), (1, 40, 24), (2, 34, 32), (2, 4, 20)])
def test_few_ffts_per_warp(fh, n_fft, n_dir, n_fdot, warps):
    inp, pp = synth.random_case(1300 + n_fft + n_fdot, n_fft=n_fft, n_bins=24, n_fdot=n_fdot,
                                n_dir=n_dir, p=0.2, vmax=2e-6)
    check(fh, inp, pp, block_warps=warps, tile_cells=96)


@pytest.mark.parametrize("n_fft", [193, 351])
def test_runs_of_ffts_weighted(fh, n_fft):
    inp, pp = synth.random_case(77 + n_fft, n_fft=n_fft, n_bins=30, n_fdot=20, n_dir=2, p=0.2)
    w = 0.25 * (1 + np.arange(2 * n_fft).reshape(2, n_fft) % 7)
    check(fh, inp, pp, weights=w, block_warps=4, tile_cells=128)


@pytest.mark.parametrize("n_bins", [13, 200, 1000, 1531])
def test_default_tile_of_few_items(fh, n_bins):
    """The library's own tile where one direction has few items: bands at and
    around the width it is narrowed to."""
    for n_dir in (1, 2):
        inp, pp = synth.random_case(31 + n_bins, n_fft=40, n_bins=n_bins, n_fdot=9, n_dir=n_dir,
                                    p=0.05, vmax=2e-6)
        check(fh, inp, pp)


# 8 cells per thread in whole warps: one warp up to 256 cells, 1024 threads from 7937,
# the profile read again per pick beyond 8192
@pytest.mark.parametrize("subband_bins, k_over", [(1, 1), (85, 3), (256, 1), (257, 1), (1023, 8),
                                                  (1024, 8), (1171, 7)])
def test_selection_block_sizes(fh, subband_bins, k_over):
    inp, pp = synth.random_case(61 + subband_bins, n_fft=12, n_bins=1200, k_over=k_over, n_fdot=3,
                                n_dir=2, p=0.1, subband_bins=subband_bins, top_k=4,
                                excl_cells=2 * k_over, sep_cells=3 * k_over)
    check(fh, inp, pp)


# maps staged through the guard cells: 16-cell groups with rows of 16 bytes (n_f0 a
# multiple of 4), written row by row where they are not (odd K and bins), more warps
# than the guard cells hold a stage for; ragged last groups, tiles and slabs
@pytest.mark.parametrize("n_bins, k_over", [(40, 4), (33, 4), (41, 3), (100, 10), (64, 1)])
@pytest.mark.parametrize("n_dir, n_fdot", [(1, 5), (1, 45), (1, 70), (2, 33), (3, 31)])
def test_written_maps(fh, n_bins, k_over, n_dir, n_fdot):
    for warps, tile in ((4, 64), (16, 0), (24, 0), (32, 0)):
        inp, pp = synth.random_case(400 + n_bins + n_fdot, n_fft=50, n_bins=n_bins, k_over=k_over,
                                    n_fdot=n_fdot, n_dir=n_dir, p=0.2, vmax=2e-6)
        check(fh, inp, pp, block_warps=warps, tile_cells=min(tile, pp["n_f0"]))
    w = 0.5 + np.arange(n_dir * 50).reshape(n_dir, 50) % 3
    check(fh, inp, pp, weights=w)


def test_plans_of_different_shapes_take_turns(fh):
    """A plan with small tiles between two passes of one with the largest."""
    import torch
    import oracle
    big, pb = synth.random_case(81, n_fft=40, n_bins=400, n_fdot=40, n_dir=2, p=0.1, vmax=2e-6)
    small, ps = synth.random_case(82, n_fft=40, n_bins=20, n_fdot=40, n_dir=2, p=0.1, vmax=2e-6)
    plans, want = [], []
    for inp, pp, tile in ((big, pb, 0), (small, ps, 32)):
        plan = fh.fh_create_plan(fh.make_desc(pp, 40, 2, inp.n_peaks, tile_cells=tile))
        dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda()
               for x in (inp.t, inp.offsets, inp.freq, inp.v, inp.sky)]
        fh.fh_correct_doppler(plan, *dev)
        plans.append((plan, dev))
        want.append(oracle.search(inp, pp))
    try:
        for k in (0, 1, 0, 1):
            fh.fh_transform(plans[k][0], 0, 2)
            c = fh.fh_select_candidates(plans[k][0], 0, 2)
            assert np.array_equal(c["count"].ravel(), want[k]["count"].ravel())
    finally:
        for plan, _ in plans:
            fh.fh_destroy_plan(plan)


# positions formed in integers and, where their bounds fail, in binary64: band edges
# at and around powers of two, T_FFT that is not one (K T odd up to 675), K up to
# 40, frequencies on and off the bin grid, far above and below the band, r on both
# sides of 1, f0 of 0 and below
@pytest.mark.parametrize("f0", [0.0, -3.0, 1e-3, 63.75, 64.0, 127.999, 900.0, 903.21, 1999.3])
@pytest.mark.parametrize("t_fft, k_over", [(1024.0, 10), (8192.0, 7), (1800.0, 12), (4096.0, 40),
                                           (3.0, 1), (1000.1, 1)])
def test_positions_in_integers(fh, f0, t_fft, k_over):
    import torch
    import oracle
    rng = np.random.RandomState(int(t_fft) + k_over)
    n_fft, base = 17, max(abs(f0), 1.0)
    parts = [np.round((base + rng.uniform(-0.2, 9.0, 40)) * t_fft) / t_fft,
             base + rng.uniform(-0.3, 12.0, 40), base * rng.uniform(0.3, 3.0, 10),
             np.nextafter(base, 1e9) * np.ones(1), np.array([base, base / 2, base * 2])]
    f = np.unique(np.abs(np.concatenate(parts)) + 1e-9)
    f[:20] = np.round(f[:20] * 1024) / 1024
    f = np.unique(f[f > 0])
    offsets = np.arange(n_fft + 1, dtype=np.int64) * len(f)
    freq = np.tile(f, n_fft)
    t = np.arange(n_fft) * 0.5 * t_fft
    v = rng.uniform(-1, 1, (n_fft, 3)) * np.array([0.0, 1e-9, 1e-4, 0.05])[np.arange(n_fft) % 4, None]
    sky = np.array([[0.6, 0.0, 0.8], [-0.6, 0.64, 0.48]])
    pp = dict(t_fft=t_fft, k_over=k_over, f0_min=f0, n_f0=50, fdot_min=0.0, fdot_step=1e-12,
              n_fdot=1, t_ref=0.0, subband_cells=50, top_k=1, excl_cells=0, sep_cells=0, n_thr=0,
              p0=0.1)
    plan = fh.fh_create_plan(fh.make_desc(pp, n_fft, 2, len(freq)))
    try:
        A = torch.empty((2, len(freq)), dtype=torch.int64, device="cuda")
        dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (t, offsets, freq, v, sky)]
        fh.fh_correct_doppler(plan, *dev, out_A=A)
        got = A.cpu().numpy()
    finally:
        fh.fh_destroy_plan(plan)
    kt = float(k_over) * t_fft
    r = oracle.doppler_factor(v, sky)
    x = (freq[None, :] * np.repeat(r, len(f), axis=1) - f0) * kt + (0.5 - 0.5 * k_over)
    near = np.abs(x) < 2.0 ** 28   # beyond that a call is refused
    want = np.floor(x * 2.0 ** 32)[near].astype(np.int64)
    assert near.sum() > 1000 and np.array_equal(got[near], want)


# correction blocks of 2 and of 8 FFTs (4800 FFT-directions), of one and of four
# directions, and window passes side by side (up to 600 blocks of 8 FFTs) or not
@pytest.mark.parametrize("n_fft, n_dir", [(1, 1), (2, 1), (9, 3), (1599, 3), (1601, 3), (2049, 7),
                                          (17, 5)])
def test_correction_and_window_blocks(fh, n_fft, n_dir):
    inp, pp = synth.random_case(500 + n_fft, n_fft=n_fft, n_bins=110, n_fdot=4, n_dir=n_dir, p=0.05,
                                vmax=2e-6)
    check(fh, inp, pp, tile_cells=32)


@pytest.mark.parametrize("n_dir, n_fdot", [(24, 40), (9, 70)])
def test_window_table_grows_between_transforms_in_flight(fh, n_dir, n_fdot):
    """One direction, then more and more of them, queued without a wait: each call
    replaces the window table that the one before may still read, while clustering
    calls on other threads' streams take and return memory of the same pool.  Every
    map equals the oracle's."""
    import threading

    import oracle
    import torch
    n_fft = 400
    inp, pp = synth.random_case(1500 + n_dir, n_fft=n_fft, n_bins=200, n_fdot=n_fdot, n_dir=n_dir,
                                p=0.2, vmax=2e-6)
    want = oracle.search(inp, pp, want_maps=True)["maps"]
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda()
           for x in (inp.t, inp.offsets, inp.freq, inp.v, inp.sky)]
    cand = torch.from_numpy(synth.candidate_set(71, 0, 20000, clusters=40)).cuda()
    labels = fh.fh_cluster(cand, 3.0)[0].clone()
    torch.cuda.synchronize()
    stop, bad = threading.Event(), []

    def cluster():
        try:
            st = torch.cuda.Stream()
            while not stop.is_set():
                lab, _ = fh.fh_cluster(cand, 3.0, stream=st)
                st.synchronize()
                if not torch.equal(lab, labels):
                    bad.append("labels")
        except Exception as e:  # noqa: BLE001
            bad.append(repr(e))

    threads = [threading.Thread(target=cluster) for _ in range(2)]
    for t in threads:
        t.start()
    try:
        st = torch.cuda.Stream()
        for _ in range(10):
            counts = [1, 2, 5, n_dir]
            maps = [torch.empty((k, n_fdot, pp["n_f0"]), dtype=torch.int32, device="cuda")
                    for k in counts]
            plan = fh.fh_create_plan(fh.make_desc(pp, n_fft, n_dir, inp.n_peaks))
            torch.cuda.synchronize()
            fh.fh_correct_doppler(plan, *dev, stream=st)
            for k, m in zip(counts, maps):
                fh.fh_transform(plan, 0, k, m, stream=st)
            st.synchronize()
            fh.fh_destroy_plan(plan)
            for k, m in zip(counts, maps):
                assert np.array_equal(m.cpu().numpy(), want[:k])
    finally:
        stop.set()
        for t in threads:
            t.join()
    assert not bad


def test_window_table_that_does_not_fit_in_memory(fh):
    """A million FFTs of one peak: the narrowed tiles of one direction want a table of
    300 MB and room for 600; with less to be had the widest tile serves."""
    import torch
    n_fft = 1_000_000
    rng = np.random.RandomState(3)
    t = np.arange(n_fft) * 512.0
    freq = 50.0 + rng.uniform(0.1, 1.9, n_fft)
    offsets = np.arange(n_fft + 1, dtype=np.int64)
    pp = dict(t_fft=1024.0, k_over=10, f0_min=50.0, n_f0=20480, fdot_min=0.0,
              fdot_step=1.0 / (1024.0 * t[-1]), n_fdot=8, t_ref=0.0, subband_cells=1024, top_k=2,
              excl_cells=20, sep_cells=40, n_thr=0, p0=0.1)
    dev = [torch.from_numpy(x).cuda() for x in
           (t, offsets, freq, np.zeros((n_fft, 3)), np.array([[0.0, 0.0, 1.0]]))]

    got = []
    for left in (0, 200 << 20):               # 0: with all the room there is
        fill = []
        plan = fh.fh_create_plan(fh.make_desc(pp, n_fft, 1, n_fft))
        try:
            fh.fh_correct_doppler(plan, *dev)
            torch.cuda.synchronize()
            while left and torch.cuda.mem_get_info()[0] > left + (2 << 20):
                fill.append(torch.empty(min(4 << 30, torch.cuda.mem_get_info()[0] - left),
                                        dtype=torch.uint8, device="cuda"))
            fh.fh_transform(plan, 0, 1)
            got.append(fh.fh_select_candidates(plan, 0, 1))
        finally:
            del fill
            torch.cuda.empty_cache()
            fh.fh_destroy_plan(plan)
    assert got[0]["count"].max() > 0 and np.array_equal(got[0], got[1])
