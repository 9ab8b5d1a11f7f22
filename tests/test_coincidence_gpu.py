"""Candidate clustering and coincidences on the GPU, through the C ABI, against
the oracle (Sec. "Candidate clustering and coincidences", Eq. norm; App.
"Theory of coincidences").  Labels, cluster counts, pairs and partner counts
bit for bit."""
import math

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


@pytest.fixture(scope="module")
def co():
    import oracle
    return oracle.coincidence


def dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()


def check_cluster(fh, co, c, d_max):
    lab, n = fh.fh_cluster(dev(c), d_max)
    want, wn = co.cluster(c, d_max)
    assert n == wn
    assert np.array_equal(lab.cpu().numpy(), want)
    return want


def check_coinc(fh, co, a, b, ta, tb, tc, win):
    p, m1, m2 = fh.fh_coincidences(dev(a), dev(b), ta, tb, tc, win)
    wp, w1, w2 = co.coincidences(a, b, ta, tb, tc, win)
    assert np.array_equal(p.cpu().numpy(), wp.reshape(-1, 2))
    assert np.array_equal(m1.cpu().numpy(), w1) and np.array_equal(m2.cpu().numpy(), w2)
    return wp


@pytest.mark.parametrize("n, clusters", [(1, 0), (2, 0), (37, 3), (1500, 30)])
def test_cluster_matches_oracle(fh, co, n, clusters):
    c = synth.candidate_set(41 + n, 0, n, clusters=clusters, cluster_size=7)
    for d_max in (0.0, 1.5, 4.0, 9.0):
        check_cluster(fh, co, c, d_max)


def test_cluster_degenerate_geometries(fh, co):
    c = synth.candidate_set(42, 0, 400, clusters=10)
    # every candidate at one frequency: a single bucket
    same = c.copy()
    same[:, 2] = 123.456
    check_cluster(fh, co, same, 3.0)
    # longitudes on both sides of 0 / 2 pi
    wrap = c.copy()
    wrap[:, 0] = np.where(np.arange(400) % 2 == 0, 0.0005 * np.arange(400) % 0.01,
                          2 * math.pi - 0.0005 * np.arange(400) % 0.01)
    check_cluster(fh, co, wrap, 4.0)
    # duplicates and an enormous d_max (one cluster)
    dup = np.concatenate([c[:50], c[:50]])
    check_cluster(fh, co, dup, 0.0)
    lab = check_cluster(fh, co, c, 1e300)
    assert np.all(lab == 0)


@pytest.mark.parametrize("win", [(0, 0, 0, 0), (1, 1, 1, 1), (2, 2, 3, 2)])
def test_coincidences_match_oracle(fh, co, win):
    seeds = synth.candidate_set(43, 0, 80, clusters=10, cluster_size=8)[::8, :4]
    a = synth.candidate_set(43, 1, 900, signals=seeds, clusters=5)
    b = synth.candidate_set(43, 2, 1100, signals=seeds, clusters=5)
    check_coinc(fh, co, a, b, 3.0e6, 4.5e6, 3.7e6, win)
    check_coinc(fh, co, a, b, 0.0, 0.0, 0.0, win)


def test_coincidences_on_a_grid_and_edge_cases(fh, co):
    m = (40, 30, 50, 20)
    a = synth.candidates_on_grid(44, 1, 3000, m)
    b = synth.candidates_on_grid(44, 2, 2500, m)
    for win in ((0, 0, 0, 0), (1, 0, 2, 1)):
        check_coinc(fh, co, a, b, 0.0, 0.0, 0.0, win)
    # empty sets
    p, m1, m2 = fh.fh_coincidences(dev(a[:0]), dev(b), 0.0, 0.0, 0.0, (1, 1, 1, 1))
    assert p.shape[0] == 0 and np.all(m2.cpu().numpy() == 0)
    p, m1, m2 = fh.fh_coincidences(dev(a), dev(b[:0]), 0.0, 0.0, 0.0, (1, 1, 1, 1))
    assert p.shape[0] == 0 and np.all(m1.cpu().numpy() == 0)
    # a window so wide that everything coincides
    check_coinc(fh, co, a[:60], b[:70], 0.0, 0.0, 0.0, (1e300, 1e300, 1e300, 1e300))


def test_capacity_and_invalid_candidates(fh):
    a = synth.candidates_on_grid(45, 1, 300, (5, 5, 5, 5))
    with pytest.raises(fh.FHError) as ei:
        fh.fh_coincidences(dev(a), dev(a), 0.0, 0.0, 0.0, (0, 0, 0, 0), capacity=10)
    assert ei.value.code == fh.FH_ERR_CAPACITY
    bad = a.copy()
    bad[7, 6] = 0.0            # a zero frequency width
    with pytest.raises(fh.FHError) as ei:
        fh.fh_cluster(dev(bad), 2.0)
    assert ei.value.code == fh.FH_ERR_INVALID_ARG
    bad[7, 6] = 1.0
    bad[9, 2] = np.nan
    with pytest.raises(fh.FHError) as ei:
        fh.fh_coincidences(dev(bad), dev(a), 0.0, 0.0, 0.0, (1, 1, 1, 1))
    assert ei.value.code == fh.FH_ERR_INVALID_ARG
    with pytest.raises(fh.FHError) as ei:
        fh.fh_cluster(dev(a), -1.0)
    assert ei.value.code == fh.FH_ERR_INVALID_ARG


def test_twenty_thousand_candidates(fh, co):
    """Sets the size of one band's output (10^4 - 10^5 candidates)."""
    seeds = synth.candidate_set(46, 0, 400, clusters=50, cluster_size=8)[::8, :4]
    # the same sources seen by the second set at its own reference time 1e6 s later
    later = seeds.copy()
    later[:, 2] += later[:, 3] * 1.0e6
    a = synth.candidate_set(46, 1, 20000, signals=seeds, clusters=200, cluster_size=6)
    b = synth.candidate_set(46, 2, 20000, signals=later, clusters=200, cluster_size=6)
    check_cluster(fh, co, a, 4.0)
    wp = check_coinc(fh, co, a, b, 1.0e6, 2.0e6, 1.5e6, (2, 2, 2, 2))
    assert {(i, i) for i in range(50)} <= {tuple(x) for x in wp}


def test_cluster_coincidences_match_oracle(fh, co):
    """Clusters of both sets, their coincident pairs, and the nearest pair of
    each coincident pair of clusters: rows and distances equal the oracle's."""
    import torch
    seeds = synth.candidate_set(47, 0, 160, clusters=20, cluster_size=8)[::8, :4]
    later = seeds.copy()
    later[:, 2] += later[:, 3] * 1.0e6
    a = synth.candidate_set(47, 1, 3000, signals=seeds, clusters=60, cluster_size=6)
    b = synth.candidate_set(47, 2, 2800, signals=later, clusters=60, cluster_size=6)
    da, db = dev(a), dev(b)
    la, _ = fh.fh_cluster(da, 4.0)
    lb, _ = fh.fh_cluster(db, 4.0)
    pairs, _, _ = fh.fh_coincidences(da, db, 1.0e6, 2.0e6, 1.5e6, (3, 3, 3, 3))
    rows, dist = fh.fh_cluster_coincidences(da, db, 1.0e6, 2.0e6, 1.5e6, la, lb, pairs)
    wla, _ = co.cluster(a, 4.0)
    wlb, _ = co.cluster(b, 4.0)
    wp, _, _ = co.coincidences(a, b, 1.0e6, 2.0e6, 1.5e6, (3, 3, 3, 3))
    wrows, wd = co.cluster_coincidences(a, b, 1.0e6, 2.0e6, 1.5e6, wla, wlb, wp)
    assert np.array_equal(rows.cpu().numpy(), wrows)
    assert np.array_equal(dist.cpu().numpy().view(np.uint64), wd.view(np.uint64))
    assert len(wrows) < len(wp)
    # pairs out of (i, j) order, or out of range, are refused
    bad = pairs.flip(0).contiguous()
    if bad.shape[0] > 1:
        with pytest.raises(fh.FHError) as ei:
            fh.fh_cluster_coincidences(da, db, 1.0e6, 2.0e6, 1.5e6, la, lb, bad)
        assert ei.value.code == fh.FH_ERR_INVALID_ARG
    out = torch.tensor([[0, 5000]], dtype=torch.int32, device="cuda")
    with pytest.raises(fh.FHError) as ei:
        fh.fh_cluster_coincidences(da, db, 1.0e6, 2.0e6, 1.5e6, la, lb, out)
    assert ei.value.code == fh.FH_ERR_INVALID_ARG


def _cells_case(name):
    """Sets at the edges of the (frequency, spin-down) cells."""
    if name == "capped":      # far more cells wanted than candidates
        a = synth.candidates_on_grid(48, 1, 150, (5, 3, 100000, 90000))
        b = a + np.array([0, 0, 1.0, -1.0, 0, 0, 0, 0])
        return np.concatenate([a, b]), np.concatenate([b[::-1], a])
    if name == "outside":     # set 1 partly far outside set 2, partly one cell away
        b = synth.candidates_on_grid(49, 1, 400, (6, 4, 40, 12))
        a = np.concatenate([b + np.array([0, 0, x, y, 0, 0, 0, 0])
                            for x, y in ((1e7, 0), (-41.0, 0), (39.0, 1.0), (0, 13.0), (0, -1e9))])
        return a, b
    if name == "crowded":     # more partners per candidate than the count keeps
        return (synth.candidates_on_grid(50, 1, 700, (3, 2, 9, 5)),
                synth.candidates_on_grid(50, 2, 500, (3, 2, 9, 5)))
    if name == "one_cell":    # no range at all in frequency and spin-down
        a = synth.candidates_on_grid(51, 1, 300, (300, 40, 1, 1))
        return a, a[::-1]
    # beyond binary32: values and widths of 1e36 to 1e40, and subnormal widths
    a = synth.candidates_on_grid(52, 1, 300, (7, 5, 30, 10))
    a[:, 2] *= 1e39
    a[:, 6] = 1e39
    a[:, 3] *= 1e-39
    a[:, 7] = 1e-39
    return a, a[::-1]


@pytest.mark.parametrize("name", ["capped", "outside", "crowded", "one_cell", "beyond"])
def test_cells_of_frequency_and_spin_down(fh, co, name):
    a, b = _cells_case(name)
    for d_max in (0.0, 1.0, 1.5):
        check_cluster(fh, co, a, d_max)
    for win in ((0, 0, 0, 0), (1, 1, 1, 1), (0, 1, 1, 2)):
        check_coinc(fh, co, a, b, 0.0, 0.0, 0.0, win)


@pytest.mark.parametrize("n", [4096, 4097, 8192, 8193])
def test_scan_tiles(fh, co, n):
    """Set sizes whose cell counts end at, and one past, the scan's tiles."""
    a = synth.candidate_set(53, 1, n, clusters=20, cluster_size=5)
    check_cluster(fh, co, a, 2.0)
    check_coinc(fh, co, a[:500], a, 0.0, 0.0, 0.0, (2, 2, 2, 2))
    check_coinc(fh, co, a, a[:300], 0.0, 0.0, 0.0, (2, 2, 2, 2))


@pytest.mark.parametrize("n", [1, 8, 63, 64, 65, 257])
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (2, 1, 3, 2), (40, 20, 30, 10)])
def test_lists_of_pairs(fh, co, n, shape):
    """Set sizes at the edges of a block's and a warp's candidates, with all,
    many or few pairs left to decide, and more and fewer partners than the
    count keeps."""
    a = synth.candidates_on_grid(54, 1, n, shape)
    b = synth.candidates_on_grid(54, 2, 90, shape)
    check_cluster(fh, co, a, 1.0)
    check_coinc(fh, co, a, b, 0.0, 0.0, 0.0, (1, 1, 1, 1))
    check_coinc(fh, co, b, a, 0.0, 0.0, 0.0, (0, 1, 1, 2))


@pytest.mark.parametrize("n", [7, 8, 9, 8191, 8200])
@pytest.mark.parametrize("skip", [0, 1, 3])
def test_counts_of_any_alignment(fh, co, n, skip):
    """The scan moves 16 bytes at a time where its arrays start on 16: a
    caller's partner counts may start on any 4."""
    import ctypes

    import torch
    a = synth.candidate_set(55, 1, n, clusters=3, cluster_size=4)
    b = synth.candidate_set(55, 2, 200, clusters=3, cluster_size=4)
    win = (2, 2, 2, 2)
    want, w1, _ = co.coincidences(a, b, 0.0, 0.0, 0.0, win)
    m1 = torch.full((n + 8,), -7, dtype=torch.int32, device="cuda")
    pairs = torch.empty((max(1, len(want)), 2), dtype=torch.int32, device="cuda")
    da, db = dev(a), dev(b)
    w = (ctypes.c_double * 4)(*win)
    k = ctypes.c_int64(0)
    rc = fh.load().fh_coincidences(
        ctypes.c_void_p(da.data_ptr()), n, 0.0, ctypes.c_void_p(db.data_ptr()), 200, 0.0, 0.0,
        ctypes.cast(w, ctypes.c_void_p), ctypes.c_void_p(pairs.data_ptr()), pairs.shape[0],
        ctypes.byref(k), ctypes.c_void_p(m1.data_ptr() + 4 * skip), None,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0 and k.value == len(want)
    got = m1.cpu().numpy()
    assert np.array_equal(got[skip:skip + n], w1)
    assert (got[:skip] == -7).all() and (got[skip + n:] == -7).all()
    assert np.array_equal(pairs.cpu().numpy()[:len(want)], want.reshape(-1, 2))


@pytest.mark.parametrize("skip", [1, 2, 5])
def test_candidates_on_any_multiple_of_8_bytes(fh, co, skip):
    """Candidate records that do not start on 16 bytes."""
    import torch

    def shifted(c):
        buf = torch.zeros(c.size + 8, dtype=torch.float64, device="cuda")
        view = buf[skip:skip + c.size].view(c.shape)
        view.copy_(torch.from_numpy(c))
        assert view.data_ptr() % 16 == 8 * (skip % 2)
        return view

    a = synth.candidate_set(56, 1, 500, clusters=10, cluster_size=4)
    b = synth.candidate_set(56, 2, 300, clusters=10, cluster_size=4)
    want, wn = co.cluster(a, 2.0)
    lab, n = fh.fh_cluster(shifted(a), 2.0)
    assert n == wn and np.array_equal(lab.cpu().numpy(), want)
    p, m1, m2 = fh.fh_coincidences(shifted(a), shifted(b), 0.0, 0.0, 0.0, (2, 2, 2, 2))
    wp, w1, w2 = co.coincidences(a, b, 0.0, 0.0, 0.0, (2, 2, 2, 2))
    assert np.array_equal(p.cpu().numpy(), wp.reshape(-1, 2))
    assert np.array_equal(m1.cpu().numpy(), w1) and np.array_equal(m2.cpu().numpy(), w2)


def test_scratch_shared_by_threads_and_streams(fh):
    """Calls of several threads, each on its own stream, share the library's
    scratch pool: every result is that of a call alone; the last plan's
    destruction between calls (which empties the pool) changes nothing."""
    import threading

    import torch
    sets = [dev(synth.candidate_set(60 + k, 0, 3000 + 500 * k, clusters=40)) for k in range(4)]
    want = [fh.fh_cluster(c, 3.0)[0].clone() for c in sets]
    torch.cuda.synchronize()
    bad = []

    def work(k):
        try:
            st = torch.cuda.Stream()
            for r in range(12):
                c = sets[(k + r) % 4]
                lab, _ = fh.fh_cluster(c, 3.0, stream=st)
                st.synchronize()
                if not torch.equal(lab, want[(k + r) % 4]):
                    bad.append((k, r))
                if r == 5:
                    _, pp = synth.random_case(3)
                    fh.fh_destroy_plan(fh.fh_create_plan(fh.make_desc(pp, 20, 1, 100)))
        except Exception as e:  # noqa: BLE001
            bad.append(repr(e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_windows_next_to_the_ends_of_binary64(fh, co):
    """A smallest subnormal apart, with windows whose product with the width lies
    within half of it: the quotient decides."""
    a = synth.candidate_set(3, 1, 40, clusters=2, cluster_size=3)
    a[:, 0] = 0.0
    a[:, 4] = 2.0 ** -474
    b = a.copy()
    b[:, 0] = 2.0 ** -1074
    for w in (0.5, 0.75, 1.0, 1.25):
        check_coinc(fh, co, a, b, 0.0, 0.0, 0.0, (w * 2.0 ** -600, 1.0, 1.0, 1.0))


# a reach below binary32's range on a very wide width, and a very wide reach on a width
# below it: a tenth of what is allowed apart, and ten times that
@pytest.mark.parametrize("width, reach", [(1e30, 1e-50), (1e-50, 1e20)])
def test_reaches_beyond_binary32(fh, co, width, reach):
    a = synth.candidate_set(4, 1, 60, clusters=2, cluster_size=3)
    a[:, 1] = 0.0
    a[:, 5] = width
    b = a.copy()
    b[:30, 1] = 0.1 * width * reach
    b[30:, 1] = 10.0 * width * reach
    check_coinc(fh, co, a, b, 0.0, 0.0, 0.0, (1.0, reach, 1.0, 1.0))
    c = np.concatenate([a, b])
    c[:, [0, 2, 3]] = c[0, [0, 2, 3]]
    check_cluster(fh, co, c, reach)


def test_sets_whose_records_do_not_fit_in_memory(fh):
    """With the device's memory taken up to what the sets' cells need, clustering and
    coincidences do without the 32-byte records (and the kept partners): labels and
    pairs are those of the calls with room."""
    import torch
    n = 16_000_000                        # records 512 MB per set, all else below 400 MB
    g = torch.Generator(device="cuda")
    g.manual_seed(11)

    def rand():
        return torch.rand(n, dtype=torch.float64, device="cuda", generator=g)

    a = torch.empty((n, 8), dtype=torch.float64, device="cuda")
    a[:, 0] = 6.28 * rand()
    a[:, 1] = 3.0 * rand() - 1.5
    a[:, 2] = 50.0 + 200.0 * rand()
    a[:, 3] = -1e-9 * rand()
    a[:, 4:] = torch.tensor([2e-2, 2e-2, 2e-4, 2e-11], dtype=torch.float64, device="cuda")
    b = a[torch.randperm(n, device="cuda", generator=g)].contiguous()
    b[:, 0] += 0.5 * 2e-2
    m = 4_000_000                         # set 1 of the coincidences
    win = (2.0, 2.0, 2.0, 2.0)
    lab, k = fh.fh_cluster(a, 3.0)
    p, m1, m2 = fh.fh_coincidences(a[:m], b, 0.0, 0.0, 0.0, win, capacity=2 * m)
    assert 0 < k < n and len(p) >= m // 4
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    outputs = torch.empty(1 << 29, dtype=torch.uint8, device="cuda")
    fill, left = [], 500 << 20
    while torch.cuda.mem_get_info()[0] > left + (2 << 20):
        step = min(4 << 30, torch.cuda.mem_get_info()[0] - left)
        fill.append(torch.empty(step, dtype=torch.uint8, device="cuda"))
    assert torch.cuda.mem_get_info()[0] < 2 * left
    del outputs                           # (into torch's cache, for the calls' outputs)
    try:
        lab2, k2 = fh.fh_cluster(a, 3.0)
        p2, n1, n2 = fh.fh_coincidences(a[:m], b, 0.0, 0.0, 0.0, win, capacity=2 * m)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert k2 == k and torch.equal(lab2, lab)
    assert torch.equal(p2, p) and torch.equal(n1, m1) and torch.equal(n2, m2)
