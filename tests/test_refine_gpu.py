"""Refined-grid search (Sec. "Refined Grid in the parameter space") on the GPU,
through the C ABI, against the oracle.

Refined direction, row, cell and count bit for bit; f0, spin-down and critical
ratio to 1e-12 relative.  Cases: random peakmaps with many candidates (several
transform batches), candidates at the edges of the coarse grid (the refined
band reaches outside it), spin-down refinements whose rows span one and
several 32-row slabs, and the 50 Hz line of the T_FFT = 8192 s workload on a
refined sky rectangle.
"""
import numpy as np
import pytest

from paper_1407_8333_gb300 import synth

pytestmark = pytest.mark.gpu

REL_TOL = 1e-12


@pytest.fixture(scope="module")
def fh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_8333_gb300 import build, fh as fhmod
    build.build()
    fhmod.load()
    return fhmod


def gpu_refine(fh, inp, pp, cells, rows, sky_ref, k_fdot, checks=None):
    plan = fh.fh_create_plan(fh.make_desc(pp, inp.t.shape[0], 1, max(1, inp.n_peaks)))
    try:
        if checks is not None:
            fh.fh_plan_set_input_checks(plan, checks)
        return fh.fh_refine(plan, inp.t, inp.offsets, inp.freq, inp.v, cells, rows, sky_ref,
                            k_fdot)
    finally:
        fh.fh_destroy_plan(plan)


def check(g, o, n_cand):
    assert g.shape == (n_cand,)
    for k in ("dir", "row", "cell", "count"):
        assert np.array_equal(g[k].astype(np.int64), o[k]), k
    assert np.array_equal(g["subband"], np.arange(n_cand))
    assert np.all(g["rank"] == 0)
    for k in ("f0", "fdot", "cr"):
        np.testing.assert_allclose(g[k], o[k], rtol=REL_TOL, atol=0.0, err_msg=k)


def random_sky_ref(seed, n_cand, n_ref):
    u = synth.uniform(seed, 11, np.arange(2 * n_cand * n_ref)).reshape(n_cand, n_ref, 2)
    z = u[..., 0] * 2.0 - 1.0
    ph = u[..., 1] * 2.0 * np.pi
    r = np.sqrt(1.0 - z * z)
    return np.stack([r * np.cos(ph), r * np.sin(ph), z], axis=-1)


@pytest.mark.parametrize("k_fdot", [1, 3, 10])
def test_random_candidates_match_the_oracle(fh, oracle_mod, k_fdot):
    inp, pp = synth.random_case(301 + k_fdot, n_fft=40, n_bins=50, n_fdot=16, n_dir=1, p=0.4)
    n_cand, n_ref = 29, 5
    cu = synth.uniform(400 + k_fdot, 3, np.arange(2 * n_cand)).reshape(2, n_cand)
    cells = (cu[0] * pp["n_f0"]).astype(np.int32)
    rows = (cu[1] * pp["n_fdot"]).astype(np.int32)
    # the edges of the coarse grid: the refined band reaches outside it
    cells[:4] = [0, 1, pp["n_f0"] - 1, pp["n_f0"] // 2]
    rows[:4] = [0, pp["n_fdot"] - 1, 1, 0]
    sky = random_sky_ref(500 + k_fdot, n_cand, n_ref)
    sky[:, 0] = inp.sky[0]
    g = gpu_refine(fh, inp, pp, cells, rows, sky, k_fdot)
    o = oracle_mod.refine(inp, pp, cells, rows, sky, k_fdot)
    check(g, o, n_cand)


def test_many_rows_several_slabs(fh, oracle_mod):
    """K_fdot = 20: 80 refined rows, two full 32-row slabs and a ragged one."""
    inp, pp = synth.random_case(333, n_fft=24, n_bins=30, n_fdot=9, n_dir=1, p=0.5)
    cells = np.array([5, pp["n_f0"] // 3, pp["n_f0"] - 7], dtype=np.int32)
    rows = np.array([4, 2, 6], dtype=np.int32)
    sky = random_sky_ref(334, 3, 2)
    g = gpu_refine(fh, inp, pp, cells, rows, sky, 20)
    o = oracle_mod.refine(inp, pp, cells, rows, sky, 20)
    check(g, o, 3)


def test_no_candidates_and_argument_errors(fh):
    inp, pp = synth.random_case(335, n_fft=8, n_bins=10, n_fdot=5, n_dir=1)
    sky = np.zeros((0, 1, 3))
    out = gpu_refine(fh, inp, pp, np.zeros(0, np.int32), np.zeros(0, np.int32), sky, 2)
    assert out.shape == (0,)
    one = inp.sky[None, :1]
    for kf in (0, 65):
        with pytest.raises(fh.FHError) as ei:
            gpu_refine(fh, inp, pp, [3], [2], one, kf)
        assert ei.value.code == fh.FH_ERR_INVALID_ARG
    with pytest.raises(fh.FHError) as ei:      # no refined direction
        gpu_refine(fh, inp, pp, [3], [2], np.zeros((1, 0, 3)), 2)
    assert ei.value.code == fh.FH_ERR_INVALID_ARG
    bad = inp.sky[None, :1] * 2.0               # not a unit vector
    with pytest.raises(fh.FHError) as ei:
        gpu_refine(fh, inp, pp, [3], [2], bad, 2)
    assert ei.value.code == fh.FH_ERR_INVALID_ARG
    with pytest.raises(fh.FHError) as ei:      # candidate outside the fixed-point range
        gpu_refine(fh, inp, pp, [1 << 28], [2], one, 2)
    assert ei.value.code == fh.FH_ERR_RANGE


@pytest.mark.parametrize("k_fdot", [1, 4])
def test_the_50Hz_line_on_a_refined_sky(fh, oracle_mod, k_fdot):
    """The injected line of the T_FFT = 8192 s, 150 d workload: the coarse
    candidate of its subband, refined on a 3 x 3 sky rectangle around the
    coarse direction and K_fdot spin-down."""
    w = synth.WORKLOADS["single_sky_T8192_150d_50Hz"]
    inp = synth.make_inputs(w)
    pp = w.plan_params()
    o = oracle_mod.search(inp, pp)
    sb = int((w.line_f0 - w.f_lo) / w.subband_hz)
    # the line's subband and two of its neighbours, best candidate of each
    sbs = [sb, sb - 1, sb + 1]
    cells = np.array([int(o["cell"][0, s, 0]) for s in sbs], dtype=np.int32)
    rows = np.array([int(o["row"][0, s, 0]) for s in sbs], dtype=np.int32)
    n_d = synth.doppler_number(w.f_hi, w.t_fft)
    sky = np.stack([synth.refined_sky(inp.sky[0], n_d, 3)] * len(sbs))
    g = gpu_refine(fh, inp, pp, cells, rows, sky, k_fdot)
    r = oracle_mod.refine(inp, pp, cells, rows, sky, k_fdot)
    check(g, r, len(sbs))
    assert g["count"][0] >= int(o["count"][0, sb, 0])


def test_refine_with_device_checks(fh, oracle_mod):
    """FH_CHECKS_DEVICE: the same refined candidates; unsorted frequencies are
    reported by the call (it synchronises) as FH_ERR_UNSORTED."""
    inp, pp = synth.random_case(336, n_fft=30, n_bins=40, n_fdot=12, n_dir=1, p=0.4)
    cells = np.array([10, pp["n_f0"] // 2, pp["n_f0"] - 3], dtype=np.int32)
    rows = np.array([3, 6, 9], dtype=np.int32)
    sky = random_sky_ref(337, 3, 4)
    g = gpu_refine(fh, inp, pp, cells, rows, sky, 3, checks=fh.FH_CHECKS_DEVICE)
    check(g, oracle_mod.refine(inp, pp, cells, rows, sky, 3), 3)
    # the two highest peaks of one FFT swapped, far from candidates near the
    # bottom of the band: found by the check of every frequency, not only of
    # the peaks near the candidates
    f = inp.freq.copy()
    b = int(inp.offsets[5]) - 1
    f[b - 1], f[b] = f[b], f[b - 1]
    low = np.array([8, 12], dtype=np.int32)
    plan = fh.fh_create_plan(fh.make_desc(pp, inp.t.shape[0], 1, inp.n_peaks))
    try:
        fh.fh_plan_set_input_checks(plan, fh.FH_CHECKS_DEVICE)
        with pytest.raises(fh.FHError) as ei:
            fh.fh_refine(plan, inp.t, inp.offsets, f, inp.v, low, rows[:2], sky[:2], 3)
        assert ei.value.code == fh.FH_ERR_UNSORTED
    finally:
        fh.fh_destroy_plan(plan)


# histograms of all directions and rows, of groups of directions (40 of them), of one
# direction (256 rows), of groups of rows (K = 16: 213 of 256); K = 1; FFT shares
# around a block's 256 FFTs; directions taken in two turns (12,000 of them)
@pytest.mark.parametrize("k_over, k_fdot, n_fft, n_cand, n_ref", [
    (10, 4, 255, 6, 9), (10, 4, 257, 3, 40), (10, 64, 40, 2, 3), (16, 64, 30, 2, 2),
    (1, 2, 300, 5, 4), (3, 1, 2049, 1, 1), (30, 64, 4, 1, 12000)])
def test_groups_and_shares(fh, oracle_mod, k_over, k_fdot, n_fft, n_cand, n_ref):
    inp, pp = synth.random_case(700 + n_fft + k_over, n_fft=n_fft, n_bins=24, k_over=k_over,
                                n_fdot=9, n_dir=1, p=0.3)
    cu = synth.uniform(800 + n_fft, 3, np.arange(2 * n_cand)).reshape(2, n_cand)
    cells = (cu[0] * pp["n_f0"]).astype(np.int32)
    rows = (cu[1] * pp["n_fdot"]).astype(np.int32)
    sky = random_sky_ref(900 + n_fft, n_cand, n_ref)
    g = gpu_refine(fh, inp, pp, cells, rows, sky, k_fdot)
    o = oracle_mod.refine(inp, pp, cells, rows, sky, k_fdot)
    check(g, o, n_cand)


def _far_case(f_cells):
    n_fft, kt, f0 = 40, 16.0, 100.0
    f = f0 + (2.0 ** 30 + f_cells) / kt
    t = np.arange(n_fft) * 1.0 + 1e5
    inp = synth.Inputs(w=None, t=t, offsets=np.arange(n_fft + 1, dtype=np.int64) * len(f),
                       freq=np.tile(f, n_fft), v=np.zeros((n_fft, 3)), sky=np.array([[0., 0., 1.]]))
    pp = dict(t_fft=1.0, k_over=16, f0_min=f0, n_f0=2000, fdot_min=0.0, fdot_step=5e-6, n_fdot=9,
              t_ref=0.0, subband_cells=100, top_k=1, excl_cells=0, sep_cells=0, n_thr=0, p0=0.1)
    return inp, pp


def test_rows_far_outside_the_plan(fh):
    """A candidate row whose shift (8 cells a row) lies 2^30 cells from the plan's band:
    peaks there are beyond the fixed-point range and reported, by the device checks
    (1) as by the host's, which look at every peak."""
    sky = np.array([[[0.0, 0.0, 1.0]]])
    for cells, refused in ((np.arange(-4000.0, 40000.0), True), (np.arange(1e6, 1e6 + 50), False)):
        inp, pp = _far_case(cells)
        plan = fh.fh_create_plan(fh.make_desc(pp, inp.t.shape[0], 1, inp.n_peaks))
        try:
            for checks in (0, 1):
                fh.fh_plan_set_input_checks(plan, checks)
                args = (plan, inp.t, inp.offsets, inp.freq, inp.v, [1000], [2 ** 27 - 2], sky, 1)
                if refused or checks == 0:
                    with pytest.raises(fh.FHError) as ei:
                        fh.fh_refine(*args)
                    assert ei.value.code == fh.FH_ERR_RANGE
                else:
                    assert fh.fh_refine(*args)["count"][0] == 0
        finally:
            fh.fh_destroy_plan(plan)


def test_a_refused_refinement_leaves_nothing_queued(fh):
    """A refined drift too wide for shared memory is refused with nothing left on the
    stream that reads the caller's page-locked arrays (256 MB), behind work that keeps
    the stream busy."""
    import torch
    n_fft, per = 64, 500_000

    def pinned(x):
        return torch.from_numpy(np.ascontiguousarray(x)).pin_memory().numpy()

    t, v = pinned(np.arange(n_fft) * 512.0), pinned(np.zeros((n_fft, 3)))
    offsets = pinned(np.arange(n_fft + 1, dtype=np.int64) * per)
    freq = pinned(np.tile(50.0 + np.arange(per) * 1e-6, n_fft))
    cells, rows = pinned(np.array([1000], np.int32)), pinned(np.array([3], np.int32))
    sky = pinned(np.array([[[0.0, 0.0, 1.0]]]))
    _, pp = synth.random_case(5)
    plan = fh.fh_create_plan(fh.make_desc(pp, n_fft, 1, 1000))   # (kernels loaded)
    fh.fh_refine(plan, t, offsets, freq, v, cells, rows, sky, 1)
    fh.fh_destroy_plan(plan)
    pp["fdot_step"] = 100.0 / (pp["k_over"] * pp["t_fft"] * t[-1])   # 100 cells a row
    pp["t_ref"] = 0.0
    plan = fh.fh_create_plan(fh.make_desc(pp, n_fft, 1, 1000))
    try:
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            torch.cuda._sleep(1_000_000_000)
        with pytest.raises(fh.FHError) as ei:
            fh.fh_refine(plan, t, offsets, freq, v, cells, rows, sky, 1, stream=st)
        assert ei.value.code == fh.FH_ERR_CUDA
        assert st.query()
    finally:
        torch.cuda.synchronize()
        fh.fh_destroy_plan(plan)


def test_starts_that_do_not_fit_in_memory(fh):
    """600 MB of stripe starts (108 candidates x 60 directions x 256 rows x 90 starts)
    with less than 450 MB to be had: taken in turns, the result is that of one turn."""
    import torch
    inp, pp = synth.random_case(77, n_fft=40, n_bins=60, k_over=30, n_fdot=9, n_dir=1, p=0.3)
    rng = np.random.RandomState(5)
    cells, rows = rng.randint(0, pp["n_f0"], 108), rng.randint(0, 9, 108)
    sky = random_sky_ref(6, 108, 60)
    plan = fh.fh_create_plan(fh.make_desc(pp, 40, 1, inp.n_peaks))
    args = (plan, inp.t, inp.offsets, inp.freq, inp.v, cells, rows, sky, 64)
    fill, left = [], 150 << 20
    try:
        want = fh.fh_refine(*args)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        while torch.cuda.mem_get_info()[0] > left + (2 << 20):
            fill.append(torch.empty(min(4 << 30, torch.cuda.mem_get_info()[0] - left),
                                    dtype=torch.uint8, device="cuda"))
        got = fh.fh_refine(*args)
    finally:
        del fill
        torch.cuda.empty_cache()
        fh.fh_destroy_plan(plan)
    assert want["count"].max() > 5 and np.array_equal(got, want)
