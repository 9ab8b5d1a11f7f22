"""A plan's step captured into a CUDA graph and replayed (batching row a7).

After one eager call of the same shape (which sizes the plan's window table),
fh_correct_doppler on device inputs, fh_transform and fh_select_candidates
into device memory enqueue only kernels, memsets and device copies, so the
sequence can be captured and replayed.  Checked here through the C ABI: each
replay's candidates equal a fresh eager plan's, bit for bit, and the CPU
oracle's (cells, rows and counts bit for bit; f0, fdot and CR to 1e-12
relative), including after the device inputs were overwritten in place (same
addresses, new contents).
"""
import numpy as np
import pytest

from paper_1407_8333_gb300 import synth

pytestmark = pytest.mark.gpu

REL_TOL = 1e-12


def _same_as_oracle(got, o, pp, n_dir):
    c = got.reshape(n_dir, -1, pp["top_k"])
    for k in ("cell", "row", "count"):
        assert np.array_equal(c[k], o[k]), k
    for k in ("f0", "fdot", "cr"):
        a, b = c[k], o[k]
        same = (a == b) | (np.isnan(a) & np.isnan(b))
        assert np.all(same | (np.abs(a - b) <= REL_TOL * np.abs(b))), k


@pytest.fixture(scope="module")
def fh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_8333_gb300 import build, fh as fhmod
    build.build()
    fhmod.load()
    return fhmod


def _eager(fh, inp, pp, n_dir, schedule):
    import torch
    plan = fh.fh_create_plan(fh.make_desc(pp, inp.t.shape[0], n_dir, inp.n_peaks,
                                          schedule=schedule))
    try:
        dev = [torch.from_numpy(x).cuda() for x in (inp.t, inp.offsets, inp.freq, inp.v, inp.sky)]
        fh.fh_correct_doppler(plan, *dev)
        fh.fh_transform(plan, 0, n_dir)
        return fh.fh_select_candidates(plan, 0, n_dir)
    finally:
        fh.fh_destroy_plan(plan)


@pytest.mark.parametrize("schedule", [0, 1])
def test_step_replays_from_a_cuda_graph(fh, oracle_mod, schedule):
    import torch
    inp, pp = synth.random_case(91, n_fft=48, n_bins=160, n_fdot=70, n_dir=3, p=0.3)
    n_dir = inp.sky.shape[0]
    # a second input of the same shape: frequencies one bin higher, other velocities
    inp2 = synth.Inputs(w=inp.w, t=inp.t, offsets=inp.offsets,
                        freq=inp.freq + 1.0 / pp["t_fft"], v=inp.v[::-1].copy(), sky=inp.sky)
    want = [_eager(fh, x, pp, n_dir, schedule) for x in (inp, inp2)]
    oracle = [oracle_mod.search(x, pp) for x in (inp, inp2)]

    plan = fh.fh_create_plan(fh.make_desc(pp, inp.t.shape[0], n_dir, inp.n_peaks,
                                          schedule=schedule))
    try:
        dev = [torch.from_numpy(x).cuda() for x in (inp.t, inp.offsets, inp.freq, inp.v, inp.sky)]
        n_sb = -(-pp["n_f0"] // pp["subband_cells"])
        cand = torch.zeros(n_dir * n_sb * pp["top_k"] * 48, dtype=torch.uint8, device="cuda")
        s = torch.cuda.Stream()

        def step():
            fh.fh_correct_doppler(plan, *dev, stream=s)
            fh.fh_transform(plan, 0, n_dir, None, stream=s)
            fh.fh_select_candidates(plan, 0, n_dir, cand, stream=s)

        with torch.cuda.stream(s):
            step()                      # eager: sizes the plan's buffers
        torch.cuda.synchronize()
        launches = fh.fh_plan_launches(plan)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            step()
        captured = fh.fh_plan_launches(plan) - launches
        assert captured > 0

        def replay():
            cand.zero_()
            g.replay()
            torch.cuda.synchronize()
            fh.fh_sync(plan)            # device-side input checks stayed clean
            return cand.cpu().numpy().view(fh.CANDIDATE_DTYPE).copy()

        for k in range(2):
            got = replay()
            assert np.array_equal(got, want[0]), k
            _same_as_oracle(got, oracle[0], pp, n_dir)
        # new contents at the same addresses
        dev[2].copy_(torch.from_numpy(inp2.freq))
        dev[3].copy_(torch.from_numpy(inp2.v))
        got = replay()
        assert np.array_equal(got, want[1])
        _same_as_oracle(got, oracle[1], pp, n_dir)
        assert not np.array_equal(want[0], want[1])
    finally:
        torch.cuda.synchronize()
        fh.fh_destroy_plan(plan)


FIRST_CALL = r'''
import sys
sys.path.insert(0, %(root)r)
import numpy as np, torch
import oracle
from paper_1407_8333_gb300 import build, fh, synth
build.build(); fh.load()
s = synth.spectra_case(7, 6, 600, wander_amp=30.0, wander_f=(50.01, 50.05), wander_width=5)
sp, sa = torch.from_numpy(s.s_p).cuda(), torch.from_numpy(s.s_ar).cuda()
ws = torch.empty(fh.fh_peakmap_select_workspace(6, 600), dtype=torch.uint8, device="cuda")
out = (torch.zeros(7, dtype=torch.int64, device="cuda"),
       torch.zeros(1800, dtype=torch.int32, device="cuda"),
       torch.zeros(1800, dtype=torch.float64, device="cuda"))
st = torch.cuda.Stream()
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=st):
    fh.fh_peakmap_select(sp, sa, 2.5, s.k0, s.t_fft, out=out, workspace=%(ws)s, stream=st)
for k in range(2):
    for x in out:
        x.zero_()
    g.replay()
    torch.cuda.synchronize()
    o, b = oracle.peakmap.select_peaks(s.s_p, s.s_ar, 2.5)
    assert np.array_equal(out[0].cpu().numpy(), o)
    assert np.array_equal(out[1].cpu().numpy()[:len(b)], b)
print("ok")
'''


@pytest.mark.parametrize("ws", ["ws", "None"])
def test_first_call_of_a_process_is_captured(ws):
    """The selection captured as a process's first call of the library, with a
    caller's workspace and with scratch of its own: making the scratch pool ends no
    capture."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FIRST_CALL % dict(root=root, ws=ws)],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]


@pytest.mark.parametrize("eager, captured", [(8, 6), (2, 1), (3, 1)])
def test_fewer_directions_are_captured_after_more(fh, oracle_mod, eager, captured):
    """An eager call sizes the window table for every smaller one: fewer directions
    make narrower and so more tiles (8 directions of 600 rows x 640 cells in 76 items,
    6 in 114), and a capture cannot allocate."""
    import torch
    inp, pp = synth.random_case(92, n_fft=30, n_bins=64, n_fdot=600, n_dir=eager, p=0.3)
    want = oracle_mod.search(inp, pp, want_maps=True)["maps"][:captured]
    plan = fh.fh_create_plan(fh.make_desc(pp, 30, eager, inp.n_peaks))
    try:
        dev = [torch.from_numpy(x).cuda() for x in (inp.t, inp.offsets, inp.freq, inp.v, inp.sky)]
        maps = torch.empty((captured, pp["n_fdot"], pp["n_f0"]), dtype=torch.int32, device="cuda")
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        fh.fh_correct_doppler(plan, *dev, stream=s)
        fh.fh_transform(plan, 0, eager, stream=s)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            fh.fh_transform(plan, 0, captured, maps, stream=s)
        for _ in range(2):
            maps.fill_(-1)
            g.replay()
            torch.cuda.synchronize()
            assert np.array_equal(maps.cpu().numpy(), want)
    finally:
        torch.cuda.synchronize()
        fh.fh_destroy_plan(plan)
