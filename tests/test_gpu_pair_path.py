"""Which sar_backproject calls take the pair path, and the path itself where
the rule and not the test's size decides: images against the copying kernel
(sar_backproject_noalloc) with the bounds of tests/test_gpu_pairs.py."""
import pytest

import synth
from tests.test_gpu_pairs import _compare, _frames

pytestmark = pytest.mark.gpu


def _plan(n_rx, M, nx, ny, spacing=0.025, bins=None, n_samples=512):
    import paper_2306_09784_gb300 as sar
    radar = synth.Radar(n_samples=n_samples, n_rx=n_rx, os=4)
    grid = synth.Grid(-spacing * nx / 2, 2.0, spacing, spacing, nx, ny)
    q_tx, q_rx = synth.trajectory(radar, 16)
    crop = (0, bins - 1) if bins else synth.crop_for(radar, grid, q_tx, q_rx)
    return sar.Plan.from_radar(radar, max_pulses=M, grid=grid, crop=crop)


@pytest.mark.parametrize("taken,kw", [
    (True, dict(n_rx=4, M=1024, nx=512, ny=512)),            # an ordinary frame
    (True, dict(n_rx=16, M=256, nx=1201, ny=601)),
    (True, dict(n_rx=1, M=4096, nx=256, ny=256, spacing=0.1)),  # one Rx: only long windows pay
    (False, dict(n_rx=1, M=2048, nx=512, ny=512, spacing=0.01)),
    (False, dict(n_rx=4, M=64, nx=128, ny=128)),             # a small call
    (False, dict(n_rx=1, M=16384, nx=64, ny=64, bins=2048)),  # few tiles of whole spectra
    (False, dict(n_rx=4, M=2048, nx=64, ny=128, bins=2048)),
    (False, dict(n_rx=1, M=16, nx=2048, ny=2048, spacing=0.01)),  # few chirps on many tiles
    (False, dict(n_rx=4, M=4, nx=2048, ny=2048, spacing=0.01)),
])
def test_calls_that_gain_take_the_pair_path(taken, kw):
    plan = _plan(**kw)
    got, nbytes = plan.pair_path(kw["M"])
    assert got == taken
    assert (nbytes > 0) == taken  # a plan whose largest call does not gain keeps no workspace
    if taken:
        rows = kw["M"] * kw["n_rx"]
        assert rows * plan.info.n_bins * 16 <= nbytes <= plan.info.device_bytes
        assert plan.pair_path(1)[0] is False  # its small calls do not take it
    import paper_2306_09784_gb300 as sar
    for bad in (0, kw["M"] + 1):
        with pytest.raises(sar.SarError):
            plan.pair_path(bad)


@pytest.mark.parametrize("n_rx,M,fd,taken", [(1, 9001, 0.0, True), (1, 3001, 0.0, False), (2, 1203, 2.0, True),
                                             (3, 1100, 0.0, True), (4, 700, 1.0, True), (6, 501, 0.0, True)])
def test_long_windows(n_rx, M, fd, taken):
    """Wide tiles, so that few channels gain too: every pixel loop of the path
    (and one call just short of the line)."""
    plan, prof, qt, qr, fdopp = _frames(n_rx, M, synth.Grid(-11.0, 2.0, 0.09, 0.1, 240, 200), precision=n_rx % 2,
                                        fd=fd)
    assert plan.pair_path(M)[0] == taken
    _compare(plan, prof, M, qt, qr, fdopp)


@pytest.mark.parametrize("case", [
    dict(heading=0.4), dict(y0=0.1), dict(fd=3.0), dict(fd=3.0, heading=-0.3), dict(sign=-1), dict(crop=(40, 90)),
    dict(crop=(0, 1023)), dict(os_factor=1), dict(os_factor=16), dict(near=True), dict(precision=1, near=True, fd=2.0)])
@pytest.mark.parametrize("n_rx,M", [(4, 2201), (6, 701)])
def test_options(case, n_rx, M):
    """The options of tests/test_gpu_pairs.py at sizes beyond the line."""
    case = dict(case)
    y0 = case.pop("y0", 1.2)
    if case.pop("near", False):
        y0 = -3.0
    plan, prof, qt, qr, fd = _frames(n_rx, M, synth.Grid(-4.1, y0, 0.033, 0.03, 250, 270), **case)
    assert plan.pair_path(M)[0]
    _compare(plan, prof, M, qt, qr, fd)
    _compare(plan, prof, M, qt, qr, fd, accumulate=True)


def test_wait_that_runs_out_is_reported():
    """With no polls every CTA gives up at its first block: the call is flagged
    as timed out, and after the check the next call is right bit for bit."""
    import torch
    import paper_2306_09784_gb300 as sar
    M = 600
    plan, prof, qt, qr, _ = _frames(4, M, synth.Grid(-4.1, 1.2, 0.033, 0.03, 250, 270))
    assert plan.pair_path(M)[0]
    ref = plan.backproject(prof, M, qt, qr)
    assert plan.check_errors() == sar.SAR_OK
    for polls in (-2, -100):
        with pytest.raises(sar.SarError):
            plan.set_wait_limit(polls)
    plan.set_wait_limit(0)
    left = torch.full_like(ref, complex(7.0, -7.0))
    plan.backproject(prof, M, qt, qr, image=left)
    assert plan.check_errors() == sar.SAR_ETIMEOUT
    assert bool((left == complex(7.0, -7.0)).all())  # nothing half-done was written
    plan.set_wait_limit()
    got = plan.backproject(prof, M, qt, qr)
    assert plan.check_errors() == sar.SAR_OK
    assert torch.equal(got, ref)


def test_nothing_is_left_behind_by_a_call_that_gave_up():
    """Split tiles are counted per call: after calls that gave up (no status
    read in between), after a captured call and across both kernels and chirp
    counts, each call equals its own first result bit for bit."""
    import torch
    M, small = 600, 90
    plan, prof, qt, qr, _ = _frames(4, M, synth.Grid(-4.1, 1.2, 0.033, 0.03, 250, 270))
    assert plan.pair_path(M)[0] and not plan.pair_path(small)[0]
    beat = torch.randn(small, 4, 256, dtype=torch.complex64, device="cuda",
                       generator=torch.Generator("cuda").manual_seed(2))
    prof_s, qt_s, qr_s = plan.range_compress(beat), qt[:small].contiguous(), qr[:small].contiguous()
    calls = {M: (prof, M, qt, qr), small: (prof_s, small, qt_s, qr_s), 41: (prof_s, 41, qt_s, qr_s)}
    ref = {n: plan.backproject(*c).clone() for n, c in calls.items()}
    img = torch.zeros_like(ref[M])
    torch.cuda.synchronize()
    graphs, stream = {}, torch.cuda.Stream()
    for n, c in calls.items():
        graphs[n] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graphs[n], stream=stream):
            plan.backproject(*c, image=img, stream=stream)
    for n in (small, M, 41, M, small, 41):
        plan.set_wait_limit(0)
        plan.backproject(*calls[M])
        plan.set_wait_limit()
        got = plan.backproject(*calls[n])
        assert torch.equal(got, ref[n]), n
        img.zero_()
        graphs[n].replay()
        assert torch.equal(img, ref[n]), n
        for k in (41, small, M):  # and ordinary calls after the replay
            assert torch.equal(plan.backproject(*calls[k]), ref[k]), (n, k)


@pytest.mark.parametrize("M0,M1", [(1101, 620), (90, 47)])  # on the pair path, and below its line
def test_calls_on_several_streams_and_ordered_replays(M0, M1):
    """Calls of one plan with different chirps, profiles and arrays alternate on
    two streams, then with replays of captured calls that the caller orders by
    events: every image is its call's own, bit for bit."""
    import torch
    plan, prof, qt, qr, _ = _frames(4, M0, synth.Grid(-4.1, 1.2, 0.033, 0.03, 250, 270))
    beat = torch.randn(M1, 4, 256, dtype=torch.complex64, device="cuda",
                       generator=torch.Generator("cuda").manual_seed(3))
    qt1 = qt[:M1].flip(0).contiguous()
    qr1 = (qt1[:, None, :] + 2.5 * (qr[:M1] - qt[:M1, None, :])).contiguous()
    frames = [(prof, M0, qt, qr), (plan.range_compress(beat), M1, qt1, qr1)]
    assert [plan.pair_path(f[1])[0] for f in frames] == [M0 > 500] * 2
    ref = [plan.backproject(*f).clone() for f in frames]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [torch.zeros_like(ref[0]) for _ in range(8)]
    for i, o in enumerate(outs):
        plan.backproject(*frames[i % 2], image=o, stream=streams[(i + i // 4) % 2])
    torch.cuda.synchronize()
    assert all(torch.equal(o, ref[i % 2]) for i, o in enumerate(outs))
    img, graph = torch.zeros_like(ref[0]), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=streams[0]):
        plan.backproject(*frames[0], image=img, stream=streams[0])
    for i, o in enumerate(outs):
        img.zero_(), o.zero_()
        torch.cuda.synchronize()
        ev = torch.cuda.Event()
        if i % 2:  # the replay, then the call
            with torch.cuda.stream(streams[0]):
                graph.replay()
            ev.record(streams[0])
            ev.wait(streams[1])
            plan.backproject(*frames[1], image=o, stream=streams[1])
        else:  # the call, then the replay
            plan.backproject(*frames[1], image=o, stream=streams[1])
            ev.record(streams[1])
            ev.wait(streams[0])
            with torch.cuda.stream(streams[0]):
                graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(img, ref[0]) and torch.equal(o, ref[1])


@pytest.mark.parametrize("minb", [2, 3])
def test_a_block_that_was_set_is_kept(minb):
    """Below the line, a set block cuts the work as it cuts sar_backproject_noalloc's
    (the same tiles split at the same chirps: the same sums, bit for bit), also
    above the largest that fits minb CTAs per SM; that one block and a new
    plan's leave the choice to the call."""
    import torch
    import paper_2306_09784_gb300 as sar
    M = 60
    plan, prof, qt, qr, _ = _frames(8, M, synth.Grid(-2.1, 1.2, 0.033, 0.03, 150, 130))
    assert not plan.pair_path(M)[0]
    lib, first = sar.load_library(), plan.launch_shape()
    img = plan.backproject(prof, M, qt, qr)
    most = plan.launch_shape()["pulses_per_block"]
    assert 3 <= most <= 12
    for mb in (1, 2, most + 1, most + 4):
        shape = plan.set_launch(4, minb, mb)
        assert shape["pulses_per_block"] == mb
        ref = torch.zeros_like(img)
        assert lib.sar_backproject_noalloc(plan.handle, prof.data_ptr(), M, qt.data_ptr(), qr.data_ptr(), None,
                                           ref.data_ptr(), 0, torch.cuda.current_stream().cuda_stream) == sar.SAR_OK
        assert torch.equal(plan.backproject(prof, M, qt, qr), ref), mb
    plan.set_launch(first["rx_group"], first["regs_ctas_per_sm"], first["pulses_per_block"])
    assert plan.launch_shape() == first
    assert torch.equal(plan.backproject(prof, M, qt, qr), img)


def test_workspace_is_given_back():
    """The memory returns to the device and to the plan's count, and calls go on
    by the other kernel; a budget that does not hold the workspace leaves a plan
    without it and without a part of it."""
    import torch
    import paper_2306_09784_gb300 as sar
    M, grid = 1101, synth.Grid(-4.1, 1.2, 0.033, 0.03, 250, 270)
    plan, prof, qt, qr, _ = _frames(4, M, grid)
    taken, nbytes = plan.pair_path(M)
    assert taken and nbytes > 0
    before = plan.backproject(prof, M, qt, qr)
    torch.cuda.synchronize()
    held, free = int(plan.info.device_bytes), torch.cuda.mem_get_info()[0]
    plan.release_pairs()
    plan.launch_shape()  # reads the plan's info
    assert plan.pair_path(M) == (False, 0)
    assert held - plan.info.device_bytes >= nbytes
    assert torch.cuda.mem_get_info()[0] >= free
    after = plan.backproject(prof, M, qt, qr)
    assert ((after - before).abs().norm() / before.abs().norm()).item() < 1e-5
    plan.release_pairs()
    left = int(plan.info.device_bytes)
    tight = sar.Plan.from_radar(synth.Radar(n_samples=256, n_rx=4, os=4), max_pulses=M, grid=grid,
                                crop=(plan.info.crop_lo, plan.info.crop_hi), hbm_budget=left + nbytes // 2)
    assert tight.pair_path(M) == (False, 0) and tight.info.device_bytes == left


def test_workspace_for_calls_whose_pairs_fit_l2():
    """A plan whose largest call does not gain, as its pairs leave the L2 cache,
    has a workspace all the same when its shorter calls gain."""
    for n_rx, side, bins, short, M in ((4, (320, 320), 1024, 1400, 8000), (6, (288, 1024), 2048, 640, 1156)):
        plan = _plan(n_rx, M, *side, spacing=0.025 if n_rx == 4 else 0.01, bins=bins)
        assert [plan.pair_path(m)[0] for m in (short, M)] == [True, False] and plan.pair_path(short)[1] > 0


def test_a_refused_call_leaves_no_error_behind():
    """A call on the legacy stream beside the capture of a blocking stream is
    refused; the same call after the capture is a call like any other."""
    import ctypes

    import torch
    import paper_2306_09784_gb300 as sar
    M = 600
    plan, prof, qt, qr, _ = _frames(4, M, synth.Grid(-4.1, 1.2, 0.033, 0.03, 250, 270))
    assert plan.pair_path(M)[0]
    ref = plan.backproject(prof, M, qt, qr)
    torch.cuda.synchronize()
    cu, lib = ctypes.CDLL("libcuda.so.1"), sar.load_library()
    stream, graph, img = ctypes.c_void_p(), ctypes.c_void_p(), torch.zeros_like(ref)

    def call():
        return lib.sar_backproject(plan.handle, prof.data_ptr(), M, qt.data_ptr(), qr.data_ptr(), None, img.data_ptr(),
                                   0, None)

    torch.cuda.synchronize()
    assert cu.cuStreamCreate(ctypes.byref(stream), 0) == 0
    assert cu.cuStreamBeginCapture_v2(stream, 2) == 0  # relaxed: only this stream's own work is captured
    refused = call()
    assert cu.cuStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert refused == sar.SAR_ECUDA
    assert call() == sar.SAR_OK
    torch.cuda.synchronize()
    assert torch.equal(img, ref) and plan.check_errors() == sar.SAR_OK
    cu.cuGraphDestroy(graph)
    cu.cuStreamDestroy_v2(stream)
