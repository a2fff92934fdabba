"""The pair path of sar_backproject (large calls) against the copying kernel
(sar_backproject_noalloc, any size): the same arithmetic per update, so the
images agree up to FP32 summation order (1e-5) for every form the path takes."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _frames(n_rx, M, grid=None, pixels=None, precision=0, heading=0.0, y0=2.0, os_factor=4, fd=0.0, crop=None,
            sign=1, speed=10.0):
    import torch
    import paper_2306_09784_gb300 as sar
    radar = synth.Radar(n_samples=256, n_rx=n_rx, os=os_factor)
    rng = np.random.Generator(np.random.PCG64(17 * n_rx + M))
    q_tx, q_rx = synth.trajectory(radar, M, speed=speed, jitter=0.01, rng=rng)
    rot = np.array([[np.cos(heading), np.sin(heading)], [-np.sin(heading), np.cos(heading)]])
    q_tx, q_rx = q_tx @ rot, q_rx @ rot
    box = grid or synth.Grid(pixels[:, 0].min(), pixels[:, 1].min(), float(np.ptp(pixels[:, 0])),
                             float(np.ptp(pixels[:, 1])), 2, 2)
    plan = sar.Plan.from_radar(radar, max_pulses=M, grid=grid, pixels_xy=pixels, precision=precision,
                               crop=crop or synth.crop_for(radar, box, q_tx, q_rx), max_doppler_bins=fd,
                               phase_sign=sign)
    g = torch.Generator(device="cuda").manual_seed(n_rx)
    beat = torch.randn(M, n_rx, 256, dtype=torch.complex64, device="cuda", generator=g)
    prof = plan.range_compress(beat)
    qt = torch.from_numpy(np.ascontiguousarray(q_tx)).cuda()
    qr = torch.from_numpy(np.ascontiguousarray(q_rx)).cuda()
    fdopp = None
    if fd:
        fdopp = (torch.rand(plan.n_pixels, device="cuda", generator=g) * 2.2 - 1.1) * fd  # some beyond the bound
    return plan, prof, qt, qr, fdopp


def _compare(plan, prof, M, qt, qr, fdopp=None, accumulate=False):
    import torch
    import paper_2306_09784_gb300 as sar
    assert plan.info.n_tiles * M * qr.shape[1] >= 65536  # the pair path
    g = torch.Generator(device="cuda").manual_seed(5)
    base = torch.randn(plan.n_pixels, dtype=torch.complex64, device="cuda", generator=g)
    got, ref = base.clone(), base.clone()
    plan.backproject(prof, M, qt, qr, image=got, accumulate=accumulate, fdopp=fdopp)
    rc = sar.load_library().sar_backproject_noalloc(
        plan.handle, prof.data_ptr(), M, qt.data_ptr(), qr.data_ptr(), fdopp.data_ptr() if fdopp is not None else None,
        ref.data_ptr(), int(accumulate), torch.cuda.current_stream().cuda_stream)
    assert rc == sar.SAR_OK
    torch.cuda.synchronize()
    assert torch.isfinite(torch.view_as_real(got)).all()
    err = ((got - ref).abs().norm() / ref.abs().norm()).item()
    assert err < 1e-5, err
    # and every 32 x 32 neighbourhood of the output order
    n = plan.n_pixels // 1024 * 1024
    d, r = (got - ref)[:n].abs().square().view(-1, 1024).sum(1), ref[:n].abs().square().view(-1, 1024).sum(1)
    assert (d / torch.maximum(r, r.mean())).max().item() < 1e-9
    return got


@pytest.mark.parametrize("n_rx,M", [(1, 1025), (2, 600), (3, 401), (4, 257), (6, 200), (8, 131), (16, 70), (64, 17)])
def test_rx_counts_and_ragged_chirps(n_rx, M):
    plan, prof, qt, qr, _ = _frames(n_rx, M, synth.Grid(-4.1, 1.2, 0.033, 0.03, 250, 270), precision=n_rx % 2)
    _compare(plan, prof, M, qt, qr)
    assert plan.check_errors() == 0


@pytest.mark.parametrize("case", [
    dict(heading=0.4), dict(y0=0.1), dict(fd=3.0), dict(fd=3.0, heading=-0.3), dict(sign=-1), dict(crop=(40, 90)),
    dict(crop=(0, 1023)), dict(os_factor=1), dict(os_factor=16), dict(near=True), dict(precision=1, near=True, fd=2.0)])
def test_options(case):
    case = dict(case)
    y0 = case.pop("y0", 1.2)
    if case.pop("near", False):  # the track runs through the image: exact loop, antennas within tiles
        y0 = -3.0
    plan, prof, qt, qr, fd = _frames(4, 300, synth.Grid(-4.1, y0, 0.033, 0.03, 250, 270), **case)
    _compare(plan, prof, 300, qt, qr, fd)
    _compare(plan, prof, 300, qt, qr, fd, accumulate=True)


def test_point_list_with_wide_runs():
    """A sparse ring and a dense patch: runs of 1024 points from narrow to
    nearly the whole scene, so windows of every length, two tables and one."""
    rng = np.random.Generator(np.random.PCG64(4))
    ring = np.stack([8.5 * np.cos(np.linspace(0.2, 2.9, 3000)), 8.5 * np.sin(np.linspace(0.2, 2.9, 3000))], 1)
    px = np.concatenate([ring, rng.uniform([-1.0, 3.0], [1.0, 5.0], (60000, 2)), rng.uniform([-7, 2], [7, 9], (3000, 2))])
    plan, prof, qt, qr, fd = _frames(8, 160, pixels=px[rng.permutation(len(px))], fd=1.5, speed=60.0)
    _compare(plan, prof, 160, qt, qr, fd)


def test_launch_shapes_and_streams():
    """Every register budget and an explicit small block give the same image;
    calls of one plan on two streams do not disturb each other."""
    import torch
    plan, prof, qt, qr, _ = _frames(4, 260, synth.Grid(-4.1, 1.2, 0.033, 0.03, 250, 270))
    ref = _compare(plan, prof, 260, qt, qr).clone()
    torch.cuda.synchronize()
    outs = [torch.zeros_like(ref) for _ in range(6)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for i, o in enumerate(outs):
        plan.backproject(prof, 260, qt, qr, image=o, stream=streams[i % 2])
    torch.cuda.synchronize()
    assert all(torch.equal(o, outs[0]) for o in outs)
    for rg, minb, mb in ((4, 3, 5), (2, 2, 7), (1, 2, 1), (4, 2, 1)):
        plan.set_launch(rg, minb, mb)
        _compare(plan, prof, 260, qt, qr)


def test_captured_call_replays_with_new_geometry():
    """A captured call keeps no result of other calls: replayed after a call with
    a much smaller array and with its own array widened in place, it still
    stages every bin that its geometry reaches."""
    import torch
    M = 260
    plan, prof, qt, qr, _ = _frames(4, M, synth.Grid(-4.1, 1.2, 0.033, 0.03, 250, 270))
    img = torch.zeros(plan.n_pixels, dtype=torch.complex64, device="cuda")
    plan.backproject(prof, M, qt, qr, image=img)  # modules loaded before the capture
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        plan.backproject(prof, M, qt, qr, image=img, stream=s)
    small = (qt[:, None, :] + 0.02 * (qr - qt[:, None, :])).contiguous()
    _compare(plan, prof, M, qt, small)
    qr.copy_(qt[:, None, :] + 6.0 * (qr - qt[:, None, :]))
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(img, _compare(plan, prof, M, qt, qr))
