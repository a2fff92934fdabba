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
