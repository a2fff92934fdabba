"""sar_doppler_offsets where the Tx and the Rx term cancel, against extended
precision: what is left shows the absolute error of each FP64 term.

Tolerance, derived: a term (e . v) / |e| with |v| = 1 and cosine 0.6 or 0.38
carries at most ~6 roundings of 2^-53 (d^2: half of 2, e . v: 2, the reciprocal
root: 2, the product: 1), below 6 * 1.11e-16 * 0.6 = 4.0e-16; two terms 8e-16
m/s; twice that is allowed, plus the FP32 rounding of the output."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("triple", [(3.0, 4.0, 5.0), (5.0, 12.0, 13.0)])
def test_cancelling_terms(triple):
    import torch
    import paper_2306_09784_gb300 as sar
    a, b, _ = triple
    radar = synth.Radar(n_samples=128, n_rx=1, os=4)
    n, step = 64, 2.0 ** -30  # every coordinate is exact in FP64, every offset in FP32
    grid = synth.Grid(-32 * step, b - 32 * step, step, step, n, n)
    plan = sar.Plan.from_radar(radar, max_pulses=1, grid=grid, max_doppler_bins=1.0)
    ix, iy = np.meshgrid(np.arange(n), np.arange(n))
    x = (grid.x0 + ix * step).astype(np.longdouble).ravel()
    y = (grid.y0 + iy * step).astype(np.longdouble).ravel()
    f0 = radar.f0
    scale = f0 / radar.c * radar.n_fft / radar.fs
    worst = 0.0
    for s in (1.5, 2.5, 3.0, 3.5, 5.0, 6.0, 7.0):  # the Rx at s times the Tx's distance, on the other side
        q_tx, q_rx = np.array([[-a, 0.0]]), np.array([[[s * a, b - s * b]]])
        out = plan.doppler_offsets(*(torch.from_numpy(v).cuda() for v in (q_tx, q_rx, np.array([[1.0, 0.0]]))))
        got = out.double().cpu().numpy().astype(np.longdouble) / -scale
        ex, ey = x + a, y
        gx, gy = x - s * a, y - (b - s * b)
        ref = ex / np.sqrt(ex * ex + ey * ey) + gx / np.sqrt(gx * gx + gy * gy)
        err = np.abs(got - ref) - np.abs(ref) * 2.0 ** -24 * 1.01
        worst = max(worst, float(err.max()))
    assert worst <= 1.6e-15, worst
