"""sar_doppler_offsets calls of one plan on several streams."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_calls_on_two_streams_keep_their_own_means():
    """Trajectories of different velocity, place and length alternate on two
    streams without a wait in between: every output equals its call's own."""
    import torch
    import paper_2306_09784_gb300 as sar
    radar = synth.Radar(n_samples=128, n_rx=8, os=4)
    M = 4000
    plan = sar.Plan.from_radar(radar, max_pulses=M, grid=synth.Grid(-3.0, 2.0, 0.05, 0.05, 130, 110),
                               max_doppler_bins=4.0)
    g = np.random.Generator(np.random.PCG64(12))
    calls = []
    for n, v in ((M, 3.0), (40, 11.0), (1701, -7.0)):
        qt = g.uniform(-1.0, 1.0, (n, 2))
        calls.append([torch.from_numpy(a).cuda() for a in
                      (qt, qt[:, None, :] + g.uniform(0, 0.02, (n, 8, 2)), g.normal([v, 0.1 * v], 0.2, (n, 2)))])
    ref = [plan.doppler_offsets(*c).clone() for c in calls]
    assert not torch.equal(ref[0], ref[1]) and not torch.equal(ref[1], ref[2])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [torch.zeros_like(ref[0]) for _ in range(60)]
    for i, o in enumerate(outs):
        plan.doppler_offsets(*calls[i % 3], out=o, stream=streams[i % 2])
    torch.cuda.synchronize()
    assert all(torch.equal(o, ref[i % 3]) for i, o in enumerate(outs))
