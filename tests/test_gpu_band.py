"""Range compression at the sizes and crops where the band kernel begins, ends
and wraps, and the spectrum by the split kernel, against a 64-bit DFT.
Tolerance: FP32 transforms of up to 1024 points keep a relative L2 error of a
few 1e-7 (1e-6 allowed); FP16 samples round to 2^-11 of the value (5e-4)."""
import math

import pytest

import synth

pytestmark = pytest.mark.gpu


def _reference(radar, beat, sign, crop):
    import torch
    N, nf = radar.n_samples, radar.n_fft
    w = torch.hann_window(N, periodic=False, dtype=torch.float64, device="cuda")
    x = beat.to(torch.complex128) * w
    S = torch.fft.ifft(x, n=nf) * nf if sign > 0 else torch.fft.fft(x, n=nf)
    k = torch.arange(crop[0], crop[1] + 1, dtype=torch.float64, device="cuda")
    cyc = k * (radar.f0 / (radar.c * radar.bins_per_metre))
    ang = sign * 2 * math.pi * (cyc - cyc.floor())
    return S, S[..., crop[0]:crop[1] + 1] * torch.complex(torch.cos(ang), torch.sin(ang))


@pytest.mark.parametrize("N,os_f", [(256, 4), (256, 8), (256, 16), (512, 4), (512, 16), (1024, 4), (1024, 8), (512, 2)])
@pytest.mark.parametrize("precision", [0, 1])
def test_profiles_at_crop_edges(N, os_f, precision):
    import torch
    import paper_2306_09784_gb300 as sar
    nf, span = N * os_f, 256 * os_f
    crops = [(0, 16), (3, 20), (15 * os_f, 16 * os_f), (nf - 40, nf - 1)]
    crops += [(1, min(nf - 1, span - 1)), (0, nf - 1)]  # the widest band, and the whole spectrum
    if nf > span:
        crops += [(span - 37, span + 61), (5, span + 4)]  # Q wraps at 256; 256 values and one more
    for i, crop in enumerate(crops):
        R, M, sign = 1 + i % 3, 19 + i, 1 if i % 2 else -1
        radar = synth.Radar(n_samples=N, n_rx=R, os=os_f)
        plan = sar.Plan.from_radar(radar, max_pulses=M, grid=synth.Grid(-1.0, 2.0, 0.05, 0.05, 8, 8), crop=crop,
                                   precision=precision, phase_sign=sign)
        g = torch.Generator(device="cuda").manual_seed(i)
        beat = torch.randn(M, R, N, dtype=torch.complex64, device="cuda", generator=g)
        w_az = torch.rand(M, device="cuda", generator=g) + 0.5
        _, ref = _reference(radar, beat, sign, crop)
        ref = ref * w_az[:, None, None]
        prof, n = plan.range_compress(beat, w_az), crop[1] - crop[0] + 1
        if precision == 0:
            got, tol = prof.view(torch.complex64).view(M, R, n).to(torch.complex128), 1e-6
        else:
            head = (M * R * 4 + 255) // 256 * 256
            h = prof[head:].view(torch.float16).view(M, R, n, 2).double() * \
                prof[:M * R * 4].view(torch.float32).view(M, R, 1, 1)
            got, tol = torch.view_as_complex(h), 5e-4
        err = ((got - ref).abs().square().sum(-1).sqrt() / ref.abs().square().sum(-1).sqrt()).max().item()
        assert err <= tol, (crop, err)  # every row by itself


@pytest.mark.parametrize("N,os_f,sign", [(256, 1, 1), (256, 16, -1), (512, 2, 1), (1024, 4, 1), (1024, 8, -1)])
def test_spectrum_of_split_sizes(N, os_f, sign):
    import torch
    import paper_2306_09784_gb300 as sar
    radar = synth.Radar(n_samples=N, n_rx=3, os=os_f)
    plan = sar.Plan.from_radar(radar, max_pulses=7, grid=synth.Grid(-1.0, 2.0, 0.05, 0.05, 8, 8), crop=(2, 40),
                               phase_sign=sign)
    beat = torch.randn(7, 3, N, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    S, _ = _reference(radar, beat, sign, (2, 40))
    got = plan.range_spectrum(beat).to(torch.complex128)
    assert ((got - S).abs().norm() / S.abs().norm()).item() <= 1e-6
