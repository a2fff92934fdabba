"""Range compression around the line between the band and the split kernel, and
a batch whose frames of one transform shape go to both.  References and
tolerances as in tests/test_gpu_band.py."""
import pytest

import synth
from tests.test_gpu_band import _reference

pytestmark = pytest.mark.gpu


def _values(plan, prof, M, R, precision):
    import torch
    n = plan.info.n_bins
    if precision == 0:
        return prof.view(torch.complex64).view(M, R, n).to(torch.complex128)
    head = (M * R * 4 + 255) // 256 * 256
    h = prof[head:].view(torch.float16).view(M, R, n, 2).double() * prof[:M * R * 4].view(torch.float32).view(M, R, 1, 1)
    return torch.view_as_complex(h)


def _case(N, os_f, crop, precision, M=21, R=2, seed=0):
    import torch
    import paper_2306_09784_gb300 as sar
    radar = synth.Radar(n_samples=N, n_rx=R, os=os_f)
    grid = synth.Grid(-1.0, 2.0, 0.05, 0.05, 40, 36)
    plan = sar.Plan.from_radar(radar, max_pulses=M, grid=grid, crop=crop, precision=precision)
    g = torch.Generator(device="cuda").manual_seed(seed)
    beat = torch.randn(M, R, N, dtype=torch.complex64, device="cuda", generator=g)
    return radar, plan, beat


@pytest.mark.parametrize("N,os_f", [(512, 4), (512, 8), (512, 16), (256, 4), (256, 16)])
@pytest.mark.parametrize("precision", [0, 1])
def test_crops_on_both_sides_of_the_line(N, os_f, precision):
    for q in (184, 232):
        for n in (q * os_f, q * os_f + 1):
            for lo in (0, 3):
                crop = (lo, lo + n - 1)
                radar, plan, beat = _case(N, os_f, crop, precision, seed=n)
                _, ref = _reference(radar, beat, 1, crop)
                got = _values(plan, plan.range_compress(beat), 21, 2, precision)
                err = ((got - ref).abs().square().sum(-1).sqrt() / ref.abs().square().sum(-1).sqrt()).max().item()
                assert err <= (1e-6 if precision == 0 else 5e-4), (crop, err)


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_of_band_and_split_frames(precision):
    """Frames of N = 512, os 8 with narrow crops (band kernel) and wide ones
    (split kernel), interleaved: profiles and images are each call's own."""
    import torch
    import paper_2306_09784_gb300 as sar
    M = 21
    batch, frames = sar.Batch(6), []
    for i in range(6):
        crop = (5, 505 + i) if i % 2 else (0, 4095 - i)
        _, plan, beat = _case(512, 8, crop, precision, seed=i)
        qt = torch.zeros(M, 2, dtype=torch.float64, device="cuda")
        qt[:, 0] = torch.arange(M, device="cuda") * 0.001
        qr = qt[:, None, :] + torch.tensor([[0.002, 0.0], [0.004, 0.0]], dtype=torch.float64, device="cuda")
        prof = torch.zeros(plan.profile_bytes(M), dtype=torch.uint8, device="cuda")
        img = torch.zeros(plan.n_pixels, dtype=torch.complex64, device="cuda")
        batch.add_frame(plan, beat, None, prof, M, qt, qr, img)
        frames.append((plan, beat, prof, qt, qr, img))
    batch.commit()
    batch.launch()
    torch.cuda.synchronize()
    for plan, beat, prof, qt, qr, img in frames:
        alone = plan.range_compress(beat)
        assert torch.equal(_values(plan, prof, M, 2, precision), _values(plan, alone, M, 2, precision))
        ref = plan.backproject(alone, M, qt, qr)
        assert ((img - ref).abs().norm() / ref.abs().norm()).item() < 1e-5


@pytest.mark.parametrize("N,os_f", [(256, 1), (256, 2), (256, 4), (256, 8), (512, 1), (1024, 16)])
@pytest.mark.parametrize("sign", [1, -1])
def test_spectrum_on_each_kernel(N, os_f, sign):
    import torch
    import paper_2306_09784_gb300 as sar
    radar = synth.Radar(n_samples=N, n_rx=2, os=os_f)
    plan = sar.Plan.from_radar(radar, max_pulses=33, grid=synth.Grid(-1.0, 2.0, 0.05, 0.05, 8, 8), crop=(2, 40),
                               phase_sign=sign)
    beat = torch.randn(33, 2, N, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(N))
    S, _ = _reference(radar, beat, sign, (2, 40))
    got = plan.range_spectrum(beat).to(torch.complex128)
    assert ((got - S).abs().square().sum(-1).sqrt() / S.abs().square().sum(-1).sqrt()).max().item() <= 1e-6
