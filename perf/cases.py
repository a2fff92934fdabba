"""Timing cases of the SAR imaging library: what its users have it do.

Each case goes through the package's public entry points, the way a program
that images one frame after another calls them: the plan, the device buffers
and the scene's inputs exist, and a pass takes a frame from beat samples to
the image (or to the profiles, the spectrum).  Scenes are seeded point
scatterers with noise seen from a jittered track, generated on the GPU.

exact() restates the same results in 64-bit torch from the definitions (the
windowed zero-padded DFT, linear interpolation of the spectrum, the phase of
the two-way path), sharing no code with the library.
"""
import math
import random
from types import SimpleNamespace

import torch

import paper_2306_09784_gb300 as sar

C0 = 299_792_458.0
T_CHIRP = 102.4e-6
PRI = 106.7e-6
WORK_MAX = 2.4e10  # pixel x chirp x Rx updates of the largest listed case
ROW_MAX = 1 << 23  # beat samples of the largest listed case


def _frame(name, **kw):
    """A frame's sizes and options; the defaults are the radar the repository's
    configurations share (77 GHz, 1 GHz, 10 m/s, Hann windows, os 4)."""
    d = dict(name=name, kind="frame", f0=77e9, bandwidth=1e9, nx=0, ny=0, spacing=0.025, y0=2.0, chirps=0, rx=1,
             samples=512, os=4, fp16=False, speed=10.0, jitter=0.02, heading=0.0, kaiser=False, centre=False,
             conjugate=False)
    d.update(kw)
    return d


def listed():
    return [
        # one-channel radar with a small preview image: the smallest whole
        # frame, where launches and latency count
        _frame("tiny_frame", nx=128, ny=128, spacing=0.05, chirps=256, rx=1, samples=256, jitter=0.0),
        # a ragged region of interest (no side a multiple of the pixel tile),
        # two channels, a short aperture
        _frame("ragged_small_frame", nx=80, ny=72, spacing=0.05, y0=1.5, chirps=96, rx=2, samples=128, jitter=0.01),
        # the ordinary frame: four channels, a 512 x 512 image, FP32 profiles
        _frame("full_frame", nx=512, ny=512, chirps=1024, rx=4, samples=512),
        # the headline frame: 1024 x 1024 at 2 cm, 2048 chirps, FP16 profiles
        _frame("precision_frame", nx=1024, ny=1024, spacing=0.02, chirps=2048, rx=4, samples=1024, fp16=True),
        # the paper's reference workload: 1201 x 1201 at 2.5 cm, 1024 chirps,
        # 16 channels, 76.6 GHz / 931 MHz: the largest frame, whose near tiles
        # see a wide array
        _frame("paper_reference_frame", f0=76.6e9, bandwidth=931e6, nx=1201, ny=1201, chirps=1024, rx=16, samples=512),
        # the paper's combined workload: a polar grid of about 165 000 points,
        # 1024 chirps, 8 channels, Doppler offsets from the mean velocity
        # (20 x 20 m: a plan takes no wider point list with 8 channels)
        _frame("polar_doppler_frame", kind="polar", f0=76.6e9, bandwidth=931e6, side=20.0, factor=2.5, chirps=1024,
               rx=8, samples=512, speed=2.06, jitter=0.005),
        # a live image that grows by sub-apertures of 128 chirps while the
        # vehicle turns (the array is not along the image axes)
        _frame("subaperture_stream", kind="stream", nx=512, ny=512, chirps=1024, sub=128, rx=4, samples=512, fp16=True,
               heading=12.0),
        # a whole frame from pinned host buffers to an image in host memory
        _frame("host_frame", kind="host", nx=512, ny=512, chirps=1024, rx=4, samples=512, fp16=True),
        # several radars' uneven frames in one batched launch
        dict(name="batched_frames", kind="batch", frames=12, mix=5, samples=512, os=4, fp16=True, m_lo=128, m_hi=1024,
             side_lo=128, side_hi=512, rx_hi=4),
        # frames of several radars queued at a server together, until every
        # image is in host memory
        dict(name="served_burst", kind="served", frames=6, mix=9, samples=512, os=4, fp16=True, m_lo=128, m_hi=512,
             side_lo=128, side_hi=384, rx_hi=4),
        # range profiles alone (another stage consumes them): the headline
        # frame's beat cube, FP32 profiles over the crop of its geometry
        _frame("range_profiles", kind="profiles", nx=1024, ny=1024, spacing=0.02, chirps=2048, rx=4, samples=1024),
        # the plain zero-padded spectrum of a chirp sequence, for inspection
        _frame("range_spectrum", kind="spectrum", nx=512, ny=512, chirps=512, rx=4, samples=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "polar", "stream", "host", "batch", "served", "profiles",
                       "profiles", "spectrum"])
    samples = rng.choice([128, 256, 512, 1024])
    os_factor = rng.choice([2, 4, 4, 8]) if samples <= 512 else rng.choice([2, 4, 4])
    fp16 = rng.random() < 0.5
    if kind in ("batch", "served"):
        lo, side = _log_int(rng, 48, 256), _log_int(rng, 40, 200)
        return dict(kind=kind, frames=rng.randint(3, 12 if kind == "batch" else 6), mix=rng.randrange(1 << 20),
                    samples=samples, os=os_factor, fp16=fp16, m_lo=lo, m_hi=lo + _log_int(rng, 32, 512), side_lo=side,
                    side_hi=side + _log_int(rng, 32, 280), rx_hi=rng.randint(1, 4))
    rx = rng.choice([1, 2, 3, 4, 4, 6, 8, 16])
    chirps = _log_int(rng, 33, 2048)
    c = _frame(None, kind=kind, nx=_log_int(rng, 24, 1200), ny=_log_int(rng, 24, 1200),
               spacing=round(rng.uniform(0.02, 0.05), 4), y0=round(rng.uniform(1.0, 6.0), 2), chirps=chirps, rx=rx,
               samples=samples, os=os_factor, fp16=fp16, jitter=round(rng.uniform(0.0, 0.02), 4),
               heading=round(rng.uniform(-20.0, 20.0), 1) if rng.random() < 0.3 else 0.0, kaiser=rng.random() < 0.2,
               centre=rng.random() < 0.25, conjugate=rng.random() < 0.15)
    del c["name"]
    if kind == "polar":
        # a point list's width is bounded by the window of bins its widest
        # run of 1024 points spans (all channels of a chirp share 227 KB)
        widest = (227 * 1024 / (42 * rx) - 32) / (2.4 * _radar(c).a1)
        c.update(side=round(rng.uniform(0.4, 0.9) * min(30.0, widest), 2), factor=round(rng.uniform(1.5, 3.0), 2),
                 speed=round(rng.uniform(2.0, 8.0), 2), jitter=0.005)
    if kind == "stream":
        c["sub"] = _log_int(rng, 16, max(17, chirps // 2))
    while c["nx"] * c["ny"] * c["chirps"] * rx > WORK_MAX / 2 or c["chirps"] * rx * samples > ROW_MAX or \
            (kind == "spectrum" and c["chirps"] * rx * samples * os_factor > ROW_MAX):
        c["chirps"] = c["chirps"] * 2 // 3
        if kind == "stream":
            c["sub"] = min(c["sub"], c["chirps"])
    return c


# --- scenes ---------------------------------------------------------------


def _radar(case):
    r = SimpleNamespace(f0=case["f0"], bandwidth=case["bandwidth"], n_samples=case["samples"], os=case["os"],
                        n_rx=case["rx"], c=C0)
    r.slope = r.bandwidth / T_CHIRP
    r.fs = r.n_samples / T_CHIRP
    r.n_fft = r.n_samples * r.os
    r.a1 = r.slope * r.n_fft / (C0 * r.fs)  # bins per metre of two-way path
    return r


def _track(case, g):
    """Antenna positions at the chirp starts: along the heading at constant
    speed with a sinusoidal lateral deviation, Rx at half wavelengths."""
    m = torch.arange(case["chirps"], dtype=torch.float64)
    s = (m - (case["chirps"] - 1) / 2.0) * (case["speed"] * PRI)
    side = case["jitter"] * torch.sin(2 * math.pi * (3.0 * m / case["chirps"] + float(torch.rand((), generator=g))))
    h = math.radians(case["heading"])
    u = torch.tensor([math.cos(h), math.sin(h)], dtype=torch.float64)
    v = torch.tensor([-math.sin(h), math.cos(h)], dtype=torch.float64)
    q_tx = s[:, None] * u + side[:, None] * v
    off = (torch.arange(case["rx"], dtype=torch.float64) + 1.0) * (C0 / case["f0"] / 2.0)
    return q_tx, q_tx[:, None, :] + off[None, :, None] * u


def _grid(case):
    return SimpleNamespace(x0=-case["spacing"] * (case["nx"] - 1) / 2.0, y0=case["y0"], dx=case["spacing"],
                           dy=case["spacing"], nx=case["nx"], ny=case["ny"])


def _box(case):
    if case["kind"] == "polar":
        return -case["side"] / 2, case["side"] / 2, 2.0, 2.0 + case["side"]
    g = _grid(case)
    return g.x0, g.x0 + g.dx * (g.nx - 1), g.y0, g.y0 + g.dy * (g.ny - 1)


def _crop(case, radar, q_tx, q_rx):
    """Bins that the geometry reaches, with a margin of 8."""
    ants = torch.cat([q_tx, q_rx.reshape(-1, 2)])
    (ax0, ay0), (ax1, ay1) = ants.amin(0).tolist(), ants.amax(0).tolist()
    x0, x1, y0, y1 = _box(case)
    dmin = math.hypot(max(0.0, x0 - ax1, ax0 - x1), max(0.0, y0 - ay1, ay0 - y1))
    dmax = math.hypot(max(abs(x1 - ax0), abs(ax1 - x0)), max(abs(y1 - ay0), abs(ay1 - y0)))
    lo = max(0, math.floor(2 * radar.a1 * dmin) - 8)
    hi = min(radar.n_fft - 1, math.ceil(2 * radar.a1 * dmax) + 8)
    return min(lo, hi - 16), hi


def _beat(case, radar, q_tx, q_rx, gen):
    """complex64 [M][R][N] beat samples (Rx times conjugate Tx) of 24 scatterers
    inside the imaged region, 20 dB above complex white noise."""
    M, R, N = case["chirps"], case["rx"], case["samples"]
    x0, x1, y0, y1 = _box(case)
    t = torch.rand(24, 2, generator=gen, device="cuda", dtype=torch.float64)
    pts = t * torch.tensor([x1 - x0, y1 - y0], device="cuda", dtype=torch.float64) + torch.tensor(
        [x0, y0], device="cuda", dtype=torch.float64)
    amp = torch.randn(24, generator=gen, device="cuda", dtype=torch.complex64)
    n = torch.arange(N, device="cuda", dtype=torch.float32)
    out = torch.zeros(M, R, N, dtype=torch.complex64, device="cuda")
    sign = -1.0 if not case["conjugate"] else 1.0
    for k in range(24):
        tau = (torch.linalg.norm(pts[k] - q_tx, dim=-1)[:, None] + torch.linalg.norm(pts[k] - q_rx, dim=-1)) / C0
        ph = radar.f0 * tau
        cyc = (ph - ph.floor()).float()[..., None] + (radar.slope * tau / radar.fs).float()[..., None] * n
        ang = (2 * math.pi * sign) * cyc
        out += amp[k] * torch.complex(torch.cos(ang), torch.sin(ang))
    noise = torch.randn(M, R, N, generator=gen, device="cuda", dtype=torch.complex64)
    return out + (0.1 * out.abs().square().mean().sqrt()) * noise


def _scene(case, seed):
    """Everything a frame needs, on the GPU (pixels only for point lists)."""
    radar = _radar(case)
    q_tx, q_rx = _track(case, torch.Generator().manual_seed(seed))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = SimpleNamespace(radar=radar, crop=_crop(case, radar, q_tx, q_rx))
    s.q_tx, s.q_rx = q_tx.cuda(), q_rx.contiguous().cuda()
    s.beat = _beat(case, radar, s.q_tx, s.q_rx, gen)
    s.w_az = torch.hann_window(case["chirps"], periodic=False, dtype=torch.float64).float().cuda()
    if case["kind"] == "polar":
        # nominal track (no jitter): the grid does not depend on the seed
        nominal, _ = _track(dict(case, jitter=0.0), torch.Generator().manual_seed(0))
        s.pixels = sar.polar_grid(radar, nominal.numpy(), _box(case), case["factor"])
        wobble = 0.05 * torch.randn(case["chirps"], 2, generator=gen, device="cuda", dtype=torch.float64)
        h = math.radians(case["heading"])
        s.vel = wobble + case["speed"] * torch.tensor([math.cos(h), math.sin(h)], device="cuda", dtype=torch.float64)
    return s


def _plan(case, s, max_pulses=None):
    where = dict(pixels_xy=s.pixels) if case["kind"] == "polar" else dict(grid=_grid(case))
    return sar.Plan.from_radar(
        s.radar, max_pulses=max_pulses or case["chirps"], crop=s.crop,
        precision=sar.PREC_FP16 if case["fp16"] else sar.PREC_FP32,
        range_window=sar.WINDOW_KAISER if case["kaiser"] else sar.WINDOW_HANN,
        time_origin=sar.ORIGIN_CHIRP_CENTRE if case["centre"] else sar.ORIGIN_FIRST_SAMPLE,
        phase_sign=-1 if case["conjugate"] else 1, max_doppler_bins=2.0 if case["kind"] == "polar" else 0.0, **where)


def _mix(case):
    """The frames of a batched or served case: sizes from the case alone."""
    rng = random.Random(case["mix"])
    frames = []
    for _ in range(case["frames"]):
        side = rng.randint(case["side_lo"], case["side_hi"])
        frames.append(_frame(None, nx=side, ny=max(16, side - rng.randint(0, 15)),
                             chirps=rng.randint(case["m_lo"], case["m_hi"]), rx=rng.randint(1, case["rx_hi"]),
                             samples=case["samples"], os=case["os"], fp16=case["fp16"]))
    return frames


# --- passes ---------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "served"):
        return _prepare_many(case, seed)
    s = _scene(case, seed)
    st = SimpleNamespace(kind=kind, fp16=case["fp16"], M=case["chirps"], R=case["rx"], plan=_plan(case, s),
                         beat=s.beat, w_az=s.w_az, q_tx=s.q_tx, q_rx=s.q_rx)
    plan = st.plan
    if kind == "host":
        st.beat, st.w_az, st.q_tx, st.q_rx = (t.cpu().pin_memory() for t in (s.beat, s.w_az, s.q_tx, s.q_rx))
        st.image = torch.zeros(plan.n_pixels, dtype=torch.complex64, pin_memory=True)
        return st
    if kind == "spectrum":
        st.out = torch.empty(st.M, st.R, s.radar.n_fft, dtype=torch.complex64, device="cuda")
        return st
    st.prof = plan.empty_profiles(st.M)
    st.n_bins = int(plan.info.n_bins)
    st.image = torch.zeros(plan.n_pixels, dtype=torch.complex64, device="cuda")
    if kind == "polar":
        st.vel = s.vel
        st.fd = torch.empty(plan.n_pixels, dtype=torch.float32, device="cuda")
    if kind == "stream":
        st.parts = [(a, min(st.M, a + case["sub"])) for a in range(0, st.M, case["sub"])]
    return st


def _prepare_many(case, seed):
    frames = _mix(case)
    st = SimpleNamespace(kind=case["kind"], items=[])
    dev = case["kind"] == "batch"
    if dev:
        st.batch = sar.Batch(len(frames))
    else:
        st.server = sar.Server(hbm_budget=1 << 30, max_inflight=len(frames))
    for i, f in enumerate(frames):
        s = _scene(f, seed * 64 + i)
        plan = _plan(f, s)
        it = SimpleNamespace(plan=plan, beat=s.beat, w_az=s.w_az, q_tx=s.q_tx, q_rx=s.q_rx)
        if dev:
            it.prof = plan.empty_profiles(f["chirps"])
            it.image = torch.zeros(plan.n_pixels, dtype=torch.complex64, device="cuda")
            st.batch.add_frame(plan, it.beat, it.w_az, it.prof, f["chirps"], it.q_tx, it.q_rx, it.image)
        else:
            it.beat, it.w_az, it.q_tx, it.q_rx = (t.cpu().pin_memory() for t in (s.beat, s.w_az, s.q_tx, s.q_rx))
            it.image = torch.zeros(plan.n_pixels, dtype=torch.complex64, pin_memory=True)
        st.items.append(it)
    if dev:
        st.batch.commit()
    return st


def run(st):
    if st.kind == "batch":
        st.batch.launch()
        return [it.image for it in st.items]
    if st.kind == "served":
        tickets = [st.server.submit(it.plan, it.beat, it.q_tx, it.q_rx, w_az=it.w_az, image=it.image)
                   for it in st.items]
        for t in tickets:
            rc = st.server.wait(t)
            if rc != sar.SAR_OK:
                raise sar.SarError(rc, "wait")
            st.server.release(t)
        return [it.image for it in st.items]
    plan = st.plan
    if st.kind == "host":
        return plan.form_image_host(st.beat, st.q_tx, st.q_rx, st.image, w_az=st.w_az)
    if st.kind == "spectrum":
        return plan.range_spectrum(st.beat, out=st.out)
    if st.kind == "stream":
        for a, b in st.parts:
            plan.range_compress(st.beat[a:b], st.w_az[a:b], out=st.prof)
            plan.backproject(st.prof, b - a, st.q_tx[a:b], st.q_rx[a:b], image=st.image, accumulate=a > 0)
        return st.image
    plan.range_compress(st.beat, st.w_az, out=st.prof)
    if st.kind == "profiles":
        rows = st.M * st.R
        if not st.fp16:
            return st.prof.view(torch.complex64).view(st.M, st.R, st.n_bins)
        head = (rows * 4 + 255) // 256 * 256
        return {"scale": st.prof[:rows * 4].view(torch.float32).view(st.M, st.R),
                "samples": st.prof[head:].view(torch.float16).view(st.M, st.R, st.n_bins, 2)}
    if st.kind == "polar":
        plan.doppler_offsets(st.q_tx, st.q_rx, st.vel, out=st.fd)
        plan.backproject(st.prof, st.M, st.q_tx, st.q_rx, image=st.image, fdopp=st.fd)
        return {"image": st.image, "offsets": st.fd}
    return plan.backproject(st.prof, st.M, st.q_tx, st.q_rx, image=st.image)


# --- what a pass cannot do without -----------------------------------------


def _n_pixels(case):
    if case["kind"] != "polar":
        return case["nx"] * case["ny"]
    q_tx, _ = _track(dict(case, jitter=0.0), torch.Generator().manual_seed(0))
    return len(sar.polar_grid(_radar(case), q_tx.numpy(), _box(case), case["factor"]))


def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: 5 n log2 n
    per range transform of the samples, and 20 per pixel, chirp and channel
    (17 of arithmetic, one square root, one sine, one cosine)."""
    if case["kind"] in ("batch", "served"):
        parts = [work(f) for f in _mix(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    M, R, N = case["chirps"], case["rx"], case["samples"]
    nbytes = M * R * N * 8 + M * 4
    flops = 5.0 * M * R * N * math.log2(N)
    if case["kind"] == "spectrum":
        return {"bytes": nbytes - M * 4 + M * R * N * case["os"] * 8, "flops": flops}
    if case["kind"] == "profiles":
        lo, hi = _crop(case, _radar(case), *_track(case, torch.Generator().manual_seed(0)))
        return {"bytes": nbytes + M * R * (hi - lo + 1) * (4 if case["fp16"] else 8), "flops": flops}
    P = _n_pixels(case)
    nbytes += M * (R + 1) * 16 + P * 8 + (P * 4 + M * 16 if case["kind"] == "polar" else 0)
    return {"bytes": nbytes, "flops": flops + 20.0 * P * M * R}


# --- the same results in 64 bits --------------------------------------------


def _window64(case):
    N = case["samples"]
    if case["kaiser"]:
        return torch.kaiser_window(N, periodic=False, beta=6.0, dtype=torch.float64, device="cuda")
    return torch.hann_window(N, periodic=False, dtype=torch.float64, device="cuda")


def _spectrum64(case, s, t0):
    """[M * R][N_fft]: sum_n w[n] beat[n] exp(sign j 2 pi (n - t0) k / N_fft)."""
    x = s.beat.to(torch.complex128).reshape(-1, case["samples"]) * _window64(case)
    n = s.radar.n_fft
    S = torch.fft.fft(x, n=n) if case["conjugate"] else torch.fft.ifft(x, n=n) * n
    if t0:
        k = torch.arange(n, dtype=torch.float64, device="cuda")
        S = S * _unit(-_sign(case) * t0 * k / n)
    return S


def _sign(case):
    return -1.0 if case["conjugate"] else 1.0


def _unit(cycles):
    a = 2 * math.pi * (cycles - cycles.floor())
    return torch.complex(torch.cos(a), torch.sin(a))


def _pixels64(case, s):
    if case["kind"] == "polar":
        return torch.from_numpy(s.pixels).cuda()
    g = _grid(case)
    x = g.x0 + g.dx * torch.arange(g.nx, dtype=torch.float64, device="cuda")
    y = g.y0 + g.dy * torch.arange(g.ny, dtype=torch.float64, device="cuda")
    return torch.stack([x.expand(g.ny, g.nx), y[:, None].expand(g.ny, g.nx)], -1).reshape(-1, 2)


def _image64(case, s, fd=None):
    r = s.radar
    t0 = 0.5 * (case["samples"] - 1) if case["centre"] else 0.0
    f0 = r.f0 + r.slope * t0 / r.fs
    S = _spectrum64(case, s, t0) * s.w_az.double().repeat_interleave(case["rx"])[:, None]
    S = S.contiguous()
    px = _pixels64(case, s)
    P, R, n = len(px), case["rx"], r.n_fft
    lo, hi = s.crop
    out = torch.zeros(P, dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 23) // P)
    for m0 in range(0, case["chirps"], step):
        m1 = min(case["chirps"], m0 + step)
        dtx = torch.hypot(px[None, :, 0] - s.q_tx[m0:m1, None, 0], px[None, :, 1] - s.q_tx[m0:m1, None, 1])
        for c in range(R):
            q = s.q_rx[m0:m1, c]
            d = dtx + torch.hypot(px[None, :, 0] - q[:, None, 0], px[None, :, 1] - q[:, None, 1])
            idx = r.a1 * d if fd is None else r.a1 * d + fd
            i0 = idx.floor()
            f = idx - i0
            f = f * ((i0 >= lo) & (i0 < hi))
            keep = ((i0 >= lo) & (i0 < hi)).to(torch.float64)
            i0 = i0.clamp(0, n - 2).long() + (torch.arange(m0, m1, device="cuda") * R + c)[:, None] * n
            a, b = S.view(-1)[i0], S.view(-1)[i0 + 1]
            out += ((a + f * (b - a)) * _unit((_sign(case) * f0 / C0) * d) * keep).sum(0)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "served"):
        return [_image64(f, _scene(f, seed * 64 + i)) for i, f in enumerate(_mix(case))]
    s = _scene(case, seed)
    r = s.radar
    if kind == "spectrum":
        return _spectrum64(case, s, 0.0).view(case["chirps"], case["rx"], r.n_fft)
    if kind == "profiles":
        k = torch.arange(s.crop[0], s.crop[1] + 1, dtype=torch.float64, device="cuda")
        P = _spectrum64(case, s, 0.0)[:, s.crop[0]:s.crop[1] + 1] * _unit(_sign(case) * k * (r.f0 / (C0 * r.a1)))
        P = P.view(case["chirps"], case["rx"], -1) * s.w_az.double()[:, None, None]
        if not case["fp16"]:
            return P
        P = torch.view_as_real(P)
        scale = P.abs().amax((2, 3)) / 16384.0
        scale = torch.where(scale > 0, scale, torch.ones_like(scale))
        return {"scale": scale, "samples": P / scale[:, :, None, None]}
    if kind == "polar":
        px = _pixels64(case, s)
        v, qt, qr = s.vel.mean(0), s.q_tx.mean(0), s.q_rx.reshape(-1, 2).mean(0)
        t0 = 0.5 * (case["samples"] - 1) if case["centre"] else 0.0
        rate = sum(((px - q) @ v) / torch.linalg.norm(px - q, dim=-1) for q in (qt, qr))
        fd = -rate * ((r.f0 + r.slope * t0 / r.fs) / C0) * (r.n_fft / r.fs)
        return {"image": _image64(case, s, fd), "offsets": fd}
    return _image64(case, s)
