"""What a user of this framework has it do: the measured cases.

Each case is one call (or the few calls that belong together) through the public entry points of
``paper_2606_04304_gb300``: a whole integration through the batched pipeline, the upchannelizer, the
X-engine, the imager, the candidate search, the drift search and a training step of the candidate
scorer.  Sizes are the ones of the repository's workloads (16 antennas and 64^2 images; 352 antennas,
1024 to 16384 fine channels, 256^2 to 1024^2 images; batches of 300 fine channels of 2400) and generic ones
between them.  Inputs are synthetic and drawn on the GPU from the seed: 4+4-bit Gaussian voltages with
plane-wave tones, int8 spectra of about 8 levels rms, visibilities of noise and a point source, images whose
noise has the mild skew that few integrated spectra give.
"""
import math

import numpy as np
import torch

from paper_2606_04304_gb300 import ovro, scorer

C_LIGHT = 299_792_458.0
F_COARSE = 24_000.0
NU0 = 60.0e6
SIGMA = 2.0                      # voltage noise, 4-bit levels per component
ROWS = {"pipeline": 4096, "detect": 16384, "drift": 1024}      # candidates a program keeps room for


# ------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest calls: a 16-antenna test array, two coarse channels of 256 points, 64^2 images; launches
        # and host work count
        dict(name="pipeline_tiny", kind="pipeline", n_ant=16, nfft="256,256", n_time=16384, image=64, n_tones=1),
        # the whole array on one coarse channel: 10 s at 2.9 Hz channels, voltages in, candidates out
        dict(name="pipeline_full", kind="pipeline", n_ant=352, nfft="8192", n_time=240000, image=256, n_tones=4),
        # its upchannelizer alone
        dict(name="upchan_8192", kind="upchan", n_ant=352, nfft="8192", n_time=240000, taps=1, lo=0, count=0,
             f32=False),
        # the paper's 10 Hz channels (2400 = 2^5 3 5^2 points) through a polyphase filter bank, with the FP32
        # spectra that a spectrometer keeps
        dict(name="upchan_2400_pfb", kind="upchan", n_ant=352, nfft="2400", n_time=240000, taps=4, lo=0, count=0,
             f32=True),
        # the X-engine on short integrations (10 s of 2.9 Hz channels), where writing the visibilities counts
        dict(name="xengine_k29", kind="xengine", n_ant=352, n_chan=2048, n_spec=29, fp32=False),
        # one batch of 300 fine channels integrated over 30 s, where the tensor cores count
        dict(name="xengine_k299", kind="xengine", n_ant=352, n_chan=300, n_spec=299, fp32=False),
        # all-sky images of an odd number of fine channels
        dict(name="image_256", kind="image", n_ant=352, n_chan=1000, n_spec=29, image=256, store="fp32",
             cal=False, uv_min=0.0, uv_max=0.0),
        # what real data take: per-input gains and a baseline cut, at the paper's image size
        dict(name="image_512_cal", kind="image", n_ant=352, n_chan=300, n_spec=299, image=512, store="fp32",
             cal=True, uv_min=4.0, uv_max=100.0),
        # the largest images, with 16-bit storage between the two transform passes
        dict(name="image_1024_bf16", kind="image", n_ant=352, n_chan=64, n_spec=58, image=1024, store="bf16",
             cal=False, uv_min=0.0, uv_max=0.0),
        # the candidate search over two coarse channels of unlike length, threshold by false discovery rate
        dict(name="detect_mixed", kind="detect", nfft="4096,1024", n_spec=58, image=256, mode="bh", n_tones=20),
        # drifting lines over eight sub-integrations
        dict(name="drift_8", kind="drift", n_sub=8, nfft="1024", image=256, n_tones=20),
        # one training step of the candidate scorer
        dict(name="scorer_step", kind="scorer", batch=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pipeline", "upchan", "upchan", "xengine", "xengine", "image", "image", "image", "detect",
                       "detect", "drift", "scorer"])
    if kind == "pipeline":
        if rng.random() < 0.5:                      # test arrays
            n = rng.choice([64, 128, 240, 256, 512])
            return dict(kind=kind, n_ant=_log_int(rng, 8, 64), nfft=",".join([str(n)] * rng.randint(1, 4)),
                        n_time=n * rng.randint(40, 90) + rng.randint(0, n - 1), image=rng.choice([32, 64, 128]),
                        n_tones=rng.randint(1, 3))
        n = rng.choice([1024, 2048, 2400, 4096])
        return dict(kind=kind, n_ant=_log_int(rng, 96, 352), nfft=str(n), n_time=rng.randint(120000, 240000),
                    image=rng.choice([128, 256]), n_tones=rng.randint(1, 6))
    if kind == "upchan":
        n = rng.choice([256, 1024, 2048, 2400, 4096, 8192, 16384])
        taps = rng.choice([1, 1, 1, 2, 4]) if n in (256, 1024, 2400, 4096) else 1
        count = rng.choice([0, 0, 0, n // 8]) if n in (1024, 2400) else 0
        n_ant = _log_int(rng, 8, 352)
        n_time = min(int(1.7e8 / (2 * n_ant)), n * rng.randint(taps + 8, 120)) + rng.randint(0, n - 1)
        return dict(kind=kind, n_ant=n_ant, nfft=str(n), n_time=n_time, taps=taps,
                    lo=rng.randint(0, n - count) if count else 0, count=count, f32=rng.random() < 0.3)
    if kind == "xengine":
        n_ant = _log_int(rng, 16, 352)
        k = _log_int(rng, 8, 400)
        n_chan = _log_int(rng, 64, 2048)
        bl = n_ant * (n_ant + 1) // 2
        n_chan = max(16, min(n_chan, int(4.0e9 / (32 * bl)), int(4.5e10 / (bl * k))))
        return dict(kind=kind, n_ant=n_ant, n_chan=n_chan, n_spec=k, fp32=rng.random() < 0.15)
    if kind == "image":
        size = rng.choice([64, 128, 256, 256, 512, 1024])
        n_ant = _log_int(rng, 16, 352)
        n_chan = min(_log_int(rng, 16, 1200), 64 * (1024 // size) ** 2)
        cal = rng.random() < 0.4
        return dict(kind=kind, n_ant=n_ant, n_chan=n_chan, n_spec=_log_int(rng, 14, 300), image=size,
                    store=rng.choice(["fp32", "fp32", "fp32", "bf16", "fp16"]), cal=cal,
                    uv_min=rng.choice([0.0, 4.0]) if cal else 0.0, uv_max=rng.choice([0.0, 60.0, 100.0]) if cal else 0.0)
    if kind == "detect":
        size = rng.choice([32, 64, 128, 256])
        nf = [rng.choice([512, 1024, 1500, 2400, 4096, 8192, 16384]) for _ in range(rng.randint(1, 3))]
        while sum(nf) * size * size > 5200 * 65536:
            nf[nf.index(max(nf))] //= 4
        return dict(kind=kind, nfft=",".join(map(str, nf)), n_spec=_log_int(rng, 58, 300), image=size,
                    mode=rng.choice(["bh", "bh", "fixed"]), n_tones=rng.randint(2, 30))
    if kind == "drift":
        size = rng.choice([32, 64, 128, 256])
        t = rng.choice([2, 4, 8, 16])
        cap = 8 * 1024 * 65536 // (t * size * size)
        nf = [min(_log_int(rng, 100, 4096), max(32, cap // 2)) for _ in range(rng.randint(1, 2))]
        return dict(kind=kind, n_sub=t, nfft=",".join(map(str, nf)), image=size, n_tones=rng.randint(2, 20))
    return dict(kind="scorer", batch=_log_int(rng, 16, 4096))


def _nfft(case):
    return [int(x) for x in case["nfft"].split(",")]


# ----------------------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _positions(n_ant, seed):
    """Antennas uniform in area: five sevenths in a 200 m core, the others out to 1.5 km (a small array has
    only the core).  ENU metres, planar."""
    r = np.random.default_rng(seed + 1)
    core = n_ant if n_ant < 100 else (n_ant * 251) // 352
    rad = np.concatenate([np.sqrt(r.uniform(0.0, 200.0 ** 2, core)),
                          np.sqrt(r.uniform(200.0 ** 2, 1500.0 ** 2, n_ant - core))])
    th = r.uniform(0.0, 2 * np.pi, n_ant)
    return np.stack([rad * np.cos(th), rad * np.sin(th), np.zeros(n_ant)], axis=1)


def _freqs(nfft):
    return np.concatenate([NU0 + c * F_COARSE + (np.arange(n) - n / 2) * (F_COARSE / n)
                           for c, n in enumerate(nfft)])


def _sky_pixels(r, count, size, r2=0.5):
    out = []
    while len(out) < count:
        row, col = int(r.integers(2, size - 2)), int(r.integers(2, size - 2))
        if ((row - size // 2) ** 2 + (col - size // 2) ** 2) * (2.0 / size) ** 2 < r2:
            out.append((row, col))
    return out


def _voltages(n_time, n_input, seed, tones=()):
    """uint8 [n_time][n_input], 4+4-bit Gaussian noise plus (amplitude, baseband Hz, phasor per input) tones."""
    g = _gen(seed)
    out = torch.empty((n_time, n_input), dtype=torch.uint8, device="cuda")
    for t0 in range(0, n_time, 1 << 16):
        nt = min(1 << 16, n_time - t0)
        x = torch.randn((nt, n_input), generator=g, device="cuda") * SIGMA
        y = torch.randn((nt, n_input), generator=g, device="cuda") * SIGMA
        tt = (t0 + torch.arange(nt, dtype=torch.float64, device="cuda")) / F_COARSE
        for amp, f0, ph in tones:
            a = 2 * math.pi * torch.remainder(f0 * tt, 1.0)
            c, s = (amp * torch.cos(a)).float()[:, None], (amp * torch.sin(a)).float()[:, None]
            pr, pi = torch.from_numpy(np.cos(ph)).cuda().float()[None], torch.from_numpy(np.sin(ph)).cuda().float()[None]
            x += c * pr - s * pi
            y += c * pi + s * pr
        x = x.round_().clamp_(-7, 7).to(torch.int16)
        y = y.round_().clamp_(-7, 7).to(torch.int16)
        out[t0:t0 + nt] = (((x & 15) << 4) | (y & 15)).to(torch.uint8)
    return out


def _visibilities(case, seed, pos, freqs):
    """int32 [chan][baseline][pol][re, im]: the noise of K integrated spectra and one point source."""
    n_ant, n_chan, k = case["n_ant"], case["n_chan"], case["n_spec"]
    g = _gen(seed)
    r = np.random.default_rng(seed + 2)
    a, b = np.triu_indices(n_ant)
    (row, col), = _sky_pixels(r, 1, case["image"])
    l0, m0 = (col - case["image"] // 2) * 2.0 / case["image"], (row - case["image"] // 2) * 2.0 / case["image"]
    d = torch.from_numpy((pos[a, 0] - pos[b, 0]) * l0 + (pos[a, 1] - pos[b, 1]) * m0).cuda() / C_LIGHT
    out = torch.empty((n_chan, a.size, 4, 2), dtype=torch.int32, device="cuda")
    for f in range(0, n_chan, 64):
        fr = torch.from_numpy(np.ascontiguousarray(freqs[f:f + 64])).cuda()
        ph = (-2 * math.pi * torch.remainder(fr[:, None] * d[None], 1.0)).float()
        v = torch.randn((fr.numel(), a.size, 4, 2), generator=g, device="cuda") * (64.0 * math.sqrt(2.0 * k))
        v[:, :, 0, 0] += 6.0 * k * torch.cos(ph)
        v[:, :, 0, 1] += 6.0 * k * torch.sin(ph)
        v[:, :, 3, 0] += 6.0 * k * torch.cos(ph)
        v[:, :, 3, 1] += 6.0 * k * torch.sin(ph)
        out[f:f + 64] = v.round_().to(torch.int32)
    return out


def _images(n_chan, size, n_spec, tones, seed):
    """float [chan][N][N]: noise with the skew sqrt(2 / K) of K integrated spectra, per-channel level and scale,
    and tones (channel, row, col, snr) of a 3 x 3 pixel beam."""
    g = _gen(seed)
    s = math.sqrt(2.0 / n_spec) / 6.0
    img = torch.empty((n_chan, size, size), device="cuda")
    for f in range(0, n_chan, 512):
        x = torch.randn((min(512, n_chan - f), size, size), generator=g, device="cuda")
        img[f:f + 512] = x + s * (x * x - 1.0)
    for chan, row, col, snr in tones:
        for dr in (-1, 0, 1):
            for dc in (-1, 0, 1):
                img[chan, row + dr, col + dc] += snr * 0.5 ** (dr * dr + dc * dc)
    lev = torch.randn((n_chan, 1, 1), generator=g, device="cuda") * 0.3
    scale = 1.0 + 0.1 * torch.rand((n_chan, 1, 1), generator=g, device="cuda")
    img.add_(lev).mul_(scale).mul_(40.0)
    d = (torch.arange(size, device="cuda", dtype=torch.float64) - size // 2) * (2.0 / size)
    img.masked_fill_((d[None, :] ** 2 + d[:, None] ** 2 >= 1.0)[None], 0.0)
    return img


def prepare(case, seed):
    kind = case["kind"]
    r = np.random.default_rng(seed)
    if kind == "pipeline":
        nfft, size = _nfft(case), case["image"]
        pos = _positions(case["n_ant"], seed)
        hz = [NU0 + c * F_COARSE for c in range(len(nfft))]
        n_bl = case["n_ant"] * (case["n_ant"] - 1) // 2
        volt = []
        for c, n in enumerate(nfft):
            tones = []
            for row, col in _sky_pixels(r, case["n_tones"], size):
                snr = float(r.uniform(30.0, 60.0))
                amp = math.sqrt(snr * 2 * SIGMA ** 2 / (n * math.sqrt(2.0 * (case["n_time"] // n) * n_bl)))
                f0 = (int(r.integers(n // 8, n - n // 8)) - n // 2) * F_COARSE / n
                l0, m0 = (col - size // 2) * 2.0 / size, (row - size // 2) * 2.0 / size
                ph = -2 * np.pi * (hz[c] + f0) * (pos[:, 0] * l0 + pos[:, 1] * m0) / C_LIGHT
                tones.append((amp, f0, np.repeat(ph, 2)))
            volt.append(_voltages(case["n_time"], 2 * case["n_ant"], seed * 64 + c, tones))
        # ten sigma; a test array's own sidelobes raise the noise in a tone's channel, so six there
        prm = ovro.detect_params(mode=ovro.DETECT_FIXED, nsigma=10.0 if case["n_ant"] >= 64 else 6.0)
        return dict(kind=kind, volt=torch.stack(volt), rows=ROWS[kind],
                    pipe=ovro.Pipeline(case["n_ant"], nfft, hz, case["n_time"], pos, size, 2.0 / size, params=prm))
    if kind == "upchan":
        n = _nfft(case)[0]
        taps = None
        if case["taps"] > 1:                        # a Hann-tapered sinc one fine channel wide
            m = np.arange(n * case["taps"]) + 0.5
            h = np.sinc(m / n - case["taps"] / 2) * (0.5 - 0.5 * np.cos(2 * np.pi * m / (n * case["taps"])))
            taps = [torch.from_numpy(h.astype(np.float32)).cuda()]
        return dict(kind=kind, volt=_voltages(case["n_time"], 2 * case["n_ant"], seed)[None], nfft=[n], taps=taps,
                    window=(case["lo"], case["count"]) if case["count"] else None, f32=case["f32"])
    if kind == "xengine":
        shape = (case["n_chan"], case["n_spec"], 2 * case["n_ant"], 2)
        q = torch.empty(shape, dtype=torch.int8, device="cuda")
        g = _gen(seed)
        for f in range(0, case["n_chan"], 64):
            x = torch.randn((min(64, case["n_chan"] - f),) + shape[1:], generator=g, device="cuda")
            q[f:f + 64] = (x * 8.0).round_().clamp_(-127, 127).to(torch.int8)
        return dict(kind=kind, q=q, case=case, mode=ovro.XENG_FP32 if case["fp32"] else ovro.XENG_TC)
    if kind == "image":
        pos = _positions(case["n_ant"], seed)
        freqs = NU0 + (np.arange(case["n_chan"]) - case["n_chan"] // 2) * 10.0
        gains = None
        if case["cal"]:
            shape = (case["n_chan"], 2 * case["n_ant"])
            gains = torch.from_numpy((r.uniform(0.8, 1.2, shape[1]) * np.exp(2j * np.pi * r.uniform(size=shape[1])))
                                     .astype(np.complex64)[None].repeat(shape[0], axis=0)).cuda()
        uv = (case["uv_min"], case["uv_max"]) if case["uv_min"] > 0 or case["uv_max"] > 0 else None
        return dict(kind=kind, vis=_visibilities(case, seed, pos, freqs), pos=pos, freqs=freqs, image=case["image"],
                    store={"fp32": ovro.STORE_FP32, "bf16": ovro.STORE_BF16, "fp16": ovro.STORE_FP16}[case["store"]],
                    gains=gains, uv=uv)
    if kind == "detect":
        nfft, size = _nfft(case), case["image"]
        tones = [(int(r.integers(0, sum(nfft))), row, col, float(r.uniform(12.0, 40.0)))
                 for row, col in _sky_pixels(r, case["n_tones"], size)]
        prm = ovro.detect_params(mode=ovro.DETECT_BH if case["mode"] == "bh" else ovro.DETECT_FIXED)
        return dict(kind=kind, img=_images(sum(nfft), size, case["n_spec"], tones, seed), cell=2.0 / size, nfft=nfft,
                    freqs=_freqs(nfft), params=prm, rows=ROWS[kind])
    if kind == "drift":
        nfft, size, t = _nfft(case), case["image"], case["n_sub"]
        g = _gen(seed)
        zp = torch.randn((t, sum(nfft), size, size), generator=g, device="cuda")
        for row, col in _sky_pixels(r, case["n_tones"], size):
            d = int(r.integers(-(t - 1), t))
            c = int(r.integers(t, sum(nfft) - t)) if sum(nfft) > 2 * t else 0
            for s in range(t):
                zp[s, min(max(c + round(d * s / max(t - 1, 1)), 0), sum(nfft) - 1), row, col] += 12.0 / math.sqrt(t)
        return dict(kind=kind, zp=zp, cell=2.0 / size, nfft=nfft, freqs=_freqs(nfft), rows=ROWS[kind])
    # a step in the middle of a training run: moments filled, weights of He size
    g = _gen(seed)
    b = case["batch"]
    master = torch.from_numpy(scorer.init_weights(seed)).cuda()
    m = torch.randn(master.shape, generator=g, device="cuda") * 1e-4
    v = (torch.randn(master.shape, generator=g, device="cuda") * 1e-3).square_() + 1e-7
    x = torch.randn((b, 1600), generator=g, device="cuda")
    y = (torch.rand(b, generator=g, device="cuda") < 0.25).float()
    x += y[:, None] * 0.1
    return dict(kind="scorer", master=master, m=m, v=v, wb=master.to(torch.bfloat16), x=x, y=y, step=1000,
                ws=ovro.workspace(ovro.lib().ovro_scorer_workspace_size(b, 1)))


def _table(c, rows):
    """A candidate table by its columns, in a table of fixed length (the rest zeros) as a program that collects
    many integrations keeps it.  log10_p is a function of the 32-bit SNR beside it, and is as precise."""
    if len(c) > rows:
        raise ValueError("%d candidates, room for %d" % (len(c), rows))
    out = {"n": len(c)}
    for k in ("coarse", "fine", "chan", "row", "col", "width", "snr", "score", "freq_hz", "log10_p"):
        v = np.zeros(rows, np.float32 if k == "log10_p" else c.dtype[k])
        v[:len(c)] = c[k]
        out[k] = v
    return out


def run(state):
    kind = state["kind"]
    if kind == "pipeline":
        return _table(state["pipe"].run(state["volt"]), state["rows"])
    if kind == "upchan":
        q, f = ovro.upchan(state["volt"], state["nfft"], want_f32=state["f32"], taps=state["taps"],
                           window=state["window"])
        return {"q": q, "f32": f}
    if kind == "xengine":
        c = state["case"]
        return ovro.correlate(state["q"], c["n_ant"], c["n_chan"], c["n_spec"], state["mode"])
    if kind == "image":
        img, kept = ovro.grid_image(state["vis"], state["pos"], state["freqs"], state["image"], 2.0 / state["image"],
                                    storage=state["store"], want_counts=True, gains=state["gains"],
                                    uv_range=state["uv"])
        return {"img": img, "kept": kept}
    if kind == "detect":
        return _table(ovro.detect(state["img"], state["cell"], state["nfft"], state["freqs"], state["params"]),
                      state["rows"])
    if kind == "drift":
        c, d, snr, dmap = ovro.drift_search(state["zp"], state["cell"], state["nfft"], state["freqs"], n_sigma=8.0,
                                            want_maps=True)
        return {"table": _table(c, state["rows"]), "drift": np.pad(d, (0, state["rows"] - len(d))), "snr_map": snr, "drift_map": dmap}
    state["step"] += 1
    grad, loss = ovro.scorer_grad(state["wb"], state["x"], state["y"], ws=state["ws"])
    ovro.scorer_adam(state["master"], state["m"], state["v"], grad, state["step"], 1e-4, state["wb"])
    return {"grad": grad, "loss": loss, "master": state["master"], "m": state["m"], "v": state["v"],
            "w_bf16": state["wb"]}


# ------------------------------------------------------------------------------------------- work
def _fft_flops(n):
    return 5.0 * n * math.log2(n)


def _image_work(n_ant, n_chan, size, uv_min=0.0, uv_max=0.0):
    """(gridded visibilities, flops) of imaging: 2 x 49 taps x 4 flops a visibility, and a 2D transform of the
    padded grid."""
    pos = _positions(n_ant, 1)
    a, b = np.triu_indices(n_ant, 1)
    lam = NU0 / C_LIGHT
    du, dv = (pos[a, 0] - pos[b, 0]) * lam, (pos[a, 1] - pos[b, 1]) * lam
    ln = np.hypot(du, dv)
    half = size / 4.0                                # wavelengths: G / 2 cells of 1 / (G cell)
    keep = (np.abs(du) < half) & (np.abs(dv) < half) & (ln >= uv_min) & (ln < (uv_max if uv_max > 0 else np.inf))
    vis = float(keep.sum()) * n_chan
    g = 2 * size
    return vis, 392.0 * vis + n_chan * g * _fft_flops(g) * 2


def work(case):
    kind = case["kind"]
    if kind == "pipeline":
        n_in = 2 * case["n_ant"]
        bl = case["n_ant"] * (case["n_ant"] + 1) // 2
        flops, pix = 0.0, case["image"] ** 2 * math.pi / 4
        for n in _nfft(case):
            k = case["n_time"] // n
            flops += n_in * k * _fft_flops(n) + 32.0 * k * bl * n
            flops += _image_work(case["n_ant"], n, case["image"])[1] + pix * n * 29 * 2
        return {"bytes": len(_nfft(case)) * case["n_time"] * n_in, "flops": flops}
    if kind == "upchan":
        n, n_in = _nfft(case)[0], 2 * case["n_ant"]
        k = case["n_time"] // n - case["taps"] + 1
        out = (case["count"] or n) * k * n_in * 2
        return {"bytes": case["n_time"] * n_in + out * (5 if case["f32"] else 1),
                "flops": n_in * k * (_fft_flops(n) + (4.0 * case["taps"] * n if case["taps"] > 1 else 0))}
    if kind == "xengine":
        bl = case["n_ant"] * (case["n_ant"] + 1) // 2
        return {"bytes": case["n_chan"] * (32 * bl + 4 * case["n_spec"] * case["n_ant"]),
                "flops": 32.0 * case["n_spec"] * bl * case["n_chan"]}
    if kind == "image":
        vis, flops = _image_work(case["n_ant"], case["n_chan"], case["image"], case["uv_min"], case["uv_max"])
        return {"bytes": 16 * vis + 4 * case["n_chan"] * case["image"] ** 2, "flops": flops}
    if kind == "detect":
        vox = sum(_nfft(case)) * case["image"] ** 2 * math.pi / 4
        return {"bytes": 4 * vox, "flops": vox * 29 * 2}
    if kind == "drift":
        vox = sum(_nfft(case)) * case["image"] ** 2
        t = case["n_sub"]
        return {"bytes": vox * (4 * t * math.pi / 4 + 8), "flops": vox * math.pi / 4 * (2 * t - 1) * math.log2(t)}
    n = 1600 * 128 + 128 + 128 * 32 + 32 + 32 + 1
    return {"bytes": case["batch"] * 6404 + n * (2 + 4 + 12 + 14), "flops": 6.0 * n * case["batch"]}


# ------------------------------------------------------------------------------------------ exact
def _pswf_table(q=1024):
    """The prolate spheroidal psi_0(7 pi / 2, x / 3.5) at x = m / q, |x| <= 3.5, 1 at the middle: the even
    Legendre series whose coefficients are the lowest eigenvector of the spheroidal operator (Bouwkamp)."""
    c2 = (3.5 * math.pi) ** 2
    k = np.arange(0, 100, 2, dtype=np.float64)
    diag = k * (k + 1) + c2 * (2 * k * (k + 1) - 1) / ((2 * k - 1) * (2 * k + 3))
    off = c2 * (k[:-1] + 1) * (k[:-1] + 2) / ((2 * k[:-1] + 3) * np.sqrt((2 * k[:-1] + 1) * (2 * k[:-1] + 5)))
    vec = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))[1][:, 0] * np.sqrt(k + 0.5)
    coef = np.zeros(100)
    coef[0::2] = vec
    x = np.arange(-7 * q // 2, 7 * q // 2 + 1) / q / 3.5
    return np.polynomial.legendre.legval(x, coef) / np.polynomial.legendre.legval(0.0, coef)


def _exact_images(case, seed):
    s = prepare(case, seed)
    q, size, g = 1024, case["image"], 2 * case["image"]
    pos, freqs = s["pos"], torch.from_numpy(s["freqs"]).cuda()
    table = _pswf_table(q)
    d = np.arange(-size // 2, size // 2)
    m = np.arange(table.size) - table.size // 2
    corr = torch.from_numpy((table[None] * np.cos(2 * np.pi * np.outer(d, m) / (q * g))).sum(1) / q).cuda()
    table = torch.from_numpy(table).cuda()
    a, b = np.triu_indices(case["n_ant"], 1)
    n_ant = case["n_ant"]
    idx = torch.from_numpy(a * n_ant - a * (a - 1) // 2 + (b - a)).cuda()
    dx = torch.from_numpy(pos[a, 0] - pos[b, 0]).cuda()
    dy = torch.from_numpy(pos[a, 1] - pos[b, 1]).cuda()
    ln = torch.sqrt(dx * dx + dy * dy)
    a, b = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    dd = torch.from_numpy(d.astype(np.float64)).cuda() * (2.0 / size)
    below = dd[None, :] ** 2 + dd[:, None] ** 2 >= 1.0
    taps = torch.arange(-3, 4, device="cuda")
    img = torch.zeros((case["n_chan"], size, size), dtype=torch.float64, device="cuda")
    du = 1.0 / (g * (2.0 / size))

    def axis(x, f):
        p = torch.round(x * (f / (C_LIGHT * du)) * q).to(torch.int64)
        c0 = torch.sign(p) * ((p.abs() + q // 2) // q)
        return p, c0, (c0.abs() <= g // 2 - 4)

    for f in range(case["n_chan"]):
        pu, cu, iu = axis(dx, freqs[f])
        pv, cv, iv = axis(dy, freqs[f])
        keep = iu & iv
        if s["uv"] is not None:
            lam = ln * (freqs[f] / C_LIGHT)
            keep &= (lam >= s["uv"][0]) & (lam < (s["uv"][1] if s["uv"][1] > 0 else math.inf))
        pu, cu, pv, cv = pu[keep], cu[keep], pv[keep], cv[keep]
        v = s["vis"][f][idx[keep]].to(torch.float64)
        xx, yy = torch.complex(v[:, 0, 0], v[:, 0, 1]), torch.complex(v[:, 3, 0], v[:, 3, 1])
        if s["gains"] is not None:
            w = s["gains"][f].to(torch.complex128)
            ka, kb = a[keep], b[keep]
            xx = xx * w[2 * ka] * w[2 * kb].conj()
            yy = yy * w[2 * ka + 1] * w[2 * kb + 1].conj()
        val = (xx + yy) / 2
        wu = table[table.numel() // 2 + taps[None] * q - (pu - cu * q)[:, None]]
        wv = table[table.numel() // 2 + taps[None] * q - (pv - cv * q)[:, None]]
        where = ((g // 2 + cv[:, None] + taps)[:, :, None] * g + (g // 2 + cu[:, None] + taps)[:, None, :]).reshape(-1)
        wt = wv[:, :, None] * wu[:, None, :]
        grid = torch.zeros((2, g * g), dtype=torch.float64, device="cuda")
        grid[0].index_add_(0, where, (wt * val.real[:, None, None]).reshape(-1))
        grid[1].index_add_(0, where, (wt * val.imag[:, None, None]).reshape(-1))
        z = torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(torch.complex(grid[0], grid[1]).view(g, g))))
        o = g // 2 - size // 2
        # the mirrors' half of the transform is the conjugate: twice the real part over twice the count
        out = z[o:o + size, o:o + size].real * (g * g) / max(int(keep.sum()), 1) / (corr[:, None] * corr[None])
        img[f] = out.masked_fill(below, 0.0)
    return {"img": img, "kept": None}


def _exact_upchan(case, seed):
    if not case["f32"]:
        return None                                 # bytes alone come back
    s = prepare(case, seed)
    n, taps = s["nfft"][0], case["taps"]
    v = s["volt"][0].to(torch.int16)
    re, im = v >> 4, v & 15
    re, im = torch.where(re >= 8, re - 16, re), torch.where(im >= 8, im - 16, im)
    k = case["n_time"] // n
    x = torch.complex(re[:k * n].double(), im[:k * n].double()).view(k, n, -1)
    if taps > 1:
        h = s["taps"][0].double().view(taps, n, 1)
        x = sum(h[p] * x[p:k - taps + 1 + p] for p in range(taps))
    out = torch.fft.fftshift(torch.fft.fft(x, dim=1), dim=1)
    if s["window"]:
        out = out[:, s["window"][0]:s["window"][0] + s["window"][1]]
    return {"q": None, "f32": torch.view_as_real(out.transpose(0, 1).contiguous()).reshape(-1)}


def _shift(d, n, t):
    """The Taylor tree's offset at row t of n of a line of total drift d."""
    if n == 1:
        return 0
    return _shift(d // 2, n // 2, t) if t < n // 2 else d - d // 2 + _shift(d // 2, n // 2, t - n // 2)


def _exact_drift(case, seed):
    s = prepare(case, seed)
    zp, t, size = s["zp"], case["n_sub"], case["image"]
    snr = torch.full(zp.shape[1:], -math.inf, dtype=torch.float64, device="cuda")
    lo = 0
    for n in s["nfft"]:
        for d in range(-(t - 1), t):
            f0, f1 = max(0, -d), n - max(0, d)      # start channels whose line ends inside the coarse channel
            if f1 <= f0:
                continue
            acc = 0.0
            for row in range(t):
                o = lo + (_shift(d, t, row) if d >= 0 else -_shift(-d, t, row))
                acc = acc + zp[row, f0 + o:f1 + o].double()
            part = snr[lo + f0:lo + f1]
            torch.maximum(part, acc / math.sqrt(t), out=part)
        lo += n
    d = (torch.arange(size, device="cuda", dtype=torch.float64) - size // 2) * (2.0 / size)
    snr.masked_fill_((d[None, :] ** 2 + d[:, None] ** 2 >= 1.0)[None], -math.inf)
    return {"table": None, "drift": None, "snr_map": snr, "drift_map": None}


def _exact_scorer(case, seed):
    s = prepare(case, seed)
    w = s["wb"].double().requires_grad_()
    h, off = s["x"].double(), 0
    for i, o in ((1600, 128), (128, 32), (32, 1)):
        h = h @ w[off:off + i * o].view(o, i).T + w[off + i * o:off + i * o + o]
        off += i * o + o
        if o > 1:
            h = torch.nn.functional.gelu(h)
    loss = torch.nn.functional.binary_cross_entropy_with_logits(h[:, 0], s["y"].double())
    g, = torch.autograd.grad(loss, w)
    m = 0.9 * s["m"].double() + 0.1 * g
    v = 0.999 * s["v"].double() + 0.001 * g * g
    t = s["step"] + 1
    master = s["master"].double() - 1e-4 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return {"grad": g, "loss": loss.detach().reshape(1), "master": master, "m": m, "v": v, "w_bf16": master}


def exact(case, seed):
    kind = case["kind"]
    if kind == "image":
        return _exact_images(case, seed)
    if kind == "upchan":
        return _exact_upchan(case, seed)
    if kind == "drift":
        return _exact_drift(case, seed)
    if kind == "scorer":
        return _exact_scorer(case, seed)
    return None          # whole numbers (xengine), or a whole search in 64 bits (minutes)
