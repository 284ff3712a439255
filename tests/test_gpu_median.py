"""GPU parity of the running-median high-pass and the boxcars where the band ranking and the
walk can go wrong: the shortest coarse channels, lengths just past a kernel's
keys per thread, many equal values, dead channels, pixels far from zero (the
finer selection) and pixels both kernels give up (the full walk)."""
import numpy as np
import pytest
import torch

from oracle import detect as OD, imaging as OI

pytestmark = pytest.mark.gpu


def _cube(kind, n_chan, n, g):
    x = g.normal(0.3, 2.0, (n_chan, n, n))
    if kind == "ties":
        x = np.round(x * 2) / 2
    elif kind == "dead":
        x[n_chan // 4: n_chan // 4 + n_chan // 5] = 0.0
    elif kind == "offset":
        x += 60.0 * g.uniform(-1, 1, (1, n, n))
    elif kind == "scale":
        x *= np.exp(2 * g.normal(size=(1, n, n)))
    elif kind == "flat":
        x[:, ::2] = 1.0                              # whole spectra of one value
    return x.astype(np.float32)


@pytest.mark.parametrize("nfft,kind", [([1, 2, 3, 5], "noise"), ([33, 64, 100], "ties"), ([511, 513], "offset"),
                                       ([1024, 1025], "dead"), ([1030], "flat"), ([2047], "scale"),
                                       ([2049], "ties"), ([2052], "offset")])
def test_highpass_vs_oracle(lib, nfft, kind):
    n, cell = 16, 0.4
    g = np.random.default_rng(sum(nfft))
    cube = _cube(kind, sum(nfft), n, g)
    mask = OI.horizon_mask(n, cell)
    d = torch.from_numpy(cube).cuda()
    st = lib.detect_stats(d, cell)
    zp, snr, _ = lib.detect_filter(d, st, cell, nfft, want_zp=True)
    plain = lib.detect_filter(d, st, cell, nfft)[1]
    assert torch.equal(plain, snr)                   # with or without the high-passed cube
    s = st.cpu().numpy()
    z = np.zeros(cube.shape)
    for f in range(cube.shape[0]):
        if s[f, 1] > 0:
            z[f][mask] = (cube[f][mask].astype(np.float64) - s[f, 0]) / (OD.MAD_TO_SIGMA * s[f, 1])
    ref = OD.highpass(z, OD.chan_bounds_of(nfft), [OD.window_channels(24000.0 / k) for k in nfft])
    ref[:, ~mask] = 0
    # z is rounded to 24 bits before and after the subtraction
    assert np.abs(zp.cpu().numpy() - ref).max() <= 1e-5 * max(1.0, np.abs(z).max())
    so, _ = OD.matched_filter(ref, OD.chan_bounds_of(nfft))
    so[:, ~mask] = 0
    # prefix sums of 107 values: at most 107 roundings of the largest sum
    tol = 107 * 2.0 ** -24 * np.abs(ref).max() * 107 + 1e-5 * 10 * max(1.0, np.abs(z).max())
    assert np.abs(snr.cpu().numpy() - so).max() <= tol
