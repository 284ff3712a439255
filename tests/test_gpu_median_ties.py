"""The running-median high-pass where many values of a spectrum are equal: flagged
channels (zero in every pixel) up to all of them, quantised values, two values
only, equal values far from zero or beyond the band, infinite channels, at the
lengths where the ranking changes its shape.  And what it costs: equal values
were compared with one another, 4096 channels with 40% flagged took five
times the call without."""
import numpy as np
import pytest
import torch

from oracle import detect as OD, imaging as OI

pytestmark = pytest.mark.gpu
N, CELL = 16, 0.6                                     # 9 pixels above the horizon


def _cube(kind, nc, g):
    x = g.normal(0.0, 2.0, (nc, N, N))
    flagged = g.uniform(size=nc)
    flagged[nc // 3] = 0.999                          # one channel at least has values
    if kind.startswith("flagged"):
        x[flagged < float(kind[7:])] = 0.0
    elif kind == "quantised":
        x = np.round(x)
    elif kind == "two":
        x = np.where(x > g.uniform(-1, 1, (1, N, N)), 3.0, -1.0)
    elif kind == "far":
        x = 4000.0 + np.round(x * 4) / 4
        x[flagged < 0.5] = 4000.25
    elif kind == "edge":                              # equal values across the band's upper end
        x[flagged < 0.45] = 1.5
    elif kind == "infinite":
        x[flagged < 0.2] = np.inf
        x[flagged > 0.9] = -np.inf
    return x.astype(np.float32)


def _filter(lib, cube, nfft, **kw):
    st = torch.zeros((cube.shape[0], 2), dtype=torch.float64, device="cuda")
    st[:, 1] = 1.0 / OD.MAD_TO_SIGMA                  # z = x
    return lib.detect_filter(torch.from_numpy(cube).cuda(), st, CELL, nfft, **kw)


KINDS = ["flagged0.1", "flagged0.3", "flagged0.7", "flagged0.99", "quantised", "two", "far", "edge", "infinite"]


@pytest.mark.parametrize("nc,kind", [(nc, k) for nc in (100, 511, 1024, 1025, 2400, 4096, 4100, 8192) for k in KINDS] +
                         [(16384, "flagged0.3"), (16384, "edge")])
def test_equal_values(lib, nc, kind):
    g = np.random.default_rng(nc + len(kind))
    cube = _cube(kind, nc, g)
    mask = OI.horizon_mask(N, CELL)
    zp, snr, width = (t.cpu().numpy()[:, mask] for t in _filter(lib, cube, [nc], want_zp=True))
    z = cube[:, mask].astype(np.float64)
    bounds = OD.chan_bounds_of([nc])
    with np.errstate(invalid="ignore"):
        ref = OD.highpass(z, bounds, [OD.window_channels(24000.0 / nc)])
    fin = np.isfinite(ref)
    assert np.abs(ref[fin]).max() > 0
    # z, the median and their difference are each rounded to 24 bits
    tol = 1e-6 * np.abs(z[np.isfinite(z)]).max()
    assert np.array_equal(np.isfinite(zp), fin)
    assert np.abs(zp[fin] - ref[fin]).max() <= tol
    if kind == "infinite":
        return
    so, _ = OD.matched_filter(ref, bounds)
    # prefix sums of 107 values: at most 107 roundings of the largest sum, and the
    # medians' own error in each term
    lim = 107 * 2.0 ** -24 * np.abs(ref).max() * 107 + 10 * tol
    assert np.abs(snr - so).max() <= lim
    # the width reported reaches the best value
    assert set(np.unique(width)) <= set(OD.WIDTHS)
    total = np.concatenate([np.zeros((1, ref.shape[1])), np.cumsum(ref, axis=0)])
    lo = np.arange(nc)[:, None] - (width - 1) // 2
    assert lo.min() >= 0 and (lo + width).max() <= nc
    got = (np.take_along_axis(total, lo + width, 0) - np.take_along_axis(total, lo, 0)) / np.sqrt(width)
    assert (so - got).max() <= 2 * lim


def test_cost_of_flagged_channels(lib):
    nc, n = 4096, 128
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    x = torch.randn((nc, n, n), generator=g, device="cuda")
    st = torch.zeros((nc, 2), dtype=torch.float64, device="cuda")
    st[:, 1] = 1.0 / OD.MAD_TO_SIGMA

    def best():
        ms = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            lib.detect_filter(x, st, 2.0 / n, [nc])
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms)
    plain = best()
    x[torch.rand(nc, generator=g, device="cuda") < 0.4] = 0.0
    assert best() <= 2.5 * plain
