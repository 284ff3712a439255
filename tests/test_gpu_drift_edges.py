"""GPU parity of the drift search at the edges of its tiles: coarse channels of
one channel, shorter than a path, and around the start channels a thread and a
CTA take; with and without the maps; by a threshold known before and after the
sums."""
import numpy as np
import pytest
import torch

from oracle import drift as ODR, imaging as OI

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [2, 4, 8, 16])
def test_short_and_ragged_coarse_channels(lib, T):
    nfft = [1, 2, T - 1, T, T + 1, 5, 31, 33, 64 + 3]
    n, cell = 16, 2.0 / 16
    g = np.random.default_rng(T)
    zp = g.normal(size=(T, sum(nfft), n, n)).astype(np.float32)
    zp[:, ::7, 5, 9] += 8.0 / np.sqrt(T)
    mask = OI.horizon_mask(n, cell)
    freqs = 60e6 + np.arange(sum(nfft)) * 10.0
    d = torch.from_numpy(zp).cuda()
    so, do, _, _ = ODR.drift_search(zp, mask, nfft, n_sigma=6.0)
    c, dr, snr, dmap = lib.drift_search(d, cell, nfft, freqs, n_sigma=6.0, want_maps=True)
    snr, dmap = snr.cpu().numpy(), dmap.cpu().numpy()
    assert np.array_equal(np.isinf(snr), np.isinf(so))
    # T roundings of a sum of at most T values of |z| < 16, then one product
    tol = (T + 1) * 2.0 ** -24 * 16 * T / np.sqrt(T)
    fin = np.isfinite(so)
    assert np.abs(snr[fin] - so[fin]).max() <= tol
    near = np.abs(snr - so) <= tol
    assert ((dmap == do) | near)[fin].all() and (dmap[~fin] == 0).all()
    assert (dmap == do)[fin].mean() > 0.999
    c2, dr2 = lib.drift_search(d, cell, nfft, freqs, n_sigma=6.0)
    assert len(c) > 0 and np.array_equal(c, c2) and np.array_equal(dr, dr2)
    prm = lib.detect_params(mode=lib.DETECT_BH, alpha=0.05)
    c3, dr3 = lib.drift_search(d, cell, nfft, freqs, params=prm)
    ref = ODR.drift_search(zp, mask, nfft, mode="bh", alpha=0.05)
    assert {(int(x["chan"]), int(x["row"]), int(x["col"])) for x in c3} == {(x.chan, x.row, x.col) for x in ref[2]}
