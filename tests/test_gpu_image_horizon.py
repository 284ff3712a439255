"""Pixels on the unit circle (0.6, 0.8 and the like, at cells that are no power of two)
are below the horizon for the imager, the search and the drift search alike: l^2 + m^2 in
FP64, each product rounded, as the oracle's mask has it."""
import numpy as np
import pytest
import torch

import synth
from oracle import imaging as OI, xengine as OX

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cell", [(16, 0.2), (64, 0.04), (128, 0.02), (256, 0.01), (64, 1 / 13), (256, 1 / 65)])
def test_one_horizon(lib, n, cell):
    mask = OI.horizon_mask(n, cell)
    n_ant, freqs = 24, 60e6 + np.arange(2) * 10.0
    g = np.random.default_rng(n)
    pos = synth.antenna_positions(synth.Config("t", n_ant, 1, [16], 16, n, 11, core_radius_m=2.0 / cell))
    vis = g.integers(-2 ** 20, 2 ** 20, (2, OX.n_baselines(n_ant), 4, 2)).astype(np.int32)
    img = lib.grid_image(torch.from_numpy(vis).cuda(), pos, freqs, n, cell).cpu().numpy()
    assert np.array_equal(img != 0, np.broadcast_to(mask, img.shape))
    z = torch.from_numpy(g.normal(size=(2, 40, n, n)).astype(np.float32)).cuda()
    st = torch.ones((40, 2), dtype=torch.float64, device="cuda")
    width = lib.detect_filter(z[0], st, cell, [40])[2].cpu().numpy()   # at least 1 for a pixel searched
    assert np.array_equal(width != 0, np.broadcast_to(mask, width.shape))
    snr = lib.drift_search(z, cell, [40], np.arange(40.0), n_sigma=50.0, want_maps=True)[2].cpu().numpy()
    assert np.array_equal(np.isfinite(snr), np.broadcast_to(mask, snr.shape))
