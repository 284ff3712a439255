"""A channel whose frequency is not a number grids nothing and leaves the other
channels of its call as they are, whatever the band."""
import numpy as np
import pytest
import torch

import synth
from oracle import imaging as OI, xengine as OX

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,step_hz", [(16, 10.0), (256, 10.0), (64, 300e3), (1024, 10.0)])
@pytest.mark.parametrize("where", [0, 1, 39])
def test_one_channel_without_a_frequency(lib, n, step_hz, where):
    n_ant, n_chan = 24, 40
    freqs = 60e6 + np.arange(n_chan) * step_hz
    g = np.random.default_rng(n + where)
    pos = synth.antenna_positions(synth.Config("t", n_ant, 1, [16], 16, n, 11, core_radius_m=40.0))
    vis = g.integers(-2 ** 20, 2 ** 20, (n_chan, OX.n_baselines(n_ant), 4, 2)).astype(np.int32)
    odd = freqs.copy()
    odd[where] = np.nan
    img, cnt = lib.grid_image(torch.from_numpy(vis).cuda(), pos, odd, n, 2.0 / n, want_counts=True)
    img, cnt = img.cpu().numpy(), cnt.cpu().numpy()
    assert cnt[where] == 0 and not img[where].any()
    chans = [c for c in (0, 1, 20, 39) if c != where]
    ref, ng, _ = OI.dirty_images(vis, pos, freqs, n, 2.0 / n, channels=chans)
    assert np.array_equal(cnt[chans], ng)
    assert (np.abs(img[chans] - ref) / np.abs(ref).max(axis=(1, 2), keepdims=True)).max() <= 1e-5
