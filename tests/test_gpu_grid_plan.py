"""GPU parity of imaging where the device-made lists can go wrong: the fewest
antennas, the smallest and the largest image, an odd channel count, channels
spread over a wide band (general records, a counted plan) and a plan that does
not fit its workspace."""
import numpy as np
import pytest
import torch

import synth
from oracle import imaging as OI, xengine as OX

pytestmark = pytest.mark.gpu


def _case(n_ant, n, freqs, seed):
    g = np.random.default_rng(seed)
    pos = synth.antenna_positions(synth.Config("t", n_ant, 1, [16], 16, n, 11, core_radius_m=200.0))
    vis = g.integers(-2 ** 20, 2 ** 20, (len(freqs), OX.n_baselines(n_ant), 4, 2)).astype(np.int32)
    return pos, vis


@pytest.mark.parametrize("n_ant,n,cell,n_chan,step_hz", [
    (1, 16, 2.0 / 16, 1, 0.0), (2, 16, 2.0 / 16, 1, 0.0), (23, 16, 0.001, 33, 10.0), (24, 64, 0.004, 65, 10.0),
    (9, 1024, 2.0 / 1024, 2, 100.0), (12, 64, 2.0 / 64, 5, 300e3), (40, 128, 0.004, 3, 400e3)])
def test_lists_vs_oracle(lib, n_ant, n, cell, n_chan, step_hz):
    freqs = 60e6 + np.arange(n_chan) * step_hz
    pos, vis = _case(n_ant, n, freqs, n + n_ant)
    img, cnt = lib.grid_image(torch.from_numpy(vis).cuda(), pos, freqs, n, cell, want_counts=True)
    chans = sorted({0, n_chan // 2, n_chan - 1})
    ref, ng, _ = OI.dirty_images(vis, pos, freqs, n, cell, channels=chans)
    assert np.array_equal(cnt.cpu().numpy()[chans], ng)
    got = img.cpu().numpy()[chans]
    scale = np.maximum(np.abs(ref).max(axis=(1, 2), keepdims=True), 1e-30)
    assert (np.abs(got - ref) / scale).max() <= 1e-5
    again = lib.grid_image(torch.from_numpy(vis).cuda(), pos, freqs, n, cell)
    assert torch.equal(img, again)                   # list order, and so rounding, is fixed


def test_plan_too_large_is_refused(lib):
    # from 1 to 80 MHz every footprint sweeps most of its quadrant
    freqs = np.array([1e6, 80e6])
    pos, vis = _case(30, 256, freqs, 5)
    with pytest.raises(lib.OvroError) as e:
        lib.grid_image(torch.from_numpy(vis).cuda(), pos, freqs, 256, 0.001)
    assert e.value.status == lib.ERR_CAPACITY
