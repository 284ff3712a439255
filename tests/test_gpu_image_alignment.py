"""Images into a buffer that starts on any float: the same bits as into an aligned
one, in every storage format, for the fewest and the most columns a CTA, an odd
number of channels and calibrated visibilities, and nothing written beyond."""
import numpy as np
import pytest
import torch

import synth
from oracle import xengine as OX

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 32, 256, 1024])
@pytest.mark.parametrize("storage", ["STORE_FP32", "STORE_BF16", "STORE_FP16"])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_image_starts_on_any_float(lib, n, storage, shift):
    n_ant, n_chan = 24, 3
    g = np.random.default_rng(n + shift)
    pos = synth.antenna_positions(synth.Config("t", n_ant, 1, [16], 16, n, 11, core_radius_m=40.0))
    freqs = 60e6 + np.arange(n_chan) * 10.0
    vis = torch.from_numpy(g.integers(-2 ** 20, 2 ** 20, (n_chan, OX.n_baselines(n_ant), 4, 2)).astype(np.int32)).cuda()
    gains = torch.from_numpy(np.exp(2j * np.pi * g.uniform(size=(n_chan, 2 * n_ant))).astype(np.complex64)).cuda()
    for kw in ({}, {"gains": gains, "uv_range": (1.0, 60.0)}):
        want = lib.grid_image(vis, pos, freqs, n, 2.0 / n, storage=getattr(lib, storage), **kw)
        flat = torch.full((want.numel() + shift + 1,), -7.0, device="cuda")
        out = flat[shift:-1].view(want.shape)
        assert out.data_ptr() % 8 == 4 * (shift % 2)
        lib.grid_image(vis, pos, freqs, n, 2.0 / n, storage=getattr(lib, storage), out=out, **kw)
        assert float(want.abs().max()) > 0.0
        assert torch.equal(out, want)
        assert bool((flat[:shift] == -7.0).all()) and float(flat[-1]) == -7.0
