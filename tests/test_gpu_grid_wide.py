"""Imaging over a wide band: the call returns before the stream reaches it, and
a plan whose tile lists outgrow the workspace is refused before anything is
launched, exactly where the lists' length says so."""
import numpy as np
import pytest
import torch

import synth
from oracle import xengine as OX

pytestmark = pytest.mark.gpu
C = 299_792_458.0


def _case(n_ant, n, freqs, seed):
    g = np.random.default_rng(seed)
    pos = synth.antenna_positions(synth.Config("t", n_ant, 1, [16], 16, n, 11, core_radius_m=200.0))
    vis = g.integers(-2 ** 20, 2 ** 20, (len(freqs), OX.n_baselines(n_ant), 4, 2)).astype(np.int32)
    return pos, torch.from_numpy(vis).cuda()


def _entries(pos, freqs, n, cell):
    """4 x 4-cell tiles of the rows v >= 0 that the footprints of every baseline and its mirror touch."""
    g, q = 2 * n, 1024
    cmax = g // 2 - 4
    s = np.array([f / (C * (1.0 / (g * cell))) * q for f in freqs])
    a, b = np.triu_indices(len(pos), 1)
    box = []
    for axis in (0, 1):
        d = pos[a, axis] - pos[b, axis]
        p = np.rint(d[:, None] * np.array([s.min(), s.max()])[None])
        c = np.sign(p) * np.floor((np.abs(p) + q // 2) / q)
        box.append((np.maximum(c.min(1), -cmax).astype(int), np.minimum(c.max(1), cmax).astype(int)))
    (u0, u1), (v0, v1) = box
    live = (u0 <= u1) & (v0 <= v1)

    def tiles(v0, v1, u0, u1):
        r = np.where(v1 + 3 < 0, 0, (v1 + 3) // 4 - np.maximum(v0 - 3, 0) // 4 + 1)
        return r * ((g // 2 + u1 + 3) // 4 - (g // 2 + u0 - 3) // 4 + 1)
    return int((tiles(v0, v1, u0, u1) + tiles(-v1, -v0, -u1, -u0))[live].sum()), a.size


def test_refused_where_the_lists_outgrow_the_workspace(lib):
    n, cell, seen = 256, 0.001, set()
    for ratio in (1.1, 1.3, 1.5, 1.6, 1.7, 1.8, 1.9, 2.0, 2.2, 2.5, 3.0, 3.3, 3.6, 4.5, 80.0):
        freqs = np.array([20e6, 20e6 * ratio])
        pos, vis = _case(30, n, freqs, 5)
        entries, n_cross = _entries(pos, freqs, n, cell)
        before = lib.launch_count()
        try:
            lib.grid_image(vis, pos, freqs, n, cell)
            ok = True
        except lib.OvroError as e:
            assert e.status == lib.ERR_CAPACITY
            assert lib.launch_count() == before
            ok = False
        assert ok == (entries <= 24 * n_cross), (ratio, entries / n_cross)
        seen.add(ok)
    assert seen == {True, False}


@pytest.mark.parametrize("step_hz", [10.0, 24e3])
def test_returns_before_the_stream_reaches_it(lib, step_hz):
    n, freqs = 1024, 60e6 + np.arange(5) * step_hz
    pos, vis = _case(64, n, freqs, 7)
    want = lib.grid_image(vis, pos, freqs, n, 2.0 / n)
    out = torch.empty_like(want)
    ws = lib.workspace(lib.grid_image_workspace_size(64, 5, n))
    torch.cuda.synchronize()
    busy = torch.cuda.Event()
    torch.cuda._sleep(2_000_000_000)                  # about a second
    busy.record()
    lib.grid_image(vis, pos, freqs, n, 2.0 / n, out=out, ws=ws)
    assert not busy.query()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
