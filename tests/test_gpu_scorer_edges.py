"""GPU parity of the scorer's forward pass and gradients at the edges of its
tiles and splits, with buffers off 16 bytes, and with a workspace sized for a
larger batch."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import scorer as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,shift", [(1, 0), (3, 1), (63, 0), (64, 2), (65, 0), (257, 3), (700, 0)])
def test_batches_vs_oracle(lib, B, shift):
    g = np.random.default_rng(B)
    x = g.normal(size=(B, 1600)).astype(np.float32)
    y = (g.uniform(size=B) < 0.4).astype(np.float32)
    theta = (S.init_params(2) + g.normal(size=S.n_params()) * 0.01).astype(np.float32)
    # rows of a buffer that starts `shift` floats past a 16-byte boundary
    xd = torch.zeros(B * 1600 + 4, device="cuda")[shift:shift + B * 1600].view(B, 1600)
    xd.copy_(torch.from_numpy(x))
    yd = torch.from_numpy(y).cuda()
    ws = lib.workspace(lib.lib().ovro_scorer_workspace_size(2 * B + 300, 1))
    w32 = torch.zeros(theta.size + 4, device="cuda")[shift:shift + theta.size]
    w32.copy_(torch.from_numpy(theta))
    wb = torch.zeros(theta.size + 8, dtype=torch.bfloat16, device="cuda")[shift:shift + theta.size]
    wb.copy_(w32)
    tb = S.bf16_round(theta)
    logit = lib.scorer_forward(wb, xd, ws=ws).cpu().numpy()
    ref, _ = S.forward(tb, x.astype(np.float64))
    # 1600-term FP32 sums of values of order 1
    assert np.abs(logit - ref).max() <= 1e-5 * max(1.0, np.abs(ref).max())
    for w, t in ((wb, tb), (w32, theta.astype(np.float64))):
        grad, loss = lib.scorer_grad(w, xd, yd, ws=ws)
        rg, rl = S.backward(t, x.astype(np.float64), y.astype(np.float64))
        assert abs(loss.item() - rl) <= 1e-5 * max(1.0, rl)
        assert np.abs(grad.cpu().numpy() - rg).max() <= 1e-5 * np.abs(rg).max()


def test_workspace_of_a_larger_batch_serves_a_smaller_one(lib):
    size = lib.lib().ovro_scorer_workspace_size
    sizes = [size(b, 1) for b in range(1, 12000, 37)]
    assert sizes == sorted(sizes)
    assert ctypes.c_size_t(size(0, 1)).value == 0
