"""CUDA-core contractions (float mode) at the edges of their tiles and splits: one conv and one FC layer's three passes against
double-precision torch on the layer's own stored inputs."""
from __future__ import annotations

import numpy as np
import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,c0,c1,width,b,R", [
    (4, 4, 4, 4, 20, 1, 1),          # smallest tile, one pixel tile, K = 36
    (5, 7, 12, 36, 24, 3, 2),        # odd image, channels that are no multiple of a reduction step or a tile
    (6, 6, 17, 33, 21, 2, 1),        # odd channel counts: the scalar loads
    (8, 8, 64, 128, 132, 9, 2),      # whole tiles
    (16, 16, 20, 260, 68, 4, 3),     # more columns than two tiles; long weight-gradient reduction (split)
    (9, 3, 132, 8, 516, 37, 1),      # few columns, long reduction: split forward and data gradient
])
def test_conv_and_fc_passes(H, W, c0, c1, width, b, R):
    import torch
    import torch.nn.functional as F

    from paper_2112_15317_b200 import binding as sb
    wl = si.Workload("contract", [(si.CONV3X3_RELU, c0), (si.CONV3X3_RELU, c1), (si.FC_RELU, width), (si.FC_RELU, 19), (si.FC, 10), (si.SOFTMAX_XENT, 10)],
                     H, W, 4, b, R, 1)
    m = tu.gpu_model(wl, si.make_params(wl, bias_std=0.2), sb.SB_FP32)
    xs, ys = tu.device_batch(wl, *si.make_batch(wl), False)
    m.forward(xs, ys)
    m.backward()
    t = lambda what, li: torch.from_numpy(np.concatenate([m.read(what, li, r, squeeze=False) for r in range(R if li < 2 else 1)])).double()  # noqa: E731
    wt = lambda what, li: torch.from_numpy(m.read(what, li, 0, squeeze=False)).double()  # noqa: E731
    checks = tu.Checks()

    x = t(sb.SB_T_ACT, 0).permute(0, 3, 1, 2).requires_grad_()
    w = wt(sb.SB_T_WEIGHT, 1).permute(0, 3, 1, 2).requires_grad_()
    bias = wt(sb.SB_T_BIAS, 1).reshape(-1).requires_grad_()
    y = F.conv2d(x, w, bias, padding=1)
    y.backward(t(sb.SB_T_DACT, 1).permute(0, 3, 1, 2))
    checks.le("conv forward", tu.maxrel(t(sb.SB_T_ACT, 1), y.relu().permute(0, 2, 3, 1).detach()), 1e-5)
    checks.le("conv input gradient", tu.maxrel(t(sb.SB_T_DACT, 0), (x.grad * (x > 0)).permute(0, 2, 3, 1).detach()), 1e-5)
    checks.le("conv weight gradient", tu.maxrel(wt(sb.SB_T_GRAD_W, 1), w.grad.permute(0, 2, 3, 1)), 1e-5)
    checks.le("conv bias gradient", tu.maxrel(wt(sb.SB_T_GRAD_B, 1).reshape(-1), bias.grad), 1e-5)

    x = t(sb.SB_T_ACT, 1).reshape(wl.B, -1).requires_grad_()
    w = wt(sb.SB_T_WEIGHT, 2)[:, :, 0, 0].requires_grad_()
    bias = wt(sb.SB_T_BIAS, 2).reshape(-1).requires_grad_()
    y = F.linear(x, w, bias)
    y.backward(t(sb.SB_T_DACT, 2)[:, :, 0, 0])
    checks.le("fc forward", tu.maxrel(t(sb.SB_T_ACT, 2)[:, :, 0, 0], y.relu().detach()), 1e-5)
    checks.le("fc input gradient", tu.maxrel(t(sb.SB_T_DACT, 1).reshape(wl.B, -1), (x.grad * (x > 0)).detach()), 1e-5)
    checks.le("fc weight gradient", tu.maxrel(wt(sb.SB_T_GRAD_W, 2)[:, :, 0, 0], w.grad), 1e-5)
    checks.le("fc bias gradient", tu.maxrel(wt(sb.SB_T_GRAD_B, 2).reshape(-1), bias.grad), 1e-5)
    m.close()
    checks.finish()
