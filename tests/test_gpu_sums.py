"""Sums of FC layers with long rows against 64-bit sums of the same stored operands: how far a chain of additions carries their rounding."""
from __future__ import annotations

import math

import pytest

pytestmark = pytest.mark.gpu


def _view(m, what, layer):
    """A float or bf16 tensor of the model as a torch view of its memory."""
    import torch

    from paper_2112_15317_b200 import binding as sb
    ptr, shape, dt = m.tensor_info(what, layer)
    dtype = {sb.SB_DT_F32: torch.float32, sb.SB_DT_BF16: torch.bfloat16}[dt]
    off, n = ptr - m.arena.data_ptr(), math.prod(shape)
    return m.arena[off:off + n * dtype.itemsize].view(dtype).view([s for i, s in enumerate(shape) if i == 0 or s > 1])


def _logits_error(m, layer, x, in_f):
    """Relative 2-norm error of FC layer `layer`, run on x [B, in_f] with He-normal weights and zero biases."""
    import torch

    from paper_2112_15317_b200 import binding as sb
    g = torch.Generator(device="cuda").manual_seed(3)
    w = _view(m, sb.SB_T_WEIGHT, layer)
    w.copy_(torch.randn(w.shape, generator=g, device="cuda") * math.sqrt(2.0 / in_f))
    _view(m, sb.SB_T_BIAS, layer).zero_()
    m.refresh_shadow()
    B, out = x.shape[0], w.numel() // in_f
    m.forward_layers(layer, layer, [torch.zeros(B, m.cfg.H, m.cfg.W, m.cfg.C, dtype=x.dtype, device="cuda")] if layer else [x],
                     [torch.zeros(B, dtype=torch.int32, device="cuda")])
    want = x.reshape(B, in_f).double() @ (w.to(torch.bfloat16) if m.bf16 else w).double().reshape(out, in_f).T
    return ((_view(m, sb.SB_T_ACT, layer).reshape(B, out).double() - want).norm() / want.norm()).item()


@pytest.mark.parametrize("in_f,out,B", [(25088, 4096, 16), (8192, 8192, 128)])
def test_streamed_fc_forward(in_f, out, B):
    import torch

    from paper_2112_15317_b200 import binding as sb
    m = sb.Model([(sb.SB_FC, out), (sb.SB_SOFTMAX_XENT, out)], 1, 1, in_f, B, 1, 1, sb.SB_BF16)
    x = torch.randn(B, in_f, generator=torch.Generator(device="cuda").manual_seed(B), device="cuda").relu().to(torch.bfloat16)
    # A tensor core adds 16 products at a time and cuts the sum off, half a unit (2^-25) on average, at partial sums of two thirds of the
    # result.  The chains are 3136 and 2048 terms long (2.4e-6 and 1.5e-6 measured, 5.3e-6 and 3.2e-6 over twice that length).
    chain = {25088: 3136, 8192: 2048}[in_f]
    assert _logits_error(m, 0, x, in_f) < chain / 16 * 2.0 ** -25 * 2 / 3
    m.close()


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("B", [2, 96])
@pytest.mark.parametrize("side,channels", [(16, 16), (56, 8)])      # 4096 and 25088 inputs
def test_narrow_logits(side, channels, B, precision):
    import torch

    from paper_2112_15317_b200 import binding as sb
    m = sb.Model([(sb.SB_CONV3X3_RELU, channels), (sb.SB_FC, 10), (sb.SB_SOFTMAX_XENT, 10)], side, side, 4, B, 1, 1,
                 sb.SB_FP32 if precision == "fp32" else sb.SB_BF16)
    in_f = side * side * channels
    act = _view(m, sb.SB_T_ACT, 0)
    act.copy_(torch.randn(act.shape, generator=torch.Generator(device="cuda").manual_seed(B), device="cuda").relu())
    # Chains of n = in_f / 128 products of either sign: every addition rounds by 2^-25 of a sum that grows with the root of its length, which
    # adds up to 2^-25 sqrt(n / 2) of the result; the seven levels of additions across chains and lanes and the bias's make it n / 2 + 8.
    # Products of bf16 operands have 16 bits and short sums of them are exact: half over long rows.  (Measured: 4096 inputs 1.1e-7 and
    # 0.9e-7, 25088 2.4e-7 and 1.0e-7; in one chain a lane 1.5 to 2.2e-7, 4.0 to 4.2e-7 and 1.7e-7.)
    bound = 2.0 ** -25 * math.sqrt(in_f / 128 / 2 + 8) * (1.0 if precision == "fp32" or in_f < 10000 else 0.5)
    err = _logits_error(m, 1, act, in_f)
    assert err < bound, (err, bound)
    m.close()
