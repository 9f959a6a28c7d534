"""The logits layer's narrow kernel with the loss layer in it (whole passes) against the two layers run one by one, and the narrow input
gradient by 16-byte columns against double-precision torch: widths of one run and of several, odd widths, one row, all classes."""
from __future__ import annotations

import numpy as np
import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("width,classes,b,R", [
    (8, 2, 1, 1),          # one 16-byte run, one row
    (4096, 10, 33, 2),     # four steps of the reduction; more rows than a warp of the mean
    (1032, 16, 7, 3),      # a ragged last step, all classes
    (77, 10, 5, 2),        # odd width: scalar loads
    (64, 3, 70, 1),        # more than 64 rows: two rows a thread in the input gradient
])
def test_head_of_whole_passes(bf16, width, classes, b, R):
    import torch

    from paper_2112_15317_b200 import binding as sb
    wl = si.Workload("head", [(si.CONV3X3_RELU, 8), (si.FC_RELU, width), (si.FC, classes), (si.SOFTMAX_XENT, classes)], 4, 4, 4, b, R, 1)
    params = si.make_params(wl, bias_std=0.2)
    x, y = si.make_batch(wl)
    y = y.copy()
    y[0] = -1              # no such class: no loss, the softmax as gradient
    xs, ys = tu.device_batch(wl, x, y, bf16)
    prec = sb.SB_BF16 if bf16 else sb.SB_FP32
    a, ref = tu.gpu_model(wl, params, prec), tu.gpu_model(wl, params, prec)
    a.forward(xs, ys)
    for i in range(4):
        ref.forward_layers(i, i, xs, ys)
    assert a.loss() == ref.loss()
    for what, li in ((sb.SB_T_ACT, 2), (sb.SB_T_DACT, 2), (sb.SB_T_ROW_LOSS, 3)):
        assert np.array_equal(a.read(what, li), ref.read(what, li)), what
    assert a.read(sb.SB_T_ROW_LOSS, 3)[0] == 0.0
    a.backward()
    dz, w, act = (torch.from_numpy(a.read(what, li, squeeze=False)).double()
                  for what, li in ((sb.SB_T_DACT, 2), (sb.SB_T_SHADOW_W if bf16 else sb.SB_T_WEIGHT, 2), (sb.SB_T_ACT, 1)))
    want = (dz.reshape(-1, classes) @ w.reshape(classes, width)) * (act.reshape(-1, width) > 0)
    # sums of at most 16 products in float; bf16 results round to 2^-9 of the value
    assert tu.maxrel(a.read(sb.SB_T_DACT, 1).reshape(-1, width), want) <= (2.0 ** -8 if bf16 else 1e-5)
    # whole iterations leave the mean to a kernel beside the chain: run directly, captured and replayed, on other labels every time
    s = torch.cuda.Stream()
    for k in range(1, 4):
        for t, part in zip(ys, si.split_replicas((y + k) % classes, R)):
            t.copy_(torch.from_numpy(np.ascontiguousarray(part)))
        for i in range(4):
            ref.forward_layers(i, i, xs, ys)
        torch.cuda.synchronize()
        before = a.loss()
        with torch.cuda.stream(s):
            a.graph_step(xs, ys, 0.0, 0.0)
            assert a.loss() == ref.loss() != before
    assert a.debug_check_guards()[0] == 0
    a.close()
    ref.close()


@pytest.mark.parametrize("bf16", [True, False])
def test_mean_loss_of_sub_iterations(bf16):
    """The mean over all rows, left to a kernel beside the last sub-iteration's chain: directly, captured and replayed, on other labels every time."""
    import torch

    from paper_2112_15317_b200 import binding as sb
    wl = si.Workload("head_modulo", [(si.CONV3X3_RELU, 8), (si.FC_RELU, 64), (si.FC, 10), (si.SOFTMAX_XENT, 10)], 4, 4, 4, 36, 2, 3)
    x, y = si.make_batch(wl)
    xs, ys = tu.device_batch(wl, x, y, bf16)
    m = tu.gpu_model(wl, si.make_params(wl, bias_std=0.2), sb.SB_BF16 if bf16 else sb.SB_FP32, sb.SB_FLAG_MODULO_SCHEDULE)
    seen = set()
    with torch.cuda.stream(torch.cuda.Stream()):
        for k in range(4):
            for t, part in zip(ys, si.split_replicas((y + k) % 10, wl.R)):
                t.copy_(torch.from_numpy(np.ascontiguousarray(part)))
            torch.cuda.synchronize()
            m.modulo_step(xs, ys, 0.0, 0.0)
            loss, rows = m.loss(), m.read(sb.SB_T_ROW_LOSS, 3).astype(np.float64)
            assert abs(loss - rows.mean()) <= 1e-6 * abs(rows).mean()      # 72 positive terms in float
            seen.add(loss)
    assert len(seen) == 4
    assert m.debug_check_guards()[0] == 0
    m.close()
