"""Input-layer tensor-core kernels against the CUDA-core ones on image shapes that exercise the staged window: rows of an odd number
of elements, many small images in a tile, rows longer than a tile, ragged last tiles, several replicas."""
from __future__ import annotations

import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,C,cout,b,R", [
    (8, 7, 3, 64, 3, 2),        # 21 elements a row: plain copies
    (16, 1, 1, 16, 11, 1),      # one pixel a row
    (2, 2, 4, 48, 70, 2),       # 32 images in a tile
    (4, 6, 3, 32, 9, 3),        # rows of 18 elements: 4-byte copies
    (32, 32, 3, 64, 2, 2),      # 16-byte copies
    (6, 200, 3, 64, 1, 2),      # rows longer than a tile
    (24, 135, 1, 64, 5, 1),     # odd rows across tiles
    (40, 96, 4, 64, 16, 1),     # several tiles and chunks per CTA
])
def test_input_layer_shapes(H, W, C, cout, b, R):
    from paper_2112_15317_b200 import binding as sb
    wl = si.Workload("conv_in", [(si.CONV3X3_RELU, cout), (si.FC_RELU, 16), (si.FC, 10), (si.SOFTMAX_XENT, 10)], H, W, C, b, R, 1)
    params = si.make_params(wl, bias_std=0.2)
    xs, ys = tu.device_batch(wl, *si.make_batch(wl), True)
    a, ref = tu.gpu_model(wl, params, sb.SB_BF16), tu.gpu_model(wl, params, sb.SB_BF16, sb.SB_FLAG_FORCE_SIMT)
    checks = tu.Checks()
    for m in (a, ref):
        m.forward(xs, ys)
    for r in range(R):
        checks.le("act", tu.maxrel(a.read(sb.SB_T_ACT, 0, r), ref.read(sb.SB_T_ACT, 0, r)), 1e-2)
    ref.backward()
    for r in range(R):      # the same output gradient on both sides
        a.write(sb.SB_T_DACT, 0, r, ref.read(sb.SB_T_DACT, 0, r))
    a.backward_layers(0, 0)
    for what in (sb.SB_T_GRAD_W, sb.SB_T_GRAD_B):
        checks.le("grad", tu.maxrel(a.read(what, 0), ref.read(what, 0)), 1e-4)
    assert a.debug_check_guards()[0] == 0
    a.loss()       # raises if a bounded wait ran out
    a.close()
    ref.close()
    checks.finish()
