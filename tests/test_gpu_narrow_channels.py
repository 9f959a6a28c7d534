"""bf16 layers whose channel counts do not fill the 64-wide boxes of the tensor-core kernels, against the CUDA-core kernels:
every stored tensor and gradient of one iteration."""
from __future__ import annotations

import numpy as np
import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,chans,b,R", [
    (8, 8, (16, 16), 1, 1),
    (10, 6, (32, 48, 16), 5, 2),         # ragged image boxes, one-slab outputs of 16 and 48 columns
    (16, 16, (64, 80, 144), 3, 1),       # a second, partly filled reduction chunk and column tile
    (32, 32, (48, 96), 9, 3),            # many tiles
    (4, 4, (16, 272), 17, 1),            # more than one 256-wide tile
    (10, 8, (16, 128, 256), 3, 1),       # with pairs forced: two taps per CTA pair of the weight gradient
    (56, 56, (64, 256, 64), 13, 1),      # more than two tiles per SM: CTA pairs on halos by themselves, 256 columns of one reduction chunk
    (24, 40, (48, 144, 32), 41, 1),      # ... with partly filled tiles and chunks, in both directions
    (136, 120, (32, 48), 33, 1),         # long enough for the nine-tap weight gradient by itself: every CTA's share of chunks, images ragged
])
@pytest.mark.parametrize("flags", [0, 8, 32, 64])     # default / CTA pairs / no halo kernel / persistent kernels, several tiles per CTA
def test_channel_counts_off_the_tiles(H, W, chans, b, R, flags):
    from paper_2112_15317_b200 import binding as sb
    layers = [(si.CONV3X3_RELU, c) for c in chans] + [(si.MAXPOOL2, 0), (si.FC_RELU, 40), (si.FC, 10), (si.SOFTMAX_XENT, 10)]
    wl = si.Workload("narrow", layers, H, W, 3 if H * W % 8 == 0 else 4, b, R, 2)
    params = si.make_params(wl, bias_std=0.2)
    xs, ys = tu.device_batch(wl, *si.make_batch(wl), True)
    umma, simt = (tu.gpu_model(wl, params, sb.SB_BF16, f) for f in (flags, sb.SB_FLAG_FORCE_SIMT))
    checks = tu.Checks()
    for m in (umma, simt):
        m.forward(xs, ys)
    n = len(chans)
    for li in range(n + 1):
        for r in range(R):
            a, ref = umma.read(sb.SB_T_ACT, li, r), simt.read(sb.SB_T_ACT, li, r)
            checks.le(f"act {li}", tu.maxrel(a, ref), 1e-2)
            if li == n:      # the pooled maxima of the kernel that pooled them, exactly
                c = umma.read(sb.SB_T_ACT, n - 1, r, squeeze=False)
                w4 = np.stack([c[:, i::2, j::2] for i in (0, 1) for j in (0, 1)])
                assert np.array_equal(a.reshape(w4.shape[1:]), w4.max(0)) and np.array_equal(umma.read(sb.SB_T_POOL_IDX, li, r, squeeze=False), w4.argmax(0))
            simt.write(sb.SB_T_ACT, li, r, a)        # (both take their ReLU and pooling decisions on the same stored values)
            if li == n:
                simt.write(sb.SB_T_POOL_IDX, li, r, umma.read(sb.SB_T_POOL_IDX, li, r))
    for li in (n + 1, n + 2):
        simt.write(sb.SB_T_ACT, li, 0, umma.read(sb.SB_T_ACT, li))
        simt.write(sb.SB_T_DACT, li, 0, umma.read(sb.SB_T_DACT, li))
    for m in (umma, simt):
        m.backward()
    for li in range(n + 1):
        for r in range(R):
            checks.le(f"dact {li}", tu.maxrel(umma.read(sb.SB_T_DACT, li, r), simt.read(sb.SB_T_DACT, li, r)), 2e-2)
    for li in range(n):
        for what in (sb.SB_T_GRAD_W, sb.SB_T_GRAD_B):
            checks.le(f"grad {li}", tu.maxrel(umma.read(what, li), simt.read(what, li)), 1e-2)
    n_bad, at = umma.debug_check_guards()
    assert n_bad == 0, at
    umma.close()
    simt.close()
    checks.finish()
