"""Pooling in the epilogue kernel of split reductions, forward and backward, bit for bit against the stand-alone pooling kernels run on the
tensors it left: float and bf16, one window an image and several, a channel count that is no multiple of eight."""
from __future__ import annotations

import numpy as np
import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16,H,W,c0,c1,b,R,fwd,bwd", [      # pooling launches that are left, of two each
    (True, 4, 8, 512, 512, 8, 2, 0, 1),        # two windows an image, tensor-core splits
    (True, 8, 8, 256, 512, 2, 2, 1, 1),        # four windows
    (False, 8, 8, 16, 32, 4, 2, 1, 0),         # float: split contractions on tensor cores
    (False, 4, 12, 12, 20, 5, 1, 1, 0),        # and on CUDA cores, channel counts that are no multiple of eight
    (False, 4, 4, 100, 132, 2, 2, 1, 0),
])
def test_pool_in_split_reduce(bf16, H, W, c0, c1, b, R, fwd, bwd):
    from paper_2112_15317_b200 import binding as sb
    # conv, pool, conv, pool, FC: both pool layers have a contraction above and below them
    net = [(si.CONV3X3_RELU, c0), (si.MAXPOOL2, 0), (si.CONV3X3_RELU, c1), (si.MAXPOOL2, 0), (si.FC_RELU, 512), (si.FC, 10), (si.SOFTMAX_XENT, 10)]
    wl = si.Workload("split_pool", net, H, W, 4, b, R, 1)
    m = tu.gpu_model(wl, si.make_params(wl, bias_std=0.2), sb.SB_BF16 if bf16 else sb.SB_FP32)
    xs, ys = tu.device_batch(wl, *si.make_batch(wl), bf16)
    m.profile_begin()
    m.forward(xs, ys)
    m.backward()
    launches = {e["name"]: e["launches"] for e in m.profile_end()}
    assert launches.get("pool_fwd", 0) <= fwd and launches.get("pool_bwd", 0) <= bwd, launches
    read = lambda what, li: np.concatenate([m.read(what, li, r) for r in range(R)])  # noqa: E731
    for pool in (1, 3):
        whole = [read(sb.SB_T_ACT, pool), read(sb.SB_T_POOL_IDX, pool), read(sb.SB_T_DACT, pool - 1)]
        assert np.any(whole[0]) and np.any(whole[2])
        m.forward_layers(pool, pool)
        m.backward_layers(pool, pool)
        alone = [read(sb.SB_T_ACT, pool), read(sb.SB_T_POOL_IDX, pool), read(sb.SB_T_DACT, pool - 1)]
        for u, v in zip(whole, alone):
            assert np.array_equal(u, v)
    # a conv layer run by itself leaves the pool layer above it alone
    left = 7.0 * np.ones((b,) + m.tensor_info(sb.SB_T_ACT, 3, 0)[1][1:], np.float32)
    for r in range(R):
        m.write(sb.SB_T_ACT, 3, r, left)
        m.write(sb.SB_T_POOL_IDX, 3, r, (left + 2).astype(np.uint8))
    m.forward_layers(2, 2)
    assert np.all(read(sb.SB_T_ACT, 3) == 7.0) and np.all(read(sb.SB_T_POOL_IDX, 3) == 9)
    assert m.debug_check_guards()[0] == 0
    m.close()
