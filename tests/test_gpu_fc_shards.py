"""FC layers whose shard boundaries fall anywhere inside a tensor-core tile: bit-identical to the unsharded layer."""
from __future__ import annotations

import numpy as np
import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,width,b", [(3, 200, 9), (5, 136, 130), (7, 264, 1)])
def test_shard_boundaries_inside_a_tile(K, width, b):
    from paper_2112_15317_b200 import binding as sb
    layers = [(si.CONV3X3_RELU, 64), (si.MAXPOOL2, 0), (si.FC_RELU, width), (si.FC_RELU, 64), (si.FC, 10), (si.SOFTMAX_XENT, 10)]
    got = []
    for k in (1, K):
        wl = si.Workload("fc_shards", layers, 8, 8, 3, b, 1, k)
        m = tu.gpu_model(wl, si.make_params(wl, bias_std=0.2), sb.SB_BF16)
        xs, ys = tu.device_batch(wl, *si.make_batch(wl), True)
        m.forward(xs, ys)
        m.backward()
        g = m.gather_params(sb.SB_T_GRAD_W, sb.SB_T_GRAD_B)
        got.append([m.read(sb.SB_T_ACT, 2), m.read(sb.SB_T_DACT, 1)] + [p[n] for p in g if p is not None for n in ("w", "b")])
        m.close()
    for a, b_ in zip(*got):
        assert np.any(a != 0) and np.array_equal(a, b_)
