"""FC layers that take their update inside the weight-gradient kernel: replayed steps against the three separate calls, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,width,b,R,K", [
    (4800, 512, 1, 1, 1),        # one row of batch
    (4800, 520, 13, 5, 3),       # 65 rows: one row in the second batch chunk; ragged last row tile, shards inside it
    (1024, 2304, 128, 2, 4),     # many row tiles, four chunks of batch
    # gradients stored by one CTA per SM that walks its tiles:
    (4096, 4096, 1, 1, 2),       # one row of batch
    (9536, 1544, 70, 1, 1),      # ragged last row and column tiles, 70 rows
    (8192, 1792, 130, 2, 4),     # five chunks of batch: more than its ring
])
def test_folded_update_is_the_separate_one(d_in, width, b, R, K):
    import torch

    from paper_2112_15317_b200 import binding as sb
    wl = si.Workload("fc_update", [(si.FC_RELU, width), (si.FC, 10), (si.SOFTMAX_XENT, 10)], 1, 1, d_in, b, R, K)
    params = si.make_params(wl, bias_std=0.1)
    xs, ys = tu.device_batch(wl, *si.make_batch(wl), True)
    x = torch.cat(xs)
    xs = list(x.split(b))
    a, g = tu.gpu_model(wl, params, sb.SB_BF16), tu.gpu_model(wl, params, sb.SB_BF16)
    with torch.cuda.stream(torch.cuda.Stream()):
        for step in range(4):
            a.forward(xs, ys)
            a.backward()
            a.sgd_step(0.01, 0.9)
            g.graph_step(xs, ys, 0.01, 0.9)
            assert a.loss() == g.loss()
    for w, bias in ((sb.SB_T_WEIGHT, sb.SB_T_BIAS), (sb.SB_T_MOM_W, sb.SB_T_MOM_B)):
        for p, q in zip(a.gather_params(w, bias), g.gather_params(w, bias)):
            if p is not None:
                assert np.array_equal(p["w"], q["w"]) and np.array_equal(p["b"], q["b"])
    # the stored gradient against double precision
    grad = a.gather_params(sb.SB_T_GRAD_W, sb.SB_T_GRAD_B)[0]
    dy, xb = a.read(sb.SB_T_DACT, 0).astype(np.float64).reshape(wl.B, width), x.float().cpu().numpy().astype(np.float64).reshape(wl.B, d_in)
    assert tu.maxrel(grad["w"], dy.T @ xb) <= 1e-5 and tu.maxrel(grad["b"], dy.sum(0)) <= 1e-5
    assert a.debug_check_guards()[0] == 0 and g.debug_check_guards()[0] == 0
    a.close()
    g.close()
