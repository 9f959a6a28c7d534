"""Replayed iterations when the inputs move and the learning rate changes from call to call: bit-identical to the three calls."""
from __future__ import annotations

import numpy as np
import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["graph", "host"])
def test_other_inputs_and_learning_rates_every_step(call):
    import torch

    from paper_2112_15317_b200 import binding as sb
    wl = si.config(0)
    params = si.make_params(wl, bias_std=0.1)
    a, b = tu.gpu_model(wl, params, sb.SB_BF16), tu.gpu_model(wl, params, sb.SB_BF16)
    batches = [si.make_batch(wl, seed=40 + k) for k in range(3)]
    dev = [tu.device_batch(wl, x, y, True) for x, y in batches]
    host = [(torch.from_numpy(x).to(torch.bfloat16).pin_memory(), torch.from_numpy(y).pin_memory()) for x, y in batches]
    rates = [0.01, 0.01, 0.01, 0.02, 0.005, 0.005, 0.005, 0.01]
    with torch.cuda.stream(torch.cuda.Stream()):
        for k, lr in enumerate(rates):
            xs, ys = dev[k % 3]
            a.forward(xs, ys)
            a.backward()
            a.sgd_step(lr, 0.9)
            if call == "graph":
                b.graph_step(xs, ys, lr, 0.9)
                loss = b.loss()
            else:
                loss = b.train_step_host(*host[k % 3], lr, 0.9)
            assert loss == a.loss(), (k, lr)
    for p, q in zip(a.gather_params(sb.SB_T_WEIGHT, sb.SB_T_BIAS), b.gather_params(sb.SB_T_WEIGHT, sb.SB_T_BIAS)):
        if p is not None:
            assert np.array_equal(p["w"], q["w"]) and np.array_equal(p["b"], q["b"])
    a.close()
    b.close()


def test_passes_replayed_on_repeated_buffers():
    """sb_forward / sb_backward on buffers that repeat (captured), then change, then come back: the same bits as a model that
    runs every pass kernel by kernel (on the legacy default stream)."""
    import torch

    from paper_2112_15317_b200 import binding as sb
    wl = si.config(0)
    params = si.make_params(wl, bias_std=0.1)
    a, b = tu.gpu_model(wl, params, sb.SB_BF16), tu.gpu_model(wl, params, sb.SB_BF16)
    dev = [tu.device_batch(wl, *si.make_batch(wl, seed=40 + k), True) for k in range(2)]
    side = torch.cuda.Stream()
    for k in [0] * 5 + [1, 0, 1] + [1] * 6 + [0] * 2:
        a.forward(*dev[k])
        a.backward()
        a.sgd_step(0.01, 0.9)
        with torch.cuda.stream(side):
            b.forward(*dev[k])
            b.backward()
            b.sgd_step(0.01, 0.9)
            assert b.loss() == a.loss() and a.launch_count() == b.launch_count(), k
    for what in ((sb.SB_T_WEIGHT, sb.SB_T_BIAS), (sb.SB_T_GRAD_W, sb.SB_T_GRAD_B)):
        for p, q in zip(a.gather_params(*what), b.gather_params(*what)):
            if p is not None:
                assert np.array_equal(p["w"], q["w"]) and np.array_equal(p["b"], q["b"])
    a.close()
    b.close()


@pytest.mark.parametrize("handle", [1, 2])     # cudaStreamLegacy (cannot be captured), cudaStreamPerThread
def test_repeated_passes_on_the_default_streams_by_handle(handle):
    import ctypes

    import torch

    from paper_2112_15317_b200 import binding as sb
    wl = si.config(0)
    params = si.make_params(wl, bias_std=0.1)
    a, b = tu.gpu_model(wl, params, sb.SB_BF16), tu.gpu_model(wl, params, sb.SB_BF16)
    xs, ys = tu.device_batch(wl, *si.make_batch(wl), True)
    ptrs = b._ptr_arrays(xs, ys)
    st = ctypes.c_void_p(handle)
    torch.cuda.synchronize()
    for _ in range(6):
        a.forward(xs, ys)
        a.backward()
        a.sgd_step(0.01, 0.9)
        for call in (lambda: sb.sb_forward(b.h, *ptrs, st), lambda: sb.sb_backward(b.h, st), lambda: sb.sb_sgd_step(b.h, 0.01, 0.9, st)):
            assert call() == 0, sb.sb_last_error()
        torch.cuda.synchronize()
        assert a.loss() == b.loss()
    for p, q in zip(a.gather_params(sb.SB_T_WEIGHT, sb.SB_T_BIAS), b.gather_params(sb.SB_T_WEIGHT, sb.SB_T_BIAS)):
        if p is not None:
            assert np.array_equal(p["w"], q["w"]) and np.array_equal(p["b"], q["b"])
    a.close()
    b.close()
