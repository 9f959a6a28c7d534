"""Float contractions on the tensor cores (every float as three bf16 terms) at the edges of their tiles, chunks and splits: one conv and
one FC layer's three passes against double-precision torch on the layer's own stored inputs, and non-finite operands against the
CUDA-core kernels."""
from __future__ import annotations

import numpy as np
import pytest

import sb_inputs as si
import sb_testutil as tu

pytestmark = pytest.mark.gpu

# Bound on the 2-norm: products left out 2^-26, truncation of the leading products over 64 steps 4 x 2^-25, the rounded running sum
# 2^-25 sqrt(chunks) of up to 60 chunks: below 4e-7 in all; the largest measured over a sweep of 25 layers is 2.1e-7.  The other products
# of 64 chunks take part with up to 1280 truncated additions to a sum of 2^-8 of the result: 1.5e-7 where all of them have one sign.
BOUND = 5e-7


def _net(H, W, c0, c1, width, b, R):
    wl = si.Workload("contract_umma", [(si.CONV3X3_RELU, c0), (si.CONV3X3_RELU, c1), (si.FC_RELU, width), (si.FC, 10), (si.SOFTMAX_XENT, 10)], H, W, 4, b, R, 1)
    return wl, si.make_params(wl, bias_std=0.2), si.make_batch(wl)


@pytest.mark.parametrize("H,W,c0,c1,width,b,R,on", [
    (9, 7, 24, 72, 40, 17, 2, 5),        # chunks that cross taps, ragged rows, columns and chunks
    (6, 6, 8, 136, 72, 29, 2, 5),        # one run of eight channels a tap; more columns than a 128-wide tile
    (8, 8, 64, 128, 128, 24, 2, 6),      # whole tiles, split reductions
    (16, 12, 64, 64, 64, 16, 2, 4),      # one column tile, long weight-gradient reduction
    (4, 4, 264, 248, 520, 3, 1, 5),      # less than a row tile, long forward and data-gradient reductions
])
def test_passes_against_double(H, W, c0, c1, width, b, R, on):
    import torch
    import torch.nn.functional as F

    from paper_2112_15317_b200 import binding as sb
    wl, params, batch = _net(H, W, c0, c1, width, b, R)
    m = tu.gpu_model(wl, params, sb.SB_FP32, sb.SB_FLAG_PROFILE_LAYERS)
    xs, ys = tu.device_batch(wl, *batch, False)
    m.profile_begin()
    m.forward(xs, ys)
    m.backward()
    names = [e["name"] for e in m.profile_end()]
    ran = {n for n in names if "f32_umma" in n}
    assert len(ran) >= on, names
    t = lambda what, li: torch.from_numpy(np.concatenate([m.read(what, li, r, squeeze=False) for r in range(R if li < 2 else 1)])).double()  # noqa: E731
    wt = lambda what, li: torch.from_numpy(m.read(what, li, 0, squeeze=False)).double()  # noqa: E731
    checks = tu.Checks()

    x = t(sb.SB_T_ACT, 0).permute(0, 3, 1, 2).requires_grad_()
    w = wt(sb.SB_T_WEIGHT, 1).permute(0, 3, 1, 2).requires_grad_()
    bias = wt(sb.SB_T_BIAS, 1).reshape(-1).requires_grad_()
    y = F.conv2d(x, w, bias, padding=1)
    y.backward(t(sb.SB_T_DACT, 1).permute(0, 3, 1, 2))
    checks.le("conv forward", tu.frob(t(sb.SB_T_ACT, 1), y.relu().permute(0, 2, 3, 1).detach()), BOUND)
    checks.le("conv input gradient", tu.frob(t(sb.SB_T_DACT, 0), (x.grad * (x > 0)).permute(0, 2, 3, 1).detach()), BOUND)
    checks.le("conv weight gradient", tu.frob(wt(sb.SB_T_GRAD_W, 1), w.grad.permute(0, 2, 3, 1)), BOUND)
    checks.le("conv bias gradient", tu.frob(wt(sb.SB_T_GRAD_B, 1).reshape(-1), bias.grad), BOUND)

    x = t(sb.SB_T_ACT, 1).reshape(wl.B, -1).requires_grad_()
    w = wt(sb.SB_T_WEIGHT, 2)[:, :, 0, 0].requires_grad_()
    bias = wt(sb.SB_T_BIAS, 2).reshape(-1).requires_grad_()
    y = F.linear(x, w, bias)
    y.backward(t(sb.SB_T_DACT, 2)[:, :, 0, 0])
    checks.le("fc forward", tu.frob(t(sb.SB_T_ACT, 2)[:, :, 0, 0], y.relu().detach()), BOUND)
    checks.le("fc input gradient", tu.frob(t(sb.SB_T_DACT, 1).reshape(wl.B, -1), (x.grad * (x > 0)).detach()), BOUND)
    checks.le("fc weight gradient", tu.frob(wt(sb.SB_T_GRAD_W, 2)[:, :, 0, 0], w.grad), BOUND)
    checks.le("fc bias gradient", tu.frob(wt(sb.SB_T_GRAD_B, 2).reshape(-1), bias.grad), BOUND)

    # weights changed between the calls: each call reads them as they are
    x = t(sb.SB_T_ACT, 0).permute(0, 3, 1, 2).requires_grad_()
    new = -0.5 * m.read(sb.SB_T_WEIGHT, 1, 0, squeeze=False) + 0.01
    m.write(sb.SB_T_WEIGHT, 1, 0, new)
    m.forward_layers(1, 1)
    m.write(sb.SB_T_WEIGHT, 1, 0, 2.0 * new)
    m.backward_layers(1, 1)
    y = F.conv2d(x, torch.from_numpy(new).double().permute(0, 3, 1, 2), bias=wt(sb.SB_T_BIAS, 1).reshape(-1), padding=1)
    (2.0 * y).backward(t(sb.SB_T_DACT, 1).permute(0, 3, 1, 2))
    checks.le("conv forward, new weights", tu.frob(t(sb.SB_T_ACT, 1), y.relu().permute(0, 2, 3, 1).detach()), BOUND)
    checks.le("conv input gradient, new weights", tu.frob(t(sb.SB_T_DACT, 0), (x.grad * (x > 0)).permute(0, 2, 3, 1).detach()), BOUND)
    assert m.debug_check_guards()[0] == 0
    m.loss()       # raises if a bounded wait ran out
    m.close()
    checks.finish()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 3.4e38])
def test_non_finite_operands_as_on_cuda_cores(bad):
    """Infinities and values that round to one in bf16 give the infinities, NaNs and numbers of plain multiply-adds."""
    from paper_2112_15317_b200 import binding as sb
    wl, params, batch = _net(8, 8, 64, 128, 128, 24, 2)
    xs, ys = tu.device_batch(wl, *batch, False)
    a, ref = tu.gpu_model(wl, params, sb.SB_FP32), tu.gpu_model(wl, params, sb.SB_FP32, sb.SB_FLAG_FORCE_SIMT)
    dy = 0.01 * np.cos(np.arange(24 * 8 * 8 * 128, dtype=np.float32)).reshape(24, 8, 8, 128)
    got = []
    for m in (a, ref):
        m.forward(xs, ys)
        act = m.read(sb.SB_T_ACT, 0, 0, squeeze=False)
        act[1, 3, 4, 5] = bad
        m.write(sb.SB_T_ACT, 0, 0, act)
        m.forward_layers(1, 1)
        y = [m.read(sb.SB_T_ACT, 1, r) for r in range(2)]
        for r in range(2):
            m.write(sb.SB_T_DACT, 1, r, dy)
        m.backward_layers(1, 1)
        got.append(y + [m.read(sb.SB_T_GRAD_W, 1), m.read(sb.SB_T_DACT, 0, 0)])
    for u, v in zip(*got):
        assert np.array_equal(np.isnan(u), np.isnan(v)) and np.array_equal(np.isinf(u), np.isinf(v))
        fin = np.isfinite(v)
        assert np.array_equal(np.sign(u[~fin & ~np.isnan(v)]), np.sign(v[~fin & ~np.isnan(v)]))
        assert tu.maxrel(u[fin], v[fin]) < 1e-5
    a.close()
    ref.close()


@pytest.mark.parametrize("where", ["all weights NaN", "one gradient pixel inf", "one gradient value inf", "one weight -inf", "inputs of one image NaN"])
def test_non_finite_operands_over_long_reductions(where):
    """Whole operands and single values, 16384 pixels: the results of plain multiply-adds, and no wait that runs out meanwhile."""
    from paper_2112_15317_b200 import binding as sb
    wl, params, batch = _net(32, 32, 64, 64, 64, 16, 1)
    xs, ys = tu.device_batch(wl, *batch, False)
    a, ref = tu.gpu_model(wl, params, sb.SB_FP32), tu.gpu_model(wl, params, sb.SB_FP32, sb.SB_FLAG_FORCE_SIMT)
    dy = 0.01 * np.cos(np.arange(16 * 32 * 32 * 64, dtype=np.float32)).reshape(16, 32, 32, 64)
    if where == "one gradient pixel inf":
        dy[9, 30, 17, :] = np.inf
    elif where == "one gradient value inf":
        dy[15, 31, 31, 63] = np.inf
    got = []
    for m in (a, ref):
        m.forward(xs, ys)
        w = m.read(sb.SB_T_WEIGHT, 1, 0, squeeze=False)
        act = m.read(sb.SB_T_ACT, 0, 0, squeeze=False)
        if where == "all weights NaN":
            w[:] = np.nan
        elif where == "one weight -inf":
            w[33, 2, 1, 40] = -np.inf
        elif where == "inputs of one image NaN":
            act[3] = np.nan
        m.write(sb.SB_T_WEIGHT, 1, 0, w)
        m.write(sb.SB_T_ACT, 0, 0, act)
        m.forward_layers(1, 1)
        y = m.read(sb.SB_T_ACT, 1, 0)
        m.write(sb.SB_T_DACT, 1, 0, dy)
        m.backward_layers(1, 1)
        m.loss()       # raises if a bounded wait ran out
        got.append([y, m.read(sb.SB_T_GRAD_W, 1), m.read(sb.SB_T_DACT, 0, 0)])
    for u, v in zip(*got):
        assert np.array_equal(np.isnan(u), np.isnan(v)) and np.array_equal(np.isinf(u), np.isinf(v))
        fin = np.isfinite(v)
        assert np.array_equal(np.sign(u[np.isinf(v)]), np.sign(v[np.isinf(v)]))
        assert not fin.any() or tu.maxrel(u[fin], v[fin]) < 1e-5
    a.close()
    ref.close()


@pytest.mark.parametrize("exps", [(-126, 40, 40), (40, -126, 40), (40, 40, -126), (-60, -58, 50), (60, 58, -50), (60, -58, 58), (-145, 60, 60)])
@pytest.mark.parametrize("c0", [64, 24])
def test_operands_of_all_magnitudes(c0, exps):
    """Inputs, weights and output gradients down to the smallest normal (and to subnormal) floats, results up to 2^124."""
    import torch
    import torch.nn.functional as F

    from paper_2112_15317_b200 import binding as sb
    wl, params, batch = _net(8, 8, c0, 128, 128, 24, 1)
    m = tu.gpu_model(wl, params, sb.SB_FP32, sb.SB_FLAG_PROFILE_LAYERS)
    m.forward(*tu.device_batch(wl, *batch, False))
    rng = np.random.default_rng(5)
    x, w, dy = (np.ldexp(rng.uniform(0.5, 1.0, s) * rng.choice([-1.0, 1.0], s), e).astype(np.float32)
                for s, e in zip(((24, 8, 8, c0), (128, 3, 3, c0), (24, 8, 8, 128)), exps))
    x = np.abs(x)
    for what, li, a in ((sb.SB_T_ACT, 0, x), (sb.SB_T_WEIGHT, 1, w), (sb.SB_T_DACT, 1, dy), (sb.SB_T_BIAS, 1, np.zeros(128, np.float32))):
        m.write(what, li, 0, a)
    m.profile_begin()
    m.forward_layers(1, 1)
    y = m.read(sb.SB_T_ACT, 1, 0, squeeze=False)
    m.backward_layers(1, 1)
    assert sum("f32_umma" in e["name"] for e in m.profile_end()) >= 2
    t = lambda a: torch.from_numpy(a).double().permute(0, 3, 1, 2).requires_grad_()  # noqa: E731
    xt, wt = t(x), t(w)
    want = F.conv2d(xt, wt, padding=1)
    want.backward(t(dy).detach())
    checks = tu.Checks()
    for name, got, ref in (("forward", y, want.detach().relu()), ("input gradient", m.read(sb.SB_T_DACT, 0, 0, squeeze=False), xt.grad),
                           ("weight gradient", m.read(sb.SB_T_GRAD_W, 1, 0, squeeze=False), wt.grad)):
        ref = ref.permute(0, 2, 3, 1).numpy()
        assert np.isfinite(got).all()
        checks.le(name, np.linalg.norm(got.astype(np.float64) / np.abs(ref).max() - ref / np.abs(ref).max()) / np.linalg.norm(ref / np.abs(ref).max()), BOUND)
    checks.finish()
    m.close()


def test_weights_split_for_the_layers_of_a_call():
    """Every call takes apart the weights that it reads as terms, and no others."""
    from paper_2112_15317_b200 import binding as sb
    convs = [64, 64, 128, 256]
    wl = si.Workload("split_weights", [(si.CONV3X3_RELU, c) for c in convs] + [(si.FC, 10), (si.SOFTMAX_XENT, 10)], 16, 16, 4, 32, 1, 1)
    m = tu.gpu_model(wl, si.make_params(wl), sb.SB_FP32)
    xs, ys = tu.device_batch(wl, *si.make_batch(wl), False)
    m.forward(xs, ys)
    n = [0, 64 * 9 * 64, 128 * 9 * 64, 256 * 9 * 128]      # (layer 0 reads images)
    bias = [64, 64, 128]                                   # (between them in memory)
    for first, last, want in [(0, 0, 0), (1, 1, n[1]), (2, 2, n[2]), (3, 3, n[3]), (2, 3, n[2] + bias[2] + n[3]), (0, 3, sum(n) + bias[1] + bias[2]), (4, 5, 0)]:
        for run in (lambda: m.forward_layers(first, last), lambda: m.backward_layers(last, first)):
            m.profile_begin()
            run()
            assert sum(e["bytes"] for e in m.profile_end() if e["name"] == "split_weights") == 10.0 * want, (first, last)
    m.close()


def test_long_reduction_of_one_sign():
    """784 chunks in one split (512 -> 1024 channels at 28x28, batch 64), all terms of all operands positive: what the accumulators cut off
    adds up.  The leading products are exact here (ones)."""
    import torch

    from paper_2112_15317_b200 import binding as sb
    m = sb.Model([(si.CONV3X3_RELU, 512), (si.CONV3X3_RELU, 1024), (si.FC, 10), (si.SOFTMAX_XENT, 10)], 28, 28, 4, 64, 1, 1, sb.SB_FP32, sb.SB_FLAG_PROFILE_LAYERS)

    def view(what, layer, shape):
        off = m.tensor_info(what, layer)[0] - m.arena.data_ptr()
        return m.arena[off:off + 4 * int(np.prod(shape))].view(torch.float32).view(shape)
    act, dy = view(sb.SB_T_ACT, 0, (64, 784, 512)), view(sb.SB_T_DACT, 1, (64, 784, 1024))
    g = torch.Generator(device="cuda").manual_seed(1)
    m.forward_layers(0, 0, [torch.zeros(64, 28, 28, 4, device="cuda")], [torch.zeros(64, dtype=torch.int32, device="cuda")])
    for t in (act, dy):
        t.copy_(1.0 + 2.0 ** -8 * (0.25 + 0.7 * torch.rand(t.shape, generator=g, device="cuda")))      # (rounds to 1 in bf16)
    m.profile_begin()
    m.backward_layers(1, 1)
    assert any(e["name"].startswith("conv_wgrad_f32_umma") for e in m.profile_end())
    want = dy.reshape(-1, 1024)[:, :64].double().T @ act.reshape(-1, 512).double()      # (the middle tap, 64 of the output channels)
    got = view(sb.SB_T_GRAD_W, 1, (1024, 9, 512))[:64, 4].double()
    assert ((got - want).norm() / want.norm()).item() < 2e-7
    m.close()


def _same(u, v):
    assert np.array_equal(np.isnan(u), np.isnan(v)) and np.array_equal(np.isinf(u), np.isinf(v))
    assert np.array_equal(np.sign(u[np.isinf(v)]), np.sign(v[np.isinf(v)]))
    fin = np.isfinite(v)
    assert not fin.any() or tu.maxrel(u[fin], v[fin]) < 1e-5


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 3.4e38, 1e30])      # (1e30: products overflow, no operand is infinite)
@pytest.mark.parametrize("layer", [1, 2])
@pytest.mark.parametrize("H,W,c0,c1,width,b", [
    (9, 7, 24, 72, 64, 40),       # chunks that cross taps, ragged rows and columns
    (16, 16, 64, 64, 136, 96),    # conv: 192 row tiles, more than one unit a CTA
])
def test_non_finite_operands_of_all_forms(H, W, c0, c1, width, b, layer, bad):
    """Convolution and FC layers, with and without whole taps a chunk: one bad input, weight and output gradient at a time."""
    from paper_2112_15317_b200 import binding as sb
    wl, params, batch = _net(H, W, c0, c1, width, b, 1)
    xs, ys = tu.device_batch(wl, *batch, False)
    got, ran = [], []
    for flags in (sb.SB_FLAG_PROFILE_LAYERS, sb.SB_FLAG_FORCE_SIMT):
        m = tu.gpu_model(wl, params, sb.SB_FP32, flags)
        m.forward(xs, ys)
        act, w = (m.read(what, li, 0, squeeze=False) for what, li in ((sb.SB_T_ACT, layer - 1), (sb.SB_T_WEIGHT, layer)))
        dy = np.random.default_rng(7).normal(0.0, 0.01, m.read(sb.SB_T_DACT, layer).size).astype(np.float32)
        out = []
        for turn in range(3):
            t = [act.copy(), w.copy(), dy.copy()]
            t[turn].reshape(-1)[int(0.37 * t[turn].size)] = bad
            if turn == 0:
                t[0].reshape(-1)[-1] = bad
            m.write(sb.SB_T_ACT, layer - 1, 0, t[0])
            m.write(sb.SB_T_WEIGHT, layer, 0, t[1])
            m.write(sb.SB_T_DACT, layer, 0, t[2])
            m.profile_begin()
            m.forward_layers(layer, layer)
            out.append(m.read(sb.SB_T_ACT, layer))
            m.backward_layers(layer, layer)
            ran += [e["name"] for e in m.profile_end() if "f32_umma" in e["name"]]
            m.loss()       # raises if a bounded wait ran out
            out += [m.read(sb.SB_T_GRAD_W, layer), m.read(sb.SB_T_GRAD_B, layer), m.read(sb.SB_T_DACT, layer - 1)]
        assert m.debug_check_guards()[0] == 0
        got.append(out)
        m.close()
    assert len(ran) >= 6, ran
    for u, v in zip(*got):
        _same(u, v)


@pytest.mark.parametrize("where,times", [("gradients of the last image NaN", 15), ("one image infinite", 15), ("all weights NaN", 15), ("all results above 2^96", 300)])
def test_non_finite_operands_do_not_stall(where, times):
    """512 -> 1024 channels at 28x28, batch 64: several units a CTA and 50176 pixels in one reduction.  The results of plain multiply-adds,
    no wait that runs out, and passes that take a few times as long as on ordinary data (where every sum is made again, some tens of times)."""
    import torch

    from paper_2112_15317_b200 import binding as sb
    wl = si.Workload("stall", [(si.CONV3X3_RELU, 512), (si.CONV3X3_RELU, 1024), (si.FC, 10), (si.SOFTMAX_XENT, 10)], 28, 28, 4, 64, 1, 1)
    x, y = torch.randn(64, 28, 28, 4, device="cuda"), torch.zeros(64, dtype=torch.int32, device="cuda")
    got, ms = [], []
    for flags in (0, sb.SB_FLAG_FORCE_SIMT):
        m = sb.Model.from_workload(wl, precision=sb.SB_FP32, flags=flags)

        def view(what, layer, shape):
            off = m.tensor_info(what, layer)[0] - m.arena.data_ptr()
            return m.arena[off:off + 4 * int(np.prod(shape))].view(torch.float32).view(shape)
        g = torch.Generator(device="cuda").manual_seed(1)
        act, w, dy = view(sb.SB_T_ACT, 0, (64, 28, 28, 512)), view(sb.SB_T_WEIGHT, 1, (1024, 9, 512)), view(sb.SB_T_DACT, 1, (64, 28, 28, 1024))
        for t, std in ((act, 1.0), (w, 0.02), (dy, 0.01)):
            t.copy_(torch.randn(t.shape, generator=g, device="cuda") * std)
        act.relu_()
        view(sb.SB_T_BIAS, 1, (1024,)).zero_()
        m.forward_layers(0, 0, [x], [y])      # (binds the inputs; its output is replaced)
        act.copy_(torch.randn(act.shape, generator=g, device="cuda").relu())

        def passes():
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            m.forward_layers(1, 1)
            m.backward_layers(1, 1)
            e[1].record()
            torch.cuda.synchronize()
            ms.append(e[0].elapsed_time(e[1]))
        passes()
        passes()
        if where == "all weights NaN":
            w.fill_(float("nan"))
        elif where == "one image infinite":
            act[37] = float("inf")
        elif where == "all results above 2^96":
            for t, e in ((act, 60), (w, 55), (dy, 58)):
                t.mul_(2.0 ** e)
        else:
            dy[63] = float("nan")
        passes()
        m.loss()       # raises if a bounded wait ran out
        got.append([t.cpu().numpy() for t in (view(sb.SB_T_ACT, 1, (64, 28, 28, 1024)), view(sb.SB_T_GRAD_W, 1, (1024, 9, 512)), view(sb.SB_T_DACT, 0, (64, 28, 28, 512)))])
        m.close()
    for u, v in zip(*got):
        _same(u, v)
    assert ms[2] < times * ms[1], ms
