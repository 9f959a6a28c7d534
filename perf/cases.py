"""The work that is timed: training iterations, evaluation passes and the sharded-FC layer, each through the calls a
user's program makes.

A case is one network at one batch, partitioning, precision and way of calling:

    net    "tiny"      2 conv + 2 FC layers (16 and 32 channels, FC 64), 32x32 images
           "paper"     the 7-conv / 3-FC network of the paper's Table 1, 32x32 images
           "vgg16"     VGG-16: 32x32 images (FC input 512), or 224x224 and the like (FC input 25088)
           "fc"        one fully-connected layer 25088 -> 4096
    call   "graph"     Model.graph_step on device buffers that the program fills (here: once)
           "host"      Model.train_step_host on a loader's ring of pinned batches, the learning rate following a schedule
           "pipeline"  prefetch_host / train_step_host_async / train_step_host_wait: the next batch is copied meanwhile
           "calls"     forward, backward, sgd_step one by one (a program that looks at gradients in between)
           "modulo"    Model.modulo_step: the paper's own schedule of K sub-iterations
           "eval"      forward only: logits and losses of a validation batch
           "layer"     forward_layers + backward_layers of one layer: forward, input gradient, weight gradient
"""
from __future__ import annotations

import itertools
import math

import torch

from paper_2112_15317_b200 import binding as sb

LR = {"tiny": 1e-2, "paper": 1e-3, "vgg16": 1e-3}
MOMENTUM = 0.9
GRADIENT = {"tiny": 3.0, "paper": 20.0, "vgg16": 10.0}    # typical norm of one layer's weight gradient, 128 small images
RING = 4          # pinned batches a loader keeps in turn
SCHEDULE = 64     # steps of the learning-rate schedule before it repeats


def _case(name, net, call, precision, side, b, R, K, classes=10, dropout=False):
    return dict(name=name, net=net, call=call, precision=precision, side=side, b=b, R=R, K=K, classes=classes, dropout=dropout)


def listed():
    return [
        # the smallest thing a user runs: the tiny network on 8 images, in float, step by step while debugging a model
        _case("tiny_b8_calls_fp32", "tiny", "calls", "fp32", 32, 4, 2, 2),
        # the same network trained for real: a small model on a few hundred images per step, channel counts below 64
        _case("tiny_b250_host_bf16", "tiny", "host", "bf16", 32, 125, 2, 2),
        # the paper's own evaluation network and partitioning (four workers x 32 images), fed from the host
        _case("paper_b128_pipeline_bf16", "paper", "pipeline", "bf16", 32, 32, 4, 4),
        # the same in float mode, where results have to agree with a float reference
        _case("paper_b96_graph_fp32", "paper", "graph", "fp32", 32, 24, 4, 4),
        # the headline configuration
        _case("vgg16_b128_graph_bf16", "vgg16", "graph", "bf16", 32, 32, 4, 4),
        # eight replicas and shards, batches straight from a data loader
        _case("vgg16_b256_host_bf16", "vgg16", "host", "bf16", 32, 32, 8, 8),
        # the last, ragged batch of an epoch, with dropout as VGG-16 is trained, gradients inspected between the calls
        _case("vgg16_b111_dropout_calls_bf16", "vgg16", "calls", "bf16", 32, 37, 3, 5, dropout=True),
        # the paper's schedule of K sub-iterations
        _case("vgg16_b128_modulo_bf16", "vgg16", "modulo", "bf16", 32, 32, 4, 4),
        # large images, 1000 classes
        _case("vgg16_224_b64_graph_bf16", "vgg16", "graph", "bf16", 224, 16, 4, 4, classes=1000),
        # validation on large images, a ragged batch
        _case("vgg16_224_b50_eval_bf16", "vgg16", "eval", "bf16", 224, 25, 2, 4, classes=1000),
        # a single image classified: the smallest forward pass of the large network
        _case("vgg16_224_b1_eval_bf16", "vgg16", "eval", "bf16", 224, 1, 1, 4, classes=1000),
        # the sharded fully-connected layer by itself
        _case("fc_b128_layer_bf16", "fc", "layer", "bf16", 1, 32, 4, 8, classes=4096),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["tiny", "tiny_fp32", "paper", "paper_fp32", "vgg16", "vgg16", "modulo", "large", "eval", "fc"])
    R, K = rng.choice([1, 2, 3, 4, 8]), rng.choice([1, 2, 3, 4, 5, 8])
    per = lambda lo, hi: max(1, _log_int(rng, lo, hi) // R)  # noqa: E731  (images of one replica, for a batch of lo..hi)
    if kind == "tiny":
        return _drawn("tiny", rng.choice(["calls", "graph", "host", "pipeline"]), "bf16", 32, per(4, 512), R, K)
    if kind == "tiny_fp32":
        return _drawn("tiny", rng.choice(["calls", "graph", "host"]), "fp32", 32, per(4, 256), R, K)
    if kind == "paper":
        return _drawn("paper", rng.choice(["calls", "graph", "host", "pipeline"]), "bf16", 32, per(16, 512), R, K)
    if kind == "paper_fp32":
        return _drawn("paper", rng.choice(["calls", "graph", "eval"]), "fp32", 32, per(8, 128), R, K)
    if kind == "vgg16":
        return _drawn("vgg16", rng.choice(["calls", "graph", "host", "pipeline", "eval"]), "bf16", 32, per(16, 512), R, K,
                      dropout=rng.random() < 0.4)
    if kind == "modulo":
        return _drawn(rng.choice(["paper", "vgg16"]), "modulo", "bf16", 32, K * max(1, per(16, 256) // K), R, K)
    if kind == "large":
        return _drawn("vgg16", rng.choice(["graph", "host"]), "bf16", rng.choice([128, 160, 192, 224]), per(4, 63), R, K, classes=1000)
    if kind == "eval":
        return _drawn("vgg16", "eval", "bf16", rng.choice([160, 192, 224]), per(1, 64), R, K, classes=1000)
    return _drawn("fc", "layer", "bf16", 1, per(16, 512), R, K, classes=4096)


def _drawn(*a, **k):
    c = _case("", *a, **k)
    del c["name"]
    return c


# ---- networks ------------------------------------------------------------------------------------------------------


def _layers(case):
    net, classes = case["net"], case["classes"]
    conv = lambda w, n=1: [(sb.SB_CONV3X3_RELU, w)] * n  # noqa: E731
    pool = [(sb.SB_MAXPOOL2, 0)]
    drop = [(sb.SB_DROPOUT, 32768)] if case["dropout"] else []
    if net == "tiny":
        body, fc = conv(16) + pool + conv(32) + pool, [64]
    elif net == "paper":
        body, fc = conv(64, 2) + pool + conv(128, 2) + pool + conv(256, 3) + pool, [1024, 1024]
    elif net == "vgg16":
        body, fc = conv(64, 2) + pool + conv(128, 2) + pool + conv(256, 3) + pool + conv(512, 3) + pool + conv(512, 3) + pool, [4096, 4096]
    else:
        return [(sb.SB_FC, classes), (sb.SB_SOFTMAX_XENT, classes)]
    for width in fc:
        body = body + [(sb.SB_FC_RELU, width)] + drop
    return body + [(sb.SB_FC, classes), (sb.SB_SOFTMAX_XENT, classes)]


def _image(case):
    return (1, 1, 25088) if case["net"] == "fc" else (case["side"], case["side"], 3)


def _walk(case):
    """Per layer: kind, multiply-adds per image, parameters, output elements per image."""
    H, W, C = _image(case)
    feat = H * W * C
    rows = []
    for kind, out in _layers(case):
        macs = params = 0
        if kind == sb.SB_CONV3X3_RELU:
            macs, params = H * W * 9 * C * out, 9 * C * out + out
            C = out
            feat = H * W * C
        elif kind == sb.SB_MAXPOOL2:
            H, W = H // 2, W // 2
            feat = H * W * C
        elif kind in (sb.SB_FC_RELU, sb.SB_FC):
            macs, params = feat * out, feat * out + out
            feat = out
        rows.append((kind, macs, params, feat if kind != sb.SB_SOFTMAX_XENT else 0))
    return rows


def work(case):
    """Multiply-adds of the passes; bytes: images, labels, parameters and their state once in and once out, and the
    activations a backward pass needs once out and once in."""
    B, rows = case["b"] * case["R"], _walk(case)
    e = 2 if case["precision"] == "bf16" else 4
    H, W, C = _image(case)
    macs, params, acts = sum(r[1] for r in rows), sum(r[2] for r in rows), sum(r[3] for r in rows)
    x = B * H * W * C * e
    if case["call"] == "eval":
        return {"bytes": x + 4 * B + e * params + 4 * B * case["classes"], "flops": 2 * B * macs}
    if case["call"] == "layer":
        # x, dy, w in; y, dx, dw out
        return {"bytes": 2 * x + B * case["classes"] * (2 + 4) + (2 + 4) * params, "flops": 6 * B * macs}
    state = 16 * params                      # weight and momentum, read and written
    if case["call"] == "calls":
        state += 4 * params                  # the gradients the program can look at
    # (the first layer has no input gradient to compute)
    return {"bytes": x + 4 * B + state + 2 * B * acts * e, "flops": 2 * B * (3 * macs - rows[0][1])}


def tolerance(case):
    """bf16: sums in another order put stored activations on the other bf16 neighbour here and there, and that flips ReLU
    masks: two correct implementations' logits differ by 0.6e-2 (VGG-16, 224x224), a gradient by 10 to 30 % of its norm and
    the momentum it is added to by 1e-2 after one or two steps.  float: 1e-6 of the sums, and 2e-4
    where masks flip in the deeper network.  A single layer on given inputs has no such decisions."""
    if case["call"] == "layer":
        return {"rel": 1e-3, "max": 2e-2}
    if case["precision"] == "fp32":
        return {"rel": 2e-4, "max": 2e-2} if case["net"] == "tiny" else {"rel": 1e-3, "max": 1e-1}
    if case["call"] == "eval":
        return {"rel": 1.5e-2, "max": 1e-1}
    return {"rel": 2e-2, "max": 0.9}


# ---- a user's program ----------------------------------------------------------------------------------------------

_side_stream = None


def _stream():
    """One side stream for everything, as a program that wants its iterations replayed as graphs uses it."""
    global _side_stream
    if _side_stream is None:
        _side_stream = torch.cuda.Stream()
    torch.cuda.set_stream(_side_stream)


def _view(m, what, layer, part=0):
    """A tensor of the model as a torch view of its memory."""
    ptr, shape, dt = m.tensor_info(what, layer, part)
    dtype = {sb.SB_DT_F32: torch.float32, sb.SB_DT_BF16: torch.bfloat16, sb.SB_DT_U8: torch.uint8, sb.SB_DT_I32: torch.int32}[dt]
    off, n = ptr - m.arena.data_ptr(), math.prod(shape)
    shape = [s for i, s in enumerate(shape) if i == 0 or s > 1]
    return m.arena[off:off + n * dtype.itemsize].view(dtype).view(shape)


def _vector(m, what_w, what_b):
    """All weights (gradients, momenta) and biases as the one vector they are stored as."""
    parts = [i for i, (kind, _) in enumerate(m.layers) if kind in (sb.SB_CONV3X3_RELU, sb.SB_FC_RELU, sb.SB_FC)]
    lo = m.tensor_info(what_w, parts[0])[0]
    shards = 1 if m.layers[parts[-1]][0] == sb.SB_CONV3X3_RELU else m.K
    last, shape, _ = m.tensor_info(what_b, parts[-1], shards - 1)
    off = lo - m.arena.data_ptr()
    return m.arena[off:off + last + 4 * shape[0] - lo].view(torch.float32)


class _State:
    pass


def prepare(case, seed):
    _stream()
    s = _State()
    g = torch.Generator(device="cuda").manual_seed(seed)
    normal = lambda *shape, std=1.0: torch.randn(*shape, generator=g, device="cuda") * std  # noqa: E731
    H, W, C = _image(case)
    R, K, b, B, call = case["R"], case["K"], case["b"], case["b"] * case["R"], case["call"]
    bf16 = case["precision"] == "bf16"
    layers = _layers(case)
    flags = {"modulo": sb.SB_FLAG_MODULO_SCHEDULE, "layer": sb.SB_FLAG_INPUT_GRAD}.get(call, 0)
    m = s.model = sb.Model(layers, H, W, C, b, R, K, sb.SB_BF16 if bf16 else sb.SB_FP32, flags)
    # He-normal weights, small biases, and the momentum of a run under way in which successive gradients agree: 1 / (1 - 0.9)
    # times one step's gradient
    large = case["side"] > 32
    momentum_norm = 10.0 * GRADIENT.get(case["net"], 0.0) * math.sqrt(128.0 / B) * (4.0 if large else 1.0) * (2.5 if case["dropout"] else 1.0)
    for i, (kind, out) in enumerate(layers):
        if kind not in (sb.SB_CONV3X3_RELU, sb.SB_FC_RELU, sb.SB_FC):
            continue
        shards = 1 if kind == sb.SB_CONV3X3_RELU else K
        for j in range(shards):
            w, bias = _view(m, sb.SB_T_WEIGHT, i, j), _view(m, sb.SB_T_BIAS, i, j)
            w.copy_(normal(*w.shape, std=math.sqrt(2.0 * w.shape[0] / w.numel())))
            bias.copy_(normal(*bias.shape, std=0.02))
            for what, norm in ((sb.SB_T_MOM_W, momentum_norm), (sb.SB_T_MOM_B, 0.02 * momentum_norm)):
                v = _view(m, what, i, j)
                v.copy_(normal(*v.shape, std=norm / math.sqrt(v.numel() * shards)))
    m.refresh_shadow()
    n_batches = RING if call in ("host", "pipeline") else 1
    dtype = torch.bfloat16 if bf16 else torch.float32
    batches = [(normal(B, H, W, C).to(dtype), torch.randint(case["classes"], (B,), generator=g, device="cuda", dtype=torch.int32))
               for _ in range(n_batches)]
    lr = s.lr = LR.get(case["net"], 0.0) * (0.1 if large else 1.0)
    s.call = call
    s.params = _vector(m, sb.SB_T_WEIGHT, sb.SB_T_BIAS)
    s.momenta = _vector(m, sb.SB_T_MOM_W, sb.SB_T_MOM_B)
    # (bf16 gradients reach the outputs through the momentum: see tolerance)
    s.grads = _vector(m, sb.SB_T_GRAD_W, sb.SB_T_GRAD_B) if not bf16 or call == "layer" else None
    loss_layer = len(layers) - 1
    s.row_loss = _view(m, sb.SB_T_ROW_LOSS, loss_layer)
    s.logits = _view(m, sb.SB_T_ACT, loss_layer - 1)
    if case["dropout"]:
        m.dropout_seed(seed)
    if call in ("host", "pipeline"):
        s.ring = itertools.cycle([(x.cpu().pin_memory(), y.cpu().pin_memory()) for x, y in batches])
        s.lrs = itertools.cycle([lr * (0.55 + 0.45 * math.cos(math.pi * k / SCHEDULE)) for k in range(SCHEDULE)])
        if call == "pipeline":
            s.batch = next(s.ring)
            m.prefetch_host(*s.batch)
    else:
        x, y = batches[0]
        s.xs, s.ys = list(x.split(b)), list(y.split(b))
    if call == "layer":
        dy = _view(m, sb.SB_T_DACT, 0)
        dy.copy_(normal(*dy.shape))
        s.dx = [_view(m, sb.SB_T_INPUT_GRAD, 0, r) for r in range(R)]
    return s


def run(s):
    m, call = s.model, s.call
    if call == "graph":
        m.graph_step(s.xs, s.ys, s.lr, MOMENTUM)
    elif call == "modulo":
        m.modulo_step(s.xs, s.ys, s.lr, MOMENTUM)
    elif call == "host":
        loss = m.train_step_host(*next(s.ring), next(s.lrs), MOMENTUM)
        return {"loss": loss, "row_loss": s.row_loss, "params": s.params, "momenta": s.momenta}
    elif call == "pipeline":
        m.train_step_host_async(*s.batch, s.lr, MOMENTUM)
        s.batch = next(s.ring)
        m.prefetch_host(*s.batch)
        loss = m.train_step_host_wait()
        return {"loss": loss, "row_loss": s.row_loss, "params": s.params, "momenta": s.momenta}
    elif call == "calls":
        m.forward(s.xs, s.ys)
        m.backward()
        m.sgd_step(s.lr, MOMENTUM)
        return {"row_loss": s.row_loss, "params": s.params, "momenta": s.momenta, "grads": s.grads}
    elif call == "eval":
        m.forward(s.xs, s.ys)
        return {"row_loss": s.row_loss, "logits": s.logits}
    else:
        m.forward_layers(0, 0, s.xs, None)
        m.backward_layers(0, 0)
        return {"y": s.logits, "dx": s.dx, "grads": s.grads}
    return {"row_loss": s.row_loss, "params": s.params, "momenta": s.momenta}
