"""Host-only: every tile plan of a 3x3 layer fits the kernel it names (N tile, ring slots, shared memory of a CTA).  The sizing call
plans each layer as model creation does and refuses a plan that could not be launched."""
from __future__ import annotations

import ctypes

import pytest

import sb_inputs as si

CHANNELS = (16, 32, 48, 64, 80, 128, 144, 160, 192, 256, 272, 320, 384, 512)
SIDES = (8, 10, 14, 16, 28, 32, 40, 56, 64, 112, 128, 160, 192, 224)


def _chain(channels):
    """Conv layers that follow one another through every ordered pair of channel counts."""
    walk = [channels[0]]
    for i, a in enumerate(channels):
        walk.append(a)
        for b in channels[i + 1:]:
            walk += [b, a]
        walk += channels[i + 1:i + 2]
    pairs = set(zip(walk, walk[1:]))
    assert pairs == {(a, b) for a in channels for b in channels}
    return [(si.CONV3X3_RELU, c) for c in walk] + [(si.FC, 4), (si.SOFTMAX_XENT, 4)]


@pytest.mark.parametrize("flags", [0, 8, 32, 64])     # default / CTA pairs / no halo kernel / persistent kernels
@pytest.mark.parametrize("batch", [1, 3, 4, 8, 16, 32, 50, 64, 128, 250])
def test_plans_fit_their_kernels(batch, flags):
    from paper_2112_15317_b200 import binding as sb
    layers = sb._layers_array(_chain(CHANNELS))
    refused = []
    for H, W in [(s, s) for s in SIDES] + [(64, 2), (6, 30), (34, 18), (112, 20)]:
        n = ctypes.c_size_t()
        if sb.sb_model_bytes(layers, len(layers), ctypes.byref(sb.sb_config(H, W, 4, batch, 1, 1, sb.SB_BF16, flags)), ctypes.byref(n)) != 0:
            refused.append(f"{H}x{W}: {sb.sb_last_error()}")
    assert not refused, refused
