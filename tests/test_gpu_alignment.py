"""Vectors that start anywhere relative to a 128-bit boundary: unpadded strides (a different offset for every worker), inputs
whose first element is not aligned, inputs that are not equally far past a boundary, and layers that end at or around the
edges of quads, sixteen-element units and chunks."""
import numpy as np
import pytest
import torch

from tests._harness import Runner

pytestmark = pytest.mark.gpu

SIZES = [5, 4097, 32640, 1, 32639, 16, 65537, 4111, 15, 32768]


def _view(flat, offset, W, stride):
    return flat[offset:offset + W * stride].view(W, stride)


@pytest.mark.parametrize("pad,g_off,s_off,value_dtype", [(0, 0, 0, 0), (1, 1, 1, 1), (2, 3, 3, 0), (3, 2, 2, 1), (1, 0, 2, 0), (0, 3, 1, 1)])
def test_any_offset_from_a_boundary(pad, g_off, s_off, value_dtype):
    rng = np.random.default_rng(17 + pad + 10 * g_off)
    W, N = 4, sum(SIZES)
    stride = N + pad
    junk = torch.full((64 << 20,), 0xff, dtype=torch.uint8, device="cuda")  # what the workspace holds before it is attached
    del junk
    r = Runner(SIZES, W, [0.001, 0.01, 0.1, 0.4, 1.0], 1000, value_dtype, stride=stride)
    grads = _view(torch.zeros(W * stride + 8, device="cuda"), g_off, W, stride)
    state = _view(torch.zeros(W * stride + 8, device="cuda"), s_off, W, stride)
    for frac in (0.01, 0.5, 0.3):
        x = rng.standard_normal((W, stride)) * np.exp(rng.uniform(-3, 3, stride))
        if frac == 0.3:
            x = np.where(rng.random((W, stride)) < 0.8, 0.0, x)  # thresholds among exact zeros
            state.zero_()
        grads.copy_(torch.from_numpy(x.astype(np.float32)))
        r.compare_step(grads, state, [frac * 8 * N * f for f in (1.0, 0.7, 1.3, 0.9)], 1.0)
