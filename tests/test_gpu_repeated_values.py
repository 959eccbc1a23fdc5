"""GPU parity where key intervals hold more entries than a layer's list: gradients whose values came from 16 or 8 bits repeat, and
every slice then keeps a list of its own (or, with most of its entries inside the interval, is counted from the inputs)."""
import numpy as np
import pytest
import torch

from tests._harness import Runner

pytestmark = pytest.mark.gpu


def _values(kind, x):
    if kind == "one":
        return torch.where(torch.rand_like(x) < 0.7, torch.sign(x) * 0.75, x)
    dtype = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp8": torch.float8_e4m3fn}[kind]
    return x.to(dtype).float()


@pytest.mark.parametrize("pad,schedule", [(0, 0), (1, 1)])
@pytest.mark.parametrize("kind", ["bf16", "fp16", "fp8", "one"])
def test_repeated_values(kind, pad, schedule):
    torch.manual_seed(5)
    sizes, grid, W = [4097, 600001, 32640, 15, 2049, 300 * 1024], [0.01, 0.05, 0.2, 0.4, 0.6, 0.8, 1.0], 3
    N = sum(sizes)
    stride = N + (-N % 4) + pad  # pad 1: the workers start at different distances from a boundary
    r = Runner(sizes, W, grid, 1000, 0, stride=stride, schedule=schedule)
    state = torch.zeros((W, stride), device="cuda")
    for budget in (0.05, 0.4, 0.15):
        grads = _values(kind, torch.randn((W, stride), device="cuda"))
        assert r.compare_step(grads, state, [budget * 8 * N, 0.5 * budget * 8 * N, 1.6 * budget * 8 * N], 1.0)["same_k"]
