"""Contexts small enough that a cluster of CTAs reads a layer's sample (eight, four and two CTAs per layer, and the first size with one
again), and layers at the edges of the ways in which tiny ones are sorted; every element against the oracle."""
import numpy as np
import pytest
import torch

from paper_2312_08053_b200 import binding as kb
from tests._harness import Runner

pytestmark = pytest.mark.gpu


def step(sizes, W, x, frac, grid):
    N = sum(sizes)
    r = Runner(sizes, W, grid, max(1000, 2 * len(sizes)), 0)
    state = torch.zeros((W, N), dtype=torch.float32, device="cuda")
    for g in x:
        assert r.compare_step(torch.from_numpy(g).cuda(), state, [frac * 4 * N] * W, 1.0)["status"] == kb.KIMAD_OK


@pytest.mark.parametrize("R,W,n", [(1, 1, 70001), (16, 1, 33000), (17, 1, 4097), (8, 4, 9000), (11, 3, 12345), (64, 1, 5000), (65, 1, 5001),
                                   (43, 3, 4500)])
def test_samples_read_by_clusters(R, W, n):
    rng = np.random.default_rng(R * W)
    sizes = [n + 3 * i for i in range(R)]
    x = rng.standard_t(3, (2, W, sum(sizes))).astype(np.float32) * np.repeat(np.exp(rng.uniform(-4, 4, R)), sizes).astype(np.float32)
    x[1, :, : n // 2] = 0.0  # untouched rows: zeros in runs
    step(sizes, W, x, 0.1, [0.01, 0.02, 0.05, 0.1, 0.2, 0.5, 1.0])


@pytest.mark.parametrize("distinct", [0, 7])
def test_tiny_layers_of_every_size_class(distinct):
    sizes = [1, 2, 3, 5, 31, 33, 64, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1000, 1023, 1024, 1025, 2047, 2048, 2049, 3072, 4095, 4096]
    rng = np.random.default_rng(11 + distinct)
    x = rng.standard_normal((1, 2, sum(sizes))).astype(np.float32)
    if distinct:  # ties: a few magnitudes of both signs, zeros among them
        x = np.round(x * distinct / 3).astype(np.float32)
    step(sizes, 2, x, 0.2, [0.01, 0.05, 0.1, 0.3, 0.7, 1.0])
