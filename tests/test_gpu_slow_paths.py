"""GPU parity of refinement and exact radix select where a layer's own CTA takes them (contexts whose layers have few
chunks) and where chunks are listed, at the sizes that separate the two."""
import numpy as np
import pytest
import torch

from paper_2312_08053_b200 import binding as kb
from tests._harness import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4097, 262143, 262144, 262145])
def test_loose_candidates_of_small_contexts(n):
    """Forty narrow clusters of magnitudes: bins that hold a cluster's thresholds have bounds too loose for the curve, from
    one step to the next (the counts of the pieces are left clean)."""
    rng = np.random.default_rng(n)
    sizes, grid, W = [n, 50000], [0.01 * i for i in range(1, 17)] + [1.0], 2
    N = sum(sizes)
    x = np.exp(np.floor(rng.random((W, N)) * 40)) * (1 + 1e-3 * np.abs(rng.standard_normal((W, N))))
    x = (x * rng.choice((-1.0, 1.0), (W, N))).astype(np.float32)
    r = Runner(sizes, W, grid, 1000, 0)
    grads = torch.from_numpy(x).cuda()
    state = torch.zeros_like(grads)
    for budget in ([0.1 * 8 * N] * 2, [0.6 * 8 * N, 0.35 * 8 * N], [0.2 * 8 * N] * 2):
        assert r.compare_step(grads, state, budget, 1.0)["same_k"]
    detail = kb.kimad_debug_exact_path_layers(r.ctx, detail=True)
    assert sum(detail[6:]) > 0, "nothing was refined"


@pytest.mark.parametrize("n", [4097, 32768, 65535, 65537])
def test_exact_path_of_small_contexts(n):
    """Every layer on the exact path, which a layer of up to two chunks takes by itself; with a layer of one magnitude."""
    rng = np.random.default_rng(n)
    sizes, grid, W = [n, 33000, 20], [0.001, 0.01, 0.1, 0.5, 1.0], 2
    N = sum(sizes)
    x = rng.standard_normal((W, N)).astype(np.float32)
    x[:, n:n + 33000] = np.sign(x[:, n:n + 33000]) * np.float32(0.75)
    r = Runner(sizes, W, grid, 1000, 0, curve_mode=1)
    grads = torch.from_numpy(x).cuda()
    state = torch.from_numpy((rng.standard_normal((W, N)) * 0.01).astype(np.float32)).cuda()
    for budget in ([0.05 * 8 * N] * 2, [0.4 * 8 * N, 0.01 * 8 * N]):
        r.compare_step(grads, state, budget, 1.0)
    assert kb.kimad_debug_exact_path_layers(r.ctx) == 2 * 4 * W  # two layers; every comparison runs two steps
