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


@pytest.mark.parametrize("n,others,W", [(32769, 0, 1), (131072, 0, 2), (131073, 1, 1), (196609, 0, 1), (262144, 2, 3), (140000, 40, 2), (240000, 40, 2), (300001, 0, 1)])
def test_bands_that_do_not_fit(n, others, W):
    """Magnitudes over 150 octaves and thirty candidates: the bands do not fit the tables and every layer takes the exact path, by one
    CTA (up to four chunks; up to six with too many layers for clusters), by clusters of two and four, or over lists."""
    rng = np.random.default_rng(n)
    sizes, grid = [n] + [n + 7 * i for i in range(others)] + [3000], [(j + 0.5) / 30 for j in range(30)]
    N = sum(sizes)
    x = np.exp(rng.uniform(-75, 30, (W, N))) * rng.choice((-1.0, 1.0), (W, N))
    r = Runner(sizes, W, grid, 1000, 0)
    grads = torch.from_numpy(x.astype(np.float32)).cuda()
    state = torch.zeros_like(grads)
    for frac in (0.3, 0.08):
        assert r.compare_step(grads, state, [frac * 8 * N] * W, 1.0, check_inject=False)["same_k"]
    taken = kb.kimad_debug_exact_path_layers(r.ctx)
    assert taken >= W * (1 + others), taken  # (the second step's state may leave some layers within the tables)


@pytest.mark.parametrize("n", [131073, 196609, 262144, 400000])
def test_loose_candidates_of_one_layer(n):
    """Clusters of magnitudes, one of two values only: loose candidates are refined, some of which share a bin or stay loose."""
    rng = np.random.default_rng(n)
    grid = [0.01 * i for i in range(1, 17)] + [1.0]
    x = np.exp(np.floor(rng.random((1, n)) * 40)) * (1 + 1e-3 * np.abs(rng.standard_normal((1, n))))
    x[0, ::3] = np.where(rng.random(x[0, ::3].size) < 0.5, 1e5, 1.00001e5)
    r = Runner([n], 1, grid, 1000, 0)
    grads = torch.from_numpy((x * rng.choice((-1.0, 1.0), x.shape)).astype(np.float32)).cuda()
    state = torch.zeros_like(grads)
    for frac in (0.1, 0.6, 0.2):
        assert r.compare_step(grads, state, [frac * 8 * n], 1.0)["same_k"]


@pytest.mark.parametrize("K", [32, 33, 64, 127])
@pytest.mark.parametrize("n", [5000, 100000])
def test_exact_path_with_many_candidates(n, K):
    """More candidates than a warp has lanes, several of them in one bin of every digit."""
    rng = np.random.default_rng(K)
    x = rng.standard_normal((1, n)) * np.where(rng.random((1, n)) < 0.3, 1e-6, 1.0)
    x[0, :n // 5] = 1.5
    r = Runner([n], 1, [(j + 1) / (K + 1) for j in range(K)], 1000, 0, curve_mode=1)
    grads = torch.from_numpy(x.astype(np.float32)).cuda()
    assert r.compare_step(grads, torch.zeros_like(grads), [0.3 * 8 * n], 1.0)["same_k"]
