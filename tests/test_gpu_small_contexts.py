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


@pytest.mark.parametrize("R,W,n,ctas", [(2, 1, 1 << 20, 8), (5, 3, 114700, 8), (16, 1, 131072, 4), (11, 3, 40000, 4), (17, 2, 98310, 2), (60, 1, 70001, 2),
                                        (15, 1, 16384, 1)])
def test_a_cluster_counts_the_sample_that_one_CTA_counts(R, W, n, ctas):
    """The bands planned from a sample that all CTAs of a cluster have read (sizes of a full round of units each) are those of the same layers
    in a context of so many layers that one CTA reads each; without zeros, no layer is left to the exact path."""
    sizes, more = [n + 3 * i for i in range(R)], [4097] * 160
    grid = [0.01, 0.02, 0.05, 0.1, 0.2, 0.5, 1.0]
    rounds = -(-min(max(n // 64, 1024), 2047, -(-n // 32)) // 256)
    resident = {8: 15, 4: 33, 2: 74, 1: 148}[ctas]
    assert R * W <= resident and ctas <= max(1, rounds + 1)  # (the size that the dispatch takes on a B200)
    rng = np.random.default_rng(n)
    x = (rng.standard_t(3, (W, sum(sizes))) * np.repeat(np.exp(rng.uniform(-4, 4, R)), sizes)).astype(np.float32)
    rest = rng.standard_normal((W, sum(more))).astype(np.float32)
    for zeros in (False, True):
        if zeros:  # in a run: their spread over the units is counted as well
            x[W - 1, : n // 2] = 0.0
        metas = []
        for layers, values in ((sizes, x), (sizes + more, np.concatenate([x, rest], axis=1))):
            N = sum(layers)
            ctx = kb.new_context(layers, W, grid)
            state = torch.zeros((W, N), dtype=torch.float32, device="cuda")
            kb.kimad_step(ctx, torch.from_numpy(np.ascontiguousarray(values)).cuda(), state, [0.1 * 4 * N] * W, 1.0, kb.Packed(ctx))
            assert zeros or kb.kimad_debug_exact_path_layers(ctx) == 0
            metas.append(kb.kimad_debug_get_band_meta(ctx, len(layers))[:, :R])
        assert (metas[0][..., 0] > 0).any() and (zeros or (metas[0][..., 2] == 0).all())
        assert np.array_equal(metas[0], metas[1])
