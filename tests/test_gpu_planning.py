"""GPU parity on magnitudes far apart: the sample kernel plans the sweep's bins from ratios of squares that span more than
binary32 does."""
import numpy as np
import pytest
import torch

from tests._harness import Runner

pytestmark = pytest.mark.gpu


def _residues(rng):  # a clipped gradient with round-off residues
    u = rng.random(1_000_000)
    x = np.where(u < 0.9, 1e-20 * rng.standard_normal(u.size), np.where(u < 0.93, 1.0, rng.uniform(1.0, 4.0, u.size)))
    return x, [0.01, 0.02, 0.07, 1.0]


def _overflowing(rng):  # squares beyond binary32
    u = rng.random(1_000_000)
    return np.where(u < 0.7, 1e10 * rng.standard_normal(u.size), rng.uniform(2e19, 4e19, u.size)), [0.01, 0.05, 0.3, 1.0]


def _three_values(rng):
    return rng.choice([1e20, 1.0, 1e-20], 24000), [0.1, 0.2, 0.4, 0.6, 0.8, 1.0]


def _three_ranges(rng):
    x = np.concatenate([rng.uniform(100, 200, 400), rng.uniform(1.0, 1.08, 4000), rng.uniform(1e-20, 2e-20, 20000)])
    return rng.permutation(x), [float(r) for r in np.linspace(0.002, 0.95, 22)]


def _tiny_beside_large(rng):  # the smaller magnitudes' squares vanish beside the larger ones'
    u = rng.random(300_000)
    return np.exp(rng.uniform(np.log(1e-38), np.log(1e-30), u.size)) * np.where(u < 0.6, 1.0, 1e50), [0.05, 0.3, 0.45, 0.7, 0.9, 1.0]


@pytest.mark.parametrize("inputs", [_residues, _overflowing, _three_values, _three_ranges, _tiny_beside_large])
def test_magnitudes_far_apart(inputs):
    rng = np.random.default_rng(3)
    x, grid = inputs(rng)
    n = x.size
    x = (x * rng.choice((-1.0, 1.0), n)).astype(np.float32)[None, :]
    r = Runner([n], 1, grid, 1000, 0)
    grads = torch.from_numpy(x).cuda()
    state = torch.zeros_like(grads)
    for frac in (0.02, 0.5):
        r.compare_step(grads, state, [frac * 8 * n], 1.0)
