"""The knapsack kernel at the edges of its dispatch: cells per thread by axis length, candidate counts around the record
widths and the lanes of a warp, axes as short as the layer list, layers whose candidates share their cells, rows that
cross the warps and the staged chunks."""
import numpy as np
import pytest
import torch

from tests._harness import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,K,D", [
    (1, 1, 1), (5, 3, 5), (7, 8, 40), (3, 9, 33), (6, 16, 1000), (6, 17, 1026),  # two cells per thread, then four
    (9, 32, 2056), (9, 33, 2057), (4, 127, 8191), (300, 5, 4500),                # four, eight; one and more candidates per lane
    (300, 12, 330), (260, 16, 1000), (70, 40, 90),                              # several chunks of records, short rows
])
def test_decisions_match_the_oracle(L, K, D):
    rng = np.random.default_rng(1000 * L + K)
    sizes = [int(v) for v in np.exp(rng.uniform(np.log(1), np.log(600), L)).astype(int) + 1]
    sizes[L // 2] += 3000  # one layer spans a good part of the axis
    grid = np.unique(np.round(np.geomspace(0.002, 1.0, K), 6)) if K > 1 else np.array([0.3])
    N = sum(sizes)
    r = Runner(sizes, 3, list(grid), D, 0)
    scale = np.exp(rng.uniform(-6, 2, L))
    x = (rng.standard_normal((3, N)) * np.repeat(scale, sizes)).astype(np.float32)
    least = float(np.maximum(1, np.ceil(grid[0] * np.array(sizes))).sum()) * 8
    for frac in (1.02, 3.0, 20.0):  # from hardly feasible to wide; one worker's budget is cut below
        bw = [frac * least, 1.7 * frac * least, 0.4 * frac * least]
        r.compare_step(torch.from_numpy(x).cuda(), torch.zeros((3, N), dtype=torch.float32, device="cuda"), bw, 1.0)
