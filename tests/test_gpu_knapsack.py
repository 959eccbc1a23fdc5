"""The knapsack kernel at the edges of its dispatch: cells per thread by axis length, candidate counts around the record
widths and the lanes of a warp, axes as short as the layer list, layers whose candidates share their cells, rows that
cross the warps and the staged chunks."""
import numpy as np
import pytest
import torch

from oracle import kimad_oracle as ko
from paper_2312_08053_b200 import binding as kb
from tests._harness import Runner, u32

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


@pytest.mark.parametrize("L,K,D", [(40, 9, 1000), (25, 40, 300), (60, 16, 2500)])
def test_given_errors_of_any_sign(L, K, D):
    """A curve given from outside may hold negative values (and infinite ones): the search only compares sums."""
    rng = np.random.default_rng(L)
    sizes = [int(v) for v in rng.integers(20, 900, L)]
    N, W = sum(sizes), 2
    r = Runner(sizes, W, list(np.geomspace(0.01, 1.0, K)), D, 0)
    g = rng.standard_normal((W, N)).astype(np.float32)
    err = rng.standard_normal((W, L, K)).astype(np.float32)
    err[1, ::7] = -abs(err[1, ::7])
    err[0, ::5, K // 2] = np.inf
    err[0, 3] = 0.0
    for frac in (0.05, 0.3):
        bw = [frac * 8 * N, 0.7 * frac * 8 * N]
        state = torch.zeros((W, N), dtype=torch.float32, device="cuda")
        kb.kimad_debug_step_with_err(r.ctx, torch.from_numpy(g).cuda(), state, bw, 1.0, r.out, torch.from_numpy(err).cuda())
        ref = ko.step(sizes, W, r.grid, D, 0, g, np.zeros_like(g), bw, 1.0, inject_err=err)
        st = r.out.stats_host()
        assert np.array_equal(st["status"], ref.status) and not ref.status.any()
        assert np.array_equal(u32(r.out.j), ref.j)
        assert np.array_equal(st["total_err"], ref.total_err)
        assert np.array_equal(u32(state), ref.state.view(np.uint32))


@pytest.mark.parametrize("schedule", [0, 1])
def test_a_wait_that_runs_out(schedule):
    """With no patience at all the warps' first wait that is not met ends the search: nothing is selected, nothing changes, and
    the next step on the same context is the oracle's."""
    rng = np.random.default_rng(4)
    sizes = [int(v) for v in rng.integers(200, 6000, 120)]
    N, W = sum(sizes), 3
    r = Runner(sizes, W, list(np.geomspace(0.01, 1.0, 12)), 1000, 0, schedule=schedule)
    grads = torch.from_numpy(rng.standard_normal((W, N)).astype(np.float32)).cuda()
    state = torch.from_numpy(rng.standard_normal((W, N)).astype(np.float32)).cuda()
    before = state.clone()
    kb.kimad_debug_set_wait_limit(r.ctx, 0)
    status, k = r.gpu_step(grads, state, [0.2 * 8 * N] * W, 1.0)
    assert status == kb.KIMAD_ERR_TIMEOUT
    st = r.out.stats_host()
    assert (st["status"] == kb.KIMAD_ERR_TIMEOUT).all() and not st["n_selected"].any() and not st["used_bytes"].any()
    assert not k.any() and not u32(r.out.j).any() and not r.out.offs.any() and torch.equal(state, before)
    kb.kimad_debug_set_wait_limit(r.ctx, 1 << 31)
    assert r.compare_step(grads, state, [0.2 * 8 * N] * W, 1.0)["status"] == kb.KIMAD_OK
    with pytest.raises(kb.KimadError):
        kb.kimad_debug_set_wait_limit(r.ctx, (1 << 31) + 1)
