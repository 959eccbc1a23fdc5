"""The knapsack's search over windows of the rows against the recursion over whole rows (which a context with a wait limit of its
own takes) and against the oracle, on given curves: chunks of records and their ends, odd layer counts, axes from no spare cell to
thousands, windows of 64 and 256 cells, ties, and what is left to the whole rows."""
import numpy as np
import pytest
import torch

from oracle import kimad_oracle as ko
from paper_2312_08053_b200 import binding as kb
from tests._harness import Runner, u32

pytestmark = pytest.mark.gpu


def curves(kind, rng, W, L, K):
    j = np.arange(K)[None, None]
    scale = np.exp(rng.uniform(-8, 4, (W, L, 1)))
    if kind == "convex":
        e = scale * (1 - np.linspace(0.02, 1, K)[None, None] ** rng.uniform(0.2, 1, (W, L, 1)))
    elif kind == "ties":  # few distinct values: many paths with the same sum
        e = np.round(np.sort(rng.uniform(0, 8, (W, L, K)), axis=2)[:, :, ::-1])
    elif kind == "random":  # not even descending
        e = rng.uniform(0, 1, (W, L, K))
    elif kind == "same":
        e = np.broadcast_to(8.0 / (j + 1), (W, L, K))
    elif kind == "zeros":
        e = np.where(rng.uniform(size=(W, L, 1)) < 0.7, 0, 1) * np.exp(-0.4 * j)
    elif kind == "range":  # sums that absorb most of their terms, subnormal ones among them
        e = np.exp(rng.uniform(-100, 5, (W, L, 1))) * np.exp(-0.3 * j)
    elif kind == "nothing":
        e = np.zeros((W, L, K))
    else:  # "odd": negative and infinite values
        e = rng.standard_normal((W, L, K)) * scale
        e[:, ::7, K // 2] = np.inf
    return np.ascontiguousarray(e, np.float32)


@pytest.mark.parametrize("L,K,D,big", [
    (99, 16, 1000, 0), (100, 16, 1000, 0), (148, 16, 1000, 40000), (161, 7, 1000, 9000),  # whole rows, windows from 100 layers on
    (40, 12, 3000, 2000), (61, 33, 2100, 0),                                              # ... from 40 on where the axis is wide
    (227, 16, 1200, 0), (228, 16, 1200, 0), (256, 8, 600, 0), (257, 8, 600, 5000),         # one chunk of records, and one layer more
    (301, 17, 301, 0), (301, 127, 302, 0), (513, 33, 1030, 0),                             # no spare cell, one, odd counts
    (1101, 16, 2202, 0), (2100, 9, 8191, 0),                                               # many chunks; steps back in pieces
])
def test_windows_decide_as_whole_rows(L, K, D, big):
    rng = np.random.default_rng(7 * L + K)
    sizes = [int(v) for v in np.exp(rng.uniform(0, np.log(200), L)).astype(int) + 1]
    sizes[L // 3] += big
    grid = np.unique(np.round(np.geomspace(0.002, 1.0, K), 6))
    N, W, K = sum(sizes), 2, len(grid)
    r = Runner(sizes, W, list(grid), D, 0)
    other = kb.Packed(r.ctx)
    g = rng.standard_normal((W, N)).astype(np.float32)
    grads = torch.from_numpy(g).cuda()
    least, full = float(r.kt[:, 0].sum()) * 8, float(r.kt[:, -1].sum()) * 8
    for kind in ("convex", "ties", "random", "same", "zeros", "range", "nothing", "odd"):
        err = curves(kind, rng, W, L, K)
        bw = [float(v) for v in np.exp(rng.uniform(np.log(1.02 * least), np.log(max(0.98 * full, 1.03 * least)), W))]
        ref = ko.step(sizes, W, r.grid, D, 0, g, np.zeros_like(g), bw, 1.0, inject_err=err)
        for out, limit in ((r.out, 1 << 31), (other, (1 << 31) - 1)):
            kb.kimad_debug_set_wait_limit(r.ctx, limit)
            state = torch.zeros((W, N), dtype=torch.float32, device="cuda")
            kb.kimad_debug_step_with_err(r.ctx, grads, state, bw, 1.0, out, torch.from_numpy(err).cuda())
            st = out.stats_host()
            assert np.array_equal(st["status"], ref.status), kind
            assert np.array_equal(u32(out.j), ref.j), (kind, limit)
            assert np.array_equal(st["total_err"].view(np.uint32), ref.total_err.view(np.uint32)), kind
    _, failed, damaged = kb.kimad_debug_check(r.ctx)
    assert failed == 0 and damaged == 0, hex(failed)
