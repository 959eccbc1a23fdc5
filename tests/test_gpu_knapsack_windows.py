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


@pytest.mark.parametrize("L,K,D,big", [
    (148, 16, 148, 0), (148, 16, 149, 0), (148, 16, 1000, 40000),  # no spare cell, one, most of a thousand
    (301, 17, 301, 0), (301, 127, 302, 0),                         # ... records in pieces
    (45, 8, 8191, 0), (100, 50, 8191, 3000),                       # 1024 threads; records in one piece and in pieces
    (400, 16, 1200, 0), (1995, 16, 3990, 0),                       # in pieces; the steps back as well
])
@pytest.mark.parametrize("schedule", [0, 1])
def test_every_way_of_searching(L, K, D, big, schedule):
    """Windows and whole rows at the same time, one after the other, and whole rows alone: the same choice.  One after the other, convex
    curves are decided by windows (but for some on the widest axis) and errors of any sign by whole rows."""
    rng = np.random.default_rng(11 * L + D)
    sizes = [int(v) for v in np.exp(rng.uniform(0, np.log(200), L)).astype(int) + 1]
    sizes[L // 3] += big
    grid = np.unique(np.round(np.geomspace(0.002, 1.0, K), 6))
    N, W, K = sum(sizes), 3, len(grid)
    r = Runner(sizes, W, list(grid), D, 0, schedule=schedule)
    grads = torch.from_numpy(rng.standard_normal((W, N)).astype(np.float32)).cuda()
    least, full = float(r.kt[:, 0].sum()) * 8, float(r.kt[:, -1].sum()) * 8
    for kind in ("convex", "ties", "same", "zeros", "odd", "nothing"):
        err = torch.from_numpy(curves(kind, rng, W, L, K)).cuda()
        bw = [float(v) for v in np.exp(rng.uniform(np.log(1.1 * least), np.log(max(0.9 * full, 1.2 * least)), W))]
        bw[1] = 2 * full if kind == "same" else bw[1]  # a worker without a search
        got = []
        for mode in (2, 1, 0, 0):
            kb.kimad_debug_set_search(r.ctx, mode)
            before = kb.kimad_debug_searches(r.ctx)
            state = torch.zeros((W, N), dtype=torch.float32, device="cuda")
            kb.kimad_debug_step_with_err(r.ctx, grads, state, bw, 1.0, r.out, err)
            st = r.out.stats_host()
            got.append((u32(r.out.j), st["status"], st["total_err"].view(np.uint32), u32(state)))
            none, first, second = (b - a for a, b in zip(before, kb.kimad_debug_searches(r.ctx)))
            if mode == 2:
                assert none + first + second == 0
            if mode == 1 and kind == "convex":
                assert none + first + second == W and (none == 0 or D == 8191), (none, first, second)
            if mode == 1 and kind in ("odd", "nothing"):
                assert none == W and first + second == 0
        for other in got[1:]:
            assert all(np.array_equal(a, b) for a, b in zip(got[0], other)), kind
        _, failed, damaged = kb.kimad_debug_check(r.ctx)
        assert failed == 0 and damaged == 0, hex(failed)


@pytest.mark.parametrize("W,schedule", [(1, 2), (3, 1), (35, 2)])
def test_both_searches_in_a_captured_step(W, schedule):
    """The two searches run beside each other in a replayed graph as on a stream, step after step, for more workers than one launch takes
    too; their flags are clear again after every step."""
    rng = np.random.default_rng(W)
    sizes = [int(v) for v in np.exp(rng.uniform(0, np.log(300), 148)).astype(int) + 1]
    N = sum(sizes)
    r = Runner(sizes, W, list(np.geomspace(0.01, 1.0, 16)), 1000, 0, schedule=schedule)
    grads = torch.from_numpy(rng.standard_normal((W, N)).astype(np.float32)).cuda()
    bw = [float(v) for v in rng.uniform(0.05, 0.5, W) * 8 * N]
    state, other = (torch.zeros((W, N), dtype=torch.float32, device="cuda") for _ in range(2))
    kb.kimad_step(r.ctx, grads, state, bw, 1.0, r.out)  # (before the capture: kernels are loaded)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        kb.kimad_step(r.ctx, grads, state, bw, 1.0, r.out)
    state.zero_()
    plain = Runner(sizes, W, r.grid, 1000, 0, schedule=2)
    kb.kimad_debug_set_search(plain.ctx, 2)
    for _ in range(4):
        graph.replay()
        kb.kimad_step(plain.ctx, grads, other, bw, 1.0, plain.out)
        torch.cuda.synchronize()
        assert torch.equal(r.out.j, plain.out.j) and torch.equal(r.out.k, plain.out.k) and torch.equal(state, other)
        assert torch.equal(r.out.stats, plain.out.stats)
    del graph
