"""What this library's users have it do, as cases that can be timed and compared.

A case is one call pattern of ``paper_2312_08053_b200.binding`` at one size:

- ``step``     one compression pass of a training step (kimad_step): EF21 difference, error curves, search over the
               layers, Top-K, packed message, estimator update (the sending direction);
- ``builtin``  the same pass for a caller that owns no device memory (kimad_step_builtin_scratch);
- ``receive``  the receiving side of a round: every worker's message into the receiver's estimators
               (kimad_apply_packed) and the model step over them (kimad_aggregate).

Tensor shapes, ratio grids, gradient distributions and budgets are those of ``workloads`` (an MLP, ResNet-18 and -50,
GPT-2 small, a 1.1 B Llama-style model), at full size or with every tensor shrunk by a divisor.

A training step meets new gradients every time.  So that a state can be run any number of times without its estimator
settling on one gradient, every pass reads the gradient buffer from another start (16-byte aligned, whole embedding
rows where the gradient is row-sparse): to the pass these are new values of the same distribution.
"""
from __future__ import annotations

import math

import torch

from paper_2312_08053_b200 import binding as kb
from paper_2312_08053_b200 import workloads

SHIFTS = 64  # starts of the gradient buffer that a state goes through


def _case(name, kind, cfg, workers, budget, divisor=1, **more):
    """``budget``: bytes a worker may send, as a share of its dense f32 bytes.  ``odd``: every tensor this many elements
    longer and the workers back to back, so that neither tensors nor workers start on a 16-byte boundary."""
    c = dict(name=name, kind=kind, cfg=cfg, divisor=divisor, workers=workers, budget=budget, bf16=False, policy=0,
             cost_model=0, block=0, odd=0, zero_rows=0.0, check_finite=False)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call in use: a gradient hook of a small model that has no workspace to give
        _case("mlp-hook", "builtin", 1, 1, 0.1),
        # a small model's step: 0.73 M elements in 62 tensors, one worker per GPU
        _case("resnet18-div16", "step", 2, 1, 0.1, divisor=16),
        # a CNN on a medium link, four workers on one GPU, one ratio for all layers sized to the budget
        _case("resnet18-w4-uniform", "step", 2, 4, 0.13, policy=3),
        # eight workers of a CNN, the sinusoidal link's middle
        _case("resnet50-w8", "step", 3, 8, 0.1),
        # odd tensor sizes and an unpadded stride, dense fallback for layers that are kept whole, a wide link, input check
        _case("resnet50-odd-dense", "step", 3, 2, 0.35, odd=5, cost_model=1, check_finite=True),
        # one worker per GPU: a language model's step on a 1 Gbit/s link (50 ms)
        _case("gpt2-w1", "step", 4, 1, 0.0126),
        # ... and four workers on one GPU (the benchmark's default workload), between bursts and in a 25 Gbit/s burst
        _case("gpt2-w4-low", "step", 4, 4, 0.0126),
        _case("gpt2-w4-burst", "step", 4, 4, 0.314),
        # blocks of 64 K elements instead of tensors (1995 segments), bf16 values
        _case("gpt2-blocks", "step", 4, 1, 0.03, block=65536, bf16=True),
        # the largest: two workers of the 1.1 B model, bf16 values, 1 % of the dense bytes
        _case("llama-w2", "step", 5, 2, 0.01, bf16=True),
        # one worker of it whose embedding gradient is half untouched rows, on a slow link
        _case("llama-w1-sparse", "step", 5, 1, 0.002, bf16=True, zero_rows=0.5),
        # the server's side of a round with four senders
        _case("gpt2-receive-w4", "receive", 4, 4, 0.05),
    ]


# elements of the five workloads' models: bounds of the divisor in draw()
_N = {cfg: workloads.workload(cfg).N for cfg in (1, 2, 3, 4, 5)}
_MAX_ELEMS = 2_200_000_000   # over all workers: the largest listed case
_MIN_ELEMS = 60_000


def draw(rng):
    kind = rng.choices(("step", "builtin", "receive"), (14, 2, 3))[0]
    block = 0
    if kind == "builtin":
        cfg, workers = rng.choice((1, 1, 2)), 1
        # built-in scratch: 32 MiB for everything, so small models only
        divisor = 1 if cfg == 1 else int(round(math.exp(rng.uniform(math.log(40), math.log(150)))))
    else:
        cfg = rng.choice((2, 3, 4, 4, 5))
        workers = rng.choice((1, 1, 2, 3, 4, 8))
        workers = max(1, min(workers, _MAX_ELEMS // _N[cfg]))
        divisor = int(math.exp(rng.uniform(0.0, math.log(_N[cfg] / _MIN_ELEMS))))
        if rng.random() < 0.4:
            divisor = 1
        if kind == "step" and _N[cfg] / divisor >= 4e6 and _N[cfg] * workers / divisor < 6e8 and rng.random() < 0.15:
            block = 65536
    budget = math.exp(rng.uniform(math.log(0.002), math.log(0.5)))
    policy = 0 if block else rng.choices((0, 1, 3), (8, 1, 2))[0]
    return dict(kind=kind, cfg=cfg, divisor=divisor, workers=workers, budget=round(budget, 5),
                bf16=rng.random() < 0.4, policy=policy, cost_model=int(policy == 0 and rng.random() < 0.25), block=block,
                odd=rng.choice((0, 0, 0, 1, 5)), check_finite=rng.random() < 0.25,
                zero_rows=rng.choice((0.0, 0.5, 0.9)) if cfg >= 4 and divisor == 1 and not block else 0.0)


def _workload(case):
    wl = workloads.workload(case["cfg"], case["divisor"], case["workers"])
    wl.layer_sizes = [n + case["odd"] for n in wl.layer_sizes]
    return wl


def _layers(case, wl):
    return workloads.block_layers(wl.layer_sizes, case["block"]) if case["block"] else wl.layer_sizes


def _cells(case, layers):
    """Cells of the budget axis: the default, or as many as a fine segment list needs."""
    return min(8191, max(1000, 2 * len(layers))) if case["block"] else 1000


def prepare(case, seed):
    wl = _workload(case)
    W, N = wl.n_workers, wl.N
    layers = _layers(case, wl)
    grid = [1.0] if case["policy"] == 3 else wl.ratio_grid
    bpe = 6 if case["bf16"] else 8
    budget = float(int(case["budget"] * 4 * N))
    stride = N if case["odd"] else (N + 3) // 4 * 4
    # a buffer as large as the budget allows (at least what the smallest candidates take)
    cap = int(min(N, max(budget / bpe, wl.ratio_grid[0] * N) + 2 * len(layers) + 16))
    if case["cost_model"]:
        cap = N  # a layer sent densely is counted by its values alone
    opts = dict(D=_cells(case, layers), value_dtype=int(case["bf16"]), check_finite=int(case["check_finite"]),
                max_packed_elems=cap, worker_stride=stride, policy=case["policy"], cost_model=case["cost_model"])
    if case["kind"] == "builtin":
        ctx = kb.kimad_create(layers, W, grid, **opts)
    else:
        ctx = kb.new_context(layers, W, grid, **opts)
    out = kb.Packed(ctx)
    step = 4 if not case["zero_rows"] else workloads.EMBED_COLS[case["cfg"]]
    zero = dict(zero_rows=case["zero_rows"]) if case["zero_rows"] else {}
    flat = torch.empty(W * stride + SHIFTS * step, dtype=torch.float32, device="cuda")
    base = flat[:W * stride].view(W, stride)
    if case["odd"] and zero:  # the sparse rows are laid out on the unextended embedding
        zero, step = {}, 4
    base.copy_(workloads.gradients(wl, seed, device="cuda", stride=stride, **zero))
    flat[W * stride:] = flat[:SHIFTS * step]
    grads = [flat[i * step:i * step + W * stride].view(W, stride) for i in range(SHIFTS)]
    state = torch.zeros((W, stride), dtype=torch.float32, device="cuda")
    s = dict(case=case, ctx=ctx, out=out, grads=grads, state=state, bw=[budget] * W, at=0)
    if case["kind"] == "receive":
        kb.kimad_step(ctx, grads[0], state, s["bw"], 1.0, out)
        s["x"] = torch.zeros(N, dtype=torch.float32, device="cuda")
        s["weights"] = [1.0 / W] * W
        s["answer"] = [s["state"], s["x"]]
    else:
        stats = out.stats.view(torch.int64)  # budget, used bytes, entries | error, status
        s["answer"] = [state, out.idx, out.val, out.offs, out.k, out.j, out.dense, stats[:, :3],
                       out.stats.view(torch.float32)[:, 6], out.stats.view(torch.int32)[:, 7]]
    return s


def run(s):
    if s["case"]["kind"] == "receive":
        kb.kimad_apply_packed(s["ctx"], s["out"], s["state"])
        kb.kimad_aggregate(s["x"], s["state"], s["weights"], 0.1)
        return s["answer"]
    grads = s["grads"][s["at"]]
    s["at"] = (s["at"] + 1) % SHIFTS
    step = kb.kimad_step_builtin_scratch if s["case"]["kind"] == "builtin" else kb.kimad_step
    step(s["ctx"], grads, s["state"], s["bw"], 1.0, s["out"])
    return s["answer"]


def work(case):
    wl = _workload(case)
    W, N = wl.n_workers, wl.N
    vb = 2 if case["bf16"] else 4
    kept = min(N, case["budget"] * 4 * N / (4 + vb))
    if case["kind"] == "receive":
        # the messages, the estimators' entries they change, and the estimators and the model once through the model step
        return {"bytes": W * kept * (4 + vb + 8) + 4 * N * W + 8 * N, "flops": W * kept + 2 * W * N + 2 * N}
    # gradients and estimators once; the message and the estimator's kept entries written
    return {"bytes": 8 * W * N + W * kept * (4 + vb + 4), "flops": 3 * W * N}


def tolerance(case):
    if case["kind"] == "receive":
        return "exact"  # the order of the binary32 operations is part of the interface
    # The curve is certified to 1e-5 relative, and the total error is a binary32 sum over it; what is selected, packed
    # and added to the estimator are whole numbers and single binary32 operations, which do not depend on the order of sums.
    return {"rel": 1e-5, "max": 1e-5, "differ": 0.0}
