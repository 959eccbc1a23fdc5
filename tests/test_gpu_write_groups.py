"""GPU parity of the select stage's sweeps where a slice changes from reading marked 16-element groups to reading whole rounds,
at ragged ends, with one and two CTAs per chunk."""
import numpy as np
import pytest
import torch

from tests._harness import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value_dtype", [0, 1])
@pytest.mark.parametrize("frac", [0.02, 0.3])  # the sparse and the dense form of the write sweep
@pytest.mark.parametrize("n", [4097, 300 * 32768 + 5])
def test_slices_with_every_number_of_marked_groups(n, frac, value_dtype):
    """Slice s holds large entries in s % 129 of its 128 groups: from none to all, the switch included."""
    rng = np.random.default_rng(n + value_dtype)
    x = (1e-3 * rng.standard_normal((1, n))).astype(np.float32)
    groups = -(-n // 16)
    slice_of, group = np.arange(groups) // 128, np.arange(groups) % 128
    marked = np.flatnonzero(group < (slice_of * 7) % 129)
    at = np.minimum(marked * 16 + rng.integers(0, 16, marked.size), n - 1)
    x[0, at] = rng.choice((-1.0, 1.0), at.size) * (1 + rng.random(at.size))
    share = max(at.size / n, 1e-3)
    r = Runner([n], 1, [round(min(0.9, s * share), 6) for s in (0.5, 1.0, 1.2)] + [1.0], 1000, value_dtype)
    grads = torch.from_numpy(x).cuda()
    state = torch.zeros_like(grads)
    bpe = 8 if value_dtype == 0 else 6
    for _ in range(2):
        assert r.compare_step(grads, state, [frac * bpe * n], 1.0)["same_k"]
