"""The selection's radix digits at their edges, against a stable sort on the CPU (exact).

The keys of a case open 0 to 32 bits (all equal, two neighbours, one exponent, every exponent, zeros), the
budgets cut inside and at the ends of runs of equal keys, and the lengths are those at which the selection
changes its form: 1 024 and 8 192 tokens in one block, 65 536 in a cluster, the workspace beyond.
"""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_2609_05821_gb300 import _build
    _build.build()
    from paper_2609_05821_gb300 import conduit
    return conduit


def _keys(kind, n, rng):
    if kind == "equal":
        return np.full(n, 0.125, np.float32)
    if kind == "neighbours":
        return np.where(rng.random(n) < 0.5, np.float32(0.125), np.nextafter(np.float32(0.125), np.float32(1)))
    if kind == "few":
        return rng.integers(0, 3, n).astype(np.float32)
    if kind == "scores":
        return rng.gamma(0.5, 1e-3, n).astype(np.float32)
    bits = rng.integers(0, 0x7F800000, n, dtype=np.int64)   # "bits": every finite non-negative float
    return bits.astype(np.uint32).view(np.float32)


@pytest.mark.parametrize("n", (1, 31, 1024, 1025, 8192, 8193, 41472, 65536, 65537))
@pytest.mark.parametrize("kind", ("equal", "neighbours", "few", "scores", "bits"))
def test_digits(C, kind, n):
    rng = np.random.default_rng(n)
    s = _keys(kind, n, rng)
    order = np.argsort(-s.astype(np.float64), kind="stable")
    batch = C.Batch([0, n], [0, n], [0, 1], [0, 1], device="cuda")
    g = torch.ones(1, device="cuda")
    runs = int((s == s.max()).sum())
    for k in sorted({0, 1, n // 10, n // 2, min(runs, n), min(runs + 1, n), n - 1, n} & set(range(n + 1))):
        off, off_dev = C.idx_offsets([k])
        mask = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
        idx, _, _, _ = C.conduit_select_topk(batch, torch.from_numpy(s).cuda(), g, 1.0, off, off_dev, mask=mask)
        want = np.sort(order[:k])
        assert np.array_equal(idx.cpu().numpy(), want), (k,)
        assert np.array_equal(np.flatnonzero(mask.cpu().numpy()), want)
