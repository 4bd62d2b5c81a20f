"""Refresh attention at the edges of its work items against the oracle.

A work item of the tensor-core kernel is two query tiles of floor(128/G)
selected rows; the cases put the selected rows just below, at and above one
and two tiles, one row alone, a last item of one row, and positions such that
the first tile needs fewer 128-key tiles than the second (or only one). The bar
is that of tests/parity.py: 2e-2 absolute + 2^-8 relative on bf16 outputs.
"""

import numpy as np
import pytest
import torch

from oracle import conduit_oracle as O

pytestmark = pytest.mark.gpu

# (Hq, Hkv, d, tokens per request, selected positions per request: a count spread evenly, or "head" / "tail")
CASES = [
    (14, 2, 128, (700, 300), (18, 19)),        # G = 7: 18 rows per tile
    (14, 2, 128, (700, 130), (36, 37)),
    (14, 2, 128, (1500,), (73,)),              # two full items and one row
    (8, 8, 128, (400, 1), (257, 1)),           # G = 1: 128 rows per tile; a one-token request
    (16, 1, 128, (640,), ("head", 9)),         # G = 16: all rows in the first key tile
    (16, 1, 128, (640,), ("tail", 17)),        # all rows in the last key tile
    (6, 2, 128, (129, 128, 127), (0, 128, 3)), # key tiles of 1, 127 and 128 keys; an empty selection
]


def _positions(spec, n):
    if isinstance(spec, tuple):
        return np.arange(spec[1]) if spec[0] == "head" else np.arange(n - spec[1], n)
    return np.unique(np.linspace(0, n - 1, spec).round().astype(np.int64)) if spec else np.zeros(0, np.int64)


def _run(C, hq, hkv, d, n_r, specs, page=0, seed=0):
    L, G = 2, hq // hkv
    if len(specs) == 2 and isinstance(specs[0], str):
        specs = (specs,)
    pos = [_positions(s, n) for s, n in zip(specs, n_r)]
    tok = np.concatenate([[0], np.cumsum(n_r)]).tolist()
    rng = torch.Generator(device="cuda").manual_seed(seed)
    draw = lambda *shape: torch.randn(shape, generator=rng, device="cuda").bfloat16()
    k, v = draw(L, hkv, tok[-1], d), draw(L, hkv, tok[-1], d)
    q_rows = draw(L, sum(map(len, pos)), hq, d)
    R = len(n_r)
    batch = C.Batch(tok, tok, list(range(R + 1)), list(range(R + 1)), device="cuda")
    kv = C.KvCache(k, v, hq)
    off, off_dev = C.idx_offsets([len(p) for p in pos])
    idx = torch.tensor(np.concatenate(pos), dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = C.conduit_refresh_attn(kv, batch, idx, off, off_dev, q_rows, status=status)
    assert C.conduit_read_status(status) == C.OK
    f = lambda t: t.double().cpu().numpy()
    i0 = 0
    for r, p in enumerate(pos):
        if len(p):
            t = slice(tok[r], tok[r + 1])
            want = O.refresh_attention(f(q_rows[:, i0:i0 + len(p)]), f(k[:, :, t]), f(v[:, :, t]), p)
            got = f(out[:, i0:i0 + len(p)])
            err = np.abs(got - want)
            assert np.all(err <= 2e-2 + 2.0 ** -8 * np.abs(want)), (r, float(err.max()))
        i0 += len(p)
    return out


@pytest.fixture(scope="module")
def C():
    from paper_2609_05821_gb300 import _build
    _build.build()
    from paper_2609_05821_gb300 import conduit
    return conduit


@pytest.mark.parametrize("case", range(len(CASES)))
def test_item_edges(C, case):
    hq, hkv, d, n_r, specs = CASES[case]
    _run(C, hq, hkv, d, n_r, specs, seed=case)
