"""Refresh attention at the edges of its work items against the oracle.

A work item of the tensor-core kernels is one or two query tiles of floor(128/G)
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
# other head sizes: below, at and above the 64-dim half, 16-dim step and 32-byte store boundaries
HEAD_DIMS = (8, 16, 24, 56, 64, 72, 80, 96, 120)


def _positions(spec, n):
    if isinstance(spec, tuple):
        return np.arange(spec[1]) if spec[0] == "head" else np.arange(n - spec[1], n)
    return np.unique(np.linspace(0, n - 1, spec).round().astype(np.int64)) if spec else np.zeros(0, np.int64)


def _run(C, hq, hkv, d, n_r, specs, seed=0, form="plain", dtype=torch.bfloat16, L=2, unused=0.0):
    """`unused`: what a page's rows without a token hold."""
    if len(specs) == 2 and isinstance(specs[0], str):
        specs = (specs,)
    pos = [_positions(s, n) for s, n in zip(specs, n_r)]
    tok = np.concatenate([[0], np.cumsum(n_r)]).tolist()
    rng = torch.Generator(device="cuda").manual_seed(seed)
    draw = lambda *shape: torch.randn(shape, generator=rng, device="cuda").to(dtype)
    k, v = draw(L, hkv, tok[-1], d), draw(L, hkv, tok[-1], d)
    q_rows = draw(L, sum(map(len, pos)), hq, d)
    R = len(n_r)
    batch = C.Batch(tok, tok, list(range(R + 1)), list(range(R + 1)), device="cuda")
    kv = C.KvCache(k, v, hq)
    off, off_dev = C.idx_offsets([len(p) for p in pos])
    idx = torch.tensor(np.concatenate(pos), dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if form == "paged":  # pages of 16 tokens, a request's in reverse order
        pages = [-(-n // 16) for n in n_r]
        first = np.concatenate([[0], np.cumsum(pages)]).tolist()
        table = torch.full((R, max(pages)), -1, dtype=torch.int32)
        pool = [torch.full((L, first[-1], hkv, 16, d), unused, dtype=dtype, device="cuda") for _ in range(2)]
        for r, n in enumerate(n_r):
            table[r, :pages[r]] = torch.arange(first[r + 1] - 1, first[r] - 1, -1, dtype=torch.int32)
            for dst, src in zip(pool, (k, v)):
                rows = torch.nn.functional.pad(src[:, :, tok[r]:tok[r + 1]], (0, 0, 0, 16 * pages[r] - n), value=unused)
                dst[:, table[r, :pages[r]].long().cuda()] = rows.view(L, hkv, pages[r], 16, d).transpose(1, 2)
        kv = C.KvCache(*pool, hq, 16, table)
    if form in ("plain", "paged"):
        out = C.conduit_refresh_attn(kv, batch, idx, off, off_dev, q_rows, status=status)
    else:  # straight through the ABI: no workspace, or rows that start 2 bytes off a 16-byte boundary
        shift = 1 if form == "misaligned" else 0
        hold = [torch.zeros(q_rows.numel() + 8, dtype=dtype, device="cuda") for _ in range(2)]
        q_s, out = (h[shift:shift + q_rows.numel()].view(q_rows.shape) for h in hold)
        q_s.copy_(q_rows)
        C._check(C._lib.conduit_refresh_attn(kv.ref(), batch.ref(), C._ptr(idx), C._ptr(off), C._ptr(off_dev),
                                             C._ptr(q_s), C._ptr(out), None, 0, C._ptr(status),
                                             C._stream_ptr(None)))
    assert C.conduit_read_status(status) == C.OK
    sub = [0, 1] if L == 2 else [0, L // 2, L - 1]
    f = lambda t: t[sub].double().cpu().numpy()
    i0 = 0
    for r, p in enumerate(pos):
        if len(p):
            t = slice(tok[r], tok[r + 1])
            want = O.refresh_attention(f(q_rows[:, i0:i0 + len(p)]), f(k[:, :, t]), f(v[:, :, t]), p)
            got = f(out[:, i0:i0 + len(p)])
            err = np.abs(got - want)
            bar = 1e-6 + 1e-5 * np.abs(want) if dtype == torch.float32 else 2e-2 + 2.0 ** -8 * np.abs(want)
            assert np.all(err <= bar), (r, float(err.max()))
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


@pytest.mark.parametrize("form,d", [("plain", 128), ("paged", 128), ("plain", 96), ("plain", 40)])
def test_many_items(C, form, d):
    """Enough items for the work counter (fewer are dealt out in a fixed order), and that a cache in small
    pages takes two query tiles per item (a contiguous one takes one); at 96 and 128 dims more K/V than half
    of L2, so both parts of the item order."""
    _run(C, 14, 2, d, (1481,), (163,), form=form, L=64)


@pytest.mark.parametrize("d", HEAD_DIMS)
def test_head_dims(C, d):
    plain = _run(C, 6, 2, d, (300, 141), (44, 17), seed=d)
    # what a caller without a workspace, or with unaligned rows, gets
    assert torch.equal(_run(C, 6, 2, d, (300, 141), (44, 17), seed=d, form="no_workspace"), plain)
    _run(C, 6, 2, d, (300, 141), (44, 17), seed=d, form="misaligned")


@pytest.mark.parametrize("d", HEAD_DIMS)
def test_scores_of_head_dims(C, d, dtype=torch.bfloat16):
    """The scoring pass and the norm side cache at the same head sizes, contiguous and paged."""
    L, hq, hkv, n_r, nq = 2, 6, 2, (160, 208), (5, 90)   # 15 and 270 scoring rows: one and two row groups
    tok, qo = [0, 160, 368], [0, 5, 95]
    rng = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=rng, device="cuda").to(dtype)
    k, v, q = draw(L, hkv, 368, d), draw(L, hkv, 368, d), draw(L, hq, 95, d)
    batch = C.Batch(tok, [0, 100, 160, 368], [0, 2, 3], qo, device="cuda")
    pages = k.shape[2] // 16
    pool = lambda t: t.view(L, hkv, pages, 16, d).transpose(1, 2).contiguous()
    table = torch.full((2, 13), -1, dtype=torch.int32)
    table[0, :10], table[1, :13] = torch.arange(10), torch.arange(10, 23)
    got = []
    for kv in (C.KvCache(k, v, hq), C.KvCache(pool(k), pool(v), hq, 16, table)):
        got.append(C.conduit_score(kv, batch, q))
        vn = C.conduit_value_norms(kv, batch)
        got.append(C.conduit_score_with_norms(kv, batch, q, vn))
    for other in got[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got[0], other))
    f = lambda t: t.double().cpu().numpy()
    s, A, g = (f(t) for t in got[0])
    for r, img in ((0, [0, 100, 160]), (1, [0, 208])):
        t, qs = slice(tok[r], tok[r + 1]), slice(qo[r], qo[r + 1])
        want = O.score_request(f(q[:, :, qs]), f(k[:, :, t]), f(v[:, :, t]), img)
        for a, b in ((s[t], want["s"]), (A[t], want["A"])):   # fp32 sums: 1e-5 relative
            assert np.all(np.abs(a - b) <= 1e-5 * np.abs(b) + 1e-7 * np.abs(b).max())


# the CUDA-core kernels: fp32, and bf16 head sizes above 128 (rows tiles of 32, key tiles of 64)
@pytest.mark.parametrize("dtype,d", [(torch.float32, 8), (torch.float32, 64), (torch.float32, 72), (torch.float32, 128),
                                     (torch.float32, 256), (torch.bfloat16, 136), (torch.bfloat16, 256)])
def test_cuda_core_tiles(C, dtype, d):
    for specs in ((44, 17), (("head", 11), ("tail", 11)), (1, 0)):
        plain = _run(C, 6, 2, d, (300, 141), specs, seed=d, dtype=dtype)
        assert torch.equal(_run(C, 6, 2, d, (300, 141), specs, seed=d, form="misaligned", dtype=dtype), plain)
    for specs in ((9,), (("head", 1),), (44,)):   # clusters of eight CTAs: keys for all, for one, two row tiles
        _run(C, 6, 2, d, (700,), specs, seed=d, dtype=dtype)
    test_scores_of_head_dims(C, d, dtype)


@pytest.mark.parametrize("d,L", [(40, 2), (64, 2), (96, 2), (128, 2), (128, 64)])
def test_rows_without_a_token_are_not_read(C, d, L):
    """NaN and Inf in the unused rows of a request's last page, and at the head of the next request's rows.

    At 128 dims 64 layers in small pages take two query tiles per item, two layers one."""
    n_r, specs = (1481, 300), (163, ("tail", 30))
    plain = _run(C, 14, 2, d, n_r, specs, form="paged", L=L)
    for unused in (float("nan"), float("inf")):
        assert torch.equal(_run(C, 14, 2, d, n_r, specs, form="paged", L=L, unused=unused), plain)
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    k, v, q_rows = draw(L, 2, 700, d), draw(L, 2, 700, d), draw(L, 75, 14, d)
    tok = [0, 300, 700]
    batch = C.Batch(tok, tok, [0, 1, 2], [0, 1, 2], device="cuda")
    off, off_dev = C.idx_offsets([75, 0])
    idx = torch.arange(3, 300, 4, dtype=torch.int32, device="cuda")[:75]
    clean = C.conduit_refresh_attn(C.KvCache(k, v, 14), batch, idx, off, off_dev, q_rows)
    assert torch.isfinite(clean).all()
    k[:, :, 300:], v[:, :, 300:] = float("nan"), float("inf")
    assert torch.equal(C.conduit_refresh_attn(C.KvCache(k, v, 14), batch, idx, off, off_dev, q_rows), clean)


def test_values_past_a_position_add_nothing(C):
    """Non-finite V past a row's position, inside its key tile, leaves the row finite (fp32)."""
    k, v = torch.randn(1, 1, 100, 64, device="cuda"), torch.randn(1, 1, 100, 64, device="cuda")
    q_rows = torch.randn(1, 2, 1, 64, device="cuda")
    batch = C.Batch([0, 100], [0, 100], [0, 1], [0, 1], device="cuda")
    off, off_dev = C.idx_offsets([2])
    idx = torch.tensor([40, 70], dtype=torch.int32, device="cuda")
    clean = C.conduit_refresh_attn(C.KvCache(k, v, 1), batch, idx, off, off_dev, q_rows)
    v[:, :, 50] = float("inf")
    got = C.conduit_refresh_attn(C.KvCache(k, v, 1), batch, idx, off, off_dev, q_rows)
    assert torch.equal(got[:, 0], clean[:, 0]) and not torch.isfinite(got[:, 1]).any()


@pytest.mark.parametrize("form", ["contiguous", "paged"])
@pytest.mark.parametrize("d", [8, 40, 64, 72, 96, 120])
def test_non_finite_values_reach_the_rows_that_see_them(C, d, form):
    """bf16 head sizes below 128: Inf and NaN in V count from their own position on, as they do in the sum itself.

    The other rows keep the module's bar, also where they share a key tile with such a value."""
    n, hq, hkv, L = 300, 6, 2, 2
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    k, v, q_rows = draw(L, hkv, n, d), draw(L, hkv, n, d), draw(L, n // 2, hq, d)
    v[0, :, 50, :d // 2] = float("inf")
    v[0, 0, 131, 3] = -float("inf")
    v[0, 1, 200, d - 1] = float("nan")
    kv = C.KvCache(k, v, hq)
    if form == "paged":
        pool = lambda t: torch.nn.functional.pad(t, (0, 0, 0, 4)).view(L, hkv, 19, 16, d).transpose(1, 2).contiguous()
        kv = C.KvCache(pool(k), pool(v), hq, 16, torch.arange(19, dtype=torch.int32)[None])
    batch = C.Batch([0, n], [0, n], [0, 1], [0, 1], device="cuda")
    off, off_dev = C.idx_offsets([n // 2])
    idx = torch.arange(1, n, 2, dtype=torch.int32, device="cuda")
    got = C.conduit_refresh_attn(kv, batch, idx, off, off_dev, q_rows).double()
    for i, p in enumerate(idx.tolist()):
        for h in range(hq):
            kk, vv = k[:, h // 3, :p + 1].double(), v[:, h // 3, :p + 1].double()
            w = torch.softmax((kk @ q_rows[:, i, h].double()[:, :, None])[..., 0] / d ** 0.5, -1)
            want = (w[:, :, None] * vv).sum(1)
            x = got[:, i, h]
            fine = torch.isfinite(want)
            assert torch.equal(fine, torch.isfinite(x)) and torch.equal(torch.isnan(want), torch.isnan(x)), (p, h)
            assert torch.equal(want[torch.isinf(want)], x[torch.isinf(want)]), (p, h)
            assert torch.all((x - want).abs()[fine] <= 2e-2 + 2.0 ** -8 * want.abs()[fine]), (p, h)


@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64), (torch.bfloat16, 96),
                                     (torch.bfloat16, 136)])
def test_masked_keys_get_no_weight(C, dtype, d):
    """Keys whose logits overflow to -inf: a row that sees others gives them no weight, a row that sees no other is NaN."""
    n, hq, hkv = 300, 4, 2
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(dtype)
    k, v, q_rows = draw(1, hkv, n, d), draw(1, hkv, n, d), draw(1, 4, hq, d)
    q_rows[..., 0], k[..., 0] = 32.0, 0.0
    k[:, :, :40, 0] = k[:, :, 128:290, 0] = torch.finfo(dtype).min
    batch = C.Batch([0, n], [0, n], [0, 1], [0, 1], device="cuda")
    off, off_dev = C.idx_offsets([4])
    idx = torch.tensor([20, 90, 270, 299], dtype=torch.int32, device="cuda")
    got = C.conduit_refresh_attn(C.KvCache(k, v, hq), batch, idx, off, off_dev, q_rows).double()
    assert torch.isnan(got[:, 0]).all()
    for i, p in ((1, 90), (2, 270), (3, 299)):
        for h in range(hq):
            x = k[0, h // 2, :p + 1].double() @ q_rows[0, i, h].double() / d ** 0.5
            want = torch.softmax(x, 0) @ v[0, h // 2, :p + 1].double()
            bar = 1e-6 + 1e-5 * want.abs() if dtype == torch.float32 else 2e-2 + 2.0 ** -8 * want.abs()
            assert torch.all((got[0, i, h] - want).abs() <= bar), (p, h)
