"""Scoring units split over a cluster of two CTAs against the oracle and one CTA.

The library takes two CTAs per unit when that trims the last wave of units, so
the cases have a little more than one wave of units on a 152-SM GPU (160 units, 20
layers x 8 KV heads) or half a wave (72), of odd and even numbers of key tiles,
the last one ragged; each asserts that the launch is split. The bar is the 1e-3 of
tests/parity.py for bf16 scores; the split itself only adds a rounding of each
row's log2-sum-exp, so 1e-5 is asked for.
"""

import ctypes

import numpy as np
import pytest
import torch

from oracle import conduit_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_2609_05821_gb300 import _build
    _build.build()
    from paper_2609_05821_gb300 import conduit
    return conduit


def _ctas(units, tiles):
    """CTAs per unit of a scoring launch, from the test build of the library."""
    from paper_2609_05821_gb300 import _build
    lib = ctypes.CDLL(_build.build_test_hooks())
    return lib.conduit_test_score_ctas(units, tiles, torch.cuda.get_device_properties(0).multi_processor_count)


@pytest.mark.parametrize("n,nq,d,extra,L", [(3713, 4, 128, False, 20), (3713, 40, 128, True, 20), (2900, 5, 128, False, 20),
                                            (2900, 3, 64, False, 9), (2900, 40, 40, True, 9), (2049, 3, 64, False, 9)])
def test_split_units(C, n, nq, d, extra, L):
    hq, hkv = 16, 8
    assert _ctas(L * hkv, -(-n // 128)) == 2
    gen = torch.Generator(device="cuda").manual_seed(n + nq)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    k, v, q = draw(L, hkv, n, d), draw(L, hkv, n, d), draw(L, hq, nq, d)
    batch = C.Batch([0, n], [0, n // 3, n], [0, 2], [0, nq], device="cuda")
    kv = C.KvCache(k, v, hq)
    lse = torch.randn((L, hq, nq), generator=gen, device="cuda") + 8.0 if extra else None
    s, A, g = C.conduit_score_ex(kv, batch, q, extra_lse=lse)
    again = C.conduit_score_ex(kv, batch, q, extra_lse=lse)
    assert all(torch.equal(a, b) for a, b in zip((s, A, g), again))
    f = lambda t: t.double().cpu().numpy()
    kw = {} if lse is None else {"extra_lse": f(lse)}
    want = O.score_request(f(q), f(k), f(v), [0, n // 3, n], **kw)
    for got, ref in ((s, want["s"]), (A, want["A"]), (g, want["g"])):
        assert np.all(np.abs(f(got) - ref) <= 1e-5 * np.abs(ref) + 1e-7 * np.abs(ref).max())
    # a NaN in one CTA's keys reaches the rows' weights in the other's
    k[:, :, 5] = float("nan")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    s, _, _ = C.conduit_score(kv, batch, q, status=status)
    assert torch.isnan(s).all() and C.conduit_read_status(status) == C.ERR_NONFINITE


@pytest.mark.parametrize("d,kw", [(128, {}), (64, {}), (128, {"statistic": "rms"}), (128, {"value_norm": "side_cache"})])
def test_short_requests_in_a_split_batch(C, d, kw):
    """Requests of one key tile in a split launch: one CTA of the pair has no tiles of them, several times in a row.

    Every request gets what it gets alone, up to the rounding of the split (1e-5)."""
    L, hq, hkv = 4, 8, 4
    n_r = [1, 128, 4000] + [1 + 17 * i % 128 for i in range(11)]   # 14 requests, 224 units: three per pair of CTAs
    assert _ctas(L * hkv * len(n_r), 32) == 2
    nq = [1 + 7 * r % 40 for r in range(len(n_r))]
    cum = lambda x: [sum(x[:i]) for i in range(len(x) + 1)]
    tok, qo = cum(n_r), cum(nq)
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    k, v, q = draw(L, hkv, tok[-1], d), draw(L, hkv, tok[-1], d), draw(L, hq, qo[-1], d)

    def score(kv, batch, q):
        vn = C.conduit_value_norms(kv, batch) if kw.get("value_norm") == "side_cache" else None
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        out = C.conduit_score_ex(kv, batch, q, vnorm=vn, status=status, **kw)
        assert C.conduit_read_status(status) == C.OK
        return out

    batch = C.Batch(tok, tok, list(range(len(n_r) + 1)), qo, device="cuda")
    got = score(C.KvCache(k, v, hq), batch, q)
    for _ in range(5):
        assert all(torch.equal(a, b) for a, b in zip(got, score(C.KvCache(k, v, hq), batch, q)))
    for r, n in enumerate(n_r):
        t, qs = slice(tok[r], tok[r + 1]), slice(qo[r], qo[r + 1])
        alone = C.Batch([0, n], [0, n], [0, 1], [0, nq[r]], device="cuda")
        cut = lambda x, s: x[:, :, s].contiguous()
        want = score(C.KvCache(cut(k, t), cut(v, t), hq), alone, cut(q, qs))
        for a, b in zip((got[0][t], got[1][t], got[2][r:r + 1]), want):
            assert torch.all((a - b).abs() <= 1e-5 * b.abs() + 1e-7 * b.abs().max()), (r, n)


@pytest.mark.parametrize("form", ["contiguous", "paged"])
@pytest.mark.parametrize("d,nq", [(128, 10), (64, 10), (40, 3), (96, 36), (128, 72)])
def test_keys_of_no_token_reach_no_score(C, d, nq, form):
    """NaN in the next request's keys and values, or in a page's unused rows, leaves a request's scores as they are.

    40, 12, 144 and 288 scoring rows: the last 32-column chunk of a row group is partly filled."""
    L, hq, hkv, tok = 2, 8, 2, [0, 168, 460]
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    k, v, q = draw(L, hkv, 460, d), draw(L, hkv, 460, d), draw(L, hq, nq + 5, d)
    batch = C.Batch(tok, tok, [0, 1, 2], [0, nq, nq + 5], device="cuda")
    if form == "paged":   # request 0: pages 0 .. 10, the last with 8 unused rows; request 1: pages 11 .. 29
        table = torch.full((2, 19), -1, dtype=torch.int32)
        table[0, :11], table[1, :19] = torch.arange(11), torch.arange(11, 30)
        def cache(x, unused):
            pool = torch.full((L, hkv, 480, d), unused, dtype=x.dtype, device="cuda")
            pool[:, :, :168], pool[:, :, 176:468] = x[:, :, :168], x[:, :, 168:]
            return pool.view(L, hkv, 30, 16, d).transpose(1, 2).contiguous()
        score = lambda unused: C.conduit_score(C.KvCache(cache(k, unused), cache(v, unused), hq, 16, table), batch, q)
        clean, got, end = score(0.0), score(float("nan")), 460
    else:
        clean = C.conduit_score(C.KvCache(k, v, hq), batch, q)
        k[:, :, 168:], v[:, :, 168:] = float("nan"), float("nan")
        got, end = C.conduit_score(C.KvCache(k, v, hq), batch, q), 168
    assert torch.isfinite(clean[0]).all()
    for a, b, n in zip(got, clean, (end, end, 2 if form == "paged" else 1)):
        assert torch.equal(a[:n], b[:n])


@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.float32, 256), (torch.bfloat16, 64),
                                     (torch.bfloat16, 128), (torch.bfloat16, 136)])
@pytest.mark.parametrize("lo,hi", [(70, 330), (0, 330), (200, 3000)])
def test_masked_keys(C, dtype, d, lo, hi):
    """Keys whose logits overflow to -inf get no weight, also where they fill a chunk of keys or a CTA's share of them."""
    L, hq, hkv, n, nq = 1, 4, 2, 400 if hi < 400 else 3000, 5
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(dtype)
    k, v, q = draw(L, hkv, n, d), draw(L, hkv, n, d), draw(L, hq, nq, d)
    q[..., 0] = 32.0
    k[..., 0] = 0.0
    k[:, :, lo:hi, 0] = torch.finfo(dtype).min
    batch = C.Batch([0, n], [0, n], [0, 1], [0, nq], device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    s, A, _ = C.conduit_score(C.KvCache(k, v, hq), batch, q, status=status)
    assert C.conduit_read_status(status) == C.OK
    x = torch.einsum("lhqd,lhtd->lhqt", q.double(), k.double().repeat_interleave(hq // hkv, 1)) / d ** 0.5
    a = torch.softmax(x, -1).mean((1, 2))[0]
    norm = v.double().square().sum((1, 3)).sqrt()[0]
    assert torch.all(s[lo:hi] == 0) and torch.all(A[lo:hi] == 0)
    for got, want in ((A, a), (s, a * norm)):
        assert torch.all((got - want).abs() <= 1e-5 * want + 1e-7 * want.max())
