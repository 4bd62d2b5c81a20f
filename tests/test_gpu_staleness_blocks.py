"""Staleness with blocks of queries that leave the first query tile empty: paged and contiguous agree bit for bit.

With G = 7 a work item holds 2 x 18 queries; 37 to 54 of them leave a last block whose first tile has no rows.
Its softmax warps scale value tiles ahead of any logits, while the copies of a paged K (one per page half) land
late. Short requests make many such items follow one another.
"""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", (128, 96, 64))
def test_paged_equals_contiguous(d):
    from paper_2609_05821_gb300 import _build
    _build.build()
    from paper_2609_05821_gb300 import conduit as C
    L, hq, hkv, R, M, page = 11, 28, 4, 16, 2, 16
    n_r = [16 * (12 + r) for r in range(R)]
    nq = [37 + r for r in range(R)]
    cum = lambda x: [sum(x[:i]) for i in range(len(x) + 1)]
    tok, qo = cum(n_r), cum(nq)
    rng = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=rng, device="cuda").bfloat16()
    k, v, q, z = draw(L, hkv, tok[-1], d), draw(L, hkv, tok[-1], d), draw(L, hq, qo[-1], d), draw(M, L, hkv, tok[-1], d)
    pages = tok[-1] // page
    order = torch.randperm(pages, generator=rng, device="cuda")
    pool = lambda t: t.view(L, hkv, pages, page, d).transpose(1, 2)[:, torch.argsort(order)].contiguous()
    table = torch.full((R, max(n_r) // page), -1, dtype=torch.int32)
    for r in range(R):
        table[r, :n_r[r] // page] = order[tok[r] // page:tok[r + 1] // page].cpu().int()
    batch = C.Batch(tok, tok, list(range(R + 1)), qo, device="cuda")
    mask = (torch.rand(tok[-1], generator=rng, device="cuda") < 0.1).to(torch.uint8)
    run = lambda kv: C.conduit_staleness_iso(kv, batch, q, mask, z, 0.5)[0]
    want = run(C.KvCache(k, v, hq))
    paged = C.KvCache(pool(k), pool(v), hq, page, table)
    for _ in range(20):
        assert torch.equal(run(paged), want)


@pytest.mark.parametrize("d", (128, 96, 64))
def test_draws_of_other_requests_are_not_read(d):
    """Non-finite draws of a request change nothing in the one before it, whose last key tile they share."""
    from paper_2609_05821_gb300 import conduit as C
    L, hq, hkv, tok, qo = 2, 8, 2, [0, 200, 500], [0, 9, 20]
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    k, v, q, z = draw(L, hkv, 500, d), draw(L, hkv, 500, d), draw(L, hq, 20, d), draw(2, L, hkv, 500, d)
    batch = C.Batch(tok, tok, [0, 1, 2], qo, device="cuda")
    mask = (torch.rand(500, generator=gen, device="cuda") < 0.1).to(torch.uint8)
    clean = C.conduit_staleness_iso(C.KvCache(k, v, hq), batch, q, mask, z, 0.5)[0]
    z[:, :, :, 200:] = float("nan")
    got = C.conduit_staleness_iso(C.KvCache(k, v, hq), batch, q, mask, z, 0.5)[0]
    assert got[0] == clean[0] and torch.isnan(got[1])


@pytest.mark.parametrize("d", (64, 96))
def test_long_sums_have_no_bias(d):
    """16 384 keys at head sizes below 128, against 64 bits from the same bf16 deviations, outputs rounded to bf16.

    What remains are fp32 sums rounded to nearest, without a common sign, and the few outputs that round the other
    way for them: below 1e-6 of the sum over 512 rows. Sums that truncate come out 7e-5 lower (64 dims)."""
    from paper_2609_05821_gb300 import conduit as C
    n, hq, nq, M, kappa = 16384, 8, 32, 2, 0.5
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    k, v, q, z = draw(1, 1, n, d), draw(1, 1, n, d), draw(1, hq, nq, d), draw(M, 1, 1, n, d)
    batch = C.Batch([0, n], [0, n], [0, 1], [0, nq], device="cuda")
    mask = (torch.rand(n, generator=gen, device="cuda") < 0.1).to(torch.uint8)
    got = float(C.conduit_staleness_iso(C.KvCache(k, v, hq), batch, q, mask, z, kappa)[0])
    scale = kappa * (v[0, 0].float().square().sum(1) / d).sqrt() * (mask == 0)
    p = torch.softmax(q[0].reshape(-1, d).double() @ k[0, 0].double().T / d ** 0.5, 1)
    want = sum(float((p @ (scale[:, None] * z[m, 0, 0].float()).bfloat16().double()).bfloat16().double().square().sum())
               for m in range(M)) / M
    assert abs(got / want - 1) <= 5e-6, got / want - 1
