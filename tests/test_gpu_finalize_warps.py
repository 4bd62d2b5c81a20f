"""The token reduction of large batches (a warp per 32 tokens) against that of small ones (a block), bit for bit.

The same requests are scored in one batch of 100 000 tokens and more, and in two halves below it. Requests of
fewer than 16 key tiles are scored alike in both, so the partials are equal; the reductions add in one order.
"""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,hkv,opts", [(15, 2, {}), (34, 1, {}), (15, 9, {"value_norm": "none"}),
                                             (16, 2, {"statistic": "rms"}), (17, 1, {"value_norm": "side_cache"})])
def test_large_batch_equals_its_halves(layers, hkv, opts):
    from paper_2609_05821_gb300 import _build
    _build.build()
    from paper_2609_05821_gb300 import conduit as C
    R, d, G = 100, 16, 3
    n_r = [983 + 17 * (r % 5) for r in range(R)]
    nq = [(1, 90, 41, 300)[r % 4] for r in range(R)]
    assert sum(n_r) >= 98304 and sum(n_r) * layers >= 1500000
    rng = torch.Generator(device="cuda").manual_seed(layers)
    draw = lambda *shape: torch.randn(shape, generator=rng, device="cuda").bfloat16()
    k, v, q = draw(layers, hkv, sum(n_r), d), draw(layers, hkv, sum(n_r), d), draw(layers, hkv * G, sum(nq), d)

    def score(r0, r1):
        cum = lambda x: [sum(x[r0:i]) for i in range(r0, r1 + 1)]
        t, qs = slice(sum(n_r[:r0]), sum(n_r[:r1])), slice(sum(nq[:r0]), sum(nq[:r1]))
        batch = C.Batch(cum(n_r), cum(n_r), list(range(r1 - r0 + 1)), cum(nq), device="cuda")
        kv = C.KvCache(k[:, :, t].contiguous(), v[:, :, t].contiguous(), hkv * G)
        more = {"vnorm": C.conduit_value_norms(kv, batch)} if opts.get("value_norm") == "side_cache" else {}
        return C.conduit_score_ex(kv, batch, q[:, :, qs].contiguous(), **opts, **more)

    halves = [torch.cat(x) for x in zip(score(0, 50), score(50, R))]
    assert all(torch.equal(a, b) for a, b in zip(score(0, R), halves))
