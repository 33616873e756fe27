"""Non-finite values stay where they belong: a NaN logit makes its token's log-prob and log-sum-exp NaN wherever in the
vocabulary it stands, a logit of minus infinity only leaves the sum, and other tokens keep their bits."""
import numpy as np
import pytest
import torch

from paper_2603_24840_b200 import binding as B

pytestmark = pytest.mark.gpu


def _logprob(ctx, H, W, y):
    (T, d), V = H.shape, W.shape[0]
    ws = torch.empty(B.arrol_token_logprob_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
    logp, lse = torch.full((T,), 7.0, device="cuda"), torch.full((T,), 7.0, device="cuda")
    B.arrol_token_logprob(ctx, H, W, y, T, d, V, logp, ws, lse=lse)
    torch.cuda.synchronize()
    assert B.arrol_poll_status(ctx, raise_on_error=False) == 0
    return logp, lse


# single blocks and pairs; V = 3,000 is 12 vocabulary segments of one chunk: a whole wave of token tiles and a cut rest
@pytest.mark.parametrize("T,d,V", [(10000, 64, 3000), (10000, 520, 3000), (300, 640, 40000)])
def test_logprob_of_non_finite_logits(T, d, V):
    ctx = B.Context(0)
    g = np.random.default_rng(d)
    H = torch.from_numpy(np.abs(g.normal(size=(T, d))).astype(np.float32) + 0.05).to(torch.bfloat16).cuda()
    W = torch.from_numpy(g.normal(0, 0.3 / d ** 0.5, size=(V, d)).astype(np.float32)).to(torch.bfloat16).cuda()
    y = torch.from_numpy(g.integers(0, V, size=T).astype(np.int32)).cuda()
    want, want_lse = _logprob(ctx, H, W, y)
    nan, inf = float("nan"), float("inf")

    for rows in (slice(1024, 2048), slice(0, 256), slice(V - 30, V), slice(0, V), slice(1500, 1501)):
        bad = W.clone()
        bad[rows] = nan
        logp, lse = _logprob(ctx, H, bad, y)
        assert logp.isnan().all() and lse.isnan().all(), rows

    tokens = torch.tensor([0, 5, 131, T - 100, T - 1], device="cuda")
    bad = H.clone()
    bad[tokens] = nan
    logp, lse = _logprob(ctx, bad, W, y)
    good = torch.ones(T, dtype=torch.bool, device="cuda")
    good[tokens] = False
    assert logp[tokens].isnan().all() and lse[tokens].isnan().all()
    assert torch.equal(logp[good], want[good]) and torch.equal(lse[good], want_lse[good])

    for rows in (slice(1024, 2048), slice(0, 256), slice(V - 30, V)):        # every hidden value is positive
        bad = W.clone()
        bad[rows] = -inf
        logp, lse = _logprob(ctx, H, bad, y)
        live = torch.ones(V, dtype=torch.bool, device="cuda")
        live[rows] = False
        some = torch.arange(0, T, 97, device="cuda")
        z = H[some].double() @ W.double().t()
        ref = torch.logsumexp(z[:, live], dim=1)
        assert (lse[some].double() - ref).abs().max() <= 2e-3
        ref_p = torch.where(live[y[some].long()], z.gather(1, y[some].long()[:, None])[:, 0] - ref, torch.tensor(-inf, device="cuda").double())
        hit = ref_p.isinf()
        assert torch.equal(logp[some][hit], ref_p[hit].float()) and (logp[some][~hit].double() - ref_p[~hit]).abs().max() <= 2e-3
    ctx.close()
