"""Non-finite values stay where they belong: a NaN logit makes its token's log-prob and log-sum-exp NaN wherever in the
vocabulary it stands, a logit of minus infinity only leaves the sum, and other tokens keep their bits; a group with a
non-finite score keeps K members like any other, and the other groups keep theirs."""
import numpy as np
import pytest
import torch

from paper_2603_24840_b200 import binding as B
from paper_2603_24840_b200 import synth
from paper_2603_24840_b200.pipeline import PruneRebatch, host_inputs

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


@pytest.mark.parametrize("G,K", [(8, 4), (12, 6), (32, 1), (5, 5), (2, 1)])
def test_a_group_with_a_non_finite_score_keeps_exactly_k(G, K):
    """All keys of such a group are NaN or infinite: whoever goes, exactly K of it stay, and the other groups keep theirs."""
    ctx = B.Context(0)
    P = 9
    q = np.random.default_rng(G).random((P, G)).astype(np.float32)
    want = torch.full((P, G), 9, dtype=torch.uint8, device="cuda")
    B.arrol_select(ctx, torch.from_numpy(q).cuda(), P, G, K, 0.5, want)
    bad = q.copy()
    bad[1, 0] = np.nan
    bad[3, :] = np.nan
    bad[4, G - 1] = np.inf
    bad[7, G // 2] = -np.inf
    keep = torch.full((P, G), 9, dtype=torch.uint8, device="cuda")
    B.arrol_select(ctx, torch.from_numpy(bad).cuda(), P, G, K, 0.5, keep)
    torch.cuda.synchronize()
    assert (keep.sum(1) == K).all() and keep.max() <= 1
    rest = [0, 2, 5, 6, 8]
    assert torch.equal(keep[rest], want[rest])
    ctx.close()


@pytest.mark.parametrize("name", ["mini", "profile-mlp"])
def test_a_rollout_with_a_nan_hidden_row_leaves_the_other_groups_alone(name):
    w = synth.WORKLOADS[name]
    pr = PruneRebatch(w, inputs=host_inputs(w))
    pr.q_lut = None                                    # q is the score's sigmoid itself: NaN for a NaN row
    pr.prune_step()
    torch.cuda.synchronize()
    want = pr.keep.clone().view(w.P, w.G)
    bad = 2 * w.G + 1
    pr.hidden_score[pr.row_index[bad]] = float("nan")
    rest = [p for p in range(w.P) if p != 2]
    for run in (pr.prune_step, lambda: B.arrol_prune_step(pr.ctx, pr.prune_step_args())):
        pr.keep.fill_(9)
        run()
        torch.cuda.synchronize()
        keep = pr.keep.view(w.P, w.G)
        assert pr.q[bad].isnan()
        assert (keep.sum(1) == w.K).all() and torch.equal(keep[rest], want[rest])
        assert pr.counts()[0] == w.P * w.K
        assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == 0
    pr.ctx.close()
