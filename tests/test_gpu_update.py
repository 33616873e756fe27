"""GPU parity of the policy-update calls against the oracle: clipped GRPO / DAPO loss and its gradient (fp32 per
token: 1e-6 relative to the weight scale), and the lm_head log-prob backward (dz is rounded to bf16 before the two
contractions: 1e-2 of the tensor's largest entry, 5e-3 in relative Frobenius norm)."""
import numpy as np
import pytest
import torch

import oracle
from oracle import update as ou
from paper_2603_24840_b200 import binding as B
from paper_2603_24840_b200 import synth
from paper_2603_24840_b200 import update as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    assert B.arrol_poll_status(c, raise_on_error=False) == 0
    c.close()


def dv(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("S,lo,hi,agg_mode,beta", [(16, 1, 40, 0, 0.0), (300, 5, 900, 1, 0.0), (64, 1, 300, 0, 0.04),
                                                   (7, 0, 3, 1, 0.1)])
def test_policy_loss_matches_oracle(ctx, S, lo, hi, agg_mode, beta):
    g = np.random.default_rng(S)
    ell = g.integers(lo, hi + 1, size=S)
    ell[0] = max(ell[0], 1)
    cu = np.concatenate([[0], np.cumsum(ell)]).astype(np.int64)
    T = int(cu[-1])
    logp_old = (-g.random(T) * 4).astype(np.float32)
    logp = (logp_old + g.normal(0, 0.25, size=T)).astype(np.float32)
    ref = (logp_old + g.normal(0, 0.2, size=T)).astype(np.float32)
    adv = np.repeat(g.normal(size=S), ell).astype(np.float32)
    seq = np.repeat(np.arange(S), ell).astype(np.int32)
    loss_ref, grad_ref = ou.policy_loss(logp, logp_old, adv, cu, logp_ref=ref if beta else None, eps_low=0.2,
                                        eps_high=0.28, beta=beta, agg_mode=agg_mode)
    cap = T + 5
    pad = lambda a, fill: np.concatenate([a, np.full(cap - T, fill, a.dtype)])
    grad = torch.full((cap,), 77.0, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    U.arrol_policy_loss(ctx, dv(pad(logp, 0)), dv(pad(logp_old, 0)), dv(pad(adv, 0)), dv(pad(seq, 0)), dv(cu),
                        dv(np.array([S, T], np.int64)), cap, grad, loss, logp_ref=dv(pad(ref, 0)) if beta else None,
                        eps_low=0.2, eps_high=0.28, beta=beta, agg_mode=agg_mode)
    torch.cuda.synchronize()
    w_max = 1.0 / T if agg_mode else 1.0 / (S * max(1, ell[ell > 0].min()))
    assert np.abs(grad.cpu().numpy()[:T] - grad_ref).max() <= 2e-5 * w_max * max(1.0, np.abs(adv).max())
    assert np.all(grad.cpu().numpy()[T:] == 77.0)
    assert abs(loss.item() - loss_ref) <= 1e-5 * max(1.0, abs(loss_ref))


def _backward_case(ctx, T, d, V, seed, T_live=None, inv_temp=1.0):
    g = np.random.default_rng(seed)
    H = torch.from_numpy(g.normal(size=(T, d)).astype(np.float32)).to(torch.bfloat16)
    W = torch.from_numpy(g.normal(0, 0.08, size=(V, d)).astype(np.float32)).to(torch.bfloat16)
    y = g.integers(0, V, size=T).astype(np.int32)
    y[:4] = [0, V - 1, -1, min(255, V - 1)][:min(4, T)] if T >= 4 else y[:4]
    gl = g.normal(size=T).astype(np.float32)
    n = T if T_live is None else T_live
    dH_ref, dW_ref = ou.lm_head_backward(synth.as_oracle_array(H[:n]), synth.as_oracle_array(W), y[:n],
                                         gl[:n].astype(np.float64), inv_temp=inv_temp)
    Hd, Wd, yd = H.cuda(), W.cuda(), dv(y)
    if T_live is not None:
        Hd[T_live:] = float("nan")               # rows past the live tokens may hold anything
    logp = torch.empty(T, device="cuda")
    lse = torch.empty(T, device="cuda")
    d_T = None if T_live is None else torch.tensor([T_live], dtype=torch.int64, device="cuda")
    ws = torch.empty(B.arrol_token_logprob_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
    B.arrol_token_logprob(ctx, Hd, Wd, yd, T, d, V, logp, ws, lse=lse, d_T=d_T, inv_temperature=inv_temp)
    dH = torch.full((T, d), 9.0, device="cuda")
    dW = torch.full((V, d), 9.0, device="cuda")
    ws2 = torch.empty(U.arrol_lm_head_backward_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
    U.arrol_lm_head_backward(ctx, Hd, Wd, yd, dv(gl), lse, T, d, V, dH, dW, ws2, d_T=d_T, inv_temperature=inv_temp)
    torch.cuda.synchronize()
    assert B.arrol_poll_status(ctx, raise_on_error=False) == 0
    dH, dW = dH.cpu().numpy().astype(np.float64), dW.cpu().numpy().astype(np.float64)
    for got, ref in ((dH[:n], dH_ref), (dW, dW_ref)):
        scale = np.abs(ref).max()
        assert np.abs(got - ref).max() <= 1e-2 * scale
        assert np.linalg.norm(got - ref) <= 5e-3 * np.linalg.norm(ref)
    assert np.all(dH[:n][y[:n] < 0] == 0.0)                    # ignored positions carry no gradient
    return dH, n


@pytest.mark.parametrize("T,d,V", [(1, 64, 256), (130, 64, 300), (300, 192, 1000), (700, 256, 3001), (257, 200, 37)])
def test_lm_head_backward_matches_oracle(ctx, T, d, V):
    _backward_case(ctx, T, d, V, seed=T + V)


def test_lm_head_backward_many_chunks_temperature_and_device_T(ctx):
    _backward_case(ctx, 10000, 64, 512, seed=1)               # two token chunks: dW accumulates across them
    _backward_case(ctx, 400, 128, 1024, seed=2, inv_temp=0.6)
    dH, n = _backward_case(ctx, 600, 128, 1024, seed=3, T_live=333)
    assert np.all(dH[n:] == 0.0)                               # rows past T inside a processed chunk are zero
    _backward_case(ctx, 600, 128, 1024, seed=4, T_live=320)    # live rows end exactly on a 64-row block
    _backward_case(ctx, 9700, 64, 512, seed=5, T_live=9500)    # the partly live block is in the second chunk


# edges of the pairs' 256 x 256 tiles: a full tile and one row more, one vocabulary column in the last chunk, a last column tile
# of 8 (half a tile for the MMA) and of 136, a chunk of 37 tiles and one row more, dead rows in whole tiles of their own
@pytest.mark.parametrize("T,d,V,T_live", [(256, 64, 256, None), (257, 264, 2305, None), (129, 392, 640, None),
                                          (9473, 72, 300, None), (1100, 136, 520, 257), (9472, 64, 257, 9471)])
def test_lm_head_backward_at_the_edges_of_a_pairs_tile(ctx, T, d, V, T_live):
    dH, n = _backward_case(ctx, T, d, V, seed=T + d, T_live=T_live)
    assert np.all(dH[n:] == 0.0)


# tile orders of wide heads: columns in two uneven groups (6 + 5 tiles, the last one ragged or whole), token tiles in two groups
# (22 pair tiles, 19 to a group); gradients on sampled rows, so that the oracle stays cheap
@pytest.mark.parametrize("d", [2808, 2816])
def test_lm_head_backward_with_groups_of_tiles(ctx, d):
    T, V = 5500, 600
    g = np.random.default_rng(d)
    H = torch.from_numpy(g.normal(size=(T, d)).astype(np.float32)).to(torch.bfloat16)
    W = torch.from_numpy(g.normal(0, 0.02, size=(V, d)).astype(np.float32)).to(torch.bfloat16)
    y = g.integers(0, V, size=T).astype(np.int32)
    rows = np.unique(np.concatenate([[0, 255, 256, 19 * 256 - 1, 19 * 256, T - 1], g.integers(0, T, size=40)]))
    gl = np.zeros(T, np.float32)
    gl[rows] = g.normal(size=len(rows))
    dH_ref, dW_ref = ou.lm_head_backward(synth.as_oracle_array(H[rows]), synth.as_oracle_array(W), y[rows], gl[rows].astype(np.float64))
    Hd, Wd, yd = H.cuda(), W.cuda(), dv(y)
    logp, lse = torch.empty(T, device="cuda"), torch.empty(T, device="cuda")
    ws = torch.empty(B.arrol_token_logprob_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
    B.arrol_token_logprob(ctx, Hd, Wd, yd, T, d, V, logp, ws, lse=lse)
    dH, dW = torch.full((T, d), 9.0, device="cuda"), torch.full((V, d), 9.0, device="cuda")
    ws2 = torch.empty(U.arrol_lm_head_backward_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
    U.arrol_lm_head_backward(ctx, Hd, Wd, yd, dv(gl), lse, T, d, V, dH, dW, ws2)
    torch.cuda.synchronize()
    dH, dW = dH.cpu().numpy().astype(np.float64), dW.cpu().numpy().astype(np.float64)
    for got, ref in ((dH[rows], dH_ref), (dW, dW_ref)):
        assert np.abs(got - ref).max() <= 1e-2 * np.abs(ref).max()
        assert np.linalg.norm(got - ref) <= 5e-3 * np.linalg.norm(ref)
    assert np.all(np.delete(dH, rows, axis=0) == 0.0)


# tiles that are cut: all of dH along K, with a last column tile of half width (600) or one column tile and dead rows (900); 10 tiles
# beyond a whole wave of 74 along K (7,000); 37 tiles without room for partial sums (9,472); a second chunk whose tiles are cut while
# dW is added to (9,900)
@pytest.mark.parametrize("T,d,V,T_live", [(600, 320, 20000, None), (900, 72, 9001, 777), (7000, 768, 12000, None), (9472, 256, 700, None),
                                          (257, 520, 5000, 256), (9900, 136, 9001, 9800)])
def test_lm_head_backward_with_cut_tiles(ctx, T, d, V, T_live):
    g = np.random.default_rng(T + d)
    n = T if T_live is None else T_live
    H = torch.from_numpy(g.normal(size=(T, d)).astype(np.float32)).to(torch.bfloat16)
    W = torch.from_numpy(g.normal(0, 0.04, size=(V, d)).astype(np.float32)).to(torch.bfloat16)
    y = g.integers(0, V, size=T).astype(np.int32)
    rows = np.unique(np.concatenate([[0, 255, n - 1], g.integers(0, n, size=40)]))
    gl = np.zeros(T, np.float32)
    gl[rows] = g.normal(size=len(rows))
    dH_ref, dW_ref = ou.lm_head_backward(synth.as_oracle_array(H[rows]), synth.as_oracle_array(W), y[rows], gl[rows].astype(np.float64))
    Hd, Wd, yd = H.cuda(), W.cuda(), dv(y)
    Hd[n:] = float("nan")
    d_T = torch.tensor([n], dtype=torch.int64, device="cuda")
    logp, lse = torch.empty(T, device="cuda"), torch.empty(T, device="cuda")
    ws = torch.empty(B.arrol_token_logprob_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
    B.arrol_token_logprob(ctx, Hd, Wd, yd, T, d, V, logp, ws, lse=lse, d_T=d_T)
    outs = []
    for _ in range(2):
        dH, dW = torch.full((T, d), 9.0, device="cuda"), torch.full((V, d), 9.0, device="cuda")
        ws2 = torch.full((U.arrol_lm_head_backward_workspace(ctx, T, d, V),), 255, dtype=torch.uint8, device="cuda")
        U.arrol_lm_head_backward(ctx, Hd, Wd, yd, dv(gl), lse, T, d, V, dH, dW, ws2, d_T=d_T)
        torch.cuda.synchronize()
        outs.append((dH, dW))
    assert B.arrol_poll_status(ctx, raise_on_error=False) == 0
    assert all(torch.equal(a, b) for a, b in zip(*outs))
    dH, dW = dH.cpu().numpy().astype(np.float64), dW.cpu().numpy().astype(np.float64)
    for got, ref in ((dH[rows], dH_ref), (dW, dW_ref)):
        assert np.abs(got - ref).max() <= 1e-2 * np.abs(ref).max()
        assert np.linalg.norm(got - ref) <= 5e-3 * np.linalg.norm(ref)
    assert np.all(np.delete(dH, rows, axis=0) == 0.0)


def test_lm_head_backward_with_a_dead_chunk_after_a_live_one(ctx):
    _backward_case(ctx, 9700, 72, 300, seed=6, T_live=300)


def test_lm_head_backward_without_a_live_token(ctx):
    T, d, V = 300, 136, 700
    Z = torch.full((T, d), float("nan"), device="cuda", dtype=torch.bfloat16)
    W = torch.zeros((V, d), device="cuda", dtype=torch.bfloat16)
    f = torch.zeros(T, device="cuda")
    dH, dW = torch.full((T, d), 9.0, device="cuda"), torch.full((V, d), 9.0, device="cuda")
    ws = torch.empty(U.arrol_lm_head_backward_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
    U.arrol_lm_head_backward(ctx, Z, W, torch.zeros(T, dtype=torch.int32, device="cuda"), f, f, T, d, V, dH, dW, ws,
                             d_T=torch.zeros(1, dtype=torch.int64, device="cuda"))
    torch.cuda.synchronize()
    assert torch.all(dW == 0.0) and torch.all((dH == 0.0) | (dH == 9.0))


def test_lm_head_backward_workspace_serves_any_number_of_tokens(ctx):
    for d, V in ((8, 300), (72, 301), (4096, 151936)):
        want = 9472 * 2 * ((V + 7) // 8 * 8) + 128 * d
        assert all(U.arrol_lm_head_backward_workspace(ctx, T, d, V) == want for T in (1, 9472, 9473, 60000, 1 << 30))
    for d, T, T_live in ((8, 9700, 9500), (16, 20000, 18945), (24, 9473, None)):   # the narrowest rows, several chunks
        _backward_case(ctx, T, d, 300, seed=d, T_live=T_live)


# 16 tiles a pair on 74 pairs, the last that are not kept in step, and two tiles more, whose counters are cleared first
@pytest.mark.parametrize("V", [592 * 256, 592 * 256 + 1])
def test_lm_head_backward_does_not_depend_on_the_workspace(ctx, V):
    T, d = 512, 64
    g = torch.Generator(device="cuda").manual_seed(V)
    H = torch.randn((T, d), generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn((V, d), generator=g, device="cuda") * 0.2).to(torch.bfloat16)
    y = torch.randint(0, V, (T,), generator=g, device="cuda", dtype=torch.int32)
    gl = torch.randn(T, generator=g, device="cuda")
    z = H.double() @ W.double().T
    lse = torch.logsumexp(z, dim=1)
    ws = torch.empty(U.arrol_lm_head_backward_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
    got = []
    for byte in (0, 255):
        ws.fill_(byte)
        dH, dW = torch.full((T, d), 9.0, device="cuda"), torch.full((V, d), 9.0, device="cuda")
        U.arrol_lm_head_backward(ctx, H, W, y, gl, lse.float(), T, d, V, dH, dW, ws)
        got.append((dH, dW))
    assert B.arrol_poll_status(ctx) == 0
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    dz = -torch.exp(z - lse[:, None]) * gl[:, None].double()
    dz[torch.arange(T, device="cuda"), y.long()] += gl.double()
    # dz is held in bf16: 2^-9 of each term; the fp32 logits, exponentials and sums err by far less than the other 2^-9
    for out, ref, bound in ((got[0][0], dz @ W.double(), dz.abs() @ W.double().abs()), (got[0][1], dz.T @ H.double(), dz.abs().T @ H.double().abs())):
        assert bool(((out.double() - ref).abs() <= 2.0 ** -8 * bound + 1e-6).all())


def test_lm_head_backward_clears_its_counters_past_16_tiles_a_pair(ctx):
    """One kernel more, which clears the counters that keep the pairs in step: results do not show whether it ran, launches do."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the line is drawn by the number of SMs")
    T, d = 512, 64
    H, gl = torch.zeros((T, d), dtype=torch.bfloat16, device="cuda"), torch.zeros(T, device="cuda")
    y = torch.zeros(T, dtype=torch.int32, device="cuda")
    launches = []
    for V in (592 * 256, 592 * 256 + 1):
        ws = torch.empty(U.arrol_lm_head_backward_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
        W, dW = torch.zeros((V, d), dtype=torch.bfloat16, device="cuda"), torch.empty((V, d), device="cuda")
        before = B.arrol_launch_count(ctx)
        U.arrol_lm_head_backward(ctx, H, W, y, gl, gl, T, d, V, torch.empty((T, d), device="cuda"), dW, ws)
        launches.append(B.arrol_launch_count(ctx) - before)
    assert B.arrol_poll_status(ctx) == 0
    assert launches[1] == launches[0] + 1


def test_lm_head_backwards_in_flight_on_two_streams(ctx):
    """Each launch fills the GPU and keeps its pairs of blocks in step; two at once get a part of the SMs each, so neither can
    count on all of its pairs running."""
    T, d, V = 6000, 1024, 12000
    g = np.random.default_rng(3)
    streams = [torch.cuda.Stream() for _ in range(2)]
    calls = []
    for i in range(2):
        H = torch.from_numpy(g.normal(size=(T, d)).astype(np.float32)).to(torch.bfloat16).cuda()
        W = torch.from_numpy(g.normal(0, 0.02, size=(V, d)).astype(np.float32)).to(torch.bfloat16).cuda()
        y = dv(g.integers(0, V, size=T).astype(np.int32))
        gl = dv(g.normal(size=T).astype(np.float32))
        lse = torch.full((T,), float(np.log(V)) + 0.2, device="cuda")
        out = [torch.full((T, d), 9.0, device="cuda"), torch.full((V, d), 9.0, device="cuda")]
        ws = torch.empty(U.arrol_lm_head_backward_workspace(ctx, T, d, V), dtype=torch.uint8, device="cuda")
        calls.append((H, W, y, gl, lse, out, ws))

    def run(i, stream=None):
        H, W, y, gl, lse, out, ws = calls[i]
        U.arrol_lm_head_backward(ctx, H, W, y, gl, lse, T, d, V, out[0], out[1], ws, stream=stream)

    want = []
    for i in range(2):
        run(i)
        torch.cuda.synchronize()
        want.append([t.clone() for t in calls[i][5]])
        for t in calls[i][5]:
            t.fill_(9.0)
    torch.cuda.synchronize()
    for _ in range(6):
        for i in range(2):
            run(i, streams[i])
    torch.cuda.synchronize()
    assert B.arrol_poll_status(ctx, raise_on_error=False) == 0
    for i in range(2):
        assert all(torch.equal(a, b) for a, b in zip(calls[i][5], want[i]))


def test_update_argument_errors(ctx):
    z = torch.zeros(8, device="cuda")
    with pytest.raises(B.ArrolError) as e:
        U.arrol_lm_head_backward(ctx, z, z, z, z, z, 8, 60, 64, z, z, None)
    assert e.value.code == -2
    with pytest.raises(B.ArrolError) as e:
        U.arrol_lm_head_backward(ctx, z, z, z, z, z, 8, 64, 64, z, torch.zeros(64 * 64, device="cuda"), None)
    assert e.value.code == -3
    with pytest.raises(B.ArrolError) as e:
        U.arrol_policy_loss(ctx, z, z, z, None, z, z, 8, z, torch.zeros(1, dtype=torch.float64, device="cuda"),
                            agg_mode=2)
    assert e.value.code == -2
