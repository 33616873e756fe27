"""arrol_prune_step (score -> select -> compact in one call) gives exactly what the three calls give."""
import pytest
import torch

from paper_2603_24840_b200 import binding as B
from paper_2603_24840_b200 import synth
from paper_2603_24840_b200.pipeline import PruneRebatch, host_inputs

pytestmark = pytest.mark.gpu

BAD_INDEX = 16


@pytest.mark.parametrize("name,rows", [("tiny", True), ("mini", True), ("mini", False), ("profile-mlp", True)])
def test_one_call_prune_step_equals_three_calls(name, rows):
    w = synth.WORKLOADS[name]
    pr = PruneRebatch(w, inputs=host_inputs(w))
    pr.prune_step(with_rows=rows)
    torch.cuda.synchronize()
    want = {k: getattr(pr, k).clone() for k in ("score", "prob", "q", "bin", "keep", "survivor_idx", "cu_seqlens", "adv",
                                                  "d_num", "dst_tokens", "tok_adv", "tok_seq", "dst_rows")}
    S, T = pr.counts()
    for k in want:
        getattr(pr, k).fill_(0)
    B.arrol_prune_step(pr.ctx, pr.prune_step_args(with_rows=rows))
    torch.cuda.synchronize()
    assert pr.counts() == (S, T)
    for k in ("score", "prob", "q", "bin", "keep", "d_num"):
        assert torch.equal(getattr(pr, k), want[k]), k
    for k in ("survivor_idx", "adv"):
        assert torch.equal(getattr(pr, k)[:S], want[k][:S]), k
    assert torch.equal(pr.cu_seqlens[:S + 1], want["cu_seqlens"][:S + 1])
    for k in ("dst_tokens", "tok_adv", "tok_seq"):
        assert torch.equal(getattr(pr, k)[:T], want[k][:T]), k
    if rows:
        assert torch.equal(pr.dst_rows[:T], want["dst_rows"][:T])
    assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == 0
    pr.ctx.close()


@pytest.mark.parametrize("name,rows", [("mini", True), ("profile-mlp", False)])
def test_prune_step_replayed_from_a_cuda_graph(name, rows):
    """The step allocates nothing and never synchronises, so it can be captured once and replayed; the kernels'
    programmatic launch dependencies survive the capture.  Replays give what the eager call gives."""
    w = synth.WORKLOADS[name]
    pr = PruneRebatch(w, inputs=host_inputs(w))
    args = pr.prune_step_args(with_rows=rows)
    B.arrol_prune_step(pr.ctx, args)
    torch.cuda.synchronize()
    keys = ["score", "q", "keep", "survivor_idx", "cu_seqlens", "adv", "d_num", "dst_tokens", "tok_adv", "tok_seq"]
    if rows:
        keys.append("dst_rows")
    want = {k: getattr(pr, k).clone() for k in keys}
    S, T = pr.counts()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        B.arrol_prune_step(pr.ctx, args)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        B.arrol_prune_step(pr.ctx, args)
    for _ in range(2):
        for k in keys:
            getattr(pr, k).fill_(0)
        graph.replay()
        torch.cuda.synchronize()
        assert pr.counts() == (S, T)
        for k in ("score", "q", "keep", "d_num"):
            assert torch.equal(getattr(pr, k), want[k]), k
        for k in ("survivor_idx", "adv"):
            assert torch.equal(getattr(pr, k)[:S], want[k][:S]), k
        assert torch.equal(pr.cu_seqlens[:S + 1], want["cu_seqlens"][:S + 1])
        for k in ("dst_tokens", "tok_adv", "tok_seq"):
            assert torch.equal(getattr(pr, k)[:T], want[k][:T]), k
        if rows:
            assert torch.equal(pr.dst_rows[:T], want["dst_rows"][:T])
    assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == 0
    del graph
    pr.ctx.close()


def test_back_to_back_steps_never_read_the_previous_steps_results():
    """The kernels of a step start while their predecessor is still running (programmatic dependent launch) and must
    wait before they read its results.  Two steps with different heads are issued back to back without a host
    synchronisation; the buffers must hold exactly what the second step alone produces, in either order."""
    w = synth.WORKLOADS["profile-mlp"]
    pr = PruneRebatch(w, inputs=host_inputs(w), with_rows=False)
    heads = [pr.head, dict(pr.head)]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    heads[1]["w2"] = (pr.head["w2"].float() * (torch.rand(w.h, generator=gen, device="cuda") * 4 - 2)).to(pr.head["w2"].dtype)
    keys = ("score", "q", "keep", "survivor_idx", "cu_seqlens", "adv", "d_num", "dst_tokens", "tok_seq")
    refs = []
    for hd in heads:
        pr.head = hd
        B.arrol_prune_step(pr.ctx, pr.prune_step_args(with_rows=False))
        torch.cuda.synchronize()
        refs.append(({k: getattr(pr, k).clone() for k in keys}, pr.counts()))
    assert not torch.equal(refs[0][0]["keep"], refs[1][0]["keep"])          # the two steps really differ
    args = []
    for hd in heads:
        pr.head = hd
        args.append(pr.prune_step_args(with_rows=False))
    for first, second in ((0, 1), (1, 0), (0, 1)):
        for _ in range(3):
            B.arrol_prune_step(pr.ctx, args[first])
            B.arrol_prune_step(pr.ctx, args[second])
        torch.cuda.synchronize()
        want, (S, T) = refs[second]
        assert pr.counts() == (S, T)
        for k in ("score", "q", "keep", "d_num"):
            assert torch.equal(getattr(pr, k), want[k]), k
        for k in ("survivor_idx", "adv"):
            assert torch.equal(getattr(pr, k)[:S], want[k][:S]), k
        assert torch.equal(pr.cu_seqlens[:S + 1], want["cu_seqlens"][:S + 1])
        for k in ("dst_tokens", "tok_seq"):
            assert torch.equal(getattr(pr, k)[:T], want[k][:T]), k
    assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == 0
    pr.ctx.close()


@pytest.mark.parametrize("P,G,K", [(1, 1, 1), (7, 1, 1), (5, 3, 2), (9, 5, 1), (3, 32, 7), (40, 32, 16), (200, 4, 4), (333, 2, 1),
                                   (150, 16, 8), (1000, 2, 1)])
def test_fused_prune_step_over_group_shapes(P, G, K):
    """Group sizes that are no power of two, one group per block and many, more blocks than one wave of the chained
    scan would hold (the call then takes the three separate launches): always what the three calls give."""
    import dataclasses
    w = dataclasses.replace(synth.WORKLOADS["mini"], P=P, G=G, K=K, h=0, seed=100 + P + G)
    pr = PruneRebatch(w, inputs=host_inputs(w), with_rows=False)
    pr.prune_step(with_rows=False)
    torch.cuda.synchronize()
    keys = ("score", "prob", "q", "bin", "keep", "survivor_idx", "cu_seqlens", "adv", "d_num", "dst_tokens", "tok_adv", "tok_seq")
    want = {k: getattr(pr, k).clone() for k in keys}
    S, T = pr.counts()
    assert S == P * K
    for _ in range(2):                                  # twice: the chained scan's published totals are cleared in between
        for k in keys:
            getattr(pr, k).fill_(0)
        B.arrol_prune_step(pr.ctx, pr.prune_step_args(with_rows=False))
        torch.cuda.synchronize()
        assert pr.counts() == (S, T)
        for k in ("score", "prob", "q", "bin", "keep", "d_num"):
            assert torch.equal(getattr(pr, k), want[k]), k
        for k in ("survivor_idx", "adv"):
            assert torch.equal(getattr(pr, k)[:S], want[k][:S]), k
        assert torch.equal(pr.cu_seqlens[:S + 1], want["cu_seqlens"][:S + 1])
        for k in ("dst_tokens", "tok_adv", "tok_seq"):
            assert torch.equal(getattr(pr, k)[:T], want[k][:T]), k
    assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == 0
    pr.ctx.close()


ROLLOUT_OUT, SURVIVOR_OUT, TOKEN_OUT = ("score", "prob", "q", "bin", "keep"), ("survivor_idx", "adv"), ("dst_tokens", "tok_adv", "tok_seq")


def _snapshot(pr):
    return {k: getattr(pr, k).clone() for k in ROLLOUT_OUT + SURVIVOR_OUT + TOKEN_OUT + ("cu_seqlens", "d_num")}


def _clear(pr):
    for k in ROLLOUT_OUT + SURVIVOR_OUT + TOKEN_OUT + ("cu_seqlens", "d_num"):
        getattr(pr, k).fill_(0)


def _assert_equals(pr, want):
    """Everything that a call writes: what lies past the survivors and their tokens belongs to nobody."""
    S, T = (int(x) for x in want["d_num"].cpu())
    assert pr.counts() == (S, T)
    for k in ROLLOUT_OUT:
        assert torch.equal(getattr(pr, k), want[k]), k
    for k in SURVIVOR_OUT:
        assert torch.equal(getattr(pr, k)[:S], want[k][:S]), k
    assert torch.equal(pr.cu_seqlens[:S + 1], want["cu_seqlens"][:S + 1])
    for k in TOKEN_OUT:
        assert torch.equal(getattr(pr, k)[:T], want[k][:T]), k


def test_fused_prune_steps_of_changing_size_on_one_context():
    """The blocks of a call find each other's totals in the context's chain.  Calls of 1 to 290 blocks (the last one: an MLP
    head, blocks of two warps) follow one another on one context without a host synchronisation: whatever a call leaves
    there must not be taken for a later and larger call's totals."""
    import dataclasses
    import random
    ctx = B.Context(0)
    states = []
    for P, h in ((1, 0), (2, 0), (40, 0), (300, 0), (580, 0), (450, 24)):
        w = dataclasses.replace(synth.WORKLOADS["mini"], P=P, G=16, K=8, h=h, seed=P)
        pr = PruneRebatch(w, inputs=host_inputs(w), with_rows=False, ctx=ctx)
        pr.prune_step(with_rows=False)
        torch.cuda.synchronize()
        states.append((pr, pr.prune_step_args(with_rows=False), _snapshot(pr)))
    rng = random.Random(3)
    for _ in range(20):
        for pr, _, _ in states:
            _clear(pr)
        order = [rng.randrange(len(states)) for _ in range(40)] + rng.sample(range(len(states)), len(states))
        for i in order:
            B.arrol_prune_step(ctx, states[i][1])
        torch.cuda.synchronize()
        for pr, _, want in states:
            _assert_equals(pr, want)
    assert B.arrol_poll_status(ctx, raise_on_error=False) == 0
    ctx.close()


def test_an_expired_wait_of_the_fused_prune_step_leaves_nothing_to_follow():
    """A block that gives up waiting for the totals before it leaves holes in the survivors' list.  The call reports it, as
    {0, 0} survivors and tokens, gathers nothing, and leaves nothing behind for the next call."""
    import dataclasses
    w = dataclasses.replace(synth.WORKLOADS["mini"], P=580, G=16, K=8, h=0, seed=12)
    pr = PruneRebatch(w, inputs=host_inputs(w), with_rows=False)
    args = pr.prune_step_args(with_rows=False)
    pr.prune_step(with_rows=False)
    torch.cuda.synchronize()
    want = _snapshot(pr)
    expired = 0
    for _ in range(8):
        _clear(pr)
        B.arrol_test_hook(pr.ctx, B.HOOK_SPIN_LIMIT, 1)          # one look at every total
        B.arrol_prune_step(pr.ctx, args)
        torch.cuda.synchronize()
        if B.arrol_poll_status(pr.ctx, raise_on_error=False) & B.DEV_WAIT_EXPIRED:
            expired += 1
            assert pr.counts() == (0, 0)
            assert all(int(getattr(pr, k).abs().max()) == 0 for k in TOKEN_OUT)
        B.arrol_test_hook(pr.ctx, B.HOOK_SPIN_LIMIT, 0)
        _clear(pr)
        B.arrol_prune_step(pr.ctx, args)
        torch.cuda.synchronize()
        _assert_equals(pr, want)
    assert expired > 0
    assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == 0
    pr.ctx.close()


# rows past the 4 KB that a warp holds in registers: one vector more (2,056 bf16, 1,032 fp32), twice as many, a block of few warps, and
# rows too long to be staged for a block of 32 of them
@pytest.mark.parametrize("P,G,K,d,dtype", [(9, 16, 8, 2056, "bf16"), (150, 16, 8, 4096, "bf16"), (1, 3, 1, 3000, "bf16"),
                                           (5, 4, 2, 1032, "f32"), (3, 32, 7, 9000, "f32")])
def test_fused_prune_step_on_wide_rows(P, G, K, d, dtype):
    import dataclasses
    w = dataclasses.replace(synth.WORKLOADS["mini"], P=P, G=G, K=K, h=0, d=d, dtype=dtype, seed=P + d)
    pr = PruneRebatch(w, inputs=host_inputs(w), with_rows=False)
    pr.prune_step(with_rows=False)
    torch.cuda.synchronize()
    want = _snapshot(pr)
    _clear(pr)
    B.arrol_prune_step(pr.ctx, pr.prune_step_args(with_rows=False))
    torch.cuda.synchronize()
    _assert_equals(pr, want)
    assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == 0
    pr.ctx.close()


def test_fused_prune_step_on_wide_rows_checks_their_numbers():
    """Rows that go through shared memory (d = 4,096): numbers outside the source are reported and scored as zeros, as by the
    three calls, and their rows are not asked for."""
    import dataclasses
    w = dataclasses.replace(synth.WORKLOADS["mini"], P=20, G=16, K=8, h=0, d=4096, seed=41)
    pr = PruneRebatch(w, inputs=host_inputs(w), with_rows=False)
    pr.row_index[5], pr.row_index[100], pr.row_index[319] = pr.T_src, -1, 1 << 40
    B.arrol_set_source_rows(pr.ctx, pr.T_src)
    pr.prune_step(with_rows=False)
    torch.cuda.synchronize()
    assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == BAD_INDEX
    want = _snapshot(pr)
    _clear(pr)
    B.arrol_prune_step(pr.ctx, pr.prune_step_args(with_rows=False))
    torch.cuda.synchronize()
    _assert_equals(pr, want)
    assert B.arrol_poll_status(pr.ctx, raise_on_error=False) == BAD_INDEX
    pr.ctx.close()
