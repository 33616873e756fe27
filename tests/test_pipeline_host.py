"""CPU-only checks of the step's orchestration: which buffers the calls are given."""
import pytest
import torch

from paper_2603_24840_b200 import binding as B
from paper_2603_24840_b200 import synth
from paper_2603_24840_b200.pipeline import PruneRebatch


def test_the_token_count_follows_a_rebound_d_num(monkeypatch):
    given = []
    monkeypatch.setattr(B, "arrol_token_logprob", lambda *a, **kw: given.append(kw["d_T"]))
    pr = PruneRebatch.__new__(PruneRebatch)
    pr.w = synth.WORKLOADS["tiny"]
    pr.ctx = pr.dst_rows = pr.W_vocab = pr.dst_tokens = pr.cap = pr.logp = pr.workspace = pr.lse = None
    for _ in range(2):
        pr.d_num = torch.zeros(2, dtype=torch.int64)
        pr.token_logprob()
        assert given[-1].data_ptr() == pr.d_num.data_ptr() + 8 and given[-1].numel() == 1


def _host_state(w):
    """A state whose buffers are host tensors: enough to look at the argument block that a step is given."""
    pr = PruneRebatch.__new__(PruneRebatch)
    pr.w, pr.ctx, pr.cap, pr.with_rows = w, None, 64, True
    pr.hidden_score = torch.zeros((64, w.d))
    pr.head = {"W1": torch.zeros(w.d), "b1": torch.zeros(1), "w2": None, "b2": None, "h": 0}
    for name in ("q_lut", "row_index", "score", "prob", "q", "bin", "keep", "lengths", "src_tok_off", "src_tokens", "src_rows", "rewards",
                 "dst_tokens", "dst_rows", "cu_seqlens", "survivor_idx", "adv", "tok_adv", "tok_seq", "W_vocab", "logp", "lse", "workspace"):
        setattr(pr, name, torch.zeros(8))
    pr.d_num = torch.zeros(2, dtype=torch.int64)
    return pr


def test_a_step_refuses_a_head_of_another_type(monkeypatch):
    calls = []
    monkeypatch.setattr(B, "arrol_prune_step", lambda *a: calls.append(a))
    monkeypatch.setattr(B, "arrol_token_logprob", lambda *a, **kw: None)
    pr = _host_state(synth.WORKLOADS["tiny"])
    pr.step()
    assert len(calls) == 1
    pr.head["W1"] = pr.head["W1"].to(torch.bfloat16)         # half as many bytes as the kernels would read
    with pytest.raises(TypeError):
        pr.step()
    assert len(calls) == 1
