"""CPU-only checks of the step's orchestration: which buffers the calls are given."""
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
