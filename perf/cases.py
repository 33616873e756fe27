"""Performance cases: what a training loop has this library do, through the calls it makes.

Seven kinds of pass, each over the range of sizes that its callers have:

  step     one prune-and-rebatch step on device-resident inputs: score, select, compact, token log-probs
           (`in_place`: the survivors' hidden rows are read from the source buffer, no packed copy)
  prune    the prune part of a step from one call (score, select, scan, token ids; `rows`: the hidden rows too)
  logprob  log-probs of a packed batch of tokens (old- or reference-policy scoring, evaluation)
  host     the whole step from pinned host buffers
  update   clipped objective and lm_head backward on a step's survivors
  learn    the online side of the method: score, stochastic survival rule, calibrator update, head training step
  vote     test time: log-probs with token confidence, trace confidence, head scores, rank-weighted vote

Inputs come from the package's own seeded generator (`synth`), so they have the distributions of its workloads.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2603_24840_b200 import binding as B
from paper_2603_24840_b200 import calibrator as C
from paper_2603_24840_b200 import confidence as CF
from paper_2603_24840_b200 import headtrain as HT
from paper_2603_24840_b200 import synth
from paper_2603_24840_b200 import update as U
from paper_2603_24840_b200 import voting as V
from paper_2603_24840_b200.pipeline import PruneRebatch, token_capacity

MAX_FLOPS = 3.6e14        # a drawn case contracts no more than the largest listed one
MAX_ROW_BYTES = 4.0e9     # hidden rows of one state
FP32, BF16 = "f32", "bf16"


def listed():
    return [
        # A debugging-size step with an fp32 head: every call is a few microseconds, so launches and host work count.
        _step("step-tiny", P=4, G=8, K=4, lo=96, hi=256, cutoff=64, d=256, V=4096, dtype=FP32),
        # The training step of the Llama-3.2-1B-shaped workload: 64 prompts x 8 rollouts, packed rows.
        _step("step-llama-1b", P=64, G=8, K=4, lo=512, hi=2048, cutoff=256, d=2048, V=128256),
        # A data-parallel rank's share of the DAPO-shaped step (d = 4096, MLP head), rows read in place.
        _step("step-dapo-rank", P=11, G=16, K=8, med=3000.0, hi=8192, cutoff=1024, d=4096, V=151936, h=512, in_place=True),
        # The prune part alone at the Qwen-3-4B-shaped batch: linear head, token ids only.
        _prune("prune-4b", P=128, G=16, K=8, med=2500.0, hi=8192, d=2560),
        # The same at the DAPO-shaped batch, all 4,096 rollouts in one call with the MLP head.
        _prune("prune-dapo", P=256, G=16, K=8, med=3000.0, hi=8192, d=4096, h=512),
        # Re-batching with the hidden-row plane: a quarter of the Qwen-3-1.7B-shaped step.
        _prune("prune-rows-1.7b", P=32, G=16, K=8, med=1500.0, hi=4096, d=2048, h=256, rows=True),
        # One long rollout scored by itself, ragged, with a sampling temperature.
        {"kind": "logprob", "name": "logprob-one-rollout", "T": 1777, "d": 2560, "V": 151936, "inv_temp": 1.25},
        # A step whose data lives in host memory: 8 prompts of the Qwen-3-1.7B-shaped workload.
        _step("host-1.7b", kind="host", P=8, G=16, K=8, med=1500.0, hi=4096, cutoff=512, d=2048, V=151936, h=256),
        # Policy update on a mini-batch of the Llama-shaped step (GRPO aggregation with a KL term).
        _update("update-llama-1b", P=16, G=8, K=4, lo=512, hi=2048, cutoff=256, d=2048, V=128256, agg=0, beta=0.04),
        # A micro-batch of the DAPO-shaped update: one prompt, token-mean aggregation, clip-higher.
        _update("update-dapo-micro", P=1, G=16, K=8, med=3000.0, hi=8192, cutoff=1024, d=4096, V=151936, agg=1, beta=0.0),
        # Online learning at the Qwen-3-1.7B-shaped batch: 2,048 rollouts, MLP head, 128 bins.
        {"kind": "learn", "name": "learn-1.7b", "N": 2048, "d": 2048, "h": 256, "dtype": BF16, "B": 128, "cap": 2048},
        # Test-time voting on two questions with 16 candidates each.
        {"kind": "vote", "name": "vote-4b", "P": 2, "G": 16, "med": 2500.0, "hi": 8192, "d": 2560, "V": 151936, "window": 2048,
         "mode": 2},
    ]


def _step(name, kind="step", P=1, G=8, K=4, lo=0, hi=2048, med=0.0, cutoff=256, d=2048, V=128256, h=0, dtype=BF16,
          in_place=False):
    return {"kind": kind, "name": name, "P": P, "G": G, "K": K, "lo": lo, "hi": hi, "med": med, "cutoff": cutoff, "d": d, "V": V,
            "h": h, "dtype": dtype, "in_place": in_place}


def _prune(name, P, G, K, d, lo=0, hi=2048, med=0.0, h=0, dtype=BF16, rows=False):
    return {"kind": "prune", "name": name, "P": P, "G": G, "K": K, "lo": lo, "hi": hi, "med": med, "d": d, "h": h,
            "dtype": dtype, "rows": rows}


def _update(name, P, G, K, cutoff, d, V, agg, beta, lo=0, hi=2048, med=0.0):
    return {"kind": "update", "name": name, "P": P, "G": G, "K": K, "lo": lo, "hi": hi, "med": med, "cutoff": cutoff, "d": d,
            "V": V, "agg": agg, "beta": beta}


# ---- more cases of the same ranges -------------------------------------------------------------------------------
def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _width(rng, lo=256, hi=4096):
    """Hidden widths: mostly multiples of 64, as models have them, else any multiple of 8."""
    d = _log(rng, lo, hi)
    return int(min(hi, max(lo, round(d / 64) * 64))) if rng.random() < 0.7 else int(min(hi, max(lo, round(d / 8) * 8)))


def _vocab(rng):
    return 151936 if rng.random() < 0.3 else int(_log(rng, 4096, 151936))


def _rollouts(rng, T, group=None):
    """Group shape and lengths whose survivors have about T tokens."""
    G = group or rng.choice([4, 8, 12, 16, 16, 24, 32])
    K = max(1, min(G, int(round(G * rng.choice([0.25, 0.5, 0.5, 0.75])))))
    mean = min(_log(rng, 60, 3000), max(8.0, T / K))
    P = max(1, int(round(T / (K * mean))))
    c = {"P": P, "G": G, "K": K, "cutoff": max(1, int(mean / 4))}
    if rng.random() < 0.5:
        c.update(lo=max(1, int(mean / 2)), hi=max(2, int(mean * 1.5)), med=0.0)
    else:
        c.update(lo=0, hi=int(mean * 3), med=mean)
    return c


def draw(rng):
    kind = rng.choice(["step", "step", "prune", "logprob", "host", "update", "update", "learn", "vote"])
    d, v = _width(rng), _vocab(rng)
    if kind in ("step", "host", "update"):
        passes = 3 if kind == "update" else 1
        top = min(MAX_FLOPS / (2.0 * passes * d * v), MAX_ROW_BYTES / (2.0 * d) / (4.0 if kind != "host" else 16.0), 3.0e5)
        T = _log(rng, min(600.0, top / 2), top)
        c = dict(_rollouts(rng, T), kind=kind, d=d, V=v)
        if kind == "update":
            c.update(agg=rng.randrange(2), beta=rng.choice([0.0, 0.0, 0.04]))
        else:
            small = kind == "step" and d <= 1024 and rng.random() < 0.4
            c.update(h=rng.choice([0, 0, 64, 256, 384]), dtype=FP32 if small else BF16, in_place=kind == "step" and rng.random() < 0.5)
        return c
    if kind == "prune":
        rows = rng.random() < 0.4
        top = min(3.0e6, MAX_ROW_BYTES / (2.0 * d) / 4.0 if rows else 3.0e6)
        c = dict(_rollouts(rng, _log(rng, 600, top)), kind=kind, d=d, h=rng.choice([0, 0, 128, 256, 512]),
                 dtype=FP32 if d <= 1024 and rng.random() < 0.25 else BF16, rows=rows)
        c["P"] = min(c["P"], 16384 // c["G"])
        del c["cutoff"]
        return c
    if kind == "logprob":
        top = min(MAX_FLOPS / (2.0 * d * v), MAX_ROW_BYTES / (2.0 * d), 3.0e5)
        return {"kind": kind, "T": int(_log(rng, min(100.0, top / 2), top)), "d": d, "V": v, "inv_temp": rng.choice([1.0, 1.0, 1.25])}
    if kind == "learn":
        return {"kind": kind, "N": int(_log(rng, 32, 8192)), "d": d, "h": rng.choice([0, 64, 256, 512]),
                "dtype": FP32 if d <= 1024 and rng.random() < 0.25 else BF16, "B": rng.choice([64, 128, 128, 256]),
                "cap": rng.choice([512, 1024, 2048])}
    G = rng.choice([8, 16, 32])
    top = min(MAX_FLOPS / (2.0 * d * v), MAX_ROW_BYTES / (2.0 * d), 2.0e5)
    T = _log(rng, min(2000.0, top / 2), top)
    mean = min(_log(rng, 100, 4000), T / G)
    return {"kind": kind, "P": max(1, int(round(T / (G * mean)))), "G": G, "med": mean, "hi": int(mean * 3) + 1, "d": d, "V": v,
            "window": rng.choice([256, 1024, 2048]), "mode": rng.randrange(3)}


# ---- inputs ------------------------------------------------------------------------------------------------------
_context = None


def _ctx():
    """One context per process, as a training program keeps it."""
    global _context
    if _context is None:
        _context = B.Context(torch.cuda.current_device())
    return _context


def _workload(case, seed, **kw):
    dist = ("lognormal", case["med"], 0.35) if case.get("med", 0.0) > 0 else ("uniform", case["lo"], case["hi"])
    f = dict(name=str(case["kind"]), P=case["P"], G=case["G"], K=case.get("K", case["G"]), cutoff=case.get("cutoff", 1),
             L_max=case["hi"], len_dist=dist, d=case["d"], V=case.get("V", 4096), dtype=case.get("dtype", BF16),
             h=case.get("h", 0), reward="beta_bernoulli", seed=int(seed))
    f.update(kw)
    return synth.Workload(**f)


def _head(w, dev="cuda"):
    head = {k: (None if t is None else t.to(dev)) for k, t in synth.head_weights(w).items()}
    head["h"] = w.h
    return head


def _lengths(w):
    """Rollout lengths: one draw per case, dealt anew inside every group for each seed, so that the buffers' sizes (all source
    rows; the K longest of every group) belong to the case while the survivors' token count follows the selection."""
    ell = synth.lengths(dataclasses.replace(w, seed=0)).reshape(w.P, w.G)
    return np.random.default_rng([w.seed, 51]).permuted(ell, axis=1).reshape(-1)


def _inputs(w):
    """`pipeline.host_inputs` with the lengths above."""
    ell = _lengths(w)
    off = synth.src_offsets(ell)
    hist_s, hist_y = synth.calib_history(w)
    return {"lengths": ell, "rewards": synth.rewards(w), "src_tok_off": off, "src_tokens": synth.token_ids(w, int(off[-1])),
            "head": synth.head_weights(w), "q_lut": B.arrol_build_q_lut(*B.arrol_calib_counts(hist_s, hist_y, w.B), 1.0)}


def _resident(w):
    """A resident workload whose outputs are zero wherever a pass writes nothing (rows past the survivors' tokens)."""
    pr = PruneRebatch(w, inputs=_inputs(w), ctx=_ctx())
    for name in STEP_OUT:
        getattr(pr, name).zero_()
    return pr


STEP_OUT = ("score", "prob", "q", "bin", "keep", "survivor_idx", "cu_seqlens", "adv", "d_num", "dst_tokens", "dst_rows",
            "tok_adv", "tok_seq", "logp", "lse")


def prepare(case, seed):
    return {"step": _prepare_step, "prune": _prepare_prune, "logprob": _prepare_logprob, "host": _prepare_host,
            "update": _prepare_update, "learn": _prepare_learn, "vote": _prepare_vote}[case["kind"]](case, seed)


def _prepare_step(case, seed):
    pr = _resident(_workload(case, seed))
    args = pr.prune_step_args(with_rows=False) if case["in_place"] else None
    return {"kind": "step", "pr": pr, "args": args}


def _prepare_prune(case, seed):
    w = _workload(case, seed)
    inp = _inputs(w)
    off = inp["src_tok_off"]
    T_src, N = int(off[-1]), w.N
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    # the hidden states at the detection length sit in the generation engine's buffer, one slot in eight per rollout
    hidden = synth.normal_tensor((8 * N, w.d), 1.0, synth.torch_dtype(w), w.seed * 1000 + 11, "cuda")
    slot = np.random.default_rng([w.seed, 21]).integers(0, 8, size=N) + 8 * np.arange(N)
    lut = up(inp["q_lut"])
    cap = token_capacity(w, inp["lengths"])
    z = lambda n, t: torch.zeros(n, dtype=t, device="cuda")
    f32, i32, i64 = torch.float32, torch.int32, torch.int64
    out = dict(score=z(N, f32), prob=z(N, f32), q=z(N, f32), bin=z(N, i32), keep=z(N, torch.uint8), survivor_idx=z(N, i32),
               cu_seqlens=z(N + 1, i64), adv=z(N, f32), d_num=z(2, i64), dst_tokens=z(cap, i32), tok_adv=z(cap, f32),
               tok_seq=z(cap, i32))
    rows = {"src_rows": None, "dst_rows": None}
    if case["rows"]:
        rows["src_rows"] = synth.normal_tensor((T_src, w.d), 1.0, torch.bfloat16, w.seed * 1000 + 13, "cuda")
        out["dst_rows"] = rows["dst_rows"] = torch.zeros((cap, w.d), dtype=torch.bfloat16, device="cuda")
    given = dict(row_index=up(slot.astype(np.int64)), lengths=up(inp["lengths"]), src_tok_off=up(off[:-1]),
                 src_tokens=up(inp["src_tokens"]), rewards=up(inp["rewards"]))
    head = _head(w)
    scal = dict(P=w.P, G=w.G, K=w.K, rho=w.rho, eps=1e-6, ddof=0, dst_capacity_tokens=cap,
                row_bytes=2 * w.d if case["rows"] else 0)
    args = B.make_prune_step(hidden, head, lut, scal, dict(out, **given, **rows))
    return {"kind": "prune", "args": args, "out": out, "alive": (hidden, head, lut, given, rows)}


def _prepare_logprob(case, seed):
    ctx, T, d, v = _ctx(), case["T"], case["d"], case["V"]
    w = synth.Workload("logprob", 1, 1, 1, 1, T, ("uniform", T, T), d, v, BF16, 0, "bernoulli_half", int(seed))
    return {"kind": "logprob", "case": case, "hidden": synth.hidden_states(w, T, "cuda"), "W": synth.vocab_weights(w, "cuda"),
            "targets": torch.from_numpy(synth.token_ids(w, T)).cuda(), "logp": torch.zeros(T, device="cuda"),
            "lse": torch.zeros(T, device="cuda"),
            "ws": torch.empty(B.arrol_token_logprob_workspace(ctx, T, d, v), dtype=torch.uint8, device="cuda")}


def _prepare_host(case, seed):
    w = _workload(case, seed)
    inp = _inputs(w)
    ell, off = inp["lengths"], inp["src_tok_off"]
    T_src, N = int(off[-1]), w.N
    cap = token_capacity(w, ell)
    f32, i32, i64 = torch.float32, torch.int32, torch.int64

    def pin(a):
        return torch.from_numpy(np.ascontiguousarray(a)).pin_memory()

    rows = torch.empty((T_src, w.d), dtype=torch.bfloat16, pin_memory=True)
    rows.copy_(synth.hidden_states(w, T_src, "cuda"))
    h = {"h_hidden": rows, "h_src_tokens": pin(inp["src_tokens"]), "h_lengths": pin(ell), "h_src_tok_off": pin(off[:-1]),
         "h_rewards": pin(inp["rewards"]), "h_logp": torch.zeros(cap).pin_memory(), "h_adv": torch.zeros(N).pin_memory(),
         "h_cu_seqlens": torch.zeros(N + 1, dtype=i64).pin_memory(), "h_survivor_idx": torch.zeros(N, dtype=i32).pin_memory(),
         "h_num": torch.zeros(2, dtype=i64).pin_memory()}
    z = lambda n, t: torch.zeros(n, dtype=t, device="cuda")
    dv = {"W_vocab": synth.vocab_weights(w, "cuda"), "d_hidden": z((N, w.d), torch.bfloat16), "d_lengths": z(N, i32),
          "d_src_tok_off": z(N, i64), "d_rewards": z(N, f32), "d_score": z(N, f32), "d_prob": z(N, f32), "d_q": z(N, f32),
          "d_keep": z(N, torch.uint8), "d_survivor_idx": z(N, i32), "d_cu_seqlens": z(N + 1, i64), "d_adv": z(N, f32),
          "d_num": z(2, i64), "d_dst_tokens": z(cap, i32), "d_dst_rows": z((cap, w.d), torch.bfloat16), "d_logp": z(cap, f32),
          "d_workspace": torch.empty(B.arrol_token_logprob_workspace(_ctx(), cap, w.d, w.V), dtype=torch.uint8, device="cuda")}
    scal = dict(P=w.P, G=w.G, K=w.K, cutoff=w.cutoff, d=w.d, V=w.V, ddof=0, rho=w.rho, eps=1e-6, inv_temperature=1.0,
                T_src=T_src, dst_capacity_tokens=cap)
    head, lut = _head(w), torch.from_numpy(inp["q_lut"]).cuda()
    step = B.make_host_step(scal, head, lut, dict(h, **dv))
    out = {k: t for k, t in h.items() if k in ("h_logp", "h_adv", "h_cu_seqlens", "h_survivor_idx", "h_num")}
    out.update({k: dv[k] for k in ("d_score", "d_prob", "d_q", "d_keep", "d_dst_tokens", "d_dst_rows")})
    return {"kind": "host", "step": step, "out": out, "alive": (h, dv, head, lut)}


def _prepare_update(case, seed):
    """A step's survivors as the update finds them: packed rows, targets, the log-probs of the step that sampled them (the
    policy has moved since: ratios of about exp(+-0.1)) and, with a KL term, a reference policy's."""
    w = _workload(case, seed)
    pr = _resident(w)
    pr.step()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1000 + 17)
    noise = lambda s: torch.randn(pr.cap, generator=gen, device="cuda") * s
    old = pr.logp + noise(0.1)
    ref = pr.logp + noise(0.2) if case["beta"] > 0 else None
    keep = {k: getattr(pr, k) for k in ("W_vocab", "dst_rows", "dst_tokens", "tok_adv", "tok_seq", "cu_seqlens", "d_num", "logp", "lse")}
    return dict(keep, kind="update", case=case, cap=pr.cap, old=old, ref=ref, grad=torch.zeros(pr.cap, device="cuda"),
                loss=torch.zeros(1, dtype=torch.float64, device="cuda"), dH=torch.zeros((pr.cap, w.d), device="cuda"),
                dW=torch.zeros((w.V, w.d), device="cuda"),
                ws=torch.empty(U.arrol_lm_head_backward_workspace(_ctx(), pr.cap, w.d, w.V), dtype=torch.uint8, device="cuda"))


def _prepare_learn(case, seed):
    ctx, N, d, h = _ctx(), case["N"], case["d"], case["h"]
    w = synth.Workload("learn", N, 1, 1, 1, 8, ("uniform", 1, 8), d, 4096, case["dtype"], h, "beta_bernoulli", int(seed), B=case["B"])
    g = np.random.default_rng([int(seed), 31])
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    hidden = synth.normal_tensor((4 * N, d), 1.0, synth.torch_dtype(w), w.seed * 1000 + 11, "cuda")
    head = _head(w)
    params = C.survival(kappa=0.5, lam=0.5, rho=0.5)
    cal = C.Calibrator(ctx, n_bins=case["B"], cap=case["cap"])
    hist_s, hist_y = synth.calib_history(w)            # earlier steps' rollouts: more than both rings hold
    cal.update(up(np.minimum(case["B"] - 1, (hist_s * case["B"]).astype(np.int32)).astype(np.int32)), up(hist_y.astype(np.float32)), params)
    z = lambda n, t: torch.zeros(n, dtype=t, device="cuda")
    f32 = torch.float32
    lay = cal.layout
    ints = lambda a, b, t: cal.state[lay[a]:lay[a] + b].view(t)
    out = dict(score=z(N, f32), prob=z(N, f32), q=z(N, f32), bin=z(N, torch.int32), keep=z(N, torch.uint8), p=z(N, f32),
               loss=z(1, torch.float64), W1=z((max(h, 1), d), f32), b1=z(max(h, 1), f32), q_lut=cal.q_lut, delta=cal.delta,
               cpos=ints("cpos", 8 * case["B"], torch.int64), cneg=ints("cneg", 8 * case["B"], torch.int64),
               ring_pos=ints("ring_pos", 2 * case["cap"], torch.int16), ring_neg=ints("ring_neg", 2 * case["cap"], torch.int16))
    if h:
        out.update(w2=z(h, f32), b2=z(1, f32))
    return {"kind": "learn", "N": N, "hidden": hidden, "head": head, "cal": cal, "params": params, "out": out,
            "rows": up((4 * np.arange(N) + g.integers(0, 4, size=N)).astype(np.int64)), "u": up(g.random(N).astype(np.float32)),
            "eligible": up((g.random(N) < 0.95).astype(np.uint8)), "rewards": up(synth.rewards(w)),
            "grads": {k: out[k] for k in ("W1", "b1", "w2", "b2") if k in out},
            "ws": torch.empty(HT.arrol_head_grad_workspace(ctx, N, d, h), dtype=torch.uint8, device="cuda")}


def _prepare_vote(case, seed):
    ctx = _ctx()
    w = _workload(case, seed, cutoff=8)
    off = synth.src_offsets(_lengths(w))
    T, S = int(off[-1]), w.N
    g = np.random.default_rng([int(seed), 41])
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    z = lambda n, t=torch.float32: torch.zeros(n, dtype=t, device="cuda")
    out = dict(logp=z(T), lse=z(T), token_conf=z(T), trace_conf=z(S), score=z(S), prob=z(S), q=z(S), weight=z(S),
               winner=z(w.P, torch.int32), winner_weight=z(w.P))
    return {"kind": "vote", "case": case, "T": T, "S": S, "hidden": synth.hidden_states(w, T, "cuda"), "W": synth.vocab_weights(w, "cuda"),
            "targets": up(synth.token_ids(w, T)), "cu": up(off), "num": up(np.array([S, T], np.int64)), "last": up(off[1:] - 1),
            "head": _head(w), "answer": up(g.integers(-1, 5, size=S).astype(np.int32)), "out": out,
            "ws": torch.empty(B.arrol_token_logprob_workspace(ctx, T, w.d, w.V), dtype=torch.uint8, device="cuda")}


# ---- one pass ----------------------------------------------------------------------------------------------------
def run(s):
    return {"step": _run_step, "prune": _run_prune, "logprob": _run_logprob, "host": _run_host, "update": _run_update,
            "learn": _run_learn, "vote": _run_vote}[s["kind"]](s)


def _run_step(s):
    pr = s["pr"]
    if s["args"] is not None:
        B.arrol_prune_step(pr.ctx, s["args"])
        pr.token_logprob_gathered()
        return {k: getattr(pr, k) for k in STEP_OUT if k != "dst_rows"}
    pr.step()
    return {k: getattr(pr, k) for k in STEP_OUT}


def _run_prune(s):
    B.arrol_prune_step(_ctx(), s["args"])
    return s["out"]


def _run_logprob(s):
    c = s["case"]
    B.arrol_token_logprob(_ctx(), s["hidden"], s["W"], s["targets"], c["T"], c["d"], c["V"], s["logp"], s["ws"], lse=s["lse"],
                          inv_temperature=c["inv_temp"])
    return {"logp": s["logp"], "lse": s["lse"]}


def _run_host(s):
    B.arrol_prune_rebatch_host(_ctx(), s["step"])
    return s["out"]


def _run_update(s):
    c = s["case"]
    U.arrol_policy_loss(_ctx(), s["logp"], s["old"], s["tok_adv"], s["tok_seq"], s["cu_seqlens"], s["d_num"], s["cap"], s["grad"],
                        s["loss"], logp_ref=s["ref"], eps_low=0.2, eps_high=0.28 if c["agg"] else 0.2, beta=c["beta"], agg_mode=c["agg"])
    U.arrol_lm_head_backward(_ctx(), s["dst_rows"], s["W_vocab"], s["dst_tokens"], s["grad"], s["lse"], s["cap"], c["d"], c["V"],
                             s["dH"], s["dW"], s["ws"], d_T=s["d_num"][1:])
    return {k: s[k] for k in ("loss", "grad", "dH", "dW")}


def _run_learn(s):
    o, cal, N = s["out"], s["cal"], s["N"]
    B.arrol_score_partial(_ctx(), s["hidden"], s["head"], N, o["score"], o["prob"], o["q"], bin=o["bin"], row_index=s["rows"],
                          q_lut=cal.q_lut)
    C.arrol_select_stochastic(_ctx(), o["q"], s["u"], o["keep"], s["params"], d_delta=cal.delta, eligible=s["eligible"], p_out=o["p"])
    cal.update(o["bin"], s["rewards"], s["params"], mask=o["keep"])
    HT.arrol_head_grad(_ctx(), s["hidden"], s["head"], N, s["rewards"], s["grads"], o["loss"], s["ws"], row_index=s["rows"],
                       mask=o["keep"])
    return o


def _run_vote(s):
    c, o = s["case"], s["out"]
    CF.arrol_token_logprob_conf(_ctx(), s["hidden"], s["W"], s["targets"], s["T"], c["d"], c["V"], o["logp"], o["token_conf"], s["ws"],
                                lse=o["lse"])
    CF.arrol_trace_confidence(_ctx(), o["token_conf"], s["cu"], s["num"], s["S"], o["trace_conf"], window=c["window"], mode=c["mode"])
    B.arrol_score_partial(_ctx(), s["hidden"], s["head"], s["S"], o["score"], o["prob"], o["q"], row_index=s["last"])
    V.arrol_rank_vote(_ctx(), o["score"], s["answer"], c["P"], c["G"], o["weight"], o["winner"], o["winner_weight"])
    return o


# ---- what a pass cannot do without, and how exact it is ----------------------------------------------------------
def _mean_length(case):
    if case.get("med", 0.0) > 0:
        return case["med"] * math.exp(0.35 ** 2 / 2)
    return (case["lo"] + case["hi"]) / 2.0


def work(case):
    kind, d = case["kind"], case["d"]
    if kind == "logprob":
        return {"bytes": 2.0 * d * (case["T"] + case["V"]) + 12.0 * case["T"], "flops": 2.0 * case["T"] * d * case["V"]}
    e = 4 if case.get("dtype") == FP32 else 2
    h = case.get("h", 0)
    if kind == "learn":
        N = case["N"]
        head = e * d * max(h, 1)
        return {"bytes": float(e * d * N + head + 4 * d * max(h, 1) + 40 * N + 8 * case["cap"]), "flops": 4.0 * N * d * max(h, 1)}
    N = case["P"] * case["G"]
    if kind == "vote":
        T = N * _mean_length(case)
        return {"bytes": 2.0 * d * (T + case["V"]) + 16.0 * T, "flops": 2.0 * T * d * case["V"]}
    T = case["P"] * case["K"] * _mean_length(case)
    if kind == "update":     # logits again, dH, dW; rows and W read once, both gradients written once
        return {"bytes": (2.0 + 4.0) * d * (T + case["V"]) + 32.0 * T, "flops": 6.0 * T * d * case["V"]}
    score = {"bytes": float(e * d * (N + max(h, 1)) + 60 * N), "flops": 2.0 * N * d * max(h, 1)}
    per_token = 16.0         # token id in and out, survivor ordinal, advantage
    if kind == "prune":
        return {"bytes": score["bytes"] + T * (per_token + (4.0 * d if case["rows"] else 0.0)), "flops": score["flops"]}
    packed = 0.0 if kind == "host" or case["in_place"] else 4.0 * d     # the packed copy that the two-call path asks for
    return {"bytes": score["bytes"] + T * (per_token + packed + 2.0 * d + 12.0) + 2.0 * d * case["V"],
            "flops": score["flops"] + 2.0 * T * d * case["V"]}


def tolerance(case):
    """Four times what one pass differed by from the same arithmetic in 64 bits on the same inputs (rel, max):
    log-probs and log-sum-exp 6.6e-7, 1.6e-6; head scores 3.1e-7, 1.5e-6; confidences 6.5e-8, 1.7e-7; head gradients 3.0e-6,
    2.4e-5 (their largest, dW1 with du as the sum of two bf16 planes); dH and dW 1.8e-3, 3.9e-2 (dz is rounded to bf16 before the
    two contractions).  Whole values (decisions, indices, token ids, counts) are the same."""
    if case["kind"] == "update":
        return {"rel": 7e-3, "max": 0.16}
    if case["kind"] == "learn":
        return {"rel": 1.2e-5, "max": 1e-4}
    return {"rel": 3e-6, "max": 1e-5}
