"""The benchmark's line on stdout: the keys that its readers look for, finite numbers, and short enough to survive a reader that
keeps the end of the output only."""
import json

import bench
from paper_2603_24840_b200 import synth


def _block(name):
    roof = {k: 1.0 / 3.0 for k in bench.ROOFLINE_KEYS}
    roof.update(kernel="token_logprob_kernel, pairs of blocks on 256-row tiles, tcgen05 cta_group::2 (+ combine_splits_kernel)",
                note="x" * 2000)
    return {"value": 1234567.8901234, "ms_per_step": 123.45678901234, "roofline": roof, "score_roofline": dict(roof), "aux": {"t": [0.1] * 300},
            "e2e": {"value": 1234567.8901234, "unit": bench.UNIT, "h2d_bytes_per_step": 10 ** 11, "d2h_bytes_per_step": 10 ** 8},
            "clocks": {"sm_mhz": 1290.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"], "samples": 400}, "gpu_launches": 400,
            "breakdown_ms": {k: 1.0 / 3.0 for k in ("score_partial", "select", "compact", "token_logprob")},
            "logprob_tokens_per_s": float("nan"), "config": bench.config_of(synth.WORKLOADS[name], 4)}


def test_the_line_is_short_and_complete():
    head = bench.DEFAULT_WORKLOAD
    out = {"metric": bench.METRIC, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic"}
    out.update(_block(head))
    out["per_workload"] = {n: _block(n) for n in synth.WORKLOAD_ORDER if n != head}
    out["per_workload"]["tiny"] = {"skipped": "y" * 500}
    out["cpu_baseline"] = {"value": 23.7, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "z" * 900}
    text = bench.contract_line(out)
    assert len(text) < 3000 and "NaN" not in text
    line = json.loads(text)
    assert line["value"] > 0 and line["e2e"]["value"] > 0 and line["logprob_tokens_per_s"] is None
    for key in ("metric", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
                "data", "config", "clocks", "e2e", "gpu_launches", "roofline", "cpu_baseline"):
        assert key in line
    assert {"h2d_bytes_per_step", "d2h_bytes_per_step", "unit"} <= set(line["e2e"]) and line["config"]["workload"] == head
