"""bench.py's line on stdout: short enough that the end of a run's output holds
all of it, with the keys that a reader of the line needs."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_the_line_stays_short_and_keeps_the_contract():
    import bench
    text = "x" * 160
    line = {"metric": text, "value": 123456789.1, "unit": "env-evals/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.01436, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "gpu_launches": 20, "roofline": {"a": text, "b": text, "c": text},
            "cpu_baseline": {"sample": text}, "per_op_ms": {"a": text}, "parity_vs_oracle": {"a": text}}
    line.update(config={"a": text, "b": text}, e2e={"value": 1.0, "unit": text, "h2d_bytes_per_step": 1,
                                                    "d2h_bytes_per_step": 2},
                clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
                plan={"mode": "fused", "us": {f"hybrid[specialized/{k}|level/256]": float(k) for k in range(1, 300)}},
                humanoid_sweep={str(k): text for k in range(20)}, sysid={str(k): text for k in range(5)})
    short = bench.short_line(line)
    assert len(json.dumps(short)) < 3000 < len(json.dumps(line))
    assert {"metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"} <= set(short)
    assert short["plan_ran"] == {"mode": "fused", "name": "hybrid[specialized/1|level/256]"}
    assert not {"plan", "humanoid_sweep", "sysid"} & set(short)
