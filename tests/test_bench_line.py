"""bench.py's result line: the keys a reader needs in a few KB, every further leg apart."""
import json

import bench


def test_result_line_is_short_and_complete():
    need = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline")
    out = {k: 1.0 for k in need}
    out["solver"] = dict(text="s" * 1300)
    for k in bench.LEGS:
        out[k] = dict(table=["x" * 100] * 80)
    ratios = {"box_1157k": {"learned/vn": {"iters": 0.6, "ms": 0.63}}}
    out["learned"]["learned_vs_plain"] = ratios
    line, legs = bench.result_lines(out)
    assert set(need) <= set(line) and not set(bench.LEGS) & set(line)
    assert line["learned_vs_plain"] == ratios
    assert set(legs) == set(bench.LEGS) and legs["poiseuille"] == out["poiseuille"]
    assert len(json.dumps(line)) < 4000 < len(json.dumps(out))
    # without the optional legs
    line, legs = bench.result_lines({k: 1.0 for k in need} | {"learned": None, "shard": None})
    assert set(line) == set(need) and legs == {"learned": None, "shard": None}
