"""The line that bench.py prints: short, with every key of its contract and the measured numbers unchanged."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

KEYS = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
        "dtype", "data", "config", "roofline", "cpu_baseline", "e2e", "gpu_launches", "clocks")


def test_line_is_short_and_whole():
    phases = {p: 0.123456789012345 for p in ("sort", "moments", "select", "collide", "moment_match")}
    roof = {p: {"roofs": {r: {"achieved": 1 / 3, "peak": 2 / 3, "source": "x" * 80} for r in "abcdef"}} for p in phases}
    path = {"collisions_per_s": 2.6198292859323688e9, "ms_per_step": 2.6270336151123046, "phase_ms": phases, "rooflines": roof,
            "autotune": {"shapes": {"gather": [256, 8]}}}
    line = {k: 1 for k in KEYS}
    line.update(value=2619829285.932369, ms_per_step=2.6270336151123046, vs_baseline=None, config={"workload": "w" * 90, "path": "neural"},
                paths={p: path for p in ("neural", "jager", "table", "vhs")}, standalone={"chi": {"t": list(range(2000))}},
                roofline={"bound": "tensor", "frac": 0.16116, "peak_source": "p" * 60},
                cpu_baseline={"value": 771904.9405653853, "sample": "s" * 120, "single_thread": {"sample": "s" * 120}},
                e2e={"value": 1448928192.9083197, "unit": "pair collisions/s", "h2d_bytes_per_step": 256039924,
                     "d2h_bytes_per_step": 256039948})
    text = json.dumps(bench.short_line(line))
    out = json.loads(text)
    assert "\n" not in text and len(text) < 1500
    assert set(KEYS) <= set(out) and "standalone" not in out
    assert out["value"] == line["value"] and out["ms_per_step"] == line["ms_per_step"]
    assert abs(out["e2e"]["value"] / line["e2e"]["value"] - 1) < 1e-4 and out["e2e"]["h2d_bytes_per_step"] == 256039924
    assert set(out["paths"]["jager"]) == {"collisions_per_s", "ms_per_step"}
