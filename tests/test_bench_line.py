"""The benchmark's line stays short enough for a reader that keeps the last kilobytes of the output."""
import json

import bench


def record():
    r = {k: 1.0 / 3.0 for k in bench.LINE_KEYS}
    text = "x" * 120
    r.update(metric=text, unit="frames/s", dtype=text, data="synthetic",
             config={k: text for k in ("workload", "image", "grid", "samples", "brick", "parallelism")} | {"l2": 2 * text},
             roofline={f"k{i}": 1.0 / 3.0 for i in range(12)} | {"kernel": text, "hbm": {"a": 1.0 / 3.0}},
             quality={f"k{i}": 1.0 / 3.0 for i in range(10)}, brick={"bf16": 4, "fp32": 8, "fp32_split": 4},
             e2e={"value": 1.0 / 3.0, "mode": text, "serialised_mode": text, "h2d_bytes_per_step": 816,
                  "d2h_bytes_per_step": 122880000},
             clocks={"sm_mhz": 2070.0, "reasons": ["sw_power_cap"]},
             cpu_baseline={"value": 0.1, "sample": text, "threads": [text] * 100},
             stages={f"stage_{i}": {"ms_per_step": 1.0 / 3.0, "launches_per_step": 1.0} for i in range(8)})
    for w, f in bench.LINE_FIGURES.values():
        r.setdefault(w, {"targets": [{"psnr_db": 1.0 / 3.0}] * 100})[f] = 1.0 / 3.0
    r["sparw_window_sweep"] = [text] * 100
    return r


def test_line_is_short_and_complete():
    r = record()
    s = bench.headline(r)
    line = json.loads(s)
    assert len(json.dumps(r)) > 20000 and len(s) <= 4096 and "\n" not in s
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert k in line
    assert abs(line["value"] - r["value"]) < 1e-6 and set(line["workloads"]) == set(bench.LINE_FIGURES)
