"""The line bench.py prints on standard output is kept by whoever records it only up to a few thousand characters."""
import json

import bench


def _measurement():
    entries = [bench.roofline_entry("kernel_%d_with_a_long_name (one launch = 512 steps)" % i, "logistic 262144 x 8192, N=32 workers, case %d" % i,
                                    1234.567 + i, 8.59e9, 6557.8, "snapshot_kernel", 1 << 26, note="n" * 120,
                                    short="a kernel of leg %02d" % i if i < 31 else None) for i in range(45)]
    out = {k: 1.0 for k in ("value", "ms_per_step", "vs_baseline", "snapshot_ms", "inner_loop_ms", "inner_step_us", "wall_s", "objective_end")}
    out.update(metric=bench.METRIC, unit=bench.UNIT, n_gpus=1, steps=20, warmup=5, higher_is_better=True, scaling="weak", dtype="f32",
               data="synthetic", gpu_launches=60, config={"workload": "w" * 40, "step": "s" * 60, "l2": "l" * 70, "n": 131072},
               clocks={"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": [], "samples": 3},
               e2e={"value": 1.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1, "job": "j" * 100},
               cpu_baseline={"value": 1.0, "cores": 1, "sample": "s" * 130}, kernels={"k": {"avg_us": 1.0}}, launch_plan={"p": 1},
               quantize_aggregate={"grid": "g" * 8000}, tiny_logistic={"step_us": 4.4}, alpc={"b2": {"step_us": 9.9}, "b8": {"step_us": 10.4}},
               fused_large_batch={"f": 1},
               roofline={"bound": "hbm", "kernel": "inner_loop", "achieved": 460.0, "peak": 6557.8, "unit": "GB/s", "frac": 0.07,
                         "traffic": 1, "traffic_source": "t" * 200, "note": "n" * 200, "kernels": entries})
    return out


def test_headline_is_short_and_complete():
    out = _measurement()
    line = json.dumps(bench.headline(out))
    assert len(line) < 3000 and "\n" not in line
    head = json.loads(line)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
              "data", "config", "clocks", "e2e", "gpu_launches", "cpu_baseline"):
        assert head[k] == out[k]
    r = head["roofline"]
    assert {k: r[k] for k in ("bound", "kernel", "achieved", "peak", "unit", "frac", "traffic")} == \
        {k: out["roofline"][k] for k in ("bound", "kernel", "achieved", "peak", "unit", "frac", "traffic")}
    assert len(r["kernels"]) == 31 and r["kernels"]["a kernel of leg 00"][0] == 1234.6
    assert len(out["roofline"]["kernels"]) == 45  # the measurement in full is left as it was


def test_headline_of_a_rank_of_many():
    out = _measurement()
    for k in ("quantize_aggregate", "alpc", "tiny_logistic", "fused_large_batch", "cpu_baseline"):
        del out[k]
    out["e2e"], out["roofline"] = None, None
    assert bench.headline(out)["e2e"] is None
