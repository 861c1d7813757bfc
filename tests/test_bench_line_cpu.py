"""The line that bench.py prints: short enough for a reader that keeps the last kilobytes of the
output, with every key of the contract."""
import json

import bench


def _record():
    interval = {"interval": [-462.5125, -49.98750000000007], "holds": False}
    plan = {k: 1.0 / 3.0 for k in ("kernel", "replicas_per_block", "blocks", "threads", "smem_bytes",
                                   "pad_ratio", "conflict_ratio", "balance", "chunks")}
    variant = {"spin_updates_per_s": 1e11 / 3.0, "steps": 5, "ms_per_step": 100.0 / 3.0,
               "autotuned": {"candidates": [[1, 2, 0.123456]] * 13}, "equal_cut_vs_plain": interval}
    roof = {"bound": "tensor", "achieved": 1e3 / 3.0, "peak": 1948.6, "unit": "TFLOP/s", "frac": 1.0 / 3.0,
            "peak_source": "measured " * 12, "kernel": "k_dense_md<128,*,2,*,*,true,*,*,*>",
            "launch_ms": 100.0 / 3.0, "plan": plan, "traffic": None}
    e2e = {"value": 1e11 / 3.0, "unit": "spin-updates/s", "steps": 5, "h2d_bytes_per_step": 1 << 26,
           "d2h_bytes_per_step": 1 << 23}
    cpu = {"value": 1e7 / 3.0, "unit": "spin-updates/s", "cores": 16, "kind": "oracle", "sample": "x" * 90}
    rec = {"metric": bench.METRIC, "value": 1e11 / 3.0, "unit": "spin-updates/s", "n_gpus": 1, "steps": 5,
           "warmup": 3, "ms_per_step": 500.0 / 3.0, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "fp16-operand/f32-accumulate", "data": "synthetic",
           "gpu_launches": 75, "config": {"workload": "w" * 120, "name": "sk2000", "N": 2000},
           "e2e": e2e, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
           "headline_variant": "fp16x2", "variants": {f"variant_{k}": variant for k in range(6)},
           "equal_cut": {"rule": "r" * 200}, "roofline": roof, "cpu_baseline": cpu}
    gated = {"value": 1e11, "unit": "spin-updates/s", "roofline": roof, "e2e": e2e,
             "sizes": {str(n): {"gated": [dict(variant, **interval)] * 4} for n in range(8)}}
    rec["nested"] = {"er800": dict(rec), "uneven512": dict(rec), "er_surrogate": gated}
    return rec


def test_line_is_short_and_complete():
    rec = _record()
    assert len(json.dumps(rec)) > 16000         # what used to be printed
    line = bench.printed_line(rec)
    text = json.dumps(line)
    assert "\n" not in text and len(text) <= 3500
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
              "scaling", "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks",
              "roofline", "cpu_baseline"):
        assert k in line, k
    assert line["e2e"]["h2d_bytes_per_step"] == 1 << 26
    assert abs(line["value"] / rec["value"] - 1.0) < 1e-5
    assert set(line["nested"]) == {"er800", "uneven512", "er_surrogate"}


def test_line_of_one_workload():
    rec = _record()
    for k in ("nested", "variants", "cpu_baseline", "roofline"):
        rec.pop(k)
    line = bench.printed_line(rec)
    assert json.loads(json.dumps(line))["value"] == line["value"] and "nested" not in line
