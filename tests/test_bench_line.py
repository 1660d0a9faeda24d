"""The benchmark's result is one short line: what the sections measured goes
beside it."""
import importlib.util
import json
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bench():
    spec = importlib.util.spec_from_file_location("bench_mod", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_result_line_is_short_and_whole():
    b = _bench()
    roof = b.roofline_obj([(1e12, 1e9, 0.02)] * 16, {"hbm_gbs": 6779.0, "bf16_tflops": 1933.3},
                          "tensor", kernel="tc_kernel")
    roof.update(share_of_step=1.0, peak_source="x" * 80, traffic_source="x" * 160)
    line = {"metric": b.METRIC, "value": 123.456, "unit": "TFLOP/s", "n_gpus": 8, "steps": 50,
            "warmup": 5, "ms_per_step": 0.5678, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f16 (fp32 accumulate)", "data": "synthetic",
            "config": b.workload_config(False, 8),
            "e2e": {"value": 1.23456789012345, "unit": "TFLOP/s", "h2d_bytes_per_step": 268435456,
                    "d2h_bytes_per_step": 268435456, "steps": 5, "host_threads": 8},
            "gpu_launches": 1600, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "roofline": roof,
            "cpu_baseline": {"value": 0.05, "unit": "TFLOP/s", "cores": 16, "kind": "oracle",
                             "sample": "x" * 200}}
    keys = set(line)
    for k in b.DETAIL:
        line[k] = {"grid": [{"speedup": 1.234, "dense_tflops": 685.2, "m": 4096}] * 60}
    line["points"] = [{"b": bb, "d": "1/%d" % d, "us": 12.34, "kernel": "tc", "more": "y" * 100}
                      for bb in (1, 4, 8, 16) for d in (32, 16, 8, 4)]
    line["serving"] = {"tc_fp16": {"saturation_rps": 27000.1, "rates": [
        {"rate_x_sat": f, "p50_us": 100.0 * f, "p99_us": 300.0 * f} for f in (0.25, 0.5, 0.9)]}}
    head, detail = b.split_line(line)
    assert len(json.dumps(head)) < 3000 and "\n" not in json.dumps(head)
    assert keys <= set(head) and all(head[k] == line[k] for k in keys)
    assert set(detail) == set(b.DETAIL) and all(detail[k] == line[k] for k in b.DETAIL)
    assert head["serve"] == {"rate_x_sat": 0.5, "p50_us": 50.0, "p99_us": 150.0,
                             "saturation_rps": 27000.1}
    assert head["points_us"]["b=16 d=1/4"] == 12.34
    for k in b.DETAIL:
        line[k] = None              # sections left out
    assert b.split_line(line)[0]["serve"] is None
