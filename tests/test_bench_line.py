"""The benchmark's stdout line stays short enough to be found whole in a kept tail of the output, whatever the
secondary legs hold, and keeps the keys a run is read by."""
import json

import bench

KEYS = {"metric": bench.METRIC, "value": 29521656.430569034, "unit": "tokens/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 0.034686400555074215, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16 in, f32 accumulate", "data": "synthetic",
        "config": bench.config_dict(bench.WL.WORKLOADS["llama32_1b_prefill"], 0.3), "impl": "ours", "gpu_launches": 60,
        "e2e": {"value": 4057261.2694039023, "unit": "tokens/s", "h2d_bytes_per_step": 6291456, "d2h_bytes_per_step": 4194304},
        "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": [], "samples": 2}}


def test_line_leaves_the_secondary_legs_to_stderr(capsys, tmp_path):
    leg = {"us_per_step_eager": 10.704499669373035, "us_per_step_graph": 3.8971249014139175,
           "us_per_step_l2_flushed": 10.059733347346386, "us_per_step_l2_flushed_by_read": 9.979733312502503,
           "roofline": {"note": "x" * 3000}}
    report = {**KEYS, **{name: [{"x": "y" * 5000}] for name in bench.SECONDARY_LEGS},
              "decode": {"batch1": leg, "batch16": leg}, "roofline": {"frac": 0.08}, "cpu_baseline": {"value": 1126.0}}
    bench.print_report(report, str(tmp_path / "report.json"))
    io = capsys.readouterr()
    lines = io.out.splitlines()
    assert len(lines) == 1 and len(lines[0]) < 2500
    line = json.loads(lines[0])
    assert {k: line[k] for k in KEYS} == KEYS and line["roofline"] and line["cpu_baseline"]
    assert line["decode"]["batch16"] == {k: v for k, v in leg.items() if k.startswith("us_")}
    assert {json.loads(x)["leg"] for x in io.err.splitlines()} == set(bench.SECONDARY_LEGS)
    assert json.load(open(tmp_path / "report.json")) == report
