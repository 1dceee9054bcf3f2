"""The line that bench.py prints has the contract's keys and stays short enough for a reader that keeps the last few
KiB of a run's output."""
import json

import bench
from paper_2609_35140_b200 import synth


def _report(index):
    w = synth.get_workload(index)
    points = max(1, len(w.decode_contexts or [0]))
    third = 1000.0 / 3
    nums = {k: third for k in ("train", "prefill", "logprob", "total", "alone_train", "alone_prefill", "logprob_decode_shaped")}
    for i in range(points):
        nums.update({"decode%d" % i: third, "alone_decode%d" % i: third, "graph_decode%d" % i: third})
    clocks = {"sm_mhz": 1087.0, "sm_mhz_min": 967.0, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 890}
    info = {"clocks": clocks, "lp_rows": 256, "dec": [{"label": "16384", "bytes": 3250294784, "logical_bytes": 3250294784,
                                                       "graph_note": None}] * points}
    rep = bench.report_workload(w, nums, info, bench.FALLBACK_PEAKS, 1)
    rep["gpu_launches"] = 180
    return rep, nums, clocks


def test_printed_line_is_short_and_complete():
    reports = {"configs[%d]" % i: _report(i) for i in range(5)}
    head, nums, clocks = reports["configs[4]"]
    roof = {"ms": 1000.0 / 3, "achieved": 1000.0 / 3, "frac": 1.0 / 3, "note": "x" * 200}
    names = ["train_fwd", "prefill", "logprob", "decode@4096", "decode@8192", "decode@16384", "logprob_decode_shaped", "qk_norm_rope_kv_write",
             "attn_train_bwd", "rmsnorm", "add_rmsnorm", "swiglu", "linear_gate_up_decode_shaped", "linear_down_decode_shaped",
             "linear_gate_up", "linear_down"]
    full = {"metric": bench.METRIC, "value": head["value_ms"], "unit": "ms", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": nums["total"], "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
            "data": "synthetic", "config": bench.workload_config(synth.get_workload(4), 1), "phases_ms": head["phases_ms"],
            "decode_tok_per_s": [d["tok_per_s"] for d in head["decode"]],
            "roofline": {"kernel": "attn_persist_kernel<128,packed>", "bound": "tensor", "achieved": 1000.0 / 3, "peak": 1357.0,
                         "unit": "TFLOP/s", "frac": 1.0 / 3, "traffic": 1e10 / 3, "traffic_source": "x" * 300,
                         "peak_source": "x" * 110, "frac_burst_peak": 1.0 / 3, "frac_sustained_peak": 1.0 / 3,
                         "frac_nominal_peak": 1.0 / 3, "algorithmic_flops_per_launch": 52100000000000},
            "rooflines": {n: roof for n in names},
            "cpu_baseline": {"value": 1e6 / 3, "unit": "ms", "cores": 16, "kind": "oracle", "sample": "x" * 140},
            "e2e": {"value": 1000.0 / 3, "unit": "ms", "h2d_bytes_per_step": 21600000000, "d2h_bytes_per_step": 17300000000,
                    "steps": 4, "pinned_host_bytes": 2 << 30, "note": "x" * 300},
            "per_config": {n: r[0] for n, r in reports.items()}, "gpu_launches": 180, "gpu_launches_other_configs": 190,
            "clocks": clocks, "device_flags": 0, "contract": "tik3-BN128-CH2048-M128N128K16-ex2ftz-lazy8-sum2x4-LP128x1024"}
    text = json.dumps(bench.printed_line(full))
    assert len(text) < 3600, len(text)
    got = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline", "cpu_baseline"):
        assert key in got
    assert abs(got["value"] / full["value"] - 1) < 1e-4 and got["e2e"]["h2d_bytes_per_step"] == 21600000000
    assert set(got["rooflines"]) == set(names) and set(got["per_config"]) == set(reports)
