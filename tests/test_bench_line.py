"""The benchmark's printed line: the contract's keys as they are, a few KB whatever the
detail (per-tensor errors, autotuner candidates) holds.  CPU only."""

import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def full_line():
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 5}
    roof = {"bound": "tensor", "achieved": 198.3817423157985, "peak": 1696.1, "unit": "TFLOP/s", "frac": 0.11696347050,
            "peak_source": "measured bf16_tflops_sustained (kernel timed inside a long step)", "kernel_class": "gemm",
            "launches": 3000, "avg_launch_us": 25.48122662057479, "timing": "t" * 80, "traffic": None, "note": "n" * 300,
            "issued": {"tflops": 386.0737914589593, "frac": 0.2276244274859733, "note": "n" * 200}}
    breakdown = {"timing": "t" * 80} | {c: {"launches_per_step": 15, "us_per_step": 380.320000089705,
                                            "us_per_launch": 25.354666672647}
                                        for c in ("insert", "relabel", "gemm", "energy", "adam", "aux")}
    grads = [{"tensor": f"phi.{i}.W", "rel_err": 0.0016585244417353648, "cos": 0.9999986248740598} for i in range(60)]
    arm = {"status": 0, "loss_rel_err": {"critic_total": 8.9e-06, "actor": 5.5e-06}, "grad_worst_rel_err": 0.0024059,
           "grad_worst_cos": 0.9999971057604876, "grads": grads}
    error = {"workload": "w" * 60, "oracle": "o" * 40, "kink_units": {"phi": 9},
             "bars": {"fp32": {"loss_rel": 1e-05, "grad_rel": 0.0001}, "bf16": {"loss_rel": 0.02, "grad_cos": 0.999}},
             "bf16_fused": arm, "fp32_plain": arm}
    comp = {"precision": "fp32", "path": "plain", "value": 116.26210119951672, "unit": "update steps/s",
            "ms_per_step": 8.601255178451538, "speedup": 14.426531666150069, "clocks": clocks, "note": "n" * 90}
    us = {f"one_tile 128x{n} s{s}": 39.81 for n in (64, 128, 256) for s in (3, 4, 6, 8)}
    e2e = {"value": 1583.123456789, "unit": "update steps/s", "h2d_bytes_per_step": 1314816, "d2h_bytes_per_step": 24,
           "timing": "t" * 140}
    w = {"workload": "w" * 50, "value": 3210.123456789, "unit": "update steps/s", "ms_per_step": 0.3115123456789,
         "e2e": e2e, "roofline": roof, "clocks": clocks, "comparator": comp, "error": error, "breakdown": breakdown}
    return {"metric": bench.METRIC, "value": 1705.123456789012, "unit": "update steps/s", "n_gpus": 1, "steps": 200,
            "warmup": 20, "ms_per_step": 0.586466123456789, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "bf16", "data": "synthetic (seeded random-walk buffer, random-init nets)",
            "samples_per_s": 13968371.123, "config": {k: "c" * 30 for k in "abcdefghijklmnopq"}, "e2e": e2e,
            "gpu_launches": 4800, "breakdown": breakdown, "roofline": roof, "clocks": clocks,
            "gemm_tuning": {"note": "n" * 200, "groups": [
                {"problems": 3, "first_mnk": [8192, 512, 1536], "picked": "one_tile 128x256 s4", "us": us}] * 15},
            "comparator": comp, "error": error, "workloads": {"humanoid": w, "ant": w, "sweep": w},
            "relabel": {"workload": "w" * 45, "kernel": "k" * 60, "results": [
                {"samples_per_launch": 1 << 20, "value": 2294420783.259263, "unit": "samples/s",
                 "us_per_launch": 457.0112, "achieved_gbs": 5295.523, "roofline": roof}] * 2},
            "collect_loop": {"env_steps_per_s": 108119.68507817204, "note": "n" * 200},
            "cpu_baseline": {"value": 0.0773504373755728, "unit": "update steps/s", "cores": 16, "kind": "oracle",
                             "sample": "s" * 130, "one_thread": {"value": None, "note": "n" * 60}}}


def test_the_printed_line_is_short_and_keeps_the_contract(capsys):
    line = full_line()
    assert len(json.dumps(line)) > 20000
    bench.print_line(line)
    got = capsys.readouterr()
    printed = got.out.strip().splitlines()
    assert len(printed) == 1 and len(printed[0]) < 4500
    out = json.loads(printed[0])
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks"):
        assert out[key] == line[key], key
    assert out["e2e"].keys() == line["e2e"].keys() and abs(out["e2e"]["value"] / line["e2e"]["value"] - 1) < 1e-6
    assert out["roofline"]["frac"] == 0.11696
    detail = [l for l in got.err.splitlines() if l.startswith("bench detail: ")]
    assert len(detail) == 1 and json.loads(detail[0][len("bench detail: "):]) == line


def test_the_sweep_workload_runs_with_the_default_arguments(monkeypatch):
    """`--workload sweep` alone: its traced pass takes a kernel class (the default, "auto", is not one)."""
    from paper_2408_11052_gb300 import api
    seen = []

    def arm(args, ws, precision, path, grouped, dev, flush, steps, full):
        seen.append(args.trace)
        return {"ms": 1.0, "e2e_ms": 1.0, "clocks": {}, "launches_per_step": 24, "trace": (10, 1.0, 1e9)}

    monkeypatch.setattr(bench, "run_sweep_arm", arm)
    args = bench.build_parser().parse_args(["--workload", "sweep", "--no-comparator"])
    line = bench.run_sweep(args, None, None)
    assert seen and all(t in api.TRACE for t in seen)
    assert line["roofline"]["kernel_class"] in api.TRACE
