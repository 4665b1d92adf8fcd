"""The benchmark's contract that can be checked without a GPU: the reference arm (the CPU
oracle on a bounded sample) prints one JSON line with the agreed keys, and a plain
`--gpus N` start would re-execute itself under torch.distributed.run."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_one_json_line_with_the_contract_keys():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference",
                          "--config", "config0", "--steps", "2", "--warmup", "1"],
                         capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert out.returncode == 0, out.stderr[-2000:]
    lines = [l for l in out.stdout.splitlines() if l.strip()]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["metric"] == "packed_attn_fwd_bwd_useful_tflops"
    assert d["unit"] == "TFLOP/s" and d["higher_is_better"] is True and d["vs_baseline"] is None
    assert d["steps"] == 2 and d["warmup"] == 1 and d["value"] > 0 and d["ms_per_step"] > 0
    assert d["dtype"] == "f64" and d["data"] == "synthetic" and d["gpu_launches"] == 0
    assert set(d["config"]) == {"workload", "step", "l2", "per_gpu_batch"}     # the GPU arm's keys
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["cpu_baseline"]["value"] == d["value"] and d["e2e"]["value"] == d["value"]
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0


def test_headline_and_target_workloads_are_the_nine_full_size_ones():
    sys.path.insert(0, ROOT)
    import bench
    assert bench.TARGET_CONFIGS == ["config1", "config2", "config3"] + [f"config4:{i}" for i in range(6)]
    assert bench.HEADLINE in bench.TARGET_CONFIGS
    flops = {n: sum(bench.get_workload(n).useful_flops()) for n in bench.TARGET_CONFIGS}
    assert max(flops, key=flops.get) == bench.HEADLINE          # the largest workload is the headline
    # every workload has a tracked DRAM-traffic figure for the roofline
    for n in bench.TARGET_CONFIGS:
        b, how = bench.dram_traffic(n)
        assert b and b > 1e8 and "ncu" in how


def test_the_result_line_is_short_and_holds_the_agreed_keys():
    """Nine workloads, every figure at full length."""
    sys.path.insert(0, ROOT)
    import bench
    x = 1234.5678901234567
    roof = {"kernel": "bwd_kernel (dS/dQ/dK/dV main)", "bound": "tensor", "achieved": x, "peak": x, "unit": "TFLOP/s",
            "frac": x, "peak_kind": "of measured (sustained)", "frac_of_burst_peak": x, "frac_of_sustained_peak": x,
            "traffic": x * 1e7, "traffic_source": "ncu capture of the two DRAM counters (1 pass)",
            "traffic_unit": "bytes (dram read + write per launch)", "algorithmic_flops_per_launch": x * 1e10,
            "avg_launch_ms": x}
    unpacked = {"ms_per_step": x, "tokens": 123998, "speedup_of_packed": 1.8, "useful_pair_ratio": x}
    one = lambda n: {"metric": bench.METRIC, "value": x, "unit": bench.UNIT, "steps": 20, "warmup": 5, "ms_per_step": x,
                     "ms_min_median": [x, x], "config": bench.workload_config(bench.get_workload(n), n),
                     "clocks": {"sm_mhz": 1462.0, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 106},
                     "gpu_launches": 100, "tokens_per_s": x * 1e6, "roofline": roof, "roofline_fwd": roof,
                     "pct_of_peak": {"measured_burst": x, "measured_sustained": x, "nominal": x},
                     "outside_main_kernels_ms": x, "unpacked_padded": unpacked, "unpacked_unpadded": unpacked,
                     "paper_cost_model_mean": {"attention_cost_ratio": x, "memory_ratio": x}}
    per = {n: one(n) for n in bench.TARGET_CONFIGS}
    head = per[bench.HEADLINE]
    extra = {"ms": x, "bytes": x * 1e8, "note": "n" * 90, "roofline": {"achieved": x, "peak": x, "unit": "GB/s", "frac": x}}
    head.update(e2e={"value": x, "unit": bench.UNIT, "h2d_bytes_per_step": 10 ** 9, "d2h_bytes_per_step": 10 ** 9},
                cpu_baseline={"value": x, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 140},
                **{k: extra for k in ("rope_qk", "preference_loss", "deterministic_bwd", "head_dim_96", "row_builder",
                                      "row_assignment", "no_kernel_events", "graph_replay")})
    text = bench.result_line(head, per, 1)
    assert len(text) < 4000 and "\n" not in text
    d = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches"):
        assert key in d
    assert abs(d["value"] - x) < 1e-5 * x and list(d["per_config"]) == bench.TARGET_CONFIGS
    assert d["packed_faster_than_unpacked_on_every_config"] is True
