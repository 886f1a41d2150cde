"""The line that bench.py prints stays short: who runs it may keep only the last 3000 characters of its output. On a record with the
shape and the lengths of a real one."""
import json

import bench
from paper_2212_01005_b200 import workloads as WL


def chain(name, mode):
    roof = {"bound": "tensor", "achieved": 1067.519, "peak": 1691.1, "unit": "TFLOP/s", "frac": 0.6313, "traffic": 29115904,
            "peak_source": "of measured (sustained bf16 figure: SM clocks were power-capped during the timed region)", "us_per_launch": 108.63,
            "roofline_us": 68.573, "algorithmic_tensor_flops": 115964116992.0, "traffic_source": "profiles/ffn_pair_kernel__ffn_12288.txt"}
    return {"chain": name, "mode": mode, "us_per_launch_set": 108.63, "kernels_per_launch_set": 2, "tile_rows": 256, "smem_bytes": 214528, "roofline": roof}


def run(name, parts):
    clocks = {"sm_mhz": 1965.0, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 600}
    cpu = {"value": 4.307994226243495, "unit": "samples/s", "cores": 16, "kind": "oracle",
           "sample": f"2 pass(es) of the oracle over 10 of the 32 samples of one {name} launch set, 4.64 s wall"}
    e2e = {"value": 62113.923176614044, "unit": "samples/s", "h2d_bytes_per_step": 150994944, "d2h_bytes_per_step": 150994944, "launch_sets_per_step": 8, "streams": 4}
    return {"value": 293393.855128703, "unit": "samples/s", "ms_per_step": 0.8725472450256347, "us_per_launch_set": 109.068, "clocks": clocks,
            "chains": [chain(p, "fused") for p in parts], "e2e": e2e, "cpu_baseline": cpu, "fused_speedup_vs_per_mini_subgraph": 0.819,
            "auto_mode_picks": ["per_mini_subgraph"] * len(parts),
            "per_mini_subgraph": {"value": 358323.0400753097, "unit": "samples/s", "us_per_launch_set": 89.305, "chains": [chain(p, "per_mini_subgraph") for p in parts]}}


def test_printed_line_is_short_and_complete():
    names = list(WL.ALL) + bench.parts_of(bench.DEFAULT_WORKLOAD)
    head = run(bench.DEFAULT_WORKLOAD, bench.parts_of(bench.DEFAULT_WORKLOAD))
    record = {"metric": "fused-subgraph samples/s", "value": head["value"], "unit": "samples/s", "n_gpus": 1, "steps": 20, "warmup": 5,
              "ms_per_step": head["ms_per_step"], "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
              "config": {"workload": bench.DEFAULT_WORKLOAD, "chains": bench.parts_of(bench.DEFAULT_WORKLOAD), "mode": "fused", "samples_per_launch_set": 32,
                         "launches_per_step": 24, "buffer_sets": 8, "l2_policy": "8 rotating buffer sets x 141.59 MB >= 4 x L2 (133 MB)", "cuda_graph": True,
                         "parallelism": "replicas x1", "us_per_launch_set": 144.5},
              "roofline": dict(head["chains"][-1]["roofline"], kernel_of="ffn_12288"), "chains": head["chains"], "e2e": head["e2e"], "gpu_launches": 480,
              "clocks": head["clocks"], "context": {"repeats_us_per_launch_set": {"median": 144.5, "best": 144.1, "n": 5}}, "cpu_baseline": head["cpu_baseline"],
              "per_mini_subgraph": head["per_mini_subgraph"], "fused_speedup_vs_per_mini_subgraph": 1.95, "auto_mode_picks": head["auto_mode_picks"],
              "workloads": {n: run(n, [n]) for n in names}}
    assert len(json.dumps(record)) > 10000
    line = bench.headline(record)
    assert len(json.dumps(line)) < 2500
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config",
                "e2e", "gpu_launches", "cpu_baseline"):
        assert line[key] == record[key], key
    assert line["roofline"]["frac"] == 0.6313 and line["clocks"]["reasons"] == ["sw_power_cap"]
    assert set(line["workloads"]) == set(names) and line["workloads"]["ffn_512"] == [109.07, 0.631, 89.31, 0.631]
