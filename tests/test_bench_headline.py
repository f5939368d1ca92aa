"""Host logic of the benchmark line, on the CPU. The headline choice
(bench.choose_headline): `value` is the rate of the fastest precision whose
final iteration met the tolerance in the run, with its step time, its
host-buffer run and its launch count; with none, the FP32 rate stays and no
at-tolerance rate is claimed. The batched workload's CPU baseline
(bench.batched_cpu_baseline): whole trajectories, one per thread."""
import copy

import bench


def line(fp32_ok, refined_ok, mixed_ok):
    return {
        "value": 3.0e9, "ms_per_step": 6.7, "steps": 20, "dtype": "f32",
        "config": {"precision": "fp32"},
        "per_method": {"ieks": "fp32 figures"},
        "fp32": {"value": 3.0e9, "ms_per_step": 6.7, "per_method": {"ieks": "fp32 figures"}},
        "refined": {"value": 2.4e9, "ms_per_step": 8.8, "per_method": {"ieks": "refined figures"}},
        "mixed": {"value": 0.96e9, "ms_per_step": 21.8},
        "e2e": {"value": 2.7e9, "precision": "fp32"},
        "e2e_by_precision": {"fp32": {"value": 2.7e9, "precision": "fp32"},
                             "refined": {"value": 2.1e9, "precision": "refined"}},
        "parity": {"within_tol": {"fp32_final_iteration": fp32_ok, "refined_final_iteration": refined_ok,
                                  "mixed_final_iteration": mixed_ok}},
    }


def test_fp32_is_the_headline_when_it_meets_the_tolerance():
    r = line(True, True, True)
    bench.choose_headline(r)
    assert r["at_oracle_tol"]["precision"] == "fp32" and r["value"] == 3.0e9
    assert r["config"]["precision"] == "fp32" and r["e2e"]["precision"] == "fp32"
    assert r["gpu_launches"] == 7 * 2 * 20


def test_refined_is_the_headline_when_fp32_misses():
    r = line(False, True, True)
    bench.choose_headline(r)
    assert r["at_oracle_tol"] == {"precision": "refined", "value": 2.4e9, "unit": bench.UNIT}
    assert r["value"] == 2.4e9 and r["ms_per_step"] == 8.8
    assert r["config"]["precision"] == "refined" and r["e2e"]["precision"] == "refined"
    assert r["per_method"] == {"ieks": "refined figures"}
    assert r["gpu_launches"] == 12 * 2 * 20


def test_mixed_only_and_none():
    r = line(False, False, True)
    bench.choose_headline(r)
    assert r["at_oracle_tol"]["precision"] == "mixed" and r["dtype"] == "f32 (final iteration f64)"
    r = line(False, False, False)
    before = copy.deepcopy(r)
    bench.choose_headline(r)
    assert r["at_oracle_tol"] is None and r["value"] == before["value"]
    assert r["config"]["precision"].startswith("fp32 (no precision met")


def test_batched_cpu_baseline_times_whole_trajectories_on_all_cores():
    from paper_2102_00514_gb300 import synth
    wl = synth.ct_bearings([30, 50, 20, 40, 10], seed=3, omega0_halfwidth=1.0)
    rec = bench.batched_cpu_baseline(wl, iters=2, budget_states=100, cores=3)
    assert rec["kind"] == "oracle" and rec["cores"] == 3 and rec["unit"] == bench.UNIT
    n = int(rec["sample"].split(" of ")[0])
    assert 1 <= n <= 5 and rec["value"] > 0
    # whole trajectories, at most the budget of states unless one alone exceeds it
    steps = int(rec["sample"].split("(")[1].split(" steps")[0])
    assert steps <= 100 or n == 1


def test_per_state_errors_are_relative_to_each_state():
    import numpy as np
    b = np.array([[1.0, 0.0, 3.0], [0.0, 2.0, 4.0]])
    a = b + np.array([[0.1, 0.0, 0.0], [0.0, 0.0, 0.5]])
    e = bench.per_state_errors(a, b)
    assert np.allclose(e, [0.1, 0.0, 0.1])
    assert bench.per_state_max(a, b) == e.max()


def full_record():
    """A record with every block that a default run fills, long ones as long as there."""
    r = line(False, True, True)
    long_block = {f"key_{i}": {"value": 1.0 / 3.0, "per_method": {"ieks": [0.1] * 40}} for i in range(40)}
    r.update({"metric": bench.METRIC, "unit": bench.UNIT, "n_gpus": 1, "warmup": 5, "higher_is_better": True,
              "scaling": "weak", "vs_baseline": None,
              "data": "synthetic coordinated-turn / bearings (seeded, seed 20210204), inputs resident in HBM",
              "launches_per_run": {"fp32": 6, "refined": 11, "mixed": 17},
              "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "nvidia_smi": long_block},
              "roofline": {"bound": "alu", "achieved": 100.0 / 3.0, "peak": 80.5, "unit": "TFLOP/s", "frac": 1.0 / 3.0,
                           "kernel": "pes_persistent_kernel<float, cubature>", "executed": long_block},
              "fp64": {"value": 1.0e8 / 3.0, "ms_per_step": 635.0 / 3.0}, "graph": {"value": 3.1e9, "ms_per_step": 6.6},
              "iters_saved": 1.46, "learned_init": long_block, "length_sweep": long_block,
              "batched": dict(long_block, N_states=41900000, B=4096, fp32={"value": 5.8e9, "ms_per_step": 144.0},
                              refined={"value": 3.8e9, "ms_per_step": 219.0}),
              "cpu_baseline": {"value": 6.3e5, "unit": bench.UNIT, "cores": 1, "kind": "oracle",
                               "sample": "first 131072 of 1048577 states (1 trajectories), IEKS + cubature, 10 "
                                         "iterations, sequential FP64 oracle"}})
    r["parity"]["rel_frobenius"] = long_block
    r["config"].update({"workload": "single trajectory T=1048576, IEKS + cubature IPLS, 10 iterations each, FP32, "
                                    "prior initialisation", "T": 1 << 20, "B": 1, "N_states": (1 << 20) + 1,
                        "iterations": 10, "methods": ["ieks", "cubature"], "l2": "flushed before every step",
                        "launch": {"ieks": {"blocks": 152, "threads": 256, "steps_per_thread": 27},
                                   "cubature": {"blocks": 304, "threads": 128, "steps_per_thread": 27},
                                   "autotuned": long_block}})
    for e in (r["e2e"], *r["e2e_by_precision"].values()):
        e.update({"unit": bench.UNIT, "h2d_bytes_per_step": 16777632, "d2h_bytes_per_step": 167772320,
                  "ms_per_step": 7.0, "serial": long_block})
    return r


def test_printed_line_is_complete_and_short():
    """stdout's line keeps the contract's keys and fits the last 2,800 characters of a log."""
    import json
    r = full_record()
    bench.choose_headline(r)
    c = bench.compact_line(r)
    assert len(json.dumps(c)) < 2800
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline"):
        assert k in c, k
    assert c["value"] == r["value"] == 2.4e9 and c["config"]["precision"] == "refined"
    assert c["e2e"]["value"] == 2.1e9 and {"h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(c["e2e"])
    assert {"sm_mhz", "sm_max_mhz", "reasons"} == set(c["clocks"])
    assert c["batched"]["refined"] == {"value": 3.8e9, "ms_per_step": 219.0}


def test_launch_counts_of_the_line_are_used():
    r = full_record()
    bench.choose_headline(r)
    assert r["gpu_launches"] == 11 * 2 * 20
