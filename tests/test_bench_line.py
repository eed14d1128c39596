"""bench.py's result line: the contract's keys, whole numbers whole, and short
enough to be found whole at the end of a cut-off output."""
import importlib.util
import json
import os
import time

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
spec = importlib.util.spec_from_file_location("bench", os.path.join(ROOT, "bench.py"))
bench = importlib.util.module_from_spec(spec)
spec.loader.exec_module(bench)

E = 123456789012.34567  # a number of the longest kind


def _full():
    """A result with every section, each far longer than the line may be."""
    noise = {f"extra_{k}": [E] * 50 for k in range(20)}
    return {
        "metric": bench.METRIC, "value": E, "unit": bench.UNIT, "n_gpus": 8, "steps": 1000, "warmup": 100,
        "ms_per_step": E, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
        "data": "synthetic",
        "config": {"workload": bench.WORKLOAD, "items_per_gpu": 4096, "accesses_per_gpu_step": 644096746,
                   "l2": "inputs larger than L2 (traces 2.58 GB per step)",
                   "parallelism": "replicas x8 (independent batches)", "plan": "x" * 4000, "tune": noise},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 288, "power_w_max": E,
                   "reasons": ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]},
        "gpu_launches": 123456,
        "e2e": {"value": E, "unit": bench.UNIT, "h2d_bytes_per_step": 12345678, "d2h_bytes_per_step": 87654321,
                "ms_per_step": E, "path": "y" * 3000},
        "roofline": {"bound": "hbm", "achieved": E, "peak": E, "unit": "GB/s", "frac": E, "kernel_ms": E, **noise},
        "phases_ms": noise, "probes": noise,
        **{k: {**{key: E for key in keys}, **noise} for k, keys in bench.CONTRACT_SUMMARY.items()},
        "cpu_baseline": {"value": E, "unit": bench.UNIT, "cores": 144, "kind": "oracle", "sample": "z" * 2000},
        "parity_ok": True, "parity_items_checked": 512, "parity_accesses_checked": 80373275,
        "parity_mismatched_items": list(range(16))}


def test_the_line_holds_the_contract_and_is_short():
    full = _full()
    full["learned_inverse"]["at_99pct"] = {"threshold": 0.7, "traces_per_s": E, "accuracy_identical_rows": E,
                                           "speedup_vs_judge": E}
    line = bench.contract_line(full)
    assert "\n" not in line and len(line) <= bench.CONTRACT_LINE_MAX <= 2400
    d = json.loads(line)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
              "scaling", "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches", "e2e", "roofline",
              "cpu_baseline", "parity_ok"):
        assert k in d, k
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert k in d["e2e"], k
    for k in ("sm_mhz", "sm_max_mhz", "reasons"):
        assert d["clocks"][k] == full["clocks"][k]
    assert d["metric"] == bench.METRIC and d["config"]["workload"] == bench.WORKLOAD
    assert abs(d["value"] - E) < 1e-5 * E
    assert d["gpu_launches"] == 123456 and d["config"]["accesses_per_gpu_step"] == 644096746


def test_sections_that_failed_or_were_skipped():
    full = {k: v for k, v in _full().items() if k not in ("e2e", "cpu_baseline", "mixed", "parity_ok")}
    full["hierarchy"] = {"error": "RuntimeError('" + "q" * 5000 + "')"}
    full["learned_inverse"] = {"error": "q"}
    d = json.loads(bench.contract_line(full))
    assert d["hierarchy"]["error"].startswith("RuntimeError(") and len(d["hierarchy"]["error"]) == 80
    assert "e2e" not in d and "mixed" not in d and d["learned_inverse"] == {"error": "q"}


def test_clock_samples_have_begun_before_the_steps(tmp_path, monkeypatch):
    """nvidia-smi takes longer to start than the timed steps take: the sampler
    says when its samples have begun to come."""
    fake = tmp_path / "nvidia-smi"
    fake.write_text("#!/bin/sh\nsleep 0.3\nwhile true; do\n"
                    "echo '0, 2000, 2070, 900.0, 0x4, Not Active, Not Active, Not Active, Active'\n"
                    "sleep 0.01\ndone\n")
    fake.chmod(0o755)
    monkeypatch.setenv("PATH", f"{tmp_path}:{os.environ['PATH']}")
    clocks = bench.ClockSampler(0)
    clocks.start()
    assert not clocks.sampling()
    t0 = time.perf_counter()
    while not clocks.sampling():
        assert time.perf_counter() - t0 < 10.0
        time.sleep(0.01)
    time.sleep(0.1)
    got = clocks.stop()
    assert got["sm_mhz"] == 2000.0 and got["sm_max_mhz"] == 2070.0 and got["reasons"] == ["sw_power_cap"]
    assert got["samples"] >= 2
