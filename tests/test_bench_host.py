"""CPU tests of bench.py's host logic: workload specs, the traffic record's guards, peaks,
the fixed-tuning option and the whole-job arithmetic (no GPU)."""
import argparse
import hashlib
import os

import pytest

import bench


def _args(**kw):
    base = dict(workload="grid3d", size=0, k=0, iters=0, dtype="", tuning="")
    base.update(kw)
    return argparse.Namespace(**base)


def test_default_workload_is_the_400_cubed_grid():
    spec = bench.workload_spec(_args())
    assert (spec["N"], spec["b"], spec["k"], spec["iters"], spec["rescale"], spec["dtype"]) == (400, 4096, 16, 20, True, "f32")
    assert bench.workload_key(spec) == "grid3d N=400 k=16 f32 rescale=1"
    r = bench.workload_spec(_args(workload="rmat"))
    assert (r["N"], r["b"], r["k"], r["iters"], r["dtype"]) == (23, 8192, 128, 8, "bf16")


def test_traffic_record_matches_source_and_workload():
    spec = bench.workload_spec(_args())
    tr = bench.kernel_traffic(bench.workload_key(spec))
    digest = bench.kernel_source_digest()
    if tr is None:
        pytest.skip("traffic record taken on another kernel source")      # reported as null then
    assert tr["kernel_source_sha256_16"] == digest
    dram = float(tr["dram_bytes_per_launch_full_size"])
    alg = float(tr["algorithmic_bytes_per_launch_full_size"])
    assert dram == pytest.approx(float(tr["dram_bytes_read_per_launch_full_size"]) +
                                 float(tr["dram_bytes_write_per_launch_full_size"]), rel=1e-6)
    assert 0.5 < dram / alg < 1.5
    # any other workload (or size) gets no traffic figure
    for other in (_args(size=200), _args(k=32), _args(workload="grid2d")):
        assert bench.kernel_traffic(bench.workload_key(bench.workload_spec(other))) is None


def test_traffic_guard_rejects_a_changed_source(tmp_path, monkeypatch):
    src = tmp_path / "k.cu"
    src.write_text("// another kernel\n")
    monkeypatch.setattr(bench, "KERNEL_SRCS", [str(src)])
    assert bench.kernel_traffic("grid3d N=400 k=16 f32 rescale=1") is None
    assert bench.kernel_traffic("rmat N=23 k=128 bf16 rescale=0") is None


def test_traffic_record_blocks_are_parsed_per_workload(tmp_path, monkeypatch):
    prof = tmp_path / "profiles"
    prof.mkdir()
    d = bench.kernel_source_digest()
    (prof / "arrow_rows_traffic.txt").write_text(
        "# header\nworkload: A\nkernel_source_sha256_16: %s\ndram_bytes_per_launch_full_size: 1\n"
        "workload: B\nkernel_source_sha256_16: 0000\ndram_bytes_per_launch_full_size: 2\n"
        "workload: C\nkernel_source_sha256_16: %s\ndram_bytes_per_launch_full_size: 3\n" % (d, d))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_traffic("A")["dram_bytes_per_launch_full_size"] == "1"
    assert bench.kernel_traffic("B") is None                          # taken on another source
    assert bench.kernel_traffic("C")["dram_bytes_per_launch_full_size"] == "3"
    assert bench.kernel_traffic("D") is None


def test_fixed_tuning_parse():
    assert bench.fixed_tuning(_args()) is None
    assert bench.fixed_tuning(_args(tuning="384,3072,3,85")) == (384, 3072, 3, 85)
    with pytest.raises(SystemExit):
        bench.fixed_tuning(_args(tuning="384,3072"))


def test_peaks_and_job_value():
    peak, kind = bench.load_peaks()
    assert peak > 1000 and kind in ("measured", "fallback")
    if os.path.exists(os.path.join(bench.ROOT, "MEASURED_PEAKS.json")):
        assert kind == "measured"
    # whole-job throughput: every rank's units over the slowest rank's time
    assert bench.job_value(20, 4, 100.0) == pytest.approx(800.0)
    assert bench.max_over_ranks(None, 3.5) == 3.5


def test_reference_arm_prints_the_contract_line():
    # the reference arm times the CPU oracle only: it runs here, without a GPU, and prints one
    # JSON line with the keys the benchmark contract names
    import json
    import subprocess
    import sys
    out = subprocess.run([sys.executable, os.path.join(bench.ROOT, "bench.py"), "--impl", "reference", "--workload",
                          "grid2d", "--steps", "2", "--warmup", "1"], capture_output=True, text=True, timeout=600,
                         cwd=bench.ROOT)
    assert out.returncode == 0, out.stderr[-2000:]
    lines = [l for l in out.stdout.splitlines() if l.startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    for key in ("impl", "metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
                "scaling", "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e"):
        assert key in d, key
    assert d["impl"] == "reference" and d["value"] > 0 and d["steps"] == 2
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["value"] == d["value"]


def test_subrecords_collect_child_lines_and_errors(monkeypatch):
    # the default run attaches the other configurations by running bench.py as child processes;
    # here the children are the CPU-only reference arm (a line comes back) and an unknown option
    # (the error is recorded, not raised)
    monkeypatch.setattr(bench, "SUBRECORDS", [
        ("ok", ["--impl", "reference", "--workload", "grid2d", "--steps", "1", "--warmup", "0"]),
        ("bad", ["--no-such-option"]),
        ("skipped", ["--impl", "reference"]),
    ])
    recs = bench.run_subrecords(["ok", "bad"], timeout_s=600)
    assert set(recs) == {"ok", "bad"}
    assert recs["ok"]["impl"] == "reference" and recs["ok"]["value"] > 0 and recs["ok"]["wall_s"] > 0
    assert "error" in recs["bad"] and recs["bad"]["error"].startswith("rc=")


def test_every_default_subrecord_is_a_known_workload():
    # the children's arguments parse: each names a workload bench.py knows
    for key, args in bench.SUBRECORDS:
        wl = args[args.index("--workload") + 1]
        assert wl in ("grid2d", "rmat", "batch", "serve", "predicates"), (key, wl)
    assert [k for k, _ in bench.SUBRECORDS] == ["grid2d", "rmat", "batch", "serve", "predicates"]


def test_short_line_fits_and_keeps_the_contract():
    """The line that a caller parses from the end of the output: every key of the headline, at most
    1,400 characters with the longest values a run gives."""
    import json
    x = 123456.789012345678
    spec = bench.workload_spec(_args())
    out = {"metric": bench.METRIC, "value": x, "unit": "iters/s", "n_gpus": 1, "steps": 100, "warmup": 10,
           "ms_per_step": x, "step_ms": {"mean": x}, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": "bf16", "data": "synthetic",
           "config": {"workload": max((bench.workload_spec(_args(workload=v))["desc"] for v in ("grid3d", "grid2d", "rmat")),
                                      key=len),
                      "n": spec["N"] ** 3, "b": 4096, "k": 128, "iters": 20, "levels": [[64000000, 353300000]] * 20,
                      "l2": "inputs smaller than L2: a 512 MiB buffer is written", "parallelism": "replicas x1"},
           "roofline": {"bound": "hbm", "achieved": x, "peak": 6784.2, "unit": "GB/s", "frac": x, "traffic": 13361697894.0,
                        "peak_kind": "measured"},
           "gpu_launches": 123456, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap", "gpu_idle"],
                                              "samples": 1000},
           "e2e": {"value": x, "unit": "iters/s", "h2d_bytes_per_step": 4096000000, "d2h_bytes_per_step": 4096000000,
                   "ms_per_step": x, "one_stream": {"value": x}},
           "cusparse": {"iters_per_s": x, "variants": [x] * 100}, "us_per_iter": x,
           "cpu_baseline": {"value": x, "unit": "iters/s", "cores": 16, "kind": "oracle", "sample": "..."},
           "configs": {"grid2d": {"us_per_iter": x}, "rmat": {"value": x, "config": {}},
                       "batch": {"value": x, "speedup_vs_fp32": x}, "serve": {"value": x, "p50_ms": x, "p99_ms": x},
                       "predicates": {"cases": []}}}
    line = bench.short_line(out)
    text = json.dumps(line)
    assert len(text) <= 1400 and "\n" not in text
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert key in line
    assert set(line["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert set(line["clocks"]) == {"sm_mhz", "sm_max_mhz", "reasons"}
    assert abs(line["value"] / x - 1) < 1e-5 and line["steps"] == 100
    # a record without the optional parts, or with a failed configuration, has a line too
    for key in ("e2e", "cusparse", "cpu_baseline", "us_per_iter"):
        del out[key]
    out["configs"] = {"rmat": {"error": "rc=1", "wall_s": x}}
    assert bench.short_line(out)["configs"] == {"rmat": {}}
