"""The benchmark's reference arm (the FP64 oracle on the host cores) keeps the
one-JSON-line contract, alone and under torchrun with two ranks (rank 0
prints, the other rank exits without work). CPU only."""
import json
import os
import socket
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _json_lines(out: str):
    return [json.loads(l) for l in out.splitlines() if l.startswith("{")]


def _check_line(d, n_gpus):
    assert d["impl"] == "reference"
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config",
              "cpu_baseline", "e2e"):
        assert k in d, k
    assert d["n_gpus"] == n_gpus and d["steps"] == 1 and d["warmup"] >= 3
    assert d["value"] > 0 and d["unit"] == "events/s" and d["higher_is_better"] is True
    assert d["dtype"] == "f64" and d["data"] == "synthetic"
    cb = d["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["cores"] >= 1 and cb["value"] == d["value"]
    assert d["e2e"] == {"value": d["value"], "unit": d["unit"], "h2d_bytes_per_step": 0,
                        "d2h_bytes_per_step": 0}
    assert isinstance(d["config"]["workload"], str)


def test_reference_arm_one_line():
    r = subprocess.run([sys.executable, "bench.py", "--impl", "reference", "--steps", "1",
                        "--warmup", "3"], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = _json_lines(r.stdout)
    assert len(lines) == 1
    _check_line(lines[0], 1)


def test_reference_arm_under_torchrun_prints_once():
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        port = s.getsockname()[1]
    r = subprocess.run([sys.executable, "-m", "torch.distributed.run", "--nnodes=1",
                        "--nproc-per-node", "2", "--master-addr", "127.0.0.1", "--master-port",
                        str(port), "bench.py", "--impl", "reference", "--gpus", "2", "--steps",
                        "1", "--warmup", "3"], cwd=ROOT, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = _json_lines(r.stdout)
    assert len(lines) == 1
    _check_line(lines[0], 2)


def test_own_arm_line_stays_short():
    """The stdout line of the library's arm has every key of the contract and stays
    short whatever the other legs report; nothing that they report is lost."""
    sys.path.insert(0, ROOT)
    import bench
    big = {f"key_{i}": 0.123456789 for i in range(400)}
    stages = {f"stage_name_{i}": {"ms_per_step": 0.1234, "bound": "hbm", "achieved": 1234.56,
                                  "unit": "GB/s", "frac": 0.1234} for i in range(16)}
    out = {"metric": bench.METRIC, "value": 100000.1, "unit": "events/s", "n_gpus": 1, "steps": 20,
           "warmup": 5, "ms_per_step": 10.1234, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "bf16", "data": "synthetic", "hits_per_s": 123456789.1,
           "p50_step_ms": 8.1234, "p99_step_ms": 8.1234,
           "config": {"workload": "w" * 300, "n_events": 1000, "hits": 1684232, "edges": 10117076,
                      "kept_edges": 8802916, "net": "embed 3-64-64-4, IN h32 K4",
                      "precision": "bf16", "rescore_band": 0.02, "band_edges": 702891,
                      "rerun_events": 1000, "rescore_rows": big, "launch": "l" * 60,
                      "autotuned_ctas_per_sm": {k: 8 for k in ("tc_node_prep", "tc_edge_encoder",
                                                               "tc_node_update", "tc_edge_update",
                                                               "f32_encoders", "f32_node_update",
                                                               "f32_edge_update", "tc_edge_tma")},
                      "l2": "l" * 40, "parallelism": "p" * 60},
           "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 8, "reasons": []},
           "roofline": {"kernel": "rescore_edge_update", "bound": "alu", "achieved": 27.8,
                        "peak": 80.54784, "unit": "TFLOP/s", "frac": 0.3452, "traffic": 1094886559,
                        "traffic_unit": "t" * 80, "counters": big, "peak_src": "p" * 80,
                        "launch_ms": 0.5767, "work": "w" * 80, "profiled_ms_per_step": 11.4174,
                        "stage_ms_per_step": big, "stages": stages},
           "e2e": {"value": 88222.0, "unit": "events/s", "h2d_bytes_per_step": 21903024,
                   "d2h_bytes_per_step": 6736928, "ms_per_step": 11.335},
           "gpu_launches": 920, "batched_over_plain": 10.12, "batched_over_plain_hits": 30.12,
           "wall_s_timed": 0.22, "serving": big, "occupancy_study": big, "fp8_report": big,
           "cpu_baseline": {"value": 104.36, "unit": "events/s", "hits_per_s": 175767.0, "cores": 16,
                            "kind": "oracle", "sample": "s" * 100, "one_core": {"sample": "s" * 60},
                            "max_score_error": 0.0070983405964239465}}
    line, legs = bench.split_line(out)
    assert len(json.dumps(line)) < bench.LINE_MAX <= 4000
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "clocks",
              "e2e", "gpu_launches", "roofline", "cpu_baseline"):
        assert k in line, k
    for k, v in out.items():
        assert {**legs[k], **line.get(k, {})} == v if k in legs else line[k] == v, k
