"""bench.py's reference arm: the FP64 oracle timed on the host cores.

It runs without a GPU, prints exactly one JSON line with the keys of the
benchmark line (plus its own `cpu_baseline` and an `e2e` equal to its value),
and under a two-rank launch only rank 0 prints while the other rank exits 0.
"""
import json
import os
import socket
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KEYS = ("impl", "metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
        "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e")


def _json_lines(text):
    return [json.loads(s) for s in text.splitlines() if s.lstrip().startswith("{")]


def _check_line(d, n_gpus, workload):
    for key in KEYS:
        assert key in d, key
    assert d["impl"] == "reference" and d["n_gpus"] == n_gpus
    assert d["value"] > 0 and d["unit"] == "solves/s" and d["higher_is_better"] is True
    assert abs(d["ms_per_step"] - 1e3 / d["value"]) <= 1e-6 * d["ms_per_step"]
    assert d["config"]["workload"] == workload
    cb = d["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["cores"] >= 1 and cb["value"] == d["value"] and cb["sample"]
    assert d["e2e"] == {"value": d["value"], "unit": d["unit"], "h2d_bytes_per_step": 0,
                        "d2h_bytes_per_step": 0}


def test_reference_arm_prints_one_line():
    r = subprocess.run([sys.executable, "bench.py", "--impl", "reference", "--steps", "1",
                        "--warmup", "1"], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = _json_lines(r.stdout)
    assert len(lines) == 1, r.stdout[-2000:]
    _check_line(lines[0], 1, "manifolds_1000000x128_L100")


def test_reference_arm_two_ranks_rank0_alone_prints():
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        port = s.getsockname()[1]
    r = subprocess.run([sys.executable, "-m", "torch.distributed.run", "--nnodes=1",
                        "--nproc-per-node", "2", "--master-addr", "127.0.0.1",
                        "--master-port", str(port), "bench.py", "--impl", "reference",
                        "--workload", "mnist_like", "--gpus", "2", "--steps", "1", "--warmup", "1"],
                       cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = _json_lines(r.stdout)
    assert len(lines) == 1, r.stdout[-2000:]
    _check_line(lines[0], 2, "mnist_like_70000x784_L10")


def test_traffic_records_match_their_kernels():
    """A recorded DRAM traffic is reported as long as its kernel is unchanged, and
    is not kept beyond that."""
    sys.path.insert(0, ROOT)
    import bench
    for (kernel, workload), rec in bench.NCU_TRAFFIC.items():
        assert bench.ncu_traffic(kernel, workload) == rec["bytes"]
