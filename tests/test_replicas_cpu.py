"""The multi-GPU path is replicas only: N independent boxes, no collective
on the data path.  What the benchmark does across ranks -- a barrier, the
slowest rank's time by a MAX all-reduce, the whole-job rate from it, and the
reference arm running on rank 0 alone -- is host logic, checked here with two
gloo ranks on the CPU."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

WORKER = r'''
import os, sys, json
sys.path.insert(0, sys.argv[1])
import torch
import torch.distributed as dist
import bench
dist.init_process_group("gloo")
rank, ws = dist.get_rank(), dist.get_world_size()
mine = [120.0, 150.0][rank]            # this rank's timed milliseconds
tmax = bench.max_over_ranks(torch, dist, ws, mine, "cpu")
rate = bench.whole_job_mlups(ws, 1000, 10, tmax)
with open(os.path.join(sys.argv[2], "rank%d.json" % rank), "w") as fh:
    json.dump({"rank": rank, "tmax": tmax, "rate": rate}, fh)
dist.destroy_process_group()
'''


def _torchrun(args, timeout=240):
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node=2",
           "--master-addr=127.0.0.1", "--master-port=29517"] + args
    env = dict(os.environ, OMP_NUM_THREADS="1")
    return subprocess.run(cmd, capture_output=True, text=True, timeout=timeout, cwd=ROOT, env=env)


def test_max_over_ranks_and_whole_job_rate(tmp_path):
    w = tmp_path / "worker.py"
    w.write_text(WORKER)
    r = _torchrun([str(w), ROOT, str(tmp_path)])
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [json.load(open(tmp_path / ("rank%d.json" % k))) for k in (0, 1)]
    assert sorted(x["rank"] for x in lines) == [0, 1]
    for x in lines:
        assert x["tmax"] == 150.0                       # the slower rank's time on both ranks
        assert x["rate"] == pytest.approx(2 * 1000 * 10 / 0.150 / 1e6)


def test_single_rank_takes_its_own_time():
    import torch
    import bench
    assert bench.max_over_ranks(torch, None, 1, 42.5, "cpu") == 42.5
    assert bench.whole_job_mlups(1, 4194304, 300, 29.0) == pytest.approx(4194304 * 300 / 0.029 / 1e6)


def test_reference_arm_prints_on_rank_zero_only():
    """Under torchrun the reference arm (the CPU oracle) runs on rank 0 alone;
    the other rank exits 0 without work.  A tiny step count keeps it short."""
    r = _torchrun(["bench.py", "--impl", "reference", "--steps", "1", "--warmup", "0"], timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [json.loads(x) for x in r.stdout.splitlines() if x.startswith("{")]
    assert len(lines) == 1
    assert lines[0]["impl"] == "reference" and lines[0]["n_gpus"] == 2 and lines[0]["value"] > 0


def test_result_line_is_short_and_complete(capsys, tmp_path):
    """The line that a recorder keeps the end of: the agreed keys, the main
    figures, under 4,000 characters however much was measured; all of it in
    the details."""
    sys.path.insert(0, ROOT)
    import bench
    keys = {"metric": bench.METRIC, "value": 72000.5, "unit": "MLUPS", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.0545, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": {"workload": bench.WORKLOAD, "l2": "x" * 100}, "gpu_launches": 20,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, "roofline": {"frac": 0.85}}
    e2e = {"value": 58000.0, "unit": "MLUPS", "h2d_bytes_per_step": 1.0, "d2h_bytes_per_step": 2.0}
    line = dict(keys, e2e=dict(e2e, note="n" * 3000), cpu_baseline={"value": 26.1, "unit": "MLUPS", "single": {"x": "y" * 2000}},
                repeats={"blocks": 5, "block_ms": [1.0] * 5, "value_from": "z" * 500})
    case = {"mlups": 1.0, "frac": 0.5, "adjoint_kernel_mlups": 3.0, "grad": [0.123456789] * 600, "rel_err_mean": 1e-4}
    out = {k: {n: dict(case) for n in ("a", "b", "c", "d")} for k in
           ("storage_variants", "adjoint", "cavity_les_f32", "cavity_sweep", "extensions_f32", "drag_error_vs_f64")}
    path = tmp_path / "details.json"
    bench.emit(line, out, str(path))
    cap = capsys.readouterr()
    assert cap.out.count("\n") == 1 and len(cap.out) < 4000
    got = json.loads(cap.out)
    assert all(got[k] == v for k, v in keys.items()) and got["e2e"] == e2e and got["cpu_baseline"]["value"] == 26.1
    assert got["adjoint"]["b"] == {"adjoint_kernel_mlups": 3.0} and got["cavity_les_f32"]["a"] == {"mlups": 1.0, "frac": 0.5}
    full = json.loads(path.read_text())
    assert full == json.loads(cap.err.split("details: ", 1)[1]) and full["cavity_sweep"] == out["cavity_sweep"]
    assert full["e2e"]["note"] == "n" * 3000
