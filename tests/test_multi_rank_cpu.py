"""The N > 1 host path of bench.py on CPU (gloo, world size 2, 127.0.0.1):
replicas synchronise on a barrier, the job's time is the slowest rank's,
and the reported value counts every rank's units; under torchrun the
reference arm prints one line from rank 0 and the other ranks exit 0."""
import json
import os
import socket
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def free_port() -> int:
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        return s.getsockname()[1]


def _rank_main(rank, world, port, q):
    os.environ.update(RANK=str(rank), WORLD_SIZE=str(world), LOCAL_RANK=str(rank), MASTER_ADDR="127.0.0.1",
                      MASTER_PORT=str(port))
    sys.path.insert(0, ROOT)
    import bench

    d = bench.Dist("gloo")
    d.barrier()
    # rank r ran 3 steps of 1000 units in 1 + r seconds
    value, ms = bench.whole_job_rate(d, 1000.0, 3, 1.0 + rank)
    d.barrier()
    d.close()
    q.put((rank, value, ms))


def test_replicas_aggregate_over_gloo_ranks():
    import torch.multiprocessing as mp

    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    port = free_port()
    procs = [ctx.Process(target=_rank_main, args=(r, 2, port, q)) for r in range(2)]
    for p in procs:
        p.start()
    for p in procs:
        p.join(timeout=120)
        assert p.exitcode == 0
    got = sorted(q.get(timeout=10) for _ in range(2))
    # slowest rank: 2 s for 3 steps; units: 2 ranks x 3 steps x 1000
    for _, value, ms in got:
        assert value == pytest.approx(6000.0 / 2.0)
        assert ms == pytest.approx(2000.0 / 3)


def test_reference_arm_under_torchrun_prints_once():
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node", "2", "--master-addr",
           "127.0.0.1", "--master-port", str(free_port()), os.path.join(ROOT, "bench.py"), "--impl", "reference",
           "--workload", "conv1x", "--gpus", "2", "--steps", "1", "--warmup", "0"]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [ln for ln in r.stdout.splitlines() if ln.startswith("{")]
    assert len(lines) == 1
    line = json.loads(lines[0])
    assert line["impl"] == "reference" and line["n_gpus"] == 2 and line["value"] > 0
    assert line["cpu_baseline"]["kind"] == "oracle" and line["e2e"]["h2d_bytes_per_step"] == 0


def test_library_sources_use_no_cluster_multicast():
    """Every rank of a run on several GPUs loads this library, and copies with
    cluster multicast are for code that runs on one GPU alone."""
    csrc = os.path.join(ROOT, "paper_1809_10572_gb300", "csrc")
    names = sorted(os.listdir(csrc))
    assert "tc_ptx.cuh" in names
    for name in names:
        with open(os.path.join(csrc, name)) as f:
            assert "multicast" not in f.read(), name
