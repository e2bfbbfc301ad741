"""bench.py's reference arm (the FP64 oracle on the host cores) and its launch
under torchrun: with two ranks only rank 0 works and prints, the other exits 0
(the GPU arm runs independent replicas per rank; nothing here needs a GPU)."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ARGS = ["--impl", "reference", "--steps", "1", "--warmup", "0", "--sample-n", "2", "--sample-nr", "2",
        "--order", "2"]


def json_lines(out):
    return [json.loads(l) for l in out.splitlines() if l.startswith("{")]


def test_reference_arm_line():
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py")] + ARGS, capture_output=True,
                       text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = json_lines(r.stdout)
    assert len(lines) == 1
    d = lines[0]
    assert d["impl"] == "reference" and d["value"] > 0 and d["unit"] == "zone-updates/s"
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["value"] == d["value"]
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0


def test_reference_arm_two_ranks_prints_once():
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node", "2",
           "--master-addr", "127.0.0.1", "--master-port", "29517", os.path.join(ROOT, "bench.py"),
           "--gpus", "2"] + ARGS
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = json_lines(r.stdout)
    assert len(lines) == 1 and lines[0]["n_gpus"] == 2


@pytest.mark.parametrize("p,n,nnz,nedge", [(2, 8, 16, 1), (3, 20, 96, 2), (4, 32, 192, 3)])
def test_roofline_counts_what_the_predictor_executes(p, n, nnz, nedge):
    """The roofline's operations are those of the kernel that ran: for the ring predictor the
    operations of its contraction (counted here by running its formulas on numbers that
    count), not the sparse rows' of geo_stage_flops, with which it came out above the peak."""
    import bench

    class Num:
        ops = 0

        def __add__(self, o):
            Num.ops += 1
            return Num()
        __sub__ = __mul__ = __rmul__ = __add__

    x = [Num() for _ in range(8)]
    if p == 2:
        x[1] - x[0]
        Num.ops *= 2  # each end takes the difference itself
    elif p == 3:
        d, g = x[2] - x[0], (x[0] + x[2]) - 2.0 * x[1]
        G, t = g + x[5], x[4] - x[3]
        d - 2.0 * g, d + 2.0 * g, t - G, t + G
    else:
        u, g = x[3] - x[0], (x[0] + x[3]) - (x[1] + x[2])
        r = u - 3.0 * (x[2] - x[1])
        A, B, t1, t2 = r + g, r - g, x[6] - x[4], x[7] - x[5]
        u + 2.25 * B, u - 0.75 * A, u - 0.75 * B, u + 2.25 * A
        for t, y in ((t1, B), (t2, B), (t1, A), (t2, A)):
            (t + 1.5 * y) + 0.75 * x[0]
    ring = 4 * Num.ops + n          # four ring edges, then a sum at every node
    levels = 1 + (p - 1) * (p - 1)
    points = (p - 1) * 12 * (nedge - 1) * 4 * 16 if p == 4 else 0
    counted = 1e6
    got = bench.executed_flops(counted, "ader", bench.kernel_name("ader", None, False, p), p)
    assert got == counted - levels * 24 * (2 * nnz - ring) - points
    assert bench.executed_flops(counted, "ader", "k_ader_team", p) == counted
    assert bench.executed_flops(counted, "weno", "k_weno", p) == counted
