"""bench.py's Legendre roofline where the FP64 mode runs the plain kernels: no tensor-core launches to divide
by (no GPU for the arithmetic; one short run of the bench on the GPU)."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_plain_legendre_figures():
    import bench
    st = {"legendre_synth": (2.0, 4), "legendre_anal": (5.0, 6), "tc_synth_kernel": (0.0, 0), "tc_anal_kernel": (0.0, 0)}
    r = bench.plain_legendre_figures(st, 2, 3, 1000, 1.0, 0.5)
    # 1000 steps x (3 flops x 6 launches + 4 flops x 3 maps x 2 round trips) in 5 ms
    assert r["kernel"] == "legendre_anal_kernel" and abs(r["achieved"] - 1000 * 42 / 5e-3 / 1e12) < 1e-18
    assert r["frac"] == r["achieved"] and abs(r["frac_of_executed"] - 0.5 * r["achieved"]) < 1e-18


@pytest.mark.gpu
def test_bench_runs_below_the_tensor_core_sizes():
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--mode", "fp64", "--nside", "32", "--lmax", "64",
                        "--maps", "2", "--steps", "2", "--warmup", "3", "--serve-requests", "0", "--batch-maps", "0",
                        "--no-c2"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    d = json.loads(r.stdout.strip().splitlines()[-1])
    assert d["roofline"]["kernel"] in ("legendre_synth_kernel", "legendre_anal_kernel") and d["roofline"]["frac"] > 0
