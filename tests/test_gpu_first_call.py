"""The first call of a process loads the kernels' code.  One file of code holds each family (scheme variants, slabs); a
first step from any of them takes no more than four times the first default step (they are of one size)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys, time, torch
from paper_1808_04960_gb300 import gpweno, workloads as W
torch.zeros(1, device="cuda")
U0, m = W.isentropic_vortex(300)
for opts in ({}, dict(flux="hllc"), dict(sigma_over_dx=12.0), dict(scheme="fdflux"), dict(beta_mean=True)):
    p = gpweno.Plan(3, 12.0, (300, 300), m["dx"], m["bc"], dtype="f32", **opts)
    U, S = torch.from_numpy(U0).to("cuda", torch.float32), p.new_scratch()
    torch.cuda.synchronize()
    t = time.perf_counter()
    p.rk3_step(U, S, dt=1e-6)
    torch.cuda.synchronize()
    print((time.perf_counter() - t) * 1e3)
"""


def test_first_step_of_each_family():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    best = None
    for _ in range(3):   # the smallest of three processes: the machine is shared
        r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, cwd=ROOT, timeout=300,
                           env=dict(os.environ, PYTHONPATH=ROOT))
        assert r.returncode == 0, r.stderr[-2000:]
        ms = [float(x) for x in r.stdout.split()]
        best = ms if best is None else [min(a, b) for a, b in zip(best, ms)]
    print("\nFIRST ms", best)
    assert max(best[1:]) <= 4.0 * best[0], best
