"""FP64 2D and 3D steps by face lists (gpweno_rk3_step, one band or several) against the strip-marching
kernels, which the allocation-free step keeps: the same face arithmetic, so the first step from a zero
remainder is equal bit for bit."""
import numpy as np
import pytest

from paper_1808_04960_gb300 import gpweno
from paper_1808_04960_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PER, OUT = ("periodic", "periodic"), ("outflow", "outflow")


@pytest.mark.parametrize("shape,R,bc,opts", [
    ((1, 1), 1, (PER, OUT), {}), ((3, 2), 3, (OUT, PER), {}), ((2, 37), 2, (PER, PER), {}),
    ((97, 33), 2, (PER, PER), {}), ((33, 300), 3, (OUT, OUT), dict(flux="hllc")),
    ((64, 31), 1, (OUT, PER), dict(flux="hll")), ((40, 45), 2, (PER, OUT), dict(scheme="fdflux")),
    ((29, 63), 3, (PER, PER), dict(ao=True)), ((50, 41), 2, (PER, PER), dict(beta_mean=True, candidates="poly")),
    ((2, 1, 3), 2, (PER, OUT, PER), {}), ((9, 14, 33), 3, (OUT, PER, OUT), {}),
    ((21, 7, 12), 2, (PER, PER, PER), dict(scheme="fdflux")),
    ((140, 31, 32), 1, (PER, PER, PER), {}),          # 31.8 MiB of face fluxes: one band
    ((140, 31, 32), 1, (OUT, PER, PER), {}),          # over 32 MiB: two bands of 70 planes, periodic across the border
    ((140, 31, 32), 2, (PER, OUT, OUT), {}),
])
def test_list_step_equals_marching_step(shape, R, bc, opts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    U0, meta = W.smooth_field(shape, seed=11)
    plan = gpweno.Plan(R, 12.0, shape, meta["dx"], bc, dtype="f64", **opts)
    dt = 0.1 * min(meta["dx"])
    a = torch.from_numpy(U0).cuda()
    b = a.clone()
    plan.rk3_step(a, plan.new_scratch(), dt=dt)
    launches = gpweno.last_launch_count()
    plan.rk3_step_noalloc(b, dt)
    torch.cuda.synchronize()
    assert launches == (12 if shape[0] == 140 and OUT in bc else 6)
    assert np.isfinite(a.cpu().numpy()).all() and torch.equal(a, b)
    assert plan.flags() == 0
