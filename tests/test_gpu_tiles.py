"""The tile kernel of small FP32 2D grids against the strip-marching kernel: a grid periodic in y and the same
grid stacked k times in y (large enough to march) have the same stencils, so their steps agree bit for bit."""
import numpy as np
import pytest

from paper_1808_04960_gb300 import gpweno
from paper_1808_04960_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,R,opts", [
    (1, 1, 2, {}), (2, 5, 3, {}), (5, 64, 1, {}), (64, 4, 2, {}), (63, 65, 3, {}), (129, 37, 1, {}), (256, 250, 2, {}),
    (300, 190, 3, {}), (61, 50, 2, dict(flux="hllc")), (61, 50, 3, dict(flux="hll")),
    (61, 50, 2, dict(scheme="fdflux")), (61, 50, 3, dict(scheme="fdflux")), (61, 50, 1, dict(scheme="fdflux")),
    (61, 50, 2, dict(ao=True)), (61, 50, 3, dict(ao=True, flux="hllc")), (61, 50, 2, dict(beta_mean=True)),
])
@pytest.mark.parametrize("xbc", ["periodic", "outflow"])
def test_tile_equals_marching(nx, ny, R, opts, xbc):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    U0, meta = W.smooth_field((ny, nx), seed=2)
    bc = ((xbc, xbc), ("periodic", "periodic"))
    k = -(-8 * 2 * 160 // ny)          # at least two CTAs of eight rows per SM: the stacked grid marches
    got = []
    for copies in (1, k):
        U = torch.from_numpy(np.concatenate([U0] * copies, axis=1)).to("cuda", torch.float32).contiguous()
        plan = gpweno.Plan(R, 12.0, U.shape[1:], meta["dx"], bc, dtype="f32", cfl=0.4, **opts)
        dt = torch.full((1,), 0.1 * min(meta["dx"]), dtype=torch.float64, device="cuda")
        S = plan.new_scratch()
        for _ in range(2):
            plan.rk3_step(U, S, dt_dev=dt)
        torch.cuda.synchronize()
        assert plan.flags() == 0
        got.append((U[:, :ny].clone(), S[3, :, :ny].clone(), float(dt)))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1]) and got[0][2] == got[1][2]
