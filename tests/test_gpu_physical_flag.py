"""The sticky non-physical flag for each way a state can be non-physical, and the batch's choice of kernel by
its members' face fluxes."""
import numpy as np
import pytest

from paper_1808_04960_gb300 import gpweno
from paper_1808_04960_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(40,), (17, 40), (9, 8, 16)])
@pytest.mark.parametrize("opts", [{}, dict(flux="hllc"), dict(scheme="fdflux")])
def test_flag(dtype, shape, opts):
    import torch
    _need_gpu()
    U0, meta = W.smooth_field(shape, seed=3)
    plan = gpweno.Plan(2, 12.0, shape, meta["dx"], meta["bc"], dtype=dtype, **opts)
    at = tuple(n // 2 for n in shape)
    for comp, value in ((None, 0.0), (0, -1.0), (0, 0.0), (-1, -1.0), (-1, 0.0), (-1, np.nan), (1, np.inf)):
        U = torch.from_numpy(U0).to("cuda", plan.dtype)
        if comp is not None:
            U[(comp,) + at] = value
        plan.rhs(U)
        assert plan.flags() == (0 if comp is None else 1), (comp, value)
        assert plan.flags() == 0


@pytest.mark.parametrize("fluxes", [("lf", "lf"), ("lf", "hllc"), ("hll", "hllc")])
def test_batch_by_flux(fluxes):
    import torch
    _need_gpu()
    shapes = [(33, 70), (60, 41)]
    plans, Us, ref = [], [], []
    for flux, shape, R in zip(fluxes, shapes, (2, 3)):
        U0, meta = W.smooth_field(shape, seed=5)
        plans.append(gpweno.Plan(R, 12.0, shape, meta["dx"], meta["bc"], dtype="f32", flux=flux))
        Us.append(torch.from_numpy(U0).to("cuda", torch.float32))
        ref.append(Us[-1].clone())
        plans[-1].rk3_step(ref[-1], plans[-1].new_scratch(), dt=1e-3)
    batch = gpweno.BatchPlan(plans)
    batch.rk3_step(Us, [p.new_scratch() for p in plans], torch.full((2,), 1e-3, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(Us, ref))
