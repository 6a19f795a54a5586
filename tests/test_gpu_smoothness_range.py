"""The nonlinear weights of small data: a shear velocity v with one jump, carried by a uniform flow (u = 0.4, rho = p = 1),
against the FP64 oracle.

FP32 keeps eps + beta at 1e-18 or above, so a jump whose windows have beta well above that has to be treated as
a jump.  The jump's size puts beta = (a1 v)^2 of those windows at about 1e-15, a1 = 1 / |difference row of K_m| the
largest coefficient of the smoothness factor's outer difference: the excess weight of a window across the jump is at most
(1e-18 / 1e-15)^2 = 1e-6 of the others' (linear weights differ by less than 50), times candidates of the jump's size:
below 1e-4 of the right-hand side's largest value (FD-Flux, whose split data are down to 0.6 of the jump: 4e-4), with
FP32 rounding (some 50 ulps of it, 6e-6) far below that; 1e-3 is asked."""
import numpy as np
import pytest

import oracle
from paper_1808_04960_gb300 import gpweno
from paper_1808_04960_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def outer_difference(R, sigma):
    """Coefficient of f_R - f_0 in the factor of K_m(sigma)^-1: square root of its form over the skew vector."""
    K = np.exp(-0.5 * (np.subtract.outer(np.arange(R + 1.0), np.arange(R + 1.0)) / sigma) ** 2)
    t = np.zeros(R + 1)
    t[0], t[-1] = -0.5, 0.5
    return float(np.sqrt(t @ np.linalg.solve(K, t)))


def shear_jump(shape, size):
    n, one = shape[-1], np.ones(shape)
    x = np.arange(n) / n
    v = np.broadcast_to(size * ((x > 0.25) & (x < 0.75)), shape)
    vel = [0.4 * one, v, 0.0 * one][:len(shape)]
    U = W.conserved(one, vel, one, 1.4).astype(np.float32).astype(np.float64)
    return np.ascontiguousarray(U), dict(dx=tuple(1.0 / m for m in reversed(shape)),
                                         bc=(("periodic", "periodic"),) * len(shape))


@pytest.mark.parametrize("R,sigma", [(1, 3.0), (1, 12.0), (2, 3.0), (2, 12.0), (3, 3.0), (3, 12.0), (3, 25.0)])
@pytest.mark.parametrize("shape,opts", [((24, 64), {}), ((24, 64), dict(flux="hllc")), ((24, 64), dict(beta_mean=True)),
                                        ((8, 9, 64), {}), ((24, 64), dict(scheme="fdflux"))])
def test_f32_jump_of_small_data(R, sigma, shape, opts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    U, meta = shear_jump(shape, np.sqrt(1e-15) / outer_difference(R, sigma))
    want = oracle.Oracle(U.shape[1:], meta["dx"], meta["bc"], R=R, sigma_over_dx=sigma, **opts).rhs(U)[2]
    plan = gpweno.Plan(R, 12.0, U.shape[1:], meta["dx"], meta["bc"], dtype="f32", sigma_over_dx=sigma, **opts)
    got = plan.rhs(torch.from_numpy(U).to("cuda", torch.float32).contiguous())[2].double().cpu().numpy()
    assert plan.flags() == 0
    err = np.abs(got - want).max() / np.abs(want).max()
    assert err <= 1e-3


@pytest.mark.parametrize("R,sigma,eps,p", [(1, 12.0, 1e-152, 2), (2, 40.0, 1e-152, 2), (3, 12.0, 1e-153, 2),
                                           (1, 900.0, 1e-303, 1), (3, 3.0, 1e-36, 2)])
def test_f64_smallest_eps(R, sigma, eps, p):
    """FP64 weights of data whose beta is exactly zero (v = 0 beside the jump) stay finite for every eps whose own
    (eps)^-p is; against the oracle, 1e-10 of the largest value, the bound of the FP64 parity tests."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    U, meta = shear_jump((24, 64), 0.1)
    want = oracle.Oracle(U.shape[1:], meta["dx"], meta["bc"], R=R, sigma_over_dx=sigma, eps=eps, p=p).rhs(U)
    plan = gpweno.Plan(R, 12.0, U.shape[1:], meta["dx"], meta["bc"], dtype="f64", sigma_over_dx=sigma, eps=eps, p=p)
    got = plan.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    assert plan.flags() == 0 and np.isfinite(got).all()
    assert np.abs(got - want).max() <= 1e-10 * np.abs(want).max()


@pytest.mark.parametrize("fluxes", [("lf", "lf"), ("hllc", "lf")])
def test_batch_of_both_scales(fluxes):
    """sigma = 3 and 12 dx take different kernels alone; a batch of both equals them bit for bit."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    plans, Us, ref = [], [], []
    for R, sigma, flux, shape in ((2, 3.0, fluxes[0], (33, 70)), (3, 12.0, fluxes[1], (60, 41)), (3, 3.0, "lf", (20, 150)),
                                  (2, 12.0, "lf", (45, 45)), (1, 12.0, "lf", (30, 31))):
        U0, meta = W.smooth_field(shape, seed=5)
        plans.append(gpweno.Plan(R, 12.0, shape, meta["dx"], meta["bc"], dtype="f32", flux=flux, sigma_over_dx=sigma))
        Us.append(torch.from_numpy(U0).to("cuda", torch.float32))
        ref.append(Us[-1].clone())
        plans[-1].rk3_step(ref[-1], plans[-1].new_scratch(), dt=1e-3)
    batch = gpweno.BatchPlan(plans)
    batch.rk3_step(Us, [p.new_scratch() for p in plans], torch.full((5,), 1e-3, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    assert batch.flags() == 0 and all(torch.equal(a, b) for a, b in zip(Us, ref))
