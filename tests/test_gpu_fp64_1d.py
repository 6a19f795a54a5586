"""FP64 1D right-hand sides and steps around the sizes where the kernel changes (field-split CTAs of 27 cells up to
three per SM, 128-thread CTAs of 123 beyond), against the oracle: 1e-10 of the largest value, the bound of the smooth FP64
parity tests; and the same grid through an LF, HLLC and non-zero-mean plan of both kernels, equal bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1808_04960_gb300 import gpweno
from paper_1808_04960_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 27, 28, 54, 55, 2 * 152 * 27, 3 * 152 * 27, 3 * 152 * 27 + 1, 152 * 123 + 1])
@pytest.mark.parametrize("R", [1, 3])
def test_rhs_1d(n, R):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    U0, meta = W.smooth_field((n,), seed=4)
    plan = gpweno.Plan(R, 12.0, (n,), meta["dx"], meta["bc"], dtype="f64")
    got = plan.rhs(torch.from_numpy(U0).cuda()).cpu().numpy()
    want = oracle.Oracle((n,), meta["dx"], meta["bc"], R=R, ell_over_dx=12.0).rhs(U0)
    assert plan.flags() == 0
    assert np.abs(got - want).max() <= 1e-10 * max(1.0, np.abs(want).max())


@pytest.mark.parametrize("opts", [{}, dict(flux="hllc"), dict(flux="hll"), dict(beta_mean=True, candidates="poly")])
@pytest.mark.parametrize("n,R", [(40, 2), (83, 3), (256, 1)])
def test_split_equals_plain(n, R, opts):
    """A periodic tube and the same tube repeated until it takes the plain kernel."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    U0, meta = W.smooth_field((n,), seed=4)
    got = []
    for copies in (1, -(-13000 // n)):
        U = torch.from_numpy(np.concatenate([U0] * copies, axis=1)).cuda().contiguous()
        plan = gpweno.Plan(R, 12.0, U.shape[1:], meta["dx"], meta["bc"], dtype="f64", cfl=0.4, **opts)
        dt = torch.full((1,), 0.1 * meta["dx"][0], dtype=torch.float64, device="cuda")
        S = plan.new_scratch()
        for _ in range(2):
            plan.rk3_step(U, S, dt_dev=dt)
        torch.cuda.synchronize()
        assert plan.flags() == 0
        got.append((U[:, :n].clone(), float(dt)))
    assert torch.equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
