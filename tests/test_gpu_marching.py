"""The marching kernels of large grids, each variant on a grid that is large enough to reach them (checked by the schedule
that the plan reports): FP32 against the tile kernel of small grids, slabs with external sides against the single domain,
the non-physical flag, and all of it in the bounds-checked build.  The same stencils give the same bits.

FP32 2D grids are 131 columns wide: two strips of 66 columns, wider than any tile, and march from 8 rows x 16 CTAs per
SM / 2 strips on, whatever the variant.  FP64 grids march in the allocation-free step, and where 24 layers of
face fluxes exceed 1 GiB."""
import hashlib
import json
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_1808_04960_gb300 import decomp, gpweno  # noqa: E402
from paper_1808_04960_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

PER, OUT = ("periodic", "periodic"), ("outflow", "outflow")
NX, NY = 131, 50
VARIANTS = [(R, {}) for R in (1, 2, 3)] + [
    (2, dict(flux="hllc")), (3, dict(flux="hll")), (1, dict(flux="hllc")), (1, dict(scheme="fdflux")),
    (2, dict(scheme="fdflux")), (3, dict(scheme="fdflux")), (2, dict(ao=True)), (3, dict(ao=True, flux="hllc")),
    (2, dict(beta_mean=True)), (3, dict(beta_mean=True, flux="hll")), (2, dict(sigma_over_dx=12.0)),
    (3, dict(sigma_over_dx=12.0, flux="hllc")), (3, dict(sigma_over_dx=12.0, scheme="fdflux")),
    (2, dict(candidates="poly"))]


def _rows():
    """Rows (a multiple of NY) of a grid of NX columns that marches in every variant."""
    import torch
    sms = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
    return -(-8 * 16 * sms // (2 * NY)) * NY


def _steps(U0, dx, bc, R, dtype, steps=2, **opts):
    import torch
    U = U0.to(torch.float32 if dtype == "f32" else torch.float64).contiguous()
    plan = gpweno.Plan(R, 12.0, U.shape[1:], dx, bc, dtype=dtype, cfl=0.4, **opts)
    dt = torch.full((1,), 0.1 * min(dx), dtype=torch.float64, device="cuda")
    S = plan.new_scratch()
    for _ in range(steps):
        plan.rk3_step(U, S, dt_dev=dt)
    torch.cuda.synchronize()
    return plan, U, S[3], float(dt)


def _field(shape, seed=2):
    import torch
    U0, meta = W.smooth_field(shape, seed=seed)
    return torch.from_numpy(U0).cuda(), meta["dx"]


@pytest.mark.parametrize("R,opts", VARIANTS)
@pytest.mark.parametrize("xbc", [PER, OUT])
def test_marching_equals_tiles(R, opts, xbc):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    U0, dx = _field((NY, NX))
    copies = _rows() // NY
    small, a, lo_a, dt_a = _steps(U0, dx, (xbc, PER), R, "f32", **opts)
    large, b, lo_b, dt_b = _steps(U0.repeat(1, copies, 1), dx, (xbc, PER), R, "f32", **opts)
    assert small.schedule()["strip_width"] <= 64 and large.schedule()["strip_width"] == 66
    assert small.flags() == 0 and large.flags() == 0 and dt_a == dt_b
    for c in (0, copies // 2, copies - 1):
        assert torch.equal(a, b[:, c * NY:(c + 1) * NY]) and torch.equal(lo_a, lo_b[:, c * NY:(c + 1) * NY])


def _slab_steps(U0, dx, bc, R, dtype, steps=2, world=2, **opts):
    """U0 cut into slabs, exchanged by device copies; the slabs' plans and the state put back together."""
    import torch
    slabs = [decomp.Slab(U0.shape[1:], bc, r, world, R + 3) for r in range(world)]
    plans = [gpweno.Plan(R, 12.0, s.local_shape, dx, s.local_bc, dtype=dtype, **opts) for s in slabs]
    steppers = [decomp.SlabStepper(p, s, exchange=lambda *a: None) for p, s in zip(plans, slabs)]
    Us = [U0[:, s.rows].to(torch.float32 if dtype == "f32" else torch.float64).clone(memory_format=torch.contiguous_format)
          for s in slabs]
    for _ in range(steps):
        for k in range(3):
            for st, U in zip(steppers, Us):
                st.pack(k, U)
            for st, s in zip(steppers, slabs):
                if s.lo_rank is not None:
                    st.recv[0].copy_(steppers[s.lo_rank].send[1])
                if s.hi_rank is not None:
                    st.recv[1].copy_(steppers[s.hi_rank].send[0])
            for st, U in zip(steppers, Us):
                st.stage(k, U, dt=0.1 * min(dx))
    torch.cuda.synchronize()
    return plans, torch.cat(Us, dim=1)


def _single_steps(U0, dx, bc, R, dtype, steps=2, **opts):
    import torch
    U = U0.to(torch.float32 if dtype == "f32" else torch.float64).contiguous()
    plan = gpweno.Plan(R, 12.0, U.shape[1:], dx, bc, dtype=dtype, **opts)
    S = plan.new_scratch()
    for _ in range(steps):
        plan.rk3_step(U, S, dt=0.1 * min(dx))
    torch.cuda.synchronize()
    return plan, U


@pytest.mark.parametrize("R,ybc,opts", [(1, PER, {}), (2, OUT, {}), (3, PER, {}), (2, PER, dict(flux="hllc")),
                                        (3, OUT, dict(sigma_over_dx=12.0)), (2, PER, dict(sigma_over_dx=12.0, flux="hll"))])
def test_slabs_of_the_marching_kernel(R, ybc, opts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rows = _rows()
    U0, dx = _field((2 * rows + 1, NX), seed=3)
    bc = (OUT, ybc)
    plans, got = _slab_steps(U0, dx, bc, R, "f32", **opts)
    plan, want = _single_steps(U0, dx, bc, R, "f32", **opts)
    assert all(p.schedule()["strip_width"] == 66 for p in plans + [plan])
    assert all(p.flags() == 0 for p in plans + [plan]) and torch.equal(got, want)


@pytest.mark.parametrize("shape,R,bc", [((49, 330_000), 2, (PER, OUT)), ((49, 330_000), 1, (OUT, PER)),
                                        ((48, 430, 430), 1, (PER, OUT, PER))])
def test_fp64_slabs_without_workspace(shape, R, bc):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    U0, dx = _field(shape[:-1] + (1000 if len(shape) == 2 else shape[-1],), seed=4)
    U0 = U0.repeat(*([1] * len(shape)), shape[-1] // U0.shape[-1])
    plans, got = _slab_steps(U0, dx, bc, R, "f64", steps=1)
    plan, want = _single_steps(U0, dx, bc, R, "f64", steps=1)
    assert all(p.workspace() == 0 and p.flags() == 0 for p in plans + [plan]) and torch.equal(got, want)


@pytest.mark.parametrize("R,opts", [(2, {}), (3, dict(flux="hllc")), (1, dict(scheme="fdflux")), (2, dict(ao=True)),
                                    (3, dict(beta_mean=True)), (2, dict(sigma_over_dx=12.0))])
def test_flag_of_the_marching_kernel(R, opts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    U0, dx = _field((_rows(), NX))
    plan = gpweno.Plan(R, 12.0, U0.shape[1:], dx, (PER, OUT), dtype="f32", **opts)
    for comp, value in ((None, 0.0), (0, -1.0), (0, 0.0), (-1, -1.0), (-1, 0.0), (-1, np.nan), (1, np.inf)):
        U = U0.to(torch.float32)
        if comp is not None:
            U[comp, U.shape[1] // 3, NX // 2] = value
        plan.rhs(U)
        assert plan.flags() == (0 if comp is None else 1), (comp, value)
        assert plan.flags() == 0
    assert plan.schedule()["strip_width"] == 66


def _digest(*tensors):
    h = hashlib.sha1()
    for t in tensors:
        h.update(t.detach().cpu().contiguous().numpy().tobytes())
    return h.hexdigest()[:16]


def run_cases():
    """{name: [digest, flags]} of the marching kernels, with whichever library is loaded."""
    import torch
    out = {}
    rows = _rows()
    U0, dx = _field((rows, NX))
    for k, (R, opts) in enumerate(VARIANTS):
        plan, U, lo, dt = _steps(U0, dx, (OUT if k % 2 else PER, OUT), R, "f32", steps=1, **opts)
        assert plan.schedule()["strip_width"] == 66
        out[f"march_{k}"] = [_digest(U, lo, plan.rhs(U)) + repr(dt), plan.flags()]
    U0, dx = _field((2 * rows + 1, NX), seed=3)
    for R, opts in ((1, {}), (2, dict(flux="hllc")), (3, dict(sigma_over_dx=12.0))):
        plans, U = _slab_steps(U0, dx, (PER, OUT), R, "f32", steps=1, **opts)
        out[f"slabs_R{R}"] = [_digest(U), max(p.flags() for p in plans)]
    for shape, R, opts in (((37, 300), 2, {}), ((260, 131), 3, dict(flux="hllc")), ((64, 31), 1, dict(scheme="fdflux")),
                           ((40, 45), 3, dict(ao=True)), ((9, 14, 33), 3, {}), ((12, 7, 21), 2, dict(beta_mean=True))):
        U, dx = _field(shape, seed=5)
        plan = gpweno.Plan(R, 12.0, shape, dx, (OUT,) * len(shape), dtype="f64", **opts)
        plan.rk3_step_noalloc(U, 0.1 * min(dx))
        torch.cuda.synchronize()
        out["noalloc_%s" % "x".join(map(str, shape))] = [_digest(U), plan.flags()]
    return out


def test_checked_build():
    """As tests/test_gpu_bounds_checked.py does for small grids: no violation, no changed bit."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_04960_gb300 import build
    build.build()
    checked = build.build(checked=True)
    child = subprocess.run([sys.executable, os.path.abspath(__file__), checked], capture_output=True, text=True,
                           timeout=900, cwd=ROOT)
    assert child.returncode == 0, child.stdout[-2000:] + child.stderr[-4000:]
    got = json.loads(child.stdout.strip().splitlines()[-1])
    ref = run_cases()
    assert sorted(got) == sorted(ref)
    assert all(v[1] == 0 for v in got.values()), {k: v[1] for k, v in got.items() if v[1]}
    assert all(got[k][0] == ref[k][0] for k in ref), [k for k in ref if got[k][0] != ref[k][0]]


if __name__ == "__main__":
    gpweno.load(sys.argv[1])
    print(json.dumps(run_cases()))
