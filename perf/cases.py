"""Performance cases of the GP-WENO framework: what its users have it do, from the smallest call to the largest.

Every pass goes through the public binding (``gpweno.Plan``, ``gpweno.BatchPlan``).  A case is a dict of plain values:

  problem   "sod" (1D shock tube), "vortex" (2D, periodic), "quadrant" (2D four-state Riemann problem, outflow),
            "smooth" (any dimension, periodic), "shock" (3D Mach-3 shock into a random density field), "batch"
            (many 2D instances of uneven size, R and l/dx, half quadrant and half vortex)
  call      "step" (one SSP-RK3 step in place) or "rhs" (one right-hand side)
  nx, ny, nz, R, ell (l/dx), dtype ("f32"/"f64"), flux, scheme, ao, candidates: the plan's options
  cfl       > 0: the step reads its time step from the device and writes the next one there; 0: fixed time step
  count, mix  batches: number of instances and the number their sizes are drawn from

``exact`` is the scheme in 64 bits with plain torch, its GP tables from exact decimal arithmetic; it shares no code
with the library.
"""
from __future__ import annotations

import decimal
import math
import random
from decimal import Decimal
from functools import lru_cache

import numpy as np
import torch

from paper_1808_04960_gb300 import costmodel, gpweno

GAMMA = 1.4
SIGMA = 3.0
EPS = 1e-36
CFL = 0.4
BATCH_CFL = 0.2      # fixed time steps: room for the wave speeds to grow
AO_GAMMA = 0.85


def listed():
    def case(name, problem, nx, ny=0, nz=0, R=2, dtype="f32", call="step", cfl=0.0, **more):
        return dict(dict(name=name, problem=problem, call=call, nx=nx, ny=ny, nz=nz, R=R, ell=12.0, dtype=dtype,
                         flux="lf", scheme="fdprim", ao=False, candidates="gp", cfl=cfl, count=0, mix=0), **more)

    return [
        # the smallest call: the 1D Sod tube of the paper's shock-tube tests, FP64, CFL time step; launches count
        case("sod_256_f64", "sod", 256, dtype="f64", cfl=CFL),
        # a grid of the vortex convergence study (Table 2), FP64 at the highest order
        case("vortex_128_f64_R3", "vortex", 128, 128, R=3, dtype="f64"),
        # a small FP32 grid: few CTAs, latency counts
        case("vortex_256_f32", "vortex", 256, 256),
        # FP64 production grid of the vortex configuration
        case("vortex_512_f64", "vortex", 512, 512, dtype="f64"),
        # the headline workload of the benchmark: FP32 vortex at the largest grid of its configuration
        case("vortex_1024_f32", "vortex", 1024, 1024),
        # the right-hand side alone (a user with an integrator of their own), R = 1, ragged sizes
        case("rhs_777x613_f32_R1", "smooth", 777, 613, R=1, call="rhs"),
        # the four-quadrant shock problem at its full size, CFL time step
        case("quadrant_4096_f32", "quadrant", 4096, 4096, cfl=CFL),
        # the paper's default solver (HLLC) at the highest order on a ragged shock problem
        case("hllc_1501x1100_f32_R3", "quadrant", 1501, 1100, R=3, flux="hllc", cfl=CFL),
        # the adaptive-order scheme (GP-AO(3,2,3)) on shocks
        case("ao_1000x900_f32_R3", "quadrant", 1000, 900, R=3, ao=True, cfl=CFL),
        # 3D FP64 right-hand side on a small ragged box
        case("rhs3d_70x61x45_f64", "smooth", 70, 61, 45, dtype="f64", call="rhs"),
        # the 3D shock-turbulence box at its full size, R = 3
        case("shock3d_512_f32_R3", "shock", 512, 512, 512, R=3, cfl=CFL),
        # the batched path: 256 uneven instances in one launch per stage
        case("batch_256_f32", "batch", 0, count=256, mix=5, R=0, ell=0.0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = dict(problem="", call="step", nx=0, ny=0, nz=0, R=rng.choice([1, 2, 2, 3]), ell=rng.choice([6.0, 12.0, 12.0, 24.0]),
             dtype="f32", flux="lf", scheme="fdprim", ao=False, candidates="gp", cfl=0.0, count=0, mix=0)
    kind = rng.choice(["1d", "vortex", "vortex64", "quadrant", "variant", "rhs", "3d", "3d64", "batch"])
    if kind == "1d":
        c.update(problem="sod", nx=log_int(50, 20000), dtype=rng.choice(["f32", "f64"]), cfl=CFL)
    elif kind == "vortex":
        c.update(problem="vortex", nx=log_int(64, 2048), ny=log_int(64, 2048), cfl=rng.choice([0.0, CFL]))
    elif kind == "vortex64":
        c.update(problem="vortex", nx=log_int(48, 1024), ny=log_int(48, 1024), dtype="f64")
    elif kind == "quadrant":
        c.update(problem="quadrant", nx=log_int(200, 4096), ny=log_int(200, 4096), cfl=CFL)
    elif kind == "variant":
        c.update(problem="quadrant", nx=log_int(200, 2048), ny=log_int(200, 2048), cfl=CFL)
        c.update(rng.choice([dict(flux="hllc"), dict(flux="hll"), dict(scheme="fdflux"), dict(candidates="poly"),
                             dict(ao=True, R=rng.choice([2, 3]))]))
    elif kind == "rhs":
        c.update(problem="smooth", call="rhs", nx=log_int(40, 2048), ny=log_int(40, 2048))
    elif kind == "3d":
        c.update(problem="shock", nx=log_int(32, 320), cfl=CFL)
        c.update(ny=c["nx"], nz=c["nx"])
    elif kind == "3d64":
        c.update(problem="smooth", nx=log_int(20, 100), ny=log_int(20, 100), nz=log_int(20, 100), dtype="f64",
                 call=rng.choice(["rhs", "step"]))
    else:
        c.update(problem="batch", count=log_int(8, 256), mix=rng.randrange(1, 1 << 20), R=0, ell=0.0)
    return c


# ---------------------------------------------------------------------------
# inputs: conserved states in FP64 on the GPU, then rounded to the plan's type


def _dev(x):
    return torch.as_tensor(x, dtype=torch.float64, device="cuda")


def _centres(n, lo=0.0, hi=1.0):
    dx = (hi - lo) / n
    return lo + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * dx, dx


def _conserved(rho, vel, p):
    ke = sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [p / (GAMMA - 1.0) + 0.5 * rho * ke])


def _field(problem, shape, seed):
    """(U, dx in (x, y, z) order, boundary conditions in the same order) of one instance."""
    rng = np.random.default_rng([int(seed), 1808])
    per, out = ("periodic", "periodic"), ("outflow", "outflow")
    if problem == "sod":
        x, dx = _centres(shape[0])
        rl, pl = 1.0 + 0.1 * rng.uniform(-1, 1), 1.0 + 0.1 * rng.uniform(-1, 1)
        left = x < 0.5
        rho = torch.where(left, _dev(rl), _dev(0.125))
        return _conserved(rho, [torch.zeros_like(x)], torch.where(left, _dev(pl), _dev(0.1))), (dx,), (out,)
    if problem == "vortex":
        ny, nx = shape
        (x, dx), (y, dy) = _centres(nx, -5.0, 5.0), _centres(ny, -5.0, 5.0)
        beta, cx, cy = rng.uniform(2.0, 6.0), rng.uniform(-0.5, 0.5), rng.uniform(-0.5, 0.5)
        X, Y = x[None, :] - cx, y[:, None] - cy
        e = torch.exp(0.5 * (1.0 - X * X - Y * Y))
        T = 1.0 - (GAMMA - 1.0) * beta ** 2 / (8.0 * GAMMA * math.pi ** 2) * e * e
        amp = beta / (2.0 * math.pi) * e
        rho = T ** (1.0 / (GAMMA - 1.0))
        return _conserved(rho, [1.0 - amp * Y, 1.0 + amp * X], rho ** GAMMA), (dx, dy), (per, per)
    if problem == "quadrant":
        ny, nx = shape
        (x, dx), (y, dy) = _centres(nx), _centres(ny)
        st = _dev(np.stack([rng.uniform(0.1, 1.5, 4), rng.uniform(-1, 1, 4), rng.uniform(-1, 1, 4),
                            rng.uniform(0.03, 1.5, 4)]))
        q = torch.where(y[:, None] >= 0.5, torch.where(x[None, :] >= 0.5, 0, 1), torch.where(x[None, :] < 0.5, 2, 3))
        return _conserved(st[0][q], [st[1][q], st[2][q]], st[3][q]), (dx, dy), (out, out)
    if problem == "smooth":
        nd = len(shape)
        ax = [_centres(n) for n in reversed(shape)]                    # x, y, z
        prims = []
        for base in [1.0] + [0.3] * nd + [1.0]:
            f = torch.full(tuple(shape), base, dtype=torch.float64, device="cuda")
            for _ in range(3):
                arg = rng.uniform(0.0, 2.0 * math.pi)
                for d in range(nd):
                    arg = arg + (2.0 * math.pi * int(rng.integers(1, 4)) * ax[d][0]).reshape([-1] + [1] * d)
                f = f + 0.2 / 3 * torch.sin(arg)
            prims.append(f)
        return _conserved(prims[0], prims[1:1 + nd], prims[-1]), tuple(a[1] for a in ax), (per,) * nd
    # shock: Mach-3 shock at x = 0.25 moving into rho = 1 + 32 random modes of RMS 0.1
    nz, ny, nx = shape
    ks = []
    while len(ks) < 32:
        k = rng.integers(-8, 9, 3)
        if 0 < int(k @ k) <= 64:
            ks.append(k)
    ks = np.array(ks, dtype=np.float64)
    amp, ph = np.linalg.norm(ks, axis=1) ** (-5.0 / 3.0), rng.uniform(0.0, 2.0 * math.pi, 32)
    x, dx = _centres(nx)
    y, dy = _centres(ny)
    z, dz = _centres(nz)
    wave = [torch.exp(2j * math.pi * _dev(ks[:, d])[:, None] * a[None, :]) for d, a in enumerate((x, y, z))]
    zy = torch.einsum("mz,my->zym", wave[2] * (_dev(amp) * torch.exp(1j * _dev(ph)))[:, None], wave[1])
    drho = torch.view_as_real(zy.reshape(nz * ny, -1) @ wave[0])[..., 0].reshape(nz, ny, nx)
    drho = drho * (0.1 / float(drho.square().mean().sqrt()))
    M = 3.0
    r2 = (GAMMA + 1) * M * M / ((GAMMA - 1) * M * M + 2)
    post = (x < 0.25)[None, None, :]
    rho = torch.where(post, _dev(r2), 1.0 + drho)
    u = torch.where(post, _dev(M * math.sqrt(GAMMA) * (1.0 - 1.0 / r2)), _dev(0.0)).expand(nz, ny, nx)
    p = torch.where(post, _dev(1.0 + 2 * GAMMA / (GAMMA + 1) * (M * M - 1)), _dev(1.0)).expand(nz, ny, nx)
    zero = torch.zeros_like(rho)
    return _conserved(rho, [u, zero, zero], p), (dx, dy, dz), (out, per, per)


def _rates(U, dx):
    """max over cells of (|u_d| + c)/dx_d, summed over the directions."""
    rho, nd = U[0], U.shape[0] - 2
    vel = [U[1 + d] / rho for d in range(nd)]
    p = (GAMMA - 1.0) * (U[-1] - 0.5 * rho * sum(v * v for v in vel))
    c = torch.sqrt(GAMMA * p / rho)
    return sum(float((vel[d].abs() + c).max()) / dx[d] for d in range(nd))


def _shape(case):
    return tuple(n for n in (case["nz"], case["ny"], case["nx"]) if n)


def _type(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _members(case):
    """The batch's instances: (problem, (ny, nx), R, l/dx), sizes log-uniform on [64, 1024]."""
    r = random.Random(case["mix"])
    size = lambda: int(round(math.exp(r.uniform(math.log(64), math.log(1024)))))   # noqa: E731
    return [("quadrant" if k % 2 == 0 else "vortex", (size(), size()), r.randint(1, 3), r.choice([6.0, 12.0, 24.0]))
            for k in range(case["count"])]


def _inputs(case, seed):
    """[(U rounded to the plan's type, dx, bc, dt)] of the case's grids (one unless a batch)."""
    if case["problem"] == "batch":
        fields = [_field(p, s, int(seed) * 1000 + k) for k, (p, s, _, _) in enumerate(_members(case))]
        cfl = BATCH_CFL
    else:
        fields, cfl = [_field(case["problem"], _shape(case), seed)], CFL
    got = []
    for U, dx, bc in fields:
        got.append((U.to(_type(case)).contiguous(), dx, bc, cfl / _rates(U, dx)))
    return got


def prepare(case, seed):
    ins = _inputs(case, seed)
    if case["problem"] == "batch":
        # one allocation holds every instance's state, one every scratch (16-byte aligned pieces)
        plans = [gpweno.Plan(R, ell, U.shape[1:], dx, bc, gamma=GAMMA, dtype=case["dtype"])
                 for (U, dx, bc, _), (_, _, R, ell) in zip(ins, _members(case))]
        at = np.cumsum([0] + [(U.numel() + 31) // 32 * 32 for U, _, _, _ in ins])
        flat = torch.zeros(int(at[-1]), dtype=_type(case), device="cuda")
        work = torch.zeros(4 * int(at[-1]), dtype=_type(case), device="cuda")
        Us, scratch = [], []
        for (U, _, _, _), a in zip(ins, at):
            Us.append(flat[int(a):int(a) + U.numel()].view(U.shape))
            Us[-1].copy_(U)
            scratch.append(work[4 * int(a):4 * int(a) + 4 * U.numel()].view((4,) + tuple(U.shape)))
        dts = torch.tensor([dt for _, _, _, dt in ins], dtype=torch.float64, device="cuda")
        return dict(kind="batch", plan=gpweno.BatchPlan(plans), U=Us, scratch=scratch, dt=dts, flat=flat)
    U, dx, bc, dt = ins[0]
    plan = gpweno.Plan(case["R"], case["ell"], U.shape[1:], dx, bc, gamma=GAMMA, dtype=case["dtype"], cfl=case["cfl"],
                       flux=case["flux"], scheme=case["scheme"], ao=case["ao"], candidates=case["candidates"])
    s = dict(kind=case["call"], plan=plan, U=U, dt=dt, dt_dev=None)
    if case["call"] == "rhs":
        s["out"] = torch.empty_like(U)
    else:
        s["scratch"] = plan.new_scratch()
        if case["cfl"] > 0:
            s["dt_dev"] = torch.full((1,), dt, dtype=torch.float64, device="cuda")
    return s


def run(s):
    if s["kind"] == "batch":
        s["plan"].rk3_step(s["U"], s["scratch"], s["dt"])
        return s["flat"]
    if s["kind"] == "rhs":
        return s["plan"].rhs(s["U"], s["out"])
    if s["dt_dev"] is None:
        return s["plan"].rk3_step(s["U"], s["scratch"], dt=s["dt"])
    s["plan"].rk3_step(s["U"], s["scratch"], dt_dev=s["dt_dev"])
    if s["U"].dtype == torch.float64:
        return {"U": s["U"], "dt": s["dt_dev"]}
    return {"U": s["U"], "dt": s["dt_dev"].float()}    # an FP32 plan's rates are FP32 numbers


def work(case):
    """Bytes: the state once in and once out, for a step its carried remainder too.  Operations: the scheme's own
    count per cell and stage."""
    stages = 1 if case["call"] == "rhs" else 3
    esz = 8 if case["dtype"] == "f64" else 4
    grids = [(s, R) for _, s, R, _ in _members(case)] if case["problem"] == "batch" else [(_shape(case), case["R"])]
    nbytes = flops = 0
    for shape, R in grids:
        cells, nd = math.prod(shape), len(shape)
        nbytes += (2 if case["call"] == "rhs" else 4) * esz * (nd + 2) * cells
        flops += stages * cells * costmodel.flops_per_cell_stage(R, nd, case["flux"], case["scheme"], False, case["ao"])
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the scheme in 64 bits


def _solve(A, b):
    """Gaussian elimination on Decimals (the systems are symmetric positive definite)."""
    n = len(A)
    M = [list(r) + [v] for r, v in zip(A, b)]
    for c in range(n):
        for r in range(n):
            if r != c:
                f = M[r][c] / M[c][c]
                M[r] = [x - f * y for x, y in zip(M[r], M[c])]
    return [M[i][n] / M[i][i] for i in range(n)]


def _series(z, ell, order):
    """`order`-fold antiderivative from 0 of exp(-z^2/(2 ell^2)) at z, by its power series."""
    a, fact, total = Decimal(1), Decimal(1), Decimal(0)
    for n in range(80):
        den = Decimal(math.prod(range(2 * n + 1, 2 * n + 1 + order)))
        total += a / fact * z ** (2 * n + order) / den
        a *= -1 / (2 * ell * ell)
        fact *= n + 1
    return total


def _weights(first, n, x, ell, recon):
    """GP weights of cells first .. first+n-1 for the point x (cell widths); recon: from cell averages."""
    pts = [Decimal(first + j) for j in range(n)]
    h = Decimal(1) / 2
    if recon:
        cov = [[_series(a - b + 1, ell, 2) - 2 * _series(a - b, ell, 2) + _series(a - b - 1, ell, 2) for b in pts] for a in pts]
        rhs = [_series(x - b + h, ell, 1) - _series(x - b - h, ell, 1) for b in pts]
    else:
        cov = [[(-(a - b) ** 2 / (2 * ell * ell)).exp() for b in pts] for a in pts]
        rhs = [(-(x - b) ** 2 / (2 * ell * ell)).exp() for b in pts]
    return _solve(cov, rhs)


def _lagrange(first, n, x, recon):
    """Polynomial weights: interpolation, or (recon) from cell averages through the moments of the cells."""
    h = Decimal(1) / 2
    rows = []
    for k in range(n):
        if recon:
            rows.append([((first + j + h) ** (k + 1) - (first + j - h) ** (k + 1)) / (k + 1) for j in range(n)])
        else:
            rows.append([Decimal(first + j) ** k if k else Decimal(1) for j in range(n)])
    AtA = [[sum(r[a] * r[b] for r in rows) for b in range(n)] for a in range(n)]
    return _solve(AtA, [sum(r[a] * (x ** k if k else 1) for k, r in enumerate(rows)) for a in range(n)])


def _factor(n, sigma):
    """G with f^T K_n(sigma)^-1 f = |G f|^2, rows in order (inverse of the Cholesky factor)."""
    K = [[(-Decimal(a - b) ** 2 / (2 * sigma * sigma)).exp() for b in range(n)] for a in range(n)]
    L = [[Decimal(0)] * n for _ in range(n)]
    for i in range(n):
        for j in range(i + 1):
            v = K[i][j] - sum(L[i][k] * L[j][k] for k in range(j))
            L[i][j] = v.sqrt() if i == j else v / L[j][j]
    cols = []
    for c in range(n):
        y = []
        for i in range(n):
            y.append(((1 if i == c else 0) - sum(L[i][k] * y[k] for k in range(i))) / L[i][i])
        cols.append(y)
    return [[cols[c][i] for c in range(n)] for i in range(n)]


@lru_cache(maxsize=None)
def _tables(R, ell, recon, poly, ao):
    """For each side (left: x* = 1/2 on the stencil of the face's left cell; right: x* = -1/2 on that of its right
    cell): sub-stencil weights, linear weights; the factor of the smoothness indicators; the GP-AO tables."""
    with decimal.localcontext() as ctx:
        ctx.prec = 120
        ell, sigma = Decimal(ell), Decimal(SIGMA)
        w = (lambda f, n, x: _lagrange(f, n, x, recon)) if poly else (lambda f, n, x: _weights(f, n, x, ell, recon))
        out = dict(sides=[], G=_factor(R + 1, sigma))
        for x in (Decimal(1) / 2, Decimal(-1) / 2):
            sub = [w(m - R, R + 1, x) for m in range(R + 1)]
            big = w(-R, 2 * R + 1, x)
            M = [[sub[m][r - m] if 0 <= r - m <= R else Decimal(0) for m in range(R + 1)] for r in range(2 * R + 1)]
            gam = _solve([[sum(r[a] * r[b] for r in M) for b in range(R + 1)] for a in range(R + 1)],
                         [sum(r[a] * v for r, v in zip(M, big)) for a in range(R + 1)])
            out["sides"].append(dict(sub=sub, gam=gam, big=big, low=w(1 - R, 2 * R - 1, x) if ao else None,
                                     three=[w(m - 2, 3, x) for m in range(3)] if ao else None))
        if ao:
            out["ao"] = {}
            for n in {3, 2 * R - 1, 2 * R + 1}:
                G = _factor(n, sigma)
                one = sum(sum(r) ** 2 for r in G)                      # 1^T K^-1 1
                s = (1 / (2 * one)).sqrt()
                out["ao"][n] = [[s * v for v in r] for r in G]

    def rounded(v):
        if isinstance(v, dict):
            return {k: rounded(x) for k, x in v.items()}
        return [rounded(x) for x in v] if isinstance(v, list) else (None if v is None else float(v))

    return rounded(out)


def _dot(w, f):
    return sum(a * x for a, x in zip(w, f) if a != 0.0)


def _square(G, f):
    return sum(_dot(row, f).square() for row in G)


def _ao_hybrid(qh, bh, q3, b3):
    g = [0.5 * (1 - AO_GAMMA) ** 2, (1 - AO_GAMMA) * AO_GAMMA, 0.5 * (1 - AO_GAMMA) ** 2]
    w = [a / (EPS + b) ** 2 for a, b in zip(g, b3)]
    wh = AO_GAMMA / (EPS + bh) ** 2
    tot = wh + w[0] + w[1] + w[2]
    q = wh / tot / AO_GAMMA * qh
    for a, v, x in zip(g, w, q3):
        q = q + (v / tot - wh / tot / AO_GAMMA * a) * x
    return q


def _state(tab, side, f, R, ao):
    """GP-WENO (or GP-AO) prediction of one side from its 2R+1 stencil values."""
    t = tab["sides"][side]
    if not ao:
        num = den = 0.0
        for m in range(R + 1):
            win = f[m:m + R + 1]
            w = t["gam"][m] / (EPS + _square(tab["G"], win)) ** 2
            num, den = num + w * _dot(t["sub"][m], win), den + w
        return num / den
    q3 = [_dot(t["three"][m], f[R - 2 + m:R + 1 + m]) for m in range(3)]
    b3 = [_square(tab["ao"][3], f[R - 2 + m:R + 1 + m]) for m in range(3)]
    bh = _square(tab["ao"][2 * R + 1], f)
    hi = _ao_hybrid(_dot(t["big"], f), bh, q3, b3)
    if R == 2:
        return hi
    bl = _square(tab["ao"][2 * R - 1], f[1:-1])
    lo = _ao_hybrid(_dot(t["low"], f[1:-1]), bl, q3, b3)
    vh, vl = AO_GAMMA / (EPS + bh) ** 2, (1 - AO_GAMMA) / (EPS + bl) ** 2
    rh = vh / (vh + vl) / AO_GAMMA
    return rh * hi + (vl / (vh + vl) - rh * (1 - AO_GAMMA)) * lo


def _prim(u):
    vel = [u[a] / u[0] for a in range(1, len(u) - 1)]
    return [u[0]] + vel + [(GAMMA - 1.0) * (u[-1] - 0.5 * u[0] * sum(v * v for v in vel))]


def _flux(V):
    """(U, F(U)) of primitive variables, normal velocity first."""
    ke = 0.5 * V[0] * sum(v * v for v in V[1:-1])
    U = [V[0]] + [V[0] * v for v in V[1:-1]] + [V[-1] / (GAMMA - 1.0) + ke]
    F = [U[1], U[1] * V[1] + V[-1]] + [U[1] * v for v in V[2:-1]] + [V[1] * (U[-1] + V[-1])]
    return U, F


def _face_flux(a, case, R, ell):
    """Numerical face flux between cells i+R and i+R+1 of the line a [nc, M] (normal-first), i = 0 .. M-2R-2."""
    nc, M = a.shape
    n = M - 2 * R - 1
    fdflux = case["scheme"] == "fdflux"
    tab = _tables(R, ell, fdflux, case["candidates"] == "poly", bool(case["ao"]))
    u = [a[c] for c in range(nc)]
    V = _prim(u)
    at = lambda f, q: f[q:q + n]                                        # noqa: E731
    VL, VR = [at(v, R) for v in V], [at(v, R + 1) for v in V]
    uL, uR = [at(v, R) for v in u], [at(v, R + 1) for v in u]
    sl, sr = torch.sqrt(VL[0]), torch.sqrt(VR[0])
    mean = lambda x, y: (sl * x + sr * y) / (sl + sr)                   # noqa: E731
    vel = [mean(x, y) for x, y in zip(VL[1:-1], VR[1:-1])]
    H = mean((uL[-1] + VL[-1]) / VL[0], (uR[-1] + VR[-1]) / VR[0])
    q2 = sum(v * v for v in vel)
    c = torch.sqrt((GAMMA - 1.0) * (H - 0.5 * q2))
    rb = sl * sr

    def left(k, W):                                                     # row k of the left eigenvectors
        if k == 0 or k == nc - 1:
            return W[-1] / (2 * c * c) + (rb / (2 * c) * W[1]) * (1.0 if k else -1.0)
        return W[0] - W[-1] / (c * c) if k == 1 else W[k]

    def right(q):
        return [q[0] + q[1] + q[-1], c / rb * (q[-1] - q[0])] + q[2:-1] + [c * c * (q[0] + q[-1])]

    if not fdflux:
        sides = []
        for side in (0, 1):
            q = []
            for k in range(nc):
                f = [left(k, [at(v, j + side) for v in V]) for j in range(2 * R + 1)]
                q.append(_state(tab, side, f, R, case["ao"]))
            sides.append(right(q))
        (UL, FL), (UR, FR) = _flux(sides[0]), _flux(sides[1])
        cL, cR = (torch.sqrt(GAMMA * s[-1] / s[0]) for s in sides)
        vL, vR = sides[0][1], sides[1][1]
        if case["flux"] == "lf":
            al = torch.maximum(vL.abs() + cL, vR.abs() + cR)
            return torch.stack([0.5 * (x + y - al * (w - v)) for x, y, v, w in zip(FL, FR, UL, UR)])
        SL, SR = torch.minimum(vL - cL, vel[0] - c), torch.maximum(vR + cR, vel[0] + c)
        if case["flux"] == "hll":
            mid = [(SR * x - SL * y + SL * SR * (w - v)) / (SR - SL) for x, y, v, w in zip(FL, FR, UL, UR)]
        else:
            (rL, pL), (rR, pR) = (sides[0][0], sides[0][-1]), (sides[1][0], sides[1][-1])
            Ss = (pR - pL + rL * vL * (SL - vL) - rR * vR * (SR - vR)) / (rL * (SL - vL) - rR * (SR - vR))

            def star(U, F, S, v, r, p):
                chi = r * (S - v) / (S - Ss)
                us = [chi, chi * Ss] + [chi * x / r for x in U[2:-1]]
                us.append(chi * (U[-1] / r + (Ss - v) * (Ss + p / (r * (S - v)))))
                return [f + S * (b - x) for f, b, x in zip(F, us, U)]

            mid = [torch.where(Ss >= 0, x, y) for x, y in zip(star(UL, FL, SL, vL, rL, pL), star(UR, FR, SR, vR, rR, pR))]
        return torch.stack([torch.where(SL >= 0, x, torch.where(SR <= 0, y, m)) for x, y, m in zip(FL, FR, mid)])
    # FD-Flux: local Lax-Friedrichs split point fluxes, reconstructed in the fields of the conservative Jacobian
    _, F = _flux(V)
    speed = V[1].abs() + torch.sqrt(GAMMA * V[-1] / V[0])
    al = at(speed, 0)
    for j in range(1, 2 * R + 2):
        al = torch.maximum(al, at(speed, j))

    def jac(X):                                                         # dV/dU at the Roe state
        k = sum(v * x for v, x in zip(vel, X[1:-1]))
        return [X[0]] + [(x - v * X[0]) / rb for v, x in zip(vel, X[1:-1])] + [(GAMMA - 1.0) * (0.5 * q2 * X[0] + X[-1] - k)]

    q = []
    for k in range(nc):
        total = 0.0
        for side, sign in ((0, 1.0), (1, -1.0)):
            f = []
            for j in range(2 * R + 1):
                lF, lU = (left(k, jac([at(x, j + side) for x in X])) for X in (F, u))
                f.append(0.5 * (lF + sign * al * lU))
            total = total + _state(tab, side, f, R, False)
        q.append(total)
    w = right(q)
    ke = sum(v * x for v, x in zip(vel, w[1:-1]))
    return torch.stack([w[0]] + [v * w[0] + rb * x for v, x in zip(vel, w[1:-1])] +
                       [0.5 * q2 * w[0] + rb * ke + w[-1] / (GAMMA - 1.0)])


def _line_difference(a, case, R, ell, chunk=6_000_000):
    """Difference of the numerical fluxes across each cell of the line a [nc, M]; only cells at least R+3 from
    either end of a padded piece mean anything."""
    nc, M = a.shape
    G = R + 3
    out = torch.zeros_like(a)
    for lo in range(0, M, chunk):
        p0, p1 = max(0, lo - G), min(M, lo + chunk + G)
        F = _face_flux(a[:, p0:p1], case, R, ell)                       # face i: between cells p0+i+R and p0+i+R+1
        if case["scheme"] != "fdflux":
            d2 = F[:, 1:-3] - 2 * F[:, 2:-2] + F[:, 3:-1]
            d4 = F[:, :-4] - 4 * F[:, 1:-3] + 6 * F[:, 2:-2] - 4 * F[:, 3:-1] + F[:, 4:]
            F = F[:, 2:-2] - d2 / 24 + 3 * d4 / 640
            first = p0 + R + 3
        else:
            first = p0 + R + 1
        D = F[:, 1:] - F[:, :-1]                                        # across cells first, first+1, ...
        a0, a1 = max(lo, first), min(lo + chunk, first + D.shape[1])
        if a1 > a0:
            out[:, a0:a1] = D[:, a0 - first:a1 - first]
    return out


def _rhs64(grids, case):
    """L(U) of every grid (U, dx, bc, R, ell): the lines of all grids of the same tables as one long line."""
    outs = [torch.zeros_like(g[0]) for g in grids]
    groups = {}
    for i, g in enumerate(grids):
        groups.setdefault((g[3], g[4]), []).append(i)
    for (R, ell), ids in groups.items():
        G = R + 3
        pieces = []
        for i in ids:
            U, dx, bc = grids[i][:3]
            nd = U.dim() - 1
            for d in range(nd):
                axis = nd - d
                n = U.shape[axis]
                k = torch.arange(-G, n + G, device=U.device)
                k = k % n if bc[d][0] == "periodic" else k.clamp(0, n - 1)
                V = U.movedim(axis, -1).index_select(-1, k)
                order = list(range(nd + 2))
                order[1], order[1 + d] = order[1 + d], order[1]
                pieces.append((i, d, axis, order, V.shape[1:], V[order].reshape(nd + 2, -1)))
            if nd == 3 or len(ids) == 1:
                _add(pieces, outs, grids, case, R, ell, G)
                pieces = []
        if pieces:
            _add(pieces, outs, grids, case, R, ell, G)
    return outs


def _add(pieces, outs, grids, case, R, ell, G):
    D = _line_difference(torch.cat([p[5] for p in pieces], 1) if len(pieces) > 1 else pieces[0][5], case, R, ell)
    at = 0
    for i, d, axis, order, shape, line in pieces:
        m = line.shape[1]
        part = D[:, at:at + m].reshape((-1,) + tuple(shape))[..., G:-G]
        at += m
        outs[i] -= part[order].movedim(-1, axis) / grids[i][1][d]


def exact(case, seed):
    ins = _inputs(case, seed)
    if case["problem"] == "batch":
        opts = [(R, ell) for _, _, R, ell in _members(case)]
    else:
        opts = [(case["R"], case["ell"])]
    grids = lambda Us: [(U, dx, bc, R, ell) for U, (_, dx, bc, _), (R, ell) in zip(Us, ins, opts)]   # noqa: E731
    U0 = [U.double() for U, _, _, _ in ins]
    dts = [dt for _, _, _, dt in ins]
    if case["call"] == "rhs":
        return _rhs64(grids(U0), case)[0]
    U = U0
    for a, b in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
        L = _rhs64(grids(U), case)
        U = [a * u0 + b * (u + dt * l) if a else u + dt * l for u0, u, l, dt in zip(U0, U, L, dts)]
    if case["problem"] == "batch":
        flat = []
        for u in U:
            flat += [u.reshape(-1), u.new_zeros(-u.numel() % 32)]
        return torch.cat(flat)
    if case["cfl"] > 0:
        return {"U": U[0], "dt": torch.full((1,), case["cfl"] / _rates(U[0], ins[0][1]), dtype=torch.float64)}
    return U[0]
