"""Host side of the launches on a stand-in for the CUDA runtime (fake_cudart.cpp: no GPU, two devices, the runtime's
rule that a kernel's limit on dynamic shared memory belongs to one device).  Each case runs in a child process
that preloads it and drives the library through its C ABI."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, threading, time
fake = ctypes.CDLL(None)
fake.fake_bytes.restype = ctypes.c_size_t
fake.fake_budget.argtypes = [ctypes.c_size_t]
from paper_1808_04960_gb300 import gpweno as g
lib = g.load()
BUF = ctypes.c_void_p(4096)     # never read: no kernel runs
V2 = ctypes.c_void_p(8192)

def plan(shape, R=2, dtype="f32", **opts):
    dims, o = g.Dims(), g.Opts()
    dims.ndim = len(shape)
    for a, n in enumerate(reversed(shape)):
        dims.n[a], dims.dx[a] = n, 0.01
        dims.bc_lo[a] = dims.bc_hi[a] = g.PERIODIC
    lib.gpweno_default_opts(ctypes.byref(o))
    o.dtype = g.F32 if dtype == "f32" else g.F64
    for k, v in opts.items():
        setattr(o, k, v)
    h = ctypes.c_void_p()
    g._check(lib.gpweno_plan_create(ctypes.byref(h), R, 12.0, ctypes.byref(dims), 1.4, ctypes.byref(o)))
    return h

def step(h):
    g._check(lib.gpweno_rk3_step(h, BUF, V2, 1e-3, None, None))

def stage(h):
    g._check(lib.gpweno_rk3_stage(h, 0, BUF, V2, 1e-3, None, None))

def rhs(h):
    g._check(lib.gpweno_rhs(h, BUF, V2, None))

def schedule(h):
    v = [ctypes.c_int() for _ in range(4)]
    g._check(lib.gpweno_plan_schedule(h, *[ctypes.byref(x) for x in v]))
    return [x.value for x in v]
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_1808_04960_gb300 import build
    build.build()
    lib = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", include, "-o", lib,
                    os.path.join(HERE, "fake_cudart.cpp"), "-lpthread"], check=True)

    def child(code):
        r = subprocess.run([sys.executable, "-c", PRELUDE + code], capture_output=True, text=True, cwd=ROOT, timeout=120,
                           env=dict(os.environ, LD_PRELOAD=lib, PYTHONPATH=ROOT))
        assert r.returncode == 0, r.stdout[-1000:] + r.stderr[-3000:]
        return r.stdout

    return child


@pytest.mark.parametrize("shape,R,dtype", [((1024, 1024), 2, "f32"), ((512, 512), 1, "f32"), ((1200, 1100), 3, "f32"),
                                           ((300, 300), 2, "f32"), ((64, 64, 64), 2, "f32"), ((64, 64, 64), 3, "f32"),
                                           ((200, 200), 3, "f64"), ((20, 20, 20), 3, "f64")])
def test_second_device(run, shape, R, dtype):
    """A plan of the same kernels on a second device of the process; FP64 also with the marching kernels
    (no memory for the face workspace)."""
    run(f"""
if "{dtype}" == "f64":
    fake.fake_budget(1 << 12)
for device in (0, 1):
    fake.fake_device(device)
    p = plan({shape}, {R}, "{dtype}")
    step(p)
    rhs(p)
assert fake.fake_launches() >= 8
""")


def test_launch_with_another_device_current(run):
    """Such a launch is the caller's mistake; the kernel's state on the plan's own device stays right."""
    run("""
p, q = plan((1024, 1024)), plan((1024, 1024))
fake.fake_device(1)
step(p)
fake.fake_device(0)
step(q)
""")


def test_residency_published_whole(run):
    """A second thread that launches while the first is still asking for a kernel's residency sees the final value
    (R = 1's three-CTA build would fit four times and is counted as three)."""
    run("""
a, b = plan((512, 512), 1), plan((512, 512), 1)
fake.fake_hold()
t = threading.Thread(target=stage, args=(a,))
t.start()
while not fake.fake_held():
    time.sleep(1e-3)
stage(b)
got = schedule(b)[3]
fake.fake_release()
t.join()
assert got == 3 == schedule(a)[3], (got, schedule(a))
""")


def test_tiles_of_different_sizes(run):
    """No launch lowers a kernel's limit on dynamic shared memory: two threads that step plans of large and small
    tiles of the same kernel may interleave anywhere."""
    run("""
plans = [plan((n, n)) for n in (480, 384, 256, 300)]
for p in plans + plans:
    step(p)
    rhs(p)
assert fake.fake_lowered() == 0, fake.fake_lowered()
""")


@pytest.mark.parametrize("shape,R,opts,ctas", [((100, 100), 2, {}, 1), ((100, 100), 2, dict(scheme=1), 1),
                                               ((100, 100), 2, dict(ao=1), 1), ((100, 100), 2, dict(ao=1), 2),
                                               ((100, 100), 3, dict(ao=1), 1), ((100, 100), 1, dict(scheme=1), 2)])
def test_schedule_reports_the_tiles_residency(run, shape, R, opts, ctas):
    """The CTAs per SM that gpweno_plan_schedule gives for a tile launch are the runtime's."""
    run(f"""
fake.fake_resident({ctas})
p = plan({shape}, {R}, **{opts})
step(p)
assert schedule(p)[3] == {ctas}, schedule(p)
""")


def test_batch_members_give_their_workspace_back(run):
    """The batch kernel reads no face workspace: members that have never stepped alone hold none once the batch is
    built (they step with the marching kernels from then on); a member that has, keeps its own, which a
    captured graph may refer to.  Lost workspaces show in gpweno_plan_workspace."""
    run("""
def held(p):
    v = ctypes.c_ulonglong()
    g._check(lib.gpweno_plan_workspace(p, ctypes.byref(v)))
    return v.value

start = fake.fake_bytes()
members = [plan((256, 256 + k), 1 + k % 3, "f64") for k in range(8)]
step(members[0])
assert all(held(p) >= 8 << 20 for p in members)
arr = (ctypes.c_void_p * 8)(*[p.value for p in members])
b = ctypes.c_void_p()
g._check(lib.gpweno_plan_batch(ctypes.byref(b), arr, 8, None))
assert fake.fake_bytes() - start < held(members[0]) + (1 << 20), fake.fake_bytes() - start
assert held(members[0]) >= 8 << 20 and not any(held(p) for p in members[1:])
for p, launches in ((members[0], 6), (members[1], 3)):   # face lists and updates, marching
    step(p)
    assert lib.gpweno_last_launch_count() == launches
lib.gpweno_plan_destroy(b)
for p in members:
    lib.gpweno_plan_destroy(p)
assert fake.fake_bytes() == start

fake.fake_budget(fake.fake_bytes() + (1 << 20))
p = plan((256, 256), 2, "f64")
assert held(p) == 0
""")


def test_flags_return_every_bit(run):
    """gpweno_flags returns the whole word: bits 1-11 are the bounds-checked build's access sites."""
    run("""
fake.fake_block.restype, fake.fake_block.argtypes = ctypes.c_void_p, [ctypes.c_size_t]
p = plan((100, 100))
word = ctypes.c_ulonglong.from_address(fake.fake_block(32) + 24)
v = ctypes.c_int()
for bits in (0, 1, 1 << 4, (1 << 11) | 1, 0xffe):
    word.value = bits
    for want in (bits, 0):
        g._check(lib.gpweno_flags(p, ctypes.byref(v)))
        assert v.value == want, (bits, v.value)
""")
