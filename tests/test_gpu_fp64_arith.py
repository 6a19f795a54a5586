"""FP64 reciprocal and reciprocal square root of the face kernels against extended precision.

One third-order step from a start of relative error <= 2^-18 leaves at most (2^-18)^3 = 2^-54 (reciprocal) and
(5/16) 2^-54 (reciprocal square root); the last FMA rounds to 2^-53.  Bound used: 2^-52, one unit in the last place."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "face.cuh"
__global__ void k(const double *a, double *r, double *s, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        r[i] = gpweno::Num<double>::rcp(a[i]);
        s[i] = gpweno::Num<double>::rsqrt(a[i]);
    }
}
extern "C" int run(const double *a, double *r, double *s, int n)
{
    k<<<64, 128>>>(a, r, s, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("lo,hi", [(-2, 2), (-120, 40), (-250, 250)])
def test_rcp_rsqrt_one_ulp(tmp_path, lo, hi):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_04960_gb300 import build
    src, lib = tmp_path / "t.cu", str(tmp_path / "t.so")
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I",
                    build.CSRC, "-o", lib, str(src)], check=True)
    rng = np.random.default_rng(1)
    a = rng.uniform(1.0, 10.0, 200_000) * 10.0 ** rng.integers(lo, hi, 200_000)
    a[:8] = [1.0, 2.0, 4.0, 0.5, np.nextafter(1.0, 2.0), np.nextafter(1.0, 0.0), np.nextafter(4.0, 0.0), 3.0]
    d = torch.from_numpy(a).cuda()
    r, s = torch.empty_like(d), torch.empty_like(d)
    fn = ctypes.CDLL(lib).run
    fn.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    assert fn(d.data_ptr(), r.data_ptr(), s.data_ptr(), d.numel()) == 0
    x = a.astype(np.longdouble)
    for got, want in ((r, 1 / x), (s, 1 / np.sqrt(x))):
        err = np.abs((got.cpu().numpy().astype(np.longdouble) - want) / want).max()
        assert err <= 2.0 ** -52, float(err)
