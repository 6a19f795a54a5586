"""FP64 square root of the face kernels against extended precision, in units in the last place of the result.

From a start of relative error d <= 2^-19 two Newton steps with a slope 1/(2 s) that is as far off leave d^2 (3/2) and then
d^3 (3/2) <= 2^-56, 0.13 units in the last place at most; with the last rounding 0.63.  Bound used: 0.7."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "face.cuh"
__global__ void k(const double *a, double *s, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) s[i] = gpweno::Num<double>::sqrt(a[i]);
}
extern "C" int run(const double *a, double *s, int n)
{
    k<<<64, 128>>>(a, s, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("lo,hi", [(-2, 2), (-30, 40), (-250, 250)])
def test_sqrt(tmp_path, lo, hi):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_04960_gb300 import build
    src, lib = tmp_path / "t.cu", str(tmp_path / "t.so")
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I",
                    build.CSRC, "-o", lib, str(src)], check=True)
    rng = np.random.default_rng(2)
    a = rng.uniform(1.0, 10.0, 200_000) * 10.0 ** rng.integers(lo, hi, 200_000)
    a[:8] = [1.0, 2.0, 4.0, 0.25, np.nextafter(1.0, 2.0), np.nextafter(1.0, 0.0), np.nextafter(4.0, 0.0), 3.0]
    d = torch.from_numpy(a).cuda()
    s = torch.empty_like(d)
    fn = ctypes.CDLL(lib).run
    fn.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int]
    assert fn(d.data_ptr(), s.data_ptr(), d.numel()) == 0
    got = s.cpu().numpy()
    err = (np.abs(got.astype(np.longdouble) - np.sqrt(a.astype(np.longdouble))) / np.spacing(got)).max()
    print(f"\nSQRT 1e{lo} .. 1e{hi}: {float(err):.3f} ulp")
    assert err <= 0.7
