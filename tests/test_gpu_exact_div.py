"""The FP64 kernels' shared-reciprocal division and integer halving give the IEEE
results bit for bit, over random operands and the edges of their fast ranges."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2002_04889_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "exact_div.cuh"
__global__ void k(int n, const double *a, const double *b, double *q, double *r, double *h)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    vg::Recip R = vg::recip(b[i]);
    q[i] = vg::quot(a[i], R);
    r[i] = vg::inverse(R);
    h[i] = vg::half_of(a[i]);
}
extern "C" int run(int n, const double *a, const double *b, double *q, double *r, double *h)
{
    k<<<(n + 255) / 256, 256>>>(n, a, b, q, r, h);
    return (int)cudaDeviceSynchronize();
}
"""


def _operands():
    rng = np.random.default_rng(1)
    n = 1 << 20
    man = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    man[::7] = (1 << 52) - 1 - rng.integers(0, 3, man[::7].shape, dtype=np.uint64)   # all ones and next to it
    man[1::7] = rng.integers(0, 3, man[1::7].shape, dtype=np.uint64)
    exp = rng.integers(1, 2046, n, dtype=np.uint64)
    exp[::3] = rng.integers(1023 - 40, 1023 + 40, exp[::3].shape, dtype=np.uint64)
    sign = rng.integers(0, 2, n, dtype=np.uint64)
    x = (man | (exp << np.uint64(52)) | (sign << np.uint64(63))).view(np.float64)
    edge = np.array([0.0, -0.0, 1.0, -1.0, 5e-324, -5e-324, 2.2250738585072014e-308, 2.225073858507201e-308,
                     4.450147717014403e-308, 1.7976931348623157e308, np.inf, -np.inf, np.nan,
                     2.0 ** 300, 2.0 ** -300, np.nextafter(2.0 ** 300, 0), 2.0 ** 600, 2.0 ** -600,
                     np.nextafter(2.0 ** -600, 0), np.nextafter(2.0 ** 600, 0), 9.81, 3.0])
    a = np.concatenate([x, np.repeat(edge, edge.size)])
    b = np.concatenate([np.roll(x, 12345), np.tile(edge, edge.size)])
    return a, b


def test_shared_reciprocal_division_is_ieee(tmp_path):
    torch = pytest.importorskip("torch")
    src, lib = tmp_path / "div.cu", tmp_path / "libdiv.so"
    src.write_text(SRC)
    nvcc = os.path.join(B._cuda_home(), "bin", "nvcc")
    subprocess.run([nvcc if os.path.exists(nvcc) else "nvcc", "-shared", *B.ARCH, "--fmad=false", "-Xcompiler", "-fPIC",
                    "-I", B.SRC, "-o", str(lib), str(src)], check=True)
    a, b = _operands()
    A, Bb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    out = [torch.empty_like(A) for _ in range(3)]
    torch.cuda.synchronize()
    fn = C.CDLL(str(lib)).run
    fn.argtypes = [C.c_int] + [C.c_void_p] * 5
    assert fn(a.size, A.data_ptr(), Bb.data_ptr(), *(o.data_ptr() for o in out)) == 0
    q, r, h = (o.cpu().numpy() for o in out)
    with np.errstate(all="ignore"):
        for got, want in ((q, a / b), (r, 1.0 / b), (h, 0.5 * a)):
            np.testing.assert_array_equal(got, want)      # NaN matches NaN, +0 matches -0
