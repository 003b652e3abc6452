"""The square roots of the contact and drag laws (csrc/common.cuh) over the
range of their arguments: squares of lengths and speeds, Heron's product of
four lengths, and the ends of the FP32 range.

rsqrt.approx.ftz.f32 is within 2^-22.9 (PTX ISA); root() adds one Newton step
whose residual is exact, which leaves its one rounding (below 0.51 ulp; 1 ulp
asked for) as long as the residual is a normal number, above 1e-28; below it
stays within 2^-22.  rsqrt(double) is within 1 ulp (CUDA C Programming Guide)."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_2303_07819_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "common.cuh"
template <class R> __global__ void k(const R *x, R *s, R *q, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    s[i] = msd::root(x[i]);
    q[i] = msd::inv_sqrt(x[i]);
}
template <class R> int run(const R *x, R *s, R *q, int n)
{
    R *d = nullptr;
    if (cudaMalloc(&d, sizeof(R) * 3 * n) != cudaSuccess) return 1;
    cudaMemcpy(d, x, sizeof(R) * n, cudaMemcpyHostToDevice);
    k<R><<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, n);
    cudaMemcpy(s, d + n, sizeof(R) * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(q, d + 2 * n, sizeof(R) * n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
extern "C" int roots32(const float *x, float *s, float *q, int n) { return run(x, s, q, n); }
extern "C" int roots64(const double *x, double *s, double *q, int n) { return run(x, s, q, n); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    (d / "roots.cu").write_text(SRC)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I" + B.CSRC, "-shared", str(d / "roots.cu"), "-o", str(d / "roots.so")], check=True)
    return C.CDLL(str(d / "roots.so"))


def roots(lib, x):
    s, q = np.empty_like(x), np.empty_like(x)
    f = lib.roots32 if x.dtype == np.float32 else lib.roots64
    p = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    assert f(p(x), p(s), p(q), len(x)) == 0
    return s.astype(np.longdouble), q.astype(np.longdouble)


@pytest.mark.parametrize("lo,hi,tol", [(1e-28, 3.4e38, 1.2e-7), (1.2e-38, 1e-28, 2.4e-7)])
def test_fp32_roots(lib, lo, hi, tol):
    rng = np.random.default_rng(1)
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), 1 << 20)).astype(np.float32)
    x = np.concatenate([x, np.float32([1.0, 4.0, 1e16, 2.0 ** -20]), np.nextafter(np.float32(1.0), np.float32([0.0, 2.0]))])
    s, q = roots(lib, x)
    r = np.sqrt(x.astype(np.longdouble))
    assert np.abs(s / r - 1).max() <= tol
    assert np.abs(q * r - 1).max() <= 1.3e-7 + 2.0 ** -24
    if lo == 1e-28:     # and within one ulp of the correctly rounded one
        near = np.sqrt(x)
        assert np.all((s <= np.nextafter(near, np.float32(np.inf))) & (s >= np.nextafter(near, np.float32(0.0))))


def test_fp32_roots_of_nothing(lib):
    """A contact at onset asks for the root of 0 or a little less: 0 to the
    law's accuracy, and a finite reciprocal."""
    s, q = roots(lib, np.float32([0.0, -0.0, -1e-12, -1.0, 1e-42]))
    assert np.all((s >= 0) & (s < 1.2e-19))
    assert np.all(np.isfinite(q) & (q > 0))


def test_fp64_roots(lib):
    rng = np.random.default_rng(2)
    x = np.exp(rng.uniform(np.log(1e-200), np.log(1e200), 1 << 20))
    s, q = roots(lib, x)
    r = np.sqrt(x.astype(np.longdouble))
    assert np.abs(s / r - 1).max() <= 2.0 ** -53 * 1.001
    assert np.abs(q * r - 1).max() <= 2.0 ** -52 * 1.001
