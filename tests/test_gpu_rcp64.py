"""The step kernels' FP64 reciprocal against CUDA's correctly rounded divide.

An estimate good to 2^-19 leaves e^3 < 2^-57 after the third-order iteration, at
most 1/16 of an ulp, on top of the final rounding's half: within 0.5625 ulp of
1/x and within one ulp of the divide's result.  Zeros, infinities and NaN give
what the divide gives.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "rcp64.cuh"
__global__ void k(const double *x, double *r, double *q, int n)
{
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < n) {
        r[i] = wblbm::rcp64(x[i]);
        q[i] = 1.0 / x[i];
    }
}
extern "C" int rcp64_probe(const double *x, double *r, double *q, int n)
{
    double *d = nullptr;
    const size_t b = (size_t)n * sizeof(double);
    if (cudaMalloc((void **)&d, 3 * b) != cudaSuccess) return 1;
    cudaError_t e = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * (size_t)n, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(r, d + n, b, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(q, d + 2 * (size_t)n, b, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build
    d = tmp_path_factory.mktemp("rcp64")
    src, lib = str(d / "probe.cu"), str(d / "probe.so")
    with open(src, "w") as fh:
        fh.write(PROBE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-o", lib, src],
                   check=True)
    fn = ctypes.CDLL(os.path.abspath(lib)).rcp64_probe
    dp = ctypes.POINTER(ctypes.c_double)
    fn.argtypes = [dp, dp, dp, ctypes.c_int]

    def run(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        r, q = np.empty_like(x), np.empty_like(x)
        assert fn(*[a.ctypes.data_as(dp) for a in (x, r, q)], x.size) == 0
        return r, q
    return run


def test_reciprocal_within_its_bound(probe):
    """Densities and relaxation times over all of the range that validation
    admits (positive, finite) in which neither x nor 1/x leaves the normal
    numbers, and the range of real use, both signs (phi may overshoot)."""
    rng = np.random.default_rng(7)
    n = 1 << 19
    wide = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-1020, 1020, n))
    used = 10.0 ** rng.uniform(-6.0, 6.0, n)
    ends = np.ldexp(np.array([1.0, 1.0 + 2.0 ** -52, 1.5, 2.0 - 2.0 ** -52])[:, None],
                    np.arange(-1020, 1020)[None]).ravel()
    x = np.concatenate([wide, used, ends, -used])
    r, q = probe(x)
    assert np.all(np.abs(r - q) <= np.spacing(np.abs(q)))
    if np.finfo(np.longdouble).nmant >= 63:
        exact = np.longdouble(1.0) / x.astype(np.longdouble)
        ulp = np.spacing(np.abs(q)).astype(np.longdouble)
        err = float((np.abs(r.astype(np.longdouble) - exact) / ulp).max())
        print(f"largest error {err:.4f} ulp; results that differ from the divide's: "
              f"{float((r != q).mean()):.4%}")
        assert err <= 0.5625


def test_special_values_as_the_divide(probe):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan])
    r, q = probe(x)
    assert np.array_equal(r, q, equal_nan=True) and np.array_equal(np.signbit(r[:4]), np.signbit(q[:4]))
