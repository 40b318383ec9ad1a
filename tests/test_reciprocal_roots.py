"""The kernels' reciprocal square roots (csrc/rsq.cuh, csrc/ffloat.cuh) over a range of arguments."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1812_10722_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "ffloat.cuh"
#include "rsq.cuh"
__global__ void k(int n, const double *x, double *d, double *f, double *ff, double *lib) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    d[i] = lspr::rsq(x[i]);
    lib[i] = rsqrt(x[i]);
    f[i] = (double)lspr::rsq((float)x[i]);
    ff[i] = (double)rsq(ffloat(x[i]));
}
extern "C" __attribute__((visibility("default"))) int roots(int n, const double *x, double *out) {
    double *b;
    if (cudaMalloc((void **)&b, 5 * sizeof(double) * n) != cudaSuccess) return 1;
    cudaMemcpy(b, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(n, b, b + n, b + 2 * n, b + 3 * n, b + 4 * n);
    const cudaError_t e = cudaMemcpy(out, b + n, 4 * sizeof(double) * n, cudaMemcpyDeviceToHost);
    cudaFree(b);
    return e != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    (d / "roots.cu").write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", "-o", str(d / "roots.so"),
                    str(d / "roots.cu")], check=True, capture_output=True)
    lib = ctypes.CDLL(str(d / "roots.so"))

    def run(x):
        x = np.ascontiguousarray(x)
        out = np.empty((4, len(x)))
        assert lib.roots(len(x), ctypes.c_void_p(x.ctypes.data), ctypes.c_void_p(out.ctypes.data)) == 0
        return dict(zip(("d", "f", "ff", "lib"), out))
    return run


def _arguments(decades):
    rng = np.random.default_rng(1)
    x = 10.0 ** rng.uniform(-decades, decades, 200000)
    edges = 2.0 ** np.arange(-3 * decades, 3 * decades + 1)   # both sides of every power of two
    return np.concatenate([x, np.linspace(1.0, 4.0, 100001), edges, np.nextafter(edges, 0), np.nextafter(edges, np.inf)])


def test_fp64(roots):
    # the rounding of h (2^-53 of x y^2, half of it in the root), of the step and of the result (2^-53)
    # and the series' remainder of 2^-55: below 2^-52 in all.  CUDA's function for comparison
    x = _arguments(250)
    r = roots(x)
    want = 1.0 / np.sqrt(x.astype(np.longdouble))
    for key in ("d", "lib"):
        assert np.abs(r[key] / want - 1.0).max() < 2.0 ** -52, key


def test_fp32(roots):
    # the hardware approximation's documented error is 2^-22.9
    x = _arguments(30).astype(np.float32)
    r = roots(x.astype(np.float64))
    want = 1.0 / np.sqrt(x.astype(np.float64))
    assert np.abs(r["f"] / want - 1.0).max() < 2.0 ** -22


def test_float_float(roots):
    # a few units of 2^-46 from the float-float product, and the FP32 rounding (2^-23) of a correction of
    # up to 2^-22: below 2^-43 in all
    x = _arguments(10)
    x = x.astype(np.float32).astype(np.float64) + (x - x.astype(np.float32)).astype(np.float32)
    r = roots(x)
    want = 1.0 / np.sqrt(x.astype(np.longdouble))
    assert np.abs(r["ff"] / want - 1.0).max() < 2.0 ** -43
