"""The square roots of the pair kernels (common.cuh) against the exact root, in
units in the last place of the result, over the range of the arguments: a
small kernel around them is compiled for the test.

The bounds: the final rounding is half an ulp; root() adds 1.5 x 2^-60 of the
value in FP64 (0.012 ulp) and less in FP32; root_and_inverse() adds a quarter
ulp (FP64) or is the hardware approximation of 2^-22.9 (FP32: about 2 ulp)
and a product."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2002_03120_gb300 import build

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "common.cuh"
template <class R> __global__ void k(int n, const R *x, R *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    R r, v;
    sdpd::root_and_inverse(x[i], r, v);
    out[i] = sdpd::root(x[i]);
    out[n + i] = r;
    out[2 * n + i] = v;
}
template <class R> int run(int n, const R *x, R *out)
{
    R *dx, *dout;
    if (cudaMalloc(&dx, n * sizeof(R)) != cudaSuccess || cudaMalloc(&dout, 3 * n * sizeof(R)) != cudaSuccess) return 1;
    cudaMemcpy(dx, x, n * sizeof(R), cudaMemcpyHostToDevice);
    k<R><<<(n + 127) / 128, 128>>>(n, dx, dout);
    const int e = cudaMemcpy(out, dout, 3 * n * sizeof(R), cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(dx);
    cudaFree(dout);
    return e;
}
extern "C" int roots64(int n, const double *x, double *out) { return run(n, x, out); }
extern "C" int roots32(int n, const float *x, float *out) { return run(n, x, out); }
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    need_gpu()
    d = tmp_path_factory.mktemp("roots")
    (d / "p.cu").write_text(PROBE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(d / "p.cu"), "-o",
                    str(d / "p.so")], check=True)
    return ctypes.CDLL(str(d / "p.so"))


@pytest.mark.parametrize("bits,span,bounds", [(64, 300, (0.52, 0.80, 1.30)), (32, 34, (0.51, 3.0, 2.5))])
def test_roots_against_the_exact_root(probe, bits, span, bounds):
    dt = np.float64 if bits == 64 else np.float32
    rng = np.random.default_rng(bits)
    n = 30000
    x = np.concatenate([rng.uniform(1.0, 4.0, n // 2),                                   # both parities of the exponent
                        rng.uniform(1.0, 10.0, n // 2) * 10.0 ** rng.integers(-span, span, n // 2)]).astype(dt)
    out = np.empty((3, n), dt)
    p = ctypes.c_void_p
    assert getattr(probe, f"roots{bits}")(n, p(x.ctypes.data), p(out.ctypes.data)) == 0
    ulp = np.spacing(np.abs(out)).astype(np.float64)
    worst = [0.0, 0.0, 0.0]
    for i in range(n):
        X = Fraction(float(x[i]))
        for c in range(3):
            r = Fraction(float(out[c, i]))
            # r - sqrt(X) and v - 1 / sqrt(X) to first order
            err = (r * r - X) / (2 * r) if c < 2 else (r * r * X - 1) / (2 * r * X)
            worst[c] = max(worst[c], abs(float(err / Fraction(float(ulp[c, i])))))
    assert all(w < b for w, b in zip(worst, bounds)), worst
