"""The square root and the reciprocals of lbm_core.cuh against FP64 (FP32 forms) and
by their exact residuals (FP64 forms), over the arguments that their callers have: 1/4 + e, |v|^2 + tiny, cc + S, S + w, 2 S - 1, |v|, and porosities.

Tolerances, in units of 2^-24 or 2^-53 of the result.  root, FP32: the reciprocal root is
good to 2^-22.9 (PTX ISA), so after Newton's step only the last two roundings
count, of s and of the result: 2.  inverse, FP32: 1 ulp (PTX ISA), 2 units.
inverse_full: the quotient's rounding and the correction's, 2.  root, FP64: t's
rounding counts half, the result's one, and the series' remainder
5/16 e^3 is below 2^-54 for e up to 2^-17.5: 2.  inverse, FP64: remainder e^3, result: 2.
Each paired form has the bits of the scalar one."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_core.cuh"
using namespace lbm;
template <class R> __global__ void k(const R* x, R* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = op::root(x[i]);
    out[n + i] = op::inverse(x[i]);
    out[2 * n + i] = op::inverse_full(x[i]);
    if constexpr (sizeof(R) == 4) {
        const F2 v(x[i], x[n - 1 - i]);
        out[3 * n + i] = op::root(v).v.x;
        out[4 * n + i] = op::inverse(v).v.x;
        out[5 * n + i] = op::inverse_full(v).v.x;
    }
}
template <class R> static int run(const R* x, R* out, int n, int sets) {
    R *dx = nullptr, *dy = nullptr;
    cudaError_t e = cudaMalloc(&dx, n * sizeof(R));
    if (e == cudaSuccess) e = cudaMalloc(&dy, sets * n * sizeof(R));
    if (e == cudaSuccess) e = cudaMemcpy(dx, x, n * sizeof(R), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k<R><<<(n + 255) / 256, 256>>>(dx, dy, n);
        e = cudaMemcpy(out, dy, sets * n * sizeof(R), cudaMemcpyDeviceToHost);
    }
    cudaFree(dx);
    cudaFree(dy);
    return (int)e;
}
extern "C" int run_f32(const float* x, float* out, int n) { return run(x, out, n, 6); }
extern "C" int run_f64(const double* x, double* out, int n) { return run(x, out, n, 3); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300.build import ARCH, FLAGS, nvcc

    d = tmp_path_factory.mktemp("core_math")
    src, so = d / "math.cu", d / "math.so"
    src.write_text(SOURCE)
    r = subprocess.run([nvcc(), *ARCH, *FLAGS, "-shared", "-cudart", "shared", "-o", str(so), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(str(so))


# (least, largest) argument; what takes it
RANGES = {"f32": [(1.1e-37, 1e2), (0.25, 8e37), (0.5, 2.0), (3.2e-19, 8e37), (1e-4, 1.0)],
          "f64": [(1.1e-36, 1e2), (0.25, 1e300), (0.5, 2.0), (1e-18, 1e300), (1e-6, 1.0)]}


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_root_and_reciprocals(precision, lib):
    R = np.float32 if precision == "f32" else np.float64
    n = 1 << 18
    rng = np.random.default_rng(3)
    for lo, hi in RANGES[precision]:
        x = np.exp(rng.uniform(np.log(lo), np.log(hi), n)).astype(R)
        x = np.clip(x, R(lo), R(hi))
        x[:4] = R(lo), R(hi), np.nextafter(R(lo), R(hi)), np.nextafter(R(hi), R(lo))
        out = np.empty((6 if precision == "f32" else 3, n), R)
        call = getattr(lib, "run_" + precision)
        assert call(x.ctypes.data_as(C.c_void_p), out.ctypes.data_as(C.c_void_p), n) == 0
        if precision == "f32":
            assert np.array_equal(out[:3], out[3:])
            wide, unit = x.astype(np.float64), 2.0 ** -24
            want = [np.sqrt(wide), 1 / wide, 1 / wide]
            err = [np.abs(out[k] / want[k] - 1).max() / unit for k in range(3)]
        else:
            err = [relative(out[0], x, root=True), relative(out[1], x, root=False), relative(out[2], x, root=False)]
        print(precision, lo, hi, err)
        assert max(err) <= 2.0, (lo, hi, err)


def split(a):
    """a as a sum of two 26-bit numbers (Veltkamp, Dekker)."""
    c = a * 134217729.0
    hi = c - (c - a)
    return hi, a - hi


def product(a, b):
    """(p, e) with p + e = a b exactly (Dekker)."""
    p = a * b
    ah, al = split(a)
    bh, bl = split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def relative(y, x, root):
    """Largest error of y as sqrt(x) or 1 / x in units of 2^-53, to first order from the exact residual."""
    if root:
        m, k = np.frexp(x)  # to order one, by an even power of two
        k = k + (k & 1)
        x, y = np.ldexp(x, -k), np.ldexp(y, -(k // 2))
        p, e = product(y, y)
        return (np.abs((p - x) + e) / (2 * x)).max() * 2.0 ** 53
    m, k = np.frexp(x)
    x, y = m, np.ldexp(y, k)
    p, e = product(x, y)
    return np.abs((p - 1.0) + e).max() * 2.0 ** 53
